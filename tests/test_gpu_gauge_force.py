"""The double-precision gauge force built from one product per plaquette.

Lattices of one block and of a ragged last block, extents of 2 (a plaquette
meets the same sites from both sides) and unequal extents (a plane index taken
for another one shows); links near and far from the unit matrix.  Tolerance of
tests/test_gpu_parity.py.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_0710_0066_gb300 import synthetic as syn

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_0710_0066_gb300 import lqcd  # noqa: E402


@pytest.mark.parametrize("eps", [0.02, 1.5])
@pytest.mark.parametrize("L,l0", [((4, 2, 2, 2), 1), ((6, 2, 4, 10), 3), ((4, 6, 14, 2), 2)])
def test_gauge_force_and_action(L, l0, eps):
    U = syn.random_links(L, eps, 6100)
    lat = lqcd.Lattice(L, l0, -1)
    lat.set_gauge(torch.from_numpy(U).cuda())
    olat = O.Lattice(L, l0, -1)
    S, pl, F = lat.gauge_force(5.6)
    ref = olat.gauge_force(U, 5.6)
    assert np.max(np.abs(F.cpu().numpy() - ref)) < 1e-12 * np.max(np.abs(ref))
    S0, pl0, _ = lat.gauge_force(5.6, force=False)
    assert abs(S - S0) < 1e-13 * 5.6 * 6 * olat.V  # a sum over 6 V plaquettes
    assert abs(pl - pl0) < 1e-13
    assert abs(pl - olat.plaquette(U)) < 1e-12
    lat.close()
