"""The double-float source and reconstruction sweeps of a single-precision solve.

A site is three work items there, a warp to each colour of 32 sites: lattices
with less than a warp, with a ragged last warp and with slabs that begin
inside one, all slab colours; sources with zeros and with entries far below
the others (outside and inside the range of the split into two floats).
Checked by the residual under the FP64 oracle's own operator, 1.5 times the
tolerance as in the other solver tests.
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


@pytest.mark.parametrize("L,l0", [((4, 2, 2, 2), 1), ((6, 2, 2, 14), 3), ((12, 6, 6, 6), 3)])
@pytest.mark.parametrize("dagger", [0, 1])
def test_slab_and_global_solves(L, l0, dagger):
    U = syn.random_links(L, 0.6, 5300)
    lat = lqcd.Lattice(L, l0, -1)
    lat.set_gauge(torch.from_numpy(U).cuda())
    olat = O.Lattice(L, l0, -1)
    b = syn.gaussian_spinor(olat.V, 5301)
    b[::3] = 0.0
    b[1::5] *= 1e-12
    b[2::7] *= 1e-30
    bd = torch.from_numpy(b).cuda()
    x = lat.solve(bd, 0.12, dagger, lqcd.PREC_F32, tol=1e-12)[0].cpu().numpy()
    assert np.linalg.norm(b - olat.M(U, 0.12, x, dagger)) <= 1.5e-12 * np.linalg.norm(b)
    colours = olat.index_maps()[3]
    for colour in (-1, 0, 1):
        x = lat.block_solve(bd, 0.12, colour, dagger, lqcd.PREC_F32, tol=1e-12)[0].cpu().numpy()
        keep = (colours == colour) | (colour < 0)
        r = (b - olat.W1(U, 0.12, x, dagger))[keep]
        assert np.linalg.norm(r) <= 1.5e-12 * np.linalg.norm(b[keep])
        assert not x[~keep].any()
    lat.close()
