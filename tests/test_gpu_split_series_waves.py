"""Series solves whose systems do not fit the L2 together: full waves only.

Two of four systems at a time, four of twelve, one of four and two of eight;
checked by the residual under the FP64 oracle's own operator (1.5 times the
tolerance, as in the other solver tests) and by the equality of repeated solves.
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


@pytest.mark.parametrize("L,l0s", [((32, 24, 24, 24), 8), ((48, 24, 24, 24), 4), ((32, 32, 32, 32), 8),
                                   ((32, 36, 32, 32), 4)])
def test_full_waves(L, l0s):
    U = syn.random_links_torch(L, 0.6, 5500, "cuda").contiguous()
    Un = U.cpu().numpy()
    lat = lqcd.Lattice(L, 2 * l0s, -1, l0s=l0s)
    lat.set_gauge(U)
    olat = O.Lattice(L, 2 * l0s, -1, l0s=l0s)
    b = syn.gaussian_spinor(olat.Vh, 5501)
    bd = torch.from_numpy(b).cuda()
    x, it = lat.solve_w3eo(bd, 0.1, 0.2, 1, lqcd.PREC_F32, tol=1e-10, method=lqcd.SOLVER_SERIES)
    r = b - olat.w3eo(Un, 0.1, 0.2, x.cpu().numpy(), 1)
    assert np.linalg.norm(r) <= 1.5e-10 * np.linalg.norm(b)
    assert torch.equal(x, lat.solve_w3eo(bd, 0.1, 0.2, 1, lqcd.PREC_F32, tol=1e-10, method=lqcd.SOLVER_SERIES)[0])
    lat.close()
