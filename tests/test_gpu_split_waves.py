"""Batched single-precision solves whose systems do not fit the L2 together.

The persistent solver then works on a part of the systems at a time.  Four
systems in two waves, six in two waves of three, eight in three waves of three
(the last one not full) by BiCGstab; two, six and four at a time by the
series; checked by the residual under the FP64 oracle's own operator (1.5 times the tolerance, as in
the other solver tests) and by the equality of repeated solves.
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

SLABS = [((32, 20, 20, 28), 8), ((48, 14, 18, 30), 8), ((64, 16, 22, 22), 8)]
SUB_SLABS = [((32, 20, 20, 28), 8), ((48, 14, 18, 30), 4), ((64, 16, 22, 22), 8)]


def field(L, seed):
    U = syn.random_links_torch(L, 0.6, seed, "cuda").contiguous()
    return U, U.cpu().numpy()


@pytest.mark.parametrize("L,l0", SLABS)
def test_slab_bicgstab(L, l0):
    U, Un = field(L, 5400)
    lat = lqcd.Lattice(L, l0, -1)
    lat.set_gauge(U)
    olat = O.Lattice(L, l0, -1)
    b = syn.gaussian_spinor(olat.V, 5401)
    bd = torch.from_numpy(b).cuda()
    x, it, rs = lat.block_solve(bd, 0.12, -1, 0, lqcd.PREC_F32, tol=1e-10)
    r = b - olat.W1(Un, 0.12, x.cpu().numpy())
    assert np.linalg.norm(r) <= 1.5e-10 * np.linalg.norm(b)
    assert torch.equal(x, lat.block_solve(bd, 0.12, -1, 0, lqcd.PREC_F32, tol=1e-10)[0])
    lat.close()


@pytest.mark.parametrize("L,l0s", SUB_SLABS)
def test_sub_slab_series(L, l0s):
    U, Un = field(L, 5402)
    lat = lqcd.Lattice(L, 2 * l0s, -1, l0s=l0s)
    lat.set_gauge(U)
    olat = O.Lattice(L, 2 * l0s, -1, l0s=l0s)
    b = syn.gaussian_spinor(olat.Vh, 5403)
    x, it = lat.solve_w3eo(torch.from_numpy(b).cuda(), 0.1, 0.2, 0, lqcd.PREC_F32, tol=1e-10,
                           method=lqcd.SOLVER_SERIES)
    r = b - olat.w3eo(Un, 0.1, 0.2, x.cpu().numpy(), 0)
    assert np.linalg.norm(r) <= 1.5e-10 * np.linalg.norm(b)
    lat.close()
