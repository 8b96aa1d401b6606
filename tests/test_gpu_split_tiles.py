"""The persistent solver's tiled order of the sites.

A CTA that makes several passes takes its groups of 32 sites in tiles (where L1,
L2 and L3 are powers of two and a plane is whole groups); schedule 2 gives every
kernel two passes on lattices small enough for the oracle.  Double precision
and every single-precision kernel, whole lattice, slabs and series, tiles that
reach over slices, planes and parts of a plane, and thicknesses of a slab that
are no power of two.  Checked by the residual under the FP64 oracle's own
operator (1.5 times the tolerance, as in the other solver tests) and by the
equality of repeated solves.
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

KAPPA = 0.1
# 32, 48, 64, 64, 96 groups (eight warps each in single precision), 256 (four), 512 (two), 1024 (one)
CASES = [((8, 4, 8, 8), 4), ((12, 4, 4, 16), 6), ((8, 8, 8, 8), 2), ((4, 2, 16, 32), 2), ((12, 8, 8, 8), 6),
         ((16, 16, 8, 8), 4), ((32, 4, 16, 16), 8), ((16, 16, 16, 16), 8)]


@pytest.mark.parametrize("L,l0", CASES)
@pytest.mark.parametrize("prec", [lqcd.PREC_F64, lqcd.PREC_F32])
def test_two_passes(L, l0, prec):
    U = syn.random_links_torch(L, 0.6, 5600, "cuda").contiguous()
    Un = U.cpu().numpy()
    sub = l0 // 2
    lat = lqcd.Lattice(L, l0, -1, l0s=sub)
    lat.set_gauge(U)
    lqcd.lqcd_set_solver_schedule(lat.h, 2)
    olat = O.Lattice(L, l0, -1, l0s=sub)
    b = syn.gaussian_spinor(olat.V, 5601)
    bd = torch.from_numpy(b).cuda()

    def check(solve, apply, rhs):
        x = solve()
        r = rhs - apply(x.cpu().numpy())
        assert np.linalg.norm(r) <= 1.5e-10 * np.linalg.norm(rhs)
        assert torch.equal(x, solve())

    check(lambda: lat.solve(bd, KAPPA, 0, prec, tol=1e-10)[0], lambda x: olat.M(Un, KAPPA, x), b)
    check(lambda: lat.block_solve(bd, KAPPA, -1, 0, prec, tol=1e-10)[0], lambda x: olat.W1(Un, KAPPA, x), b)
    half = bd[: olat.Vh].contiguous()
    for method in (lqcd.SOLVER_BICGSTAB, lqcd.SOLVER_SERIES):
        check(lambda: lat.solve_w3eo(half, KAPPA, 0.2, 0, prec, tol=1e-10, method=method)[0],
              lambda x: olat.w3eo(Un, KAPPA, 0.2, x, 0), b[: olat.Vh])
    lat.close()


def test_whole_lattice_of_many_passes():
    """64x32^3 in single precision: five passes of the widest kernel"""
    L = (64, 32, 32, 32)
    U = syn.random_links_torch(L, 0.6, 5602, "cuda").contiguous()
    lat = lqcd.Lattice(L, 8, -1)
    lat.set_gauge(U)
    olat = O.Lattice(L, 8, -1)
    b = syn.gaussian_spinor(olat.V, 5603)
    x = lat.solve(torch.from_numpy(b).cuda(), KAPPA, 0, lqcd.PREC_F32, tol=1e-10)[0].cpu().numpy()
    lat.close()
    r = b - olat.M(U.cpu().numpy(), KAPPA, x)
    assert np.linalg.norm(r) <= 1.5e-10 * np.linalg.norm(b)
