"""The persistent solver's kernels at the sizes where they can go wrong.

The single- and double-precision solves pick a kernel by the number of
groups of 32 sites (how many warps share a group, one or several passes of a
CTA over its groups, tiled or plain order), so the lattices below cover every
kernel, both sides of the rule's lines, a last group that is not full, slabs
that do not start on a group, and groups that are all lanes of one system.
Checked by the residual under the FP64 oracle's own operator (a solve to
1e-10 that stops on its own residual may be off by the residual's rounding,
1.5 times as in the other solver tests) and by the equality of repeated
solves (fixed reduction order).
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

KAPPA = 0.12
# (L, l0) of 16 even sites (half a group), 84 (ragged), 256, 1296 (40.5 groups),
# 4256 (133 groups: the last size with eight warps per group and a group per
# SM), 4560, 9600 and 9728 (304: the line to two warps), 10032, 19456 (608: the
# line to one), 20160, 77824 (2432: the line to one CTA per SM), 78400, and
# 65536 with its two slab systems in one launch
CASES = [((4, 2, 2, 2), 1), ((6, 2, 2, 14), 1), ((8, 4, 4, 4), 2), ((12, 6, 6, 6), 3), ((14, 4, 4, 38), 7),
         ((10, 6, 4, 38), 5), ((16, 12, 10, 10), 4), ((16, 8, 4, 38), 4), ((12, 4, 11 * 2, 19 * 2), 2),
         ((16, 8, 8, 38), 4), ((18, 16, 10, 14), 3), ((64, 8, 8, 38), 8), ((20, 28, 20, 14), 2),
         ((32, 16, 16, 16), 16)]

def field(L, seed):
    U = syn.random_links_torch(L, 0.6, seed, "cuda").contiguous()
    return U, U.cpu().numpy()


def check(r, b):
    assert np.linalg.norm(r) <= 1.5e-10 * np.linalg.norm(b)


@pytest.mark.parametrize("L,l0", CASES)
def test_global_and_slab_solves(L, l0):
    U, Un = field(L, 5000 + L[0])
    lat = lqcd.Lattice(L, l0, -1)
    lat.set_gauge(U)
    olat = O.Lattice(L, l0, -1)
    b = syn.gaussian_spinor(olat.V, 5001)
    bd = torch.from_numpy(b).cuda()
    precs = (lqcd.PREC_F32, lqcd.PREC_F64) if olat.V < 50000 else (lqcd.PREC_F32,)
    for p in precs:
        x = lat.solve(bd, KAPPA, 0, p, tol=1e-10)[0]
        check(b - olat.M(Un, KAPPA, x.cpu().numpy()), b)
        assert torch.equal(x, lat.solve(bd, KAPPA, 0, p, tol=1e-10)[0])
        x = lat.block_solve(bd, KAPPA, -1, 0, p, tol=1e-10)[0]
        check(b - olat.W1(Un, KAPPA, x.cpu().numpy()), b)
    lat.close()


@pytest.mark.parametrize("L,l0", [((4, 2, 2, 2), 2), ((12, 6, 6, 6), 6), ((16, 12, 10, 10), 4), ((16, 16, 16, 18), 8),
                                  ((64, 16, 16, 16), 16)])
@pytest.mark.parametrize("rho", [0.0, 0.2])
def test_series_solves(L, l0, rho):
    """kappa = 0.1, where the series converges; the sub-slab systems"""
    U, Un = field(L, 5100 + L[0])
    lat = lqcd.Lattice(L, l0, -1, l0s=l0 // 2)
    lat.set_gauge(U)
    olat = O.Lattice(L, l0, -1, l0s=l0 // 2)
    b = syn.gaussian_spinor(olat.Vh, 5101)
    for p in (lqcd.PREC_F32, lqcd.PREC_F64) if olat.V < 50000 else (lqcd.PREC_F32,):
        for dagger in (0, 1):
            x, it = lat.solve_w3eo(torch.from_numpy(b).cuda(), 0.1, rho, dagger, p, tol=1e-10,
                                   method=lqcd.SOLVER_SERIES)
            check(b - olat.w3eo(Un, 0.1, rho, x.cpu().numpy(), dagger), b)
    lat.close()


@pytest.mark.parametrize("prec", [lqcd.PREC_F32, lqcd.PREC_F64])
def test_extreme_source_scales(prec):
    """sources far from one in magnitude, and one slab without a source"""
    L, l0 = (8, 4, 4, 6), 2
    U, Un = field(L, 5200)
    lat = lqcd.Lattice(L, l0, -1)
    lat.set_gauge(U)
    olat = O.Lattice(L, l0, -1)
    b = syn.gaussian_spinor(olat.V, 5201)
    for scale in (1e-10, 1e10):
        x = lat.solve(torch.from_numpy(scale * b).cuda(), KAPPA, 0, prec, tol=1e-10)[0]
        check(b - olat.M(Un, KAPPA, x.cpu().numpy() / scale), b)
    slab = olat.index_maps()[2] == 1
    b[slab] = 0.0
    x, it, rs = lat.block_solve(torch.from_numpy(b).cuda(), KAPPA, -1, 0, prec, tol=1e-10)
    check(b - olat.W1(Un, KAPPA, x.cpu().numpy()), b)
    assert it[1] == 0 and rs[1] == 0.0 and not x[torch.from_numpy(slab)].any()
    lat.close()
