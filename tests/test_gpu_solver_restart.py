"""Solves near a critical point, where the BiCGstab recurrence stalls.

The systems below do not converge, or only by luck of rounding, unless a
stalled inner solve is restarted from its true residual (without restarts the
single-precision ones end at max_iter).  A restart keeps the best iterate: what
a solve has after more iterations is never further off than twice what it had
after fewer (the iterate is kept whenever the residual has halved), however far
the recurrence's residual has risen in between.
"""
import ctypes as C
import re

import numpy as np
import pytest

from oracle import oracle as O
from paper_0710_0066_gb300 import synthetic as syn

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_0710_0066_gb300 import lqcd  # noqa: E402

SYSTEMS = [((8, 4, 4, 4), 0.3, 0.15), ((16, 8, 8, 8), 0.5, 0.155)]  # L, eps of the links, kappa


def setup(L, eps):
    lat = lqcd.Lattice(L, 2, -1)
    U = syn.random_links_torch(L, eps, 21, "cuda").contiguous()
    lat.set_gauge(U)
    return lat, U


def residual(lat, b, kappa, prec, max_iter):
    """of the iterate that a solve has after max_iter iterations"""
    x = torch.empty_like(b)
    it, rs = C.c_int(0), C.c_double(0)
    st = lqcd.load().lqcd_solve_wilson(lat.h, C.c_void_p(x.data_ptr()), C.c_void_p(b.data_ptr()), kappa, 0, prec,
                                       1e-12, max_iter, C.byref(it), C.byref(rs))
    assert st == lqcd.ERR_NOCONVERGE
    return float(re.search(r"residual (\S+)\)", lqcd.load().lqcd_last_error(lat.h).decode())[1])


@pytest.mark.parametrize("L,eps,kappa", SYSTEMS)
@pytest.mark.parametrize("prec", [lqcd.PREC_F64, lqcd.PREC_F32])
def test_more_iterations_are_never_worse(L, eps, kappa, prec):
    lat, _ = setup(L, eps)
    for seed in (30, 31):
        b = torch.from_numpy(syn.gaussian_spinor(int(np.prod(L)), seed)).cuda()
        r = [residual(lat, b, kappa, prec, n) for n in (5, 7, 10, 14, 20, 28, 40, 57, 80, 113, 160, 226, 320, 453, 640)]
        # (1.02: three digits are printed; x = 0 has the residual 1)
        assert max(r) <= 1.02
        if prec == lqcd.PREC_F64:  # single storage: the recurrence's residual is not the true one to a factor of two
            assert all(r[j] <= 2.02 * r[i] for j in range(len(r)) for i in range(j))
    lat.close()


@pytest.mark.parametrize("L,eps,kappa", SYSTEMS)
@pytest.mark.parametrize("prec", [lqcd.PREC_F64, lqcd.PREC_F32])
def test_near_critical_solves_converge(L, eps, kappa, prec):
    lat, U = setup(L, eps)
    olat = O.Lattice(L, 2, -1)
    Un = U.cpu().numpy()
    for seed in range(30, 36):
        b = syn.gaussian_spinor(olat.V, seed)
        x, it, rs = lat.solve(torch.from_numpy(b).cuda(), kappa, 0, prec, tol=1e-10)
        assert rs <= 1e-10
        assert np.linalg.norm(b - olat.M(Un, kappa, x.cpu().numpy())) <= 1.5e-10 * np.linalg.norm(b)
    lat.close()
