"""The dot products of a single-precision solve are double-precision sums.

On the links diag(1, 0, 0) and the source below, A = 1 - kappa^2 H_eo H_oe at
kappa = 1/4 is -3 on colour 0 (constant over the sites, in the first spin
component) and 1 on the other colours, so the first <r, A r> is the sum of
-3 a^2 + |c|^2 over the sites.  Every site's term is exact in single precision:
in units of a^2 the first 32 sites give 2^-46, 1 + 2^-20 and thirty times 1, the
next 32 -2^-20 and 31 times -1, all others 1 and -1 in turn; the sum is 2^-46.
It spans 51 bits: FP64 keeps it in any order of the sites, a sum of fewer bits
may lose it, and then the iteration has no step to take.
"""
import ctypes as C
import itertools
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_0710_0066_gb300 import lqcd  # noqa: E402


def four_squares(n):
    top = math.isqrt(n)
    for a, b, c in itertools.product(range(top, top // 2, -1), range(top, -1, -1), range(top, -1, -1)):
        d = n - a * a - b * b - c * c
        if d >= 0 and math.isqrt(d) ** 2 == d:
            return a, b, c, math.isqrt(d)


def source(V):
    b = np.zeros((V, 4, 3), dtype=np.complex128)
    Vh = V // 2
    b[:Vh, 0, 0] = 1.0
    plus = np.zeros(Vh, dtype=bool)
    plus[:32] = True
    plus[64::2] = True
    b[:Vh, 0, 1] = np.where(plus, 2.0, 1.0 + 1.0j)  # |c|^2 = 4 or 2: a term of 1 or -1
    b[0, 0, 1:] = 1.0 + 1.0j, 1.0  # |c|^2 = 3
    b[0, 1, 1] = 2.0**-23
    b[1, 0, 2] = 2.0**-10
    p, q, r, s = four_squares(3 * 2**20 - 1)
    b[32, 0, 1:] = complex(p, q) / 2**10, complex(r, s) / 2**10  # |c|^2 = 3 - 2^-20
    return b


# 64, 16384 and 65536 even sites: eight, two and one warps per group of 32 sites
@pytest.mark.parametrize("L", [(4, 4, 4, 2), (16, 16, 16, 8), (32, 16, 16, 16)])
def test_first_step_of_a_cancelling_sum(L):
    V = int(np.prod(L))
    b = source(V)
    weight = np.array([-3.0, 1.0, 1.0])
    assert math.fsum(np.concatenate(((weight * b.real**2).ravel(), (weight * b.imag**2).ravel()))) == 2.0**-46
    lat = lqcd.Lattice(L, 2, 1)
    U = torch.zeros((4, V, 3, 3), dtype=torch.complex128, device="cuda")
    U[..., 0, 0] = 1.0
    lat.set_gauge(U)
    bd = torch.from_numpy(b).cuda()
    x = torch.empty_like(bd)
    it, rs = C.c_int(0), C.c_double(0)
    st = lqcd.load().lqcd_solve_wilson(lat.h, C.c_void_p(x.data_ptr()), C.c_void_p(bd.data_ptr()), 0.25, 0,
                                       lqcd.PREC_F32, 1e-10, 1, C.byref(it), C.byref(rs))
    message = lqcd.load().lqcd_last_error(lat.h).decode()
    lat.close()
    # one step is all it may take, and it takes it (a step of 2^54: not converged)
    assert st == lqcd.ERR_NOCONVERGE and " 1 inner iterations" in message
