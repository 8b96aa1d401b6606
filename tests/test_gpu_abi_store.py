"""Operator calls whose sweep stores straight into the C-ABI layout.

The warps hand their 32 sites to the store through shared memory, so the
lattices below end in a partial warp, have fewer sites than a warp, and have
slabs that begin inside one; every storage precision, the operators with and
without a second field, all slab colours (zeros on the others), and a result
that overwrites its own source.  Tolerances of tests/test_gpu_parity.py.
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

TOL = {lqcd.PREC_F64: 1e-13, lqcd.PREC_F32: 1e-6, lqcd.PREC_F16: 5e-3, lqcd.PREC_BF16: 2e-2}


def rel(a, b):
    return float(np.max(np.abs(a - b)) / np.max(np.abs(b)))


@pytest.mark.parametrize("L,l0", [((4, 2, 2, 2), 1), ((6, 2, 2, 14), 3), ((12, 6, 6, 6), 3)])
@pytest.mark.parametrize("prec", list(TOL))
def test_operator_calls(L, l0, prec):
    U = syn.random_links(L, 0.6, 6000)
    lat = lqcd.Lattice(L, l0, -1)
    lat.set_gauge(torch.from_numpy(U).cuda())
    olat = O.Lattice(L, l0, -1)
    x = syn.gaussian_spinor(olat.V, 6001)
    xd = torch.from_numpy(x).cuda()
    xe = np.ascontiguousarray(x[:olat.Vh])
    for dagger in (0, 1):
        for parity in (0, 1):
            out = lat.dslash_eo(xd[:lat.Vh], parity, 0.0, dagger, lqcd.OP_HOP, prec).cpu().numpy()
            assert rel(out, olat.dslash_eo(U, xe, parity, dagger)) < TOL[prec]
        io = xd[:lat.Vh].clone()
        ref = lat.dslash_eo(io, 0, 0.15, dagger, lqcd.OP_MHAT, prec)
        lqcd.lqcd_dslash_eo(lat.h, io, io, 0.15, 0, dagger, lqcd.OP_MHAT, prec)
        assert torch.equal(io, ref)
        ref = olat.W1(U, 0.15, x, dagger)
        colours = olat.index_maps()[3]
        for colour in (-1, 0, 1):
            out = lat.block_dslash(xd, 0.15, colour, dagger, prec).cpu().numpy()
            keep = (colours == colour) | (colour < 0)
            assert rel(out[keep], ref[keep]) < TOL[prec]
            assert not out[~keep].any()
    lat.close()
