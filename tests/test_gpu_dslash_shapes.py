"""D in FP64 and FP32 where CTAs are small or end inside the lattice, for one
and several right-hand sides, and after the links of a handle were replaced
from host and from device buffers (FP64 links keep their rebuilt third row)."""
import numpy as np
import pytest
import torch

import synthetic as syn
from tests.gpu_common import TOL32, TOL64, assert_close, make, oracle_op, t

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,block", [((4, 4, 4, 4), (2, 2, 2, 2)), ((8, 4, 4, 12), (4, 2, 2, 6)),
                                     ((8, 8, 8, 8), (4, 4, 4, 4)), ((16, 8, 12, 8), (4, 4, 6, 2))])
@pytest.mark.parametrize("nrhs", [1, 5])
def test_D(L, block, nrhs):
    op = oracle_op(L, 0.3, 4, -0.2, 1.0)
    x = syn.gaussian_spinors(nrhs, L, 14)
    ref = op.apply(t(x)).numpy()
    s = make((L, block, 0.3, -0.2, 1.0, 1, 4), 1)
    U = syn.gauge_field(L, 0.3, 4)
    for U2 in (None, U, torch.from_numpy(U).cuda()):
        if U2 is not None:
            s.set_gauge(syn.gauge_field(L, 0.2, 6))      # other links in between
            s.set_gauge(U2)
        assert_close(s.apply_D(x, 0), ref, TOL64)
        assert_close(s.apply_D(x, 1), ref, TOL32)
        assert_close(s.get_clover(), op.packed_clover().numpy(), TOL64)
    s.close()


def test_fp64_D_in_place_and_unaligned():
    """FP64 D on device buffers reads and writes them directly: also where the
    output is the input (the neighbours are read first), overlaps it, or is
    aligned to 8 bytes only; through the C interface, as the binding allocates
    its own output."""
    import ctypes as C
    L, block = (8, 4, 4, 12), (4, 2, 2, 6)
    x = syn.gaussian_spinors(2, L, 15)
    ref = oracle_op(L, 0.3, 4, -0.2, 1.0).apply(t(x)).numpy()
    s = make((L, block, 0.3, -0.2, 1.0, 1, 4), 1)
    n = 2 * x.size
    for prec, tol in ((0, TOL64), (1, TOL32)):
        for shift, out_at in ((0, 0), (1, 1), (0, n), (1, n + 1), (0, n // 2), (1, n + 2)):
            buf = torch.zeros(2 * n + 4, dtype=torch.float64, device="cuda")
            buf[shift:shift + n] = torch.from_numpy(x.view(np.float64).reshape(-1)).cuda()
            torch.cuda.synchronize()
            at = lambda k: C.c_void_p(buf.data_ptr() + 8 * k)      # noqa: E731
            assert s.lib.ddamg_apply_D(s.h, prec, 2, at(shift), at(out_at), 1) == 0
            got = buf[out_at:out_at + n].cpu().numpy().view(np.complex128).reshape(x.shape)
            assert_close(got, ref, tol, f"precision {prec} in {shift} out {out_at}")
    s.close()
