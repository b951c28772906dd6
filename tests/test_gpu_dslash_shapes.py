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


def test_fp32_D_call_is_measured_as_it_runs():
    """The FP32 D call records its own choice, made of both whole calls (the
    four-threads form needs a pass to unpack, the other does not), and either
    form on host, device and overlapping buffers gives the oracle's result."""
    import ctypes as C
    import paper_1811_00355_gb300 as P
    L, block = (8, 4, 4, 12), (4, 2, 2, 6)
    x = syn.gaussian_spinors(3, L, 18)
    ref = oracle_op(L, 0.3, 4, -0.2, 1.0).apply(t(x)).numpy()
    s = make((L, block, 0.3, -0.2, 1.0, 1, 4), 1)
    for variant in (-1, 0, 1):
        P.pin_variant("D fp32", variant)
        try:
            assert_close(s.apply_D(x, 1), ref, TOL32, f"host, variant {variant}")
            buf = torch.from_numpy(x).cuda()
            torch.cuda.synchronize()
            assert_close(s.apply_D(buf, 1).cpu().numpy(), ref, TOL32, f"device, variant {variant}")
            p = C.c_void_p(buf.data_ptr())
            assert s.lib.ddamg_apply_D(s.h, 1, 3, p, p, 1) == 0
            assert_close(buf.cpu().numpy(), ref, TOL32, f"in place, variant {variant}")
        finally:
            P.pin_variant("D fp32", -1)
    rec = [r for r in P.tuning() if r["kernel"] == "D fp32" and r["problem"].startswith("8x4x4x12/4x2x2x6")
           and r["problem"].endswith("nrhs 3 call")]
    assert len(rec) == 1 and len(rec[0]["us"]) == 2, P.tuning()
    assert rec[0]["us"][rec[0]["best"]] == min(rec[0]["us"])
    s.close()
