"""The coarse GMRES for five or more right-hand sides when a bounded wait gives
up, in its block ring or at a grid barrier (wait limits from no poll to many, so
that both kinds give up): DDAMG_ETIMEOUT or the result, and with the default
limits the same handle returns the same bits as before."""
import numpy as np
import pytest
import torch

import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cL,n_v,nrhs", [((2, 2, 2, 2), 16, 5), ((4, 4, 4, 8), 24, 12), ((4, 4, 4, 6), 32, 12)])
def test_wide_waits(cL, n_v, nrhs):
    import paper_1811_00355_gb300 as P
    L = tuple(2 * v for v in cL)
    p = P.default_params(L=L, sap_block=(2, 2, 2, 2), n_v=n_v, precision=P.FP32)
    s = P.DDAMG(p, syn.unit_gauge(L))
    try:
        s.set_coarse_op(syn.coarse_stencil(s.NX, 2 * n_v, 8, 1.0, 0.21))
        gen = np.random.default_rng(92)
        bc = gen.standard_normal((nrhs, s.NX, 2 * n_v)) + 1j * gen.standard_normal((nrhs, s.NX, 2 * n_v))
        bc = torch.from_numpy(bc).cuda()
        torch.cuda.synchronize()
        ref, its = s.coarse_solve(bc, 5e-2, P.FP32)
        for polls in (0, 0, 1, 2, 4, 8, 16, 32, 64, 128, 256, 512):
            s.set_wait_limit(polls)
            try:
                s.coarse_solve(bc, 5e-2, P.FP32)
                assert polls > 0
            except P.DDAMGError as e:
                assert e.status == 6, e
            s.set_wait_limit(-1)
            x, n = s.coarse_solve(bc, 5e-2, P.FP32)
            assert np.array_equal(n, its) and torch.equal(x, ref), polls
    finally:
        s.close()
