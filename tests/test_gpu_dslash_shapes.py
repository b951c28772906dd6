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
