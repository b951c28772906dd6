"""The Schwarz kernel that keeps a block's operators in registers, against the
oracle's smoother: every block volume it takes (64, 128, 192, 256 sites, with
faces of different sizes), two blocks in a direction (both neighbours the same
block), blocks at the antiperiodic time boundary, one or several right-hand
sides per CTA, and few cycles or iterations.

Bounds: FP32 2e-5 (eight sweeps of about twelve dependent applies); half
storage 2e-2, the bound of one rounded apply, as the sweeps contract it."""
import numpy as np
import pytest

import synthetic as syn
from tests.gpu_common import assert_close, make, smoother, t

pytestmark = pytest.mark.gpu

SHAPES = [((8, 8, 4, 4), (4, 4, 2, 2)), ((4, 4, 8, 16), (2, 2, 4, 8)), ((8, 12, 8, 4), (4, 6, 4, 2)),
          ((12, 4, 8, 16), (6, 2, 2, 8)), ((8, 8, 8, 8), (4, 4, 4, 4)), ((4, 16, 8, 8), (2, 8, 4, 4)),
          ((16, 8, 8, 16), (4, 4, 4, 4))]


@pytest.mark.parametrize("L,block", SHAPES)
@pytest.mark.parametrize("nrhs", [1, 3])
def test_blocks(L, block, nrhs):
    cfg = (L, block, 0.3, -0.2, 1.0, 1, 0)
    s = make(cfg, 1)
    x = syn.gaussian_spinors(nrhs, L, 12)
    ref = smoother(cfg)
    got = s.sap(x, 1)
    for k in range(nrhs):
        assert_close(got[k], ref.apply(t(x[k]), 4, 4).numpy(), 2e-5)
    for prec in (2, 3):
        assert_close(s.sap(x, prec)[-1], ref.apply(t(x[-1]), 4, 4).numpy(), 2e-2)
    s.close()


@pytest.mark.parametrize("n_sap,mr", [(1, 0), (1, 4), (2, 1), (3, 2)])
def test_cycles_and_iterations(n_sap, mr):
    L = (8, 8, 8, 8)
    cfg = (L, (4, 4, 4, 4), 0.3, -0.2, 1.0, 1, 0)
    s = make(cfg, 1, n_sap=n_sap, mr_iters=mr)
    x = syn.gaussian_spinors(2, L, 13)
    x[1] *= 1e-12                                  # and a field of another scale
    got = s.sap(x, 1)
    for k in range(2):
        assert_close(got[k], smoother(cfg).apply(t(x[k]), n_sap, mr).numpy(), 2e-5)
    assert not np.any(s.sap(np.zeros_like(x), 1))  # <p,p> = 0: the step is skipped
    s.close()
