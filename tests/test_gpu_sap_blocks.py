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


@pytest.mark.parametrize("cfg", [((8, 8, 8, 8), (4, 4, 4, 4), 0.3, -0.2, 1.0, 1, 0),
                                 ((4, 4, 8, 64), (2, 2, 4, 4), 0.3, 1.0, 1.0, 1, 0)])
@pytest.mark.parametrize("prec", [1, 2, 3])
def test_residuals_near_underflow(cfg, prec):
    """Fields so small that <p,p> of a block becomes subnormal, and point
    sources whose far blocks do: finite everywhere.  Squares of components
    underflow below 4e-23, so at 1e-17 the residuals that the sums still
    resolve are 4e-6 of the field and the bounds hold; at 1e-19 the smoother
    still brings the error below that of x = 0."""
    L = cfg[0]
    s, ref = make(cfg, prec), smoother(cfg)
    v = syn.gaussian_spinors(1, L, 12)[0]
    point = np.zeros_like(v)
    point[0, 0, 0] = 1.0
    y, yp = ref.apply(t(v), 4, 4).numpy(), ref.apply(t(point), 4, 4).numpy()
    tol = 2e-5 if prec == 1 else 2e-2
    for b, want, scales in ((v, y, (1e-15, 1e-17, 1e-19, 1e-21, 1e-23)), (point, yp, (1.0, 1e-10, 1e-15))):
        got = s.sap(np.stack([k * b for k in scales]), prec)
        for k, g in zip(scales, got):
            assert np.isfinite(g).all(), k
            if k >= 1e-17:
                assert_close(g, k * want, tol, f"scale {k}")
            elif k >= 1e-19:
                assert np.linalg.norm(g - k * want) < np.linalg.norm(k * want)
    s.close()


@pytest.mark.parametrize("L,block", [SHAPES[0], SHAPES[3], SHAPES[6]])
def test_bounded_waits(L, block):
    """Sweeps whose waits for staged data give up (wait limits from no poll to
    many): DDAMG_ETIMEOUT or the result, and with the default limits the same
    handle returns the same bits as before."""
    import paper_1811_00355_gb300 as P
    s = make((L, block, 0.3, -0.2, 1.0, 1, 0), 1)
    x = syn.gaussian_spinors(3, L, 19)
    P.pin_variant("SAP fp32", 0)
    try:
        ref = s.sap(x, 1)
        for polls in (0, 0, 1, 2, 4, 8, 16):
            s.set_wait_limit(polls)
            try:
                s.sap(x, 1)
                assert polls > 0
            except P.DDAMGError as e:
                assert e.status == 6, e
            s.set_wait_limit(-1)
            assert np.array_equal(s.sap(x, 1), ref), polls
    finally:
        P.pin_variant("SAP fp32", -1)
        s.close()
