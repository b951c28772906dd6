"""The coarse GMRES for five or more right-hand sides and blocks of 32 to 64
rows, against the oracle's coarse solver on the same operator: every block
width class (rows that fill the lanes' pairs and rows that do not), one site
per CTA and several (the last CTA with fewer), fewer right-hand sides than a
lockstep group and several groups, restarts, and a zero right-hand side.

Bounds as in test_gpu_coarse_plans: iteration counts at 5e-2 within one, the
Krylov iterate after six iterations to 1e-4."""
import numpy as np
import pytest
import torch

import synthetic as syn
from oracle.coarse import CoarseOperator
from oracle.lattice import Geometry
from tests.gpu_common import assert_close

pytestmark = pytest.mark.gpu

DIAG, HOP = 1.0, 0.21
# (coarse lattice of 2^4 blocks, n_v, nrhs, restart)
CASES = [((2, 2, 2, 2), 16, 5, 30), ((4, 4, 4, 8), 17, 8, 30), ((4, 4, 4, 6), 20, 9, 30), ((4, 4, 4, 8), 24, 12, 30),
         ((2, 4, 6, 8), 25, 13, 4), ((4, 4, 4, 8), 32, 12, 30), ((2, 2, 4, 4), 29, 25, 30)]


def _solve(cL, n_v, restart, max_iter, Dc, bc, tol):
    import paper_1811_00355_gb300 as P
    L = tuple(2 * v for v in cL)
    p = P.default_params(L=L, sap_block=(2, 2, 2, 2), n_v=n_v, precision=P.FP32, coarse_restart=restart,
                         coarse_max_iter=max_iter)
    s = P.DDAMG(p, syn.unit_gauge(L))
    try:
        s.set_coarse_op(Dc)
        plan = s.coarse_plan(bc.shape[0])
        assert plan["rhs_per_pass"] == (12 if bc.shape[0] > 8 else 8) and plan["block_ring"] == 1, plan
        return s.coarse_solve(bc, tol, P.FP32)
    finally:
        s.close()


@pytest.mark.parametrize("cL,n_v,nrhs,restart", CASES)
def test_wide(cL, n_v, nrhs, restart):
    geom = Geometry(cL)
    Dc = syn.coarse_stencil(geom.V, 2 * n_v, 8, DIAG, HOP)
    cop = CoarseOperator(torch.from_numpy(Dc), geom)
    gen = np.random.default_rng(70 + nrhs)
    bc = gen.standard_normal((nrhs, geom.V, 2 * n_v)) + 1j * gen.standard_normal((nrhs, geom.V, 2 * n_v))
    bc[1] = 0.0
    bc[2] *= 1e-8
    x, its = _solve(cL, n_v, restart, 300, Dc, bc, 5e-2)
    x6, its6 = _solve(cL, n_v, restart, 6, Dc, bc, 1e-30)
    assert its[1] == 0 and not x[1].any() and not x6[1].any()
    for r in [0] + list(range(2, nrhs)):
        _, ir = cop.solve(torch.from_numpy(bc[r]), 5e-2, restart, 300)
        assert abs(int(its[r]) - ir) <= 1, (r, its, ir)
        xr, ir = cop.solve(torch.from_numpy(bc[r]), 1e-30, restart, 6)
        assert its6[r] == ir == 6
        assert_close(x6[r], xr.numpy(), 1e-4, f"rhs {r}")


def test_all_zero():
    Dc = syn.coarse_stencil(32, 40, 9, DIAG, HOP)
    x, its = _solve((2, 2, 2, 4), 20, 30, 300, Dc, np.zeros((6, 32, 40), complex), 5e-2)
    assert not its.any() and not x.any()


@pytest.mark.parametrize("cL,resident", [((2, 2, 2, 2), 1), ((4, 4, 4, 4), 1), ((4, 4, 4, 6), 0)])
def test_eight_with_32_row_blocks(cL, resident):
    """Eight right-hand sides, n_v 16: resident blocks where a CTA owns one
    site, else the ring."""
    import paper_1811_00355_gb300 as P
    geom = Geometry(cL)
    Dc = syn.coarse_stencil(geom.V, 32, 10, DIAG, HOP)
    cop = CoarseOperator(torch.from_numpy(Dc), geom)
    gen = np.random.default_rng(74)
    bc = gen.standard_normal((8, geom.V, 32)) + 1j * gen.standard_normal((8, geom.V, 32))
    L = tuple(2 * v for v in cL)
    s = P.DDAMG(P.default_params(L=L, sap_block=(2, 2, 2, 2), n_v=16, precision=P.FP32, coarse_max_iter=6),
                syn.unit_gauge(L))
    try:
        s.set_coarse_op(Dc)
        plan = s.coarse_plan(8)
        assert plan["rhs_per_pass"] == 8 and plan["resident_blocks"] == resident, plan
        assert plan["block_ring"] == 1 - resident, plan
        x, its = s.coarse_solve(bc, 1e-30, P.FP32)
        assert np.all(its == 6)
        for r in range(8):
            xr, _ = cop.solve(torch.from_numpy(bc[r]), 1e-30, 30, 6)
            assert_close(x[r], xr.numpy(), 1e-4, f"rhs {r}")
    finally:
        s.close()
