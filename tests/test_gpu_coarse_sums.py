"""The sums over all CTAs in the coarse GMRES where one reduction follows
another without a grid barrier in between: the explicit norm of a nearly
cancelled w (FP32), and the second Gram-Schmidt pass and the norm (FP64), in
both kernels, at every lockstep width, with one site per CTA and 128 CTAs.

A coarse operator close to the identity, D_c = 1 + G with |G v| = 0.007 |v|,
makes ||w||^2 - |h|^2 cancel to 5e-5 ||w||^2 (the explicit norm is taken below
1e-3) in every iteration.  Six iterations reduce the residual to 1e-12: the
FP32 solution is then off by the rounding of a few block products, each within
1e-6 (bound 1e-5), the FP64 one by the residual (bound 1e-11).  The sums run in
a fixed order, so repeated calls and equal right-hand sides agree bit by bit."""
import numpy as np
import pytest
import torch

import synthetic as syn
from oracle.coarse import CoarseOperator
from oracle.lattice import Geometry
from tests.gpu_common import assert_close

pytestmark = pytest.mark.gpu

L, BLOCK, GRID = (8, 8, 8, 8), (2, 2, 2, 2), (4, 4, 4, 4)


def _case(n_v, prec, nrhs, restart, max_iter, hop, seed):
    import paper_1811_00355_gb300 as P
    geom = Geometry(GRID)
    Dc = syn.coarse_stencil(geom.V, 2 * n_v, seed, 1.0, hop)
    p = P.default_params(L=L, sap_block=BLOCK, n_v=n_v, precision=prec, coarse_restart=restart,
                         coarse_max_iter=max_iter)
    s = P.DDAMG(p, syn.unit_gauge(L))
    s.set_coarse_op(Dc)
    gen = np.random.default_rng(60 + nrhs)
    bc = gen.standard_normal((nrhs, geom.V, 2 * n_v)) + 1j * gen.standard_normal((nrhs, geom.V, 2 * n_v))
    if nrhs > 1:
        bc[-1] = bc[0]
    return s, CoarseOperator(torch.from_numpy(Dc), geom), bc


@pytest.mark.parametrize("noalloc", [False, True])
@pytest.mark.parametrize("n_v,prec,nrhs,restart", [(16, 1, 1, 30), (6, 1, 4, 30), (20, 1, 5, 30), (16, 1, 8, 8),
                                                   (24, 1, 12, 8), (6, 1, 12, 8), (4, 0, 1, 30), (4, 0, 12, 8)])
def test_nearly_cancelled(n_v, prec, nrhs, restart, noalloc):
    s, cop, bc = _case(n_v, prec, nrhs, restart, 6, 0.005, 21)
    try:
        call = s.coarse_solve_noalloc if noalloc else lambda b, tol: s.coarse_solve(b, tol, prec)
        dev = torch.from_numpy(bc).cuda()
        torch.cuda.synchronize()
        first = None
        for _ in range(8):
            x, its = call(dev, 1e-30)
            x = x.cpu().numpy()
            assert np.all(its == 6), its
            if first is None:
                first = x
            assert np.array_equal(x, first)
        assert np.array_equal(x[-1], x[0])
        for r in (0, nrhs // 2):
            ref, _ = cop.solve(torch.from_numpy(bc[r]), 1e-13, 30, 30)
            assert_close(x[r], ref.numpy(), 1e-11 if prec == 0 else 1e-5, f"rhs {r}")
    finally:
        s.close()


def test_fp64_more_vectors_than_the_buffer_holds_twice():
    """Twelve right-hand sides in lockstep with 36 basis vectors: beyond 33 the
    sums' buffer has no room for both passes.  A Krylov iterate of a solve that
    is at 1e-4 by then; the oracle's Gram-Schmidt loses 2^-53 / 1e-4 of its
    orthogonality (bound 1e-10)."""
    s, cop, bc = _case(4, 0, 12, 36, 36, 0.21, 22)
    try:
        plan = s.coarse_plan(12)
        assert plan["rhs_per_pass"] == 12 and plan["ctas"] == 128, plan
        x, its = s.coarse_solve(bc, 1e-30, 0)
        assert np.all(its == 36), its
        assert np.array_equal(x[-1], x[0])
        for r in (0, 5):
            ref, _ = cop.solve(torch.from_numpy(bc[r]), 1e-30, 36, 36)
            assert_close(x[r], ref.numpy(), 1e-10, f"rhs {r}")
    finally:
        s.close()


@pytest.mark.parametrize("nrhs,restart", [(8, 8), (12, 4)])
def test_narrow_ring_at_full_width(nrhs, restart):
    """The narrow kernel's block ring with 8 and 12 right-hand sides in
    lockstep, two sites per CTA, which the no-allocation call alone reaches:
    the oracle's Krylov iterate after six iterations (bound 1e-4 as in
    test_gpu_coarse_plans)."""
    import paper_1811_00355_gb300 as P
    fine = (8, 8, 8, 16)
    geom = Geometry((4, 4, 4, 8))
    Dc = syn.coarse_stencil(geom.V, 32, 23, 1.0, 0.21)
    cop = CoarseOperator(torch.from_numpy(Dc), geom)
    gen = np.random.default_rng(66)
    bc = gen.standard_normal((nrhs, geom.V, 32)) + 1j * gen.standard_normal((nrhs, geom.V, 32))
    s = P.DDAMG(P.default_params(L=fine, sap_block=BLOCK, n_v=16, precision=P.FP32, coarse_restart=restart,
                                 coarse_max_iter=6), syn.unit_gauge(fine))
    try:
        s.set_coarse_op(Dc)
        dev = torch.from_numpy(bc).cuda()
        torch.cuda.synchronize()
        x, its = s.coarse_solve_noalloc(dev, 1e-30)
        assert np.all(its == 6), its
        for r in range(nrhs):
            ref, _ = cop.solve(torch.from_numpy(bc[r]), 1e-30, restart, 6)
            assert_close(x[r].cpu().numpy(), ref.numpy(), 1e-4, f"rhs {r}")
    finally:
        s.close()
