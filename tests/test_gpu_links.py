"""Gauge links as a user hands them in."""
import numpy as np
import pytest

import synthetic as syn
from oracle.dirac import WilsonClover
from tests.gpu_common import TOL64, assert_close, t

pytestmark = pytest.mark.gpu
L, BLOCK = (4, 4, 4, 8), (2, 2, 2, 4)


def test_links_at_the_tolerance():
    """Links that are SU(3) to 5e-10 only (1e-9 is accepted): the clover term
    and the FP64 D are those of the links as given, third rows included."""
    import paper_1811_00355_gb300 as P
    U = syn.gauge_field(L, 0.3, 4)
    gen = np.random.default_rng(5)
    U = U + 5e-11 * (gen.standard_normal(U.shape) + 1j * gen.standard_normal(U.shape))
    off = np.abs(U @ U.conj().swapaxes(-1, -2) - np.eye(3)).max()
    assert 1e-10 < off < 9e-10, off
    op = WilsonClover(t(U), L, -0.2, 1.0)
    s = P.DDAMG(P.default_params(L=L, sap_block=BLOCK, n_v=1, m0=-0.2, csw=1.0, precision=P.FP64), U)
    try:
        x = syn.gaussian_spinors(2, L, 16)
        assert_close(s.get_clover(), op.packed_clover().numpy(), TOL64)
        assert_close(s.apply_D(x, P.FP64), op.apply(t(x)).numpy(), TOL64)
        s.set_gauge(syn.gauge_field(L, 0.2, 6))
        s.set_gauge(U)
        assert_close(s.apply_D(x, P.FP64), op.apply(t(x)).numpy(), TOL64)
    finally:
        s.close()


@pytest.mark.parametrize("n_v", [1, 8])
def test_host_links_within_a_device_memory_budget(n_v):
    """Links from the host need no more device memory than the links in the
    exchange layout beside a handle with two rows a link did (120 doubles a
    site; the links are now kept as 72): two fields beyond what the handle
    holds, at the first links and after ddamg_trim, in one piece or several."""
    import torch
    import paper_1811_00355_gb300 as P
    U = syn.gauge_field(L, 0.3, 4)
    kw = dict(L=L, sap_block=BLOCK, n_v=n_v, m0=-0.2, csw=1.0, precision=P.FP32)
    s = P.DDAMG(P.default_params(**kw), torch.from_numpy(U).cuda())
    x = syn.gaussian_spinors(2, L, 17)
    ref = s.apply_D(x, P.FP64)
    s.close()
    s = P.DDAMG(P.default_params(**kw), torch.from_numpy(U).cuda())
    held = s.stats()["device_bytes"]
    s.close()
    s = P.DDAMG(P.default_params(hbm_budget=held + 2 * x[0].nbytes, **kw), U)
    try:
        s.trim()
        s.set_gauge(syn.gauge_field(L, 0.2, 6))
        s.trim()
        s.set_gauge(U)
        dev = torch.from_numpy(x).cuda()
        torch.cuda.synchronize()
        assert np.array_equal(s.apply_D(dev, P.FP64).cpu().numpy(), ref)
    finally:
        s.close()
