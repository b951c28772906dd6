"""The orthonormalisation that forms the second pass's small update in FP32
(handles with an FP32 inner solver) against the one that is FP64 throughout
(FP64 handles), on vectors from independent to nearly parallel: the vectors
equally orthonormal, and equal up to what the Gram-Schmidt of vectors that
close amplifies.

Bounds: an inner product of 6 |aggregate| = 1536 terms rounds to
sqrt(1536) 2^-53 = 4e-15, the deviation from orthonormality to a few of
those, 2e-14; two results differ by that times the norm lost to the first
pass, 1 / spread."""
import numpy as np
import pytest

import synthetic as syn
from tests.gpu_common import make

pytestmark = pytest.mark.gpu
CFG = ((8, 8, 8, 8), (4, 4, 4, 4), 0.3, -0.2, 1.0, 24, 0)


def _basis(v):
    """[n][V][4][3] -> [aggregate][chirality][n][6 |aggregate|]"""
    n = v.shape[0]
    w = v.reshape(n, 2, 4, 2, 4, 2, 4, 2, 4, 2, 6).transpose(1, 3, 5, 7, 9, 0, 2, 4, 6, 8, 10)
    return w.reshape(16, 2, n, -1)


@pytest.mark.parametrize("spread,scale", [(1.0, 1.0), (1e-3, 1.0), (1e-5, 1.0), (1e-8, 1.0), (1e-11, 1.0),
                                          (1e-5, 1e-34), (1e-5, 1e34)])
def test_split_update(spread, scale):
    v = spread * syn.gaussian_spinors(24, CFG[0], 21) + syn.gaussian_spinors(1, CFG[0], 22)
    out = []
    for prec in (0, 1):
        s = make(CFG, prec)
        s.set_test_vectors(scale * v)
        s.orthonormalize()
        out.append(_basis(s.get_test_vectors()))
        s.close()
    dev = [np.abs(b.conj() @ b.swapaxes(-1, -2) - np.eye(24)).max() for b in out]
    assert max(dev) < 2e-14 and dev[1] < 2 * dev[0] + 2e-15, dev
    assert np.abs(out[0] - out[1]).max() < 2e-14 / spread
