"""Exchange layout <-> device layout: tiles of pairs of sites that end inside a
block, span several blocks or end at the lattice's end, and buffers that are
aligned to 8 bytes only."""
import numpy as np
import pytest
import torch

import synthetic as syn
from tests.gpu_common import TOL32, assert_close, make, oracle_op, t

pytestmark = pytest.mark.gpu

# blocks of 16, 96, 192 and 256 sites (8 to 128 pairs; a tile has 64)
SHAPES = [((4, 4, 4, 4), (2, 2, 2, 2)), ((8, 4, 4, 12), (4, 2, 2, 6)), ((8, 12, 8, 4), (4, 6, 4, 2)),
          ((8, 8, 8, 8), (4, 4, 4, 4))]


@pytest.mark.parametrize("L,block", SHAPES)
@pytest.mark.parametrize("shift", [0, 1])
def test_vectors_in_and_out_keep_their_bits(L, block, shift):
    s = make((L, block, 0.3, -0.2, 1.0, 3, 0), 0)
    v = syn.gaussian_spinors(3, L, 9)
    flat = torch.zeros(2 * v.size + 1, dtype=torch.float64, device="cuda")
    part = flat[shift:shift + 2 * v.size]
    part.copy_(torch.from_numpy(v.view(np.float64).reshape(-1)))
    s.set_test_vectors(part)
    np.testing.assert_array_equal(s.get_test_vectors(), v)
    s.close()


@pytest.mark.parametrize("L,block", SHAPES)
def test_fp32_fields_in_and_out(L, block):
    cfg = (L, block, 0.3, -0.2, 1.0, 3, 0)
    s = make(cfg, 1)
    x = syn.gaussian_spinors(2, L, 10)
    op = oracle_op(L, 0.3, 0, -0.2, 1.0)
    dev = torch.from_numpy(x).cuda()
    for got in (s.apply_clover(x, False, 1), s.apply_clover(dev, False, 1).cpu().numpy()):
        assert_close(got, op.site(t(x)).numpy(), TOL32)
    s.close()


def test_fp32_projections_follow_the_vectors():
    """R and P in FP32 use the vectors set last, also on an FP64 handle (whose
    FP32 copy is made for the call) and after an orthonormalisation."""
    cfg = ((8, 8, 8, 8), (4, 4, 4, 4), 0.3, -0.2, 1.0, 4, 0)
    for prec in (0, 1):
        s = make(cfg, prec)
        x = syn.gaussian_spinors(1, cfg[0], 11)
        for seed in (1, 2):
            s.set_test_vectors(syn.gaussian_spinors(4, cfg[0], seed))
            for _ in range(2):
                assert_close(s.restrict(x, 1), s.restrict(x, 0), 5 * TOL32)
                s.orthonormalize()
        s.close()
