"""GPU parity of the tiled CUDA-core kernels (forward and backward) where their tiling can go wrong: lists of exactly
one step and one token more, patches other than 8 x 8, head sizes at the edges of the padded sizes, lists cut over a
cluster and not cut."""
import math

import numpy as np
import pytest
import torch

from oracle import clear_oracle as oracle
from oracle import clear_oracle_bwd as oracle_bwd
from paper_2412_16112_b200 import binding as clear
from paper_2412_16112_b200 import workloads

pytestmark = pytest.mark.gpu

# B * H, grid, text tokens, radius, head size
SHAPES = [
    (1, 8, 8, 0, 20.0, 64),      # one tile, a list of exactly 64 keys: one step
    (1, 8, 8, 1, 20.0, 68),      # 65 keys, the first head size padded to 128
    (1, 5, 3, 63, 2.0, 4),       # a grid smaller than a patch, the smallest head size, 64-row text tile one short
    (2, 4, 70, 65, 3.5, 128),    # 4 x 16 patches, a second text tile of one row
    (2, 70, 2, 10, 3.0, 40),     # 32 x 2 patches
    (40, 17, 23, 20, 4.0, 64),   # more tiles than blocks the device holds: lists not cut
    (3, 24, 40, 130, 8.0, 128),  # cut lists, some of the parts empty
]


def _inputs(bh, gh, gw, T, d, n, seed):
    g = torch.Generator(device="cpu").manual_seed(seed)
    return [torch.randn((1, bh, T + gh * gw, d), generator=g) for _ in range(n)]


@pytest.mark.parametrize("bh,gh,gw,T,r,d", SHAPES + [(2, 9, 21, 33, 3.0, 132), (1, 20, 20, 5, 4.0, 256)])
def test_forward_tiles(bh, gh, gw, T, r, d):
    q, k, v = _inputs(bh, gh, gw, T, d, 3, 11)
    scale = 1 / math.sqrt(d)
    want = oracle.attn(q, k, v, gh, gw, T, r, scale)
    qd, kd, vd = (t.cuda() for t in (q, k, v))
    out = torch.full_like(qd, float("nan"))
    clear.clear_attn_fwd_f32(qd, kd, vd, out, gh, gw, T, r, scale)
    assert np.abs(out.cpu().double().numpy() - want).max() <= 1e-5
    clear.clear_cache_clear()


@pytest.mark.parametrize("bh,gh,gw,T,r,d", SHAPES)
def test_backward_tiles(bh, gh, gw, T, r, d):
    q, k, v, g = _inputs(bh, gh, gw, T, d, 4, 12)
    scale = 1 / math.sqrt(d)
    want = oracle_bwd.attn_bwd(q, k, v, g, gh, gw, T, r, scale)
    qd, kd, vd, gd = (t.cuda() for t in (q, k, v, g))
    outs = [torch.full_like(qd, float("nan")) for _ in range(3)]
    clear.clear_attn_bwd_f32(qd, kd, vd, gd, *outs, gh, gw, T, r, scale)
    for name, got, ref in zip(("dq", "dk", "dv"), outs, want):
        err = np.abs(got.cpu().double().numpy() - ref)
        # fp32 sums of a few hundred terms of order one (the bound of the small-shape tests)
        assert err.max() <= 1e-4, f"{name}: max {err.max():.3e}"
    clear.clear_cache_clear()
