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


@pytest.mark.parametrize("negative", [False, True])
@pytest.mark.parametrize("bh,gh,gw,T,r,d", [
    (1, 8, 8, 1, 20.0, 72),      # one block with two steps: 8 rows a warp
    (40, 17, 23, 20, 4.0, 72),   # more blocks than SMs: 4 x 4 results a thread
    (40, 13, 19, 0, 4.0, 8),
    (3, 24, 40, 130, 8.0, 40),   # cut lists, more blocks than SMs
    (2, 9, 21, 33, 3.0, 136),
])
def test_forward_tiles_of_bf16_tensors(bh, gh, gw, T, r, d, negative):
    """Head sizes that the tensor-core kernels do not take, and a scale that they do not: fp32 arithmetic (1e-5, as above), the output
    rounded to 8 bits."""
    q, k, v = (x.to(torch.bfloat16) for x in _inputs(bh, gh, gw, T, d, 3, 15))
    scale = (-1 if negative else 1) / math.sqrt(d)
    want = oracle.attn(q, k, v, gh, gw, T, r, scale)
    out = torch.full_like(q, float("nan"), device="cuda:0")
    clear.clear_attn_fwd(*(t.cuda() for t in (q, k, v)), out, gh, gw, T, r, scale)
    assert (np.abs(out.cpu().double().numpy() - want) <= 1e-5 + 2.0 ** -8 * np.abs(want)).all()
    clear.clear_cache_clear()


@pytest.mark.parametrize("rise", [10, 17, 90, -17])
@pytest.mark.parametrize("bh,gh,gw,T,r,d", [(1, 24, 40, 130, 8.0, 64), (40, 19, 23, 0, 6.0, 128), (2, 3, 90, 70, 9.0, 40)])
def test_forward_tiles_with_scores_that_climb(bh, gh, gw, T, r, d, rise):
    """Scores that climb (or fall) by `rise` every 32 text tokens and every four rows or 16 columns of the grid: rows whose reference stays, and
    rows whose reference moves, at every step.  Scores of size L are good to a few 2^-24 L, and so are the weights."""
    q, k, v = _inputs(bh, gh, gw, T, d, 3, 14)
    ys, xs = torch.arange(gh).repeat_interleave(gw), torch.arange(gw).repeat(gh)
    q[..., 0], k[..., 0] = 1.0, rise * torch.cat([torch.arange(T) // 32, T // 32 + ys // 4 + xs // 16]).float()
    want = oracle.attn(q, k, v, gh, gw, T, r, 1.0)
    out = torch.full_like(q, float("nan"), device="cuda:0")
    clear.clear_attn_fwd_f32(*(t.cuda() for t in (q, k, v)), out, gh, gw, T, r, 1.0)
    logit = float(q.norm(dim=-1).max() * k.norm(dim=-1).max())
    assert np.abs(out.cpu().double().numpy() - want).max() <= 1e-5 + 2.0 ** -21 * logit * float(v.abs().max())
    clear.clear_cache_clear()


def _low_keys_first(bh, d, n_low, seed, low=-12.0):
    """An 8 x 8 grid at r = 1 behind n_low + 2 text tokens: the first n_low keys of every query score `low`, the next two q0 k0, below 1
    and with all of fp32's bits, and the image keys -112.  A row's softmax is that of the two."""
    T, gen = n_low + 2, torch.Generator(device="cpu").manual_seed(seed)
    q, k, v = (torch.zeros(1, bh, T + 64, d) for _ in range(3))
    q[..., 0], q[..., 1] = torch.rand(q.shape[:-1], generator=gen), 1.0
    k[..., n_low, 0], k[..., n_low + 1, 0] = 0.7, -0.3
    k[..., :n_low, 1], k[..., T:, 1] = low, -112.0
    v[..., n_low, :], v[..., n_low + 1, :] = 1.0, -1.0
    return T, q, k, v


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("bh,n_low", [(100, 64), (1, 1024)])   # whole lists; lists cut eight ways, a block to an SM
def test_forward_weights_of_rows_whose_first_keys_score_low(bh, n_low, d):
    """out = tanh((s1 - s2) / 2), nearly.  A weight expf(s - m) is good to the rounding of s and of s - m and to expf's last bit: for s - m
    within [-1, 2] at most 2^-25 + 2^-24 + 2^-23 of it, two of which a row has at half weight: 2.1e-7 and the output's 3e-8 at the most; a
    third of that, for errors spread evenly, over all rows.  Against the -12 of the first tiles s - m is rounded at 2^-21: 1.9e-7 over all
    rows."""
    T, q, k, v = _low_keys_first(bh, d, n_low, 21)
    want = oracle.attn(q, k, v, 8, 8, T, 1.0, 1.0)
    out = torch.full_like(q, float("nan"), device="cuda:0")
    clear.clear_attn_fwd_f32(*(t.cuda() for t in (q, k, v)), out, 8, 8, T, 1.0, 1.0)
    err = np.abs(out.cpu().double().numpy() - want)
    assert err.max() <= 2.4e-7 and np.sqrt((err ** 2).mean()) <= 0.8e-7, (err.max(), np.sqrt((err ** 2).mean()))
    clear.clear_cache_clear()


# more tiles than SMs above 64 channels: lists not cut, results stored without a merge
_WHOLE_LISTS = [(40, 19, 23, 0, 6.0, 68), (40, 19, 23, 0, 6.0, 96), (40, 19, 23, 0, 6.0, 128)]


@pytest.mark.parametrize("bh,gh,gw,T,r,d", SHAPES + _WHOLE_LISTS)
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


@pytest.mark.parametrize("rise", [10, 17, 90, -17])
@pytest.mark.parametrize("bh,gh,gw,T,r,d", [(40, 19, 23, 0, 6.0, 128), (1, 24, 40, 130, 8.0, 96), (2, 3, 90, 70, 9.0, 40), (40, 19, 23, 0, 6.0, 64)])
def test_backward_tiles_with_scores_that_climb(bh, gh, gw, T, r, d, rise):
    """As in the forward test: references, and the sums against them, that move at every step, and that differ between the blocks of a
    cut list.  Weights are good to eps, a few 2^-24 of the largest score and the rounding of fp32 sums, and each gradient to eps times
    its sum with every term taken positive."""
    q, k, v, g = _inputs(bh, gh, gw, T, d, 4, 16)
    ys, xs = torch.arange(gh).repeat_interleave(gw), torch.arange(gw).repeat(gh)
    q[..., 0], k[..., 0] = 1.0, rise * torch.cat([torch.arange(T) // 32, T // 32 + ys // 4 + xs // 16]).float()
    want = oracle_bwd.attn_bwd(q, k, v, g, gh, gw, T, r, 1.0)
    outs = [torch.full_like(q, float("nan"), device="cuda:0") for _ in range(3)]
    clear.clear_attn_bwd_f32(*(t.cuda() for t in (q, k, v, g)), *outs, gh, gw, T, r, 1.0)
    eps = 2.0 ** -21 * float(q.norm(dim=-1).max() * k.norm(dim=-1).max()) + 4e-6
    q, k, v, g = (t.double() for t in (q, k, v, g))
    P = (q @ k.mT).masked_fill(~torch.from_numpy(_mask(gh, gw, T, r)), -math.inf).softmax(-1)
    dP = (g @ v.mT).abs()
    dS = P * (dP + (P * dP).sum(-1, keepdim=True))
    for name, got, ref, size in zip(("dq", "dk", "dv"), outs, want, (dS @ k.abs(), dS.mT @ q.abs(), P.mT @ g.abs())):
        err = np.abs(got.cpu().double().numpy() - ref)
        assert (err <= eps * size.numpy() + 1e-6).all(), f"{name}: {np.max(err - eps * size.numpy()):.3e}"
    clear.clear_cache_clear()


@pytest.mark.parametrize("d", [96, 128])
@pytest.mark.parametrize("bh,n_low", [(100, 64), (1, 1024)])   # whole lists; lists cut eight ways
def test_backward_weights_of_rows_whose_first_keys_score_low(bh, n_low, d):
    """dO = 1 in channel c of row c alone: dV of a key is its weight p in the first d rows.  p = e1 / (e1 + e2) at about a half is good to
    half of e1's and the sum's errors (2^-25 for s, 2^-25 for s - m, 2^-23 for expf, twice) and two roundings of 2^-24: 2.4e-7 at the
    most, and a quarter of that, for errors spread evenly, over all rows.  Against the -12 of the first tiles: 1.0e-7 over all rows."""
    T, q, k, v = _low_keys_first(bh, d, n_low, 22)
    g = torch.zeros_like(q)
    g[..., torch.arange(d), torch.arange(d)] = 1.0
    want = oracle_bwd.attn_bwd(q, k, v, g, 8, 8, T, 1.0, 1.0)[2]
    outs = [torch.full_like(q, float("nan"), device="cuda:0") for _ in range(3)]
    clear.clear_attn_bwd_f32(*(t.cuda() for t in (q, k, v, g)), *outs, 8, 8, T, 1.0, 1.0)
    err = np.abs(outs[2].cpu().double().numpy() - want)[..., n_low:n_low + 2, :]
    assert err.max() <= 2.4e-7 and np.sqrt((err ** 2).mean()) <= 0.6e-7, (err.max(), np.sqrt((err ** 2).mean()))
    clear.clear_cache_clear()


@pytest.mark.parametrize("d", [64, 96, 128])
@pytest.mark.parametrize("bh,n_low", [(100, 64), (1, 1024)])
def test_backward_sums_stay_in_range_where_first_keys_score_low(bh, n_low, d):
    """dP of 1e34: times a weight, which no maximum keeps at one, it would leave fp32's range.  Bound: 1e-5 of the largest gradient, for
    fp32 sums of up to a thousand terms."""
    T, q, k, v = _low_keys_first(bh, d, n_low, 23, low=-15.0)
    v, g = v * 0.0, torch.zeros_like(q)
    v[..., n_low, 3], v[..., n_low + 1, 3], g[..., 3] = 1e17, -1e17, 1e17
    want = oracle_bwd.attn_bwd(q, k, v, g, 8, 8, T, 1.0, 1.0)
    outs = [torch.full_like(q, float("nan"), device="cuda:0") for _ in range(3)]
    clear.clear_attn_bwd_f32(*(t.cuda() for t in (q, k, v, g)), *outs, 8, 8, T, 1.0, 1.0)
    for name, got, ref in zip(("dq", "dk", "dv"), outs, want):
        err = np.abs(got.cpu().double().numpy() - ref)
        assert err.max() <= 1e-5 * np.abs(ref).max(), f"{name}: max {err.max():.3e} of {np.abs(ref).max():.3e}"
    clear.clear_cache_clear()


@pytest.mark.parametrize("d", [8, 40, 96, 128])
@pytest.mark.parametrize("gh,gw,r", [(9, 13, 1.0), (24, 21, 3.0), (24, 21, 3.2), (1, 70, 12.9)])
def test_backward_with_few_keys_and_no_text(gh, gw, r, d):
    """Both sides of the line between the kernel with a warp per token (1 and 25 keys, and 25 in a row) and the tiles (37)."""
    q, k, v, g = _inputs(2, gh, gw, 0, d, 4, 13)
    scale = 1 / math.sqrt(d)
    want = oracle_bwd.attn_bwd(q, k, v, g, gh, gw, 0, r, scale)
    outs = [torch.full_like(q, float("nan"), device="cuda:0") for _ in range(3)]
    clear.clear_attn_bwd_f32(*(t.cuda() for t in (q, k, v, g)), *outs, gh, gw, 0, r, scale)
    for name, got, ref in zip(("dq", "dk", "dv"), outs, want):
        err = np.abs(got.cpu().double().numpy() - ref)
        assert err.max() <= 1e-4, f"{name}: max {err.max():.3e}"
    clear.clear_cache_clear()


def _mask(gh, gw, T, r):
    ys, xs = np.repeat(np.arange(gh), gw), np.tile(np.arange(gw), gh)
    M = np.ones((T + gh * gw,) * 2, dtype=bool)
    M[T:, T:] = (ys[:, None] - ys) ** 2 + (xs[:, None] - xs) ** 2 < r * r
    return M


# B * H, grid, text tokens, radius, head size: lists cut over a cluster; whole ones; the two wider padded head sizes
_ISOLATION = [(2, 24, 40, 20, 3.0, 64), (40, 24, 40, 0, 3.0, 8), (2, 13, 19, 7, 2.5, 128), (1, 9, 33, 5, 2.0, 256)]


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("which", ["q", "k", "v"])
@pytest.mark.parametrize("H,gh,gw,T,r,d", _ISOLATION)
def test_forward_tiles_keep_non_finite_values_to_the_rows_that_see_them(H, gh, gw, T, r, d, which, bad):
    """One non-finite element: the rows that see its token are non-finite, all others are what they are without it (same
    terms in fp32; the rows of its tile are summed in another order)."""
    ts = dict(zip("qkv", workloads.make_custom(1, H, gh, gw, T, d, dtype="f32", qk_norm=False, seed=gh)))
    scale, token = 1 / math.sqrt(d), T + (gh // 2) * gw + gw // 2
    want = oracle.attn(ts["q"], ts["k"], ts["v"], gh, gw, T, r, scale)
    ts[which][0, 0, token, 3] = bad
    out = torch.full_like(ts["q"], 7.0, device="cuda:0")
    clear.clear_attn_fwd_f32(*(t.to("cuda:0") for t in ts.values()), out, gh, gw, T, r, scale)
    got = out.cpu().double().numpy()
    M = _mask(gh, gw, T, r)
    hit = np.zeros((H, M.shape[0]), dtype=bool)
    hit[0] = np.arange(M.shape[0]) == token if which == "q" else M[:, token]
    # (an infinite score of the right sign is a softmax on that key alone, or none: not every row has to be non-finite)
    finite = np.isfinite(got[0]).all(-1)
    assert finite[~hit].all()
    if bad != bad or which == "v":
        assert not finite[hit].any()
    assert np.abs(got[0] - want[0])[~hit].max() <= 1e-5
    clear.clear_cache_clear()


@pytest.mark.parametrize("which", ["q", "k", "v", "g"])
@pytest.mark.parametrize("H,gh,gw,T,r,d", _ISOLATION[:3] + _WHOLE_LISTS[2:])
def test_backward_tiles_keep_non_finite_values_to_the_rows_that_see_them(H, gh, gw, T, r, d, which):
    """The same for the gradients.  A NaN in q or dO makes row t of P, or of dS, NaN; one in k or v does so for every query
    that sees it (the row's sum, or delta), v leaving P alone."""
    ts = dict(zip("qkv", workloads.make_custom(1, H, gh, gw, T, d, dtype="f32", qk_norm=False, seed=gh)))
    gen = torch.Generator(device="cpu").manual_seed(gh + gw)
    ts["g"] = torch.randn(ts["q"].shape, generator=gen, dtype=torch.float32)
    scale, token = 1 / math.sqrt(d), T + (gh // 2) * gw + gw // 2
    want = oracle_bwd.attn_bwd(*ts.values(), gh, gw, T, r, scale)
    ts[which][0, 0, token, 3] = float("nan")
    outs = [torch.full_like(ts["q"], 7.0, device="cuda:0") for _ in range(3)]
    clear.clear_attn_bwd_f32(*(t.to("cuda:0") for t in ts.values()), *outs, gh, gw, T, r, scale)
    M = _mask(gh, gw, T, r)
    rows = np.arange(M.shape[0]) == token if which in "qg" else M[:, token]
    keys = M[rows].any(0)
    hit = {"dq": rows, "dk": keys, "dv": np.zeros_like(keys) if which == "v" else keys}
    for (name, bad_rows), got, ref in zip(hit.items(), outs, want):
        x = got.cpu().double().numpy()[0]
        finite = np.isfinite(x).all(-1)
        assert (finite[0] == ~bad_rows).all() and finite[1:].all(), name
        assert np.abs(x - ref[0])[finite].max() <= 1e-4, name
    clear.clear_cache_clear()
