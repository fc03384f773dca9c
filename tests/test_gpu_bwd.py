"""GPU parity of the backward pass (`clear_attn_bwd_f32`, through the C ABI) against its fp64 CPU oracle,
element by element on small shapes."""
import math

import numpy as np
import pytest
import torch

from oracle import clear_oracle_bwd as oracle_bwd
from paper_2412_16112_b200 import binding as clear
from paper_2412_16112_b200 import workloads

pytestmark = pytest.mark.gpu

# fp32 arithmetic with fp32 atomic sums of up to a few hundred terms of order one
BWD_ATOL = 1e-4


@pytest.mark.parametrize("gh,gw,T,r,d", [
    (16, 16, 16, 4.0, 64),      # the tiny fp32 configuration
    (13, 19, 7, 4.0, 128),      # ragged on both axes
    (8, 16, 0, 1.0, 128),       # no text, self only: dv = d_out, dq = dk = 0
    (9, 33, 0, 5.5, 40),        # head size that is no multiple of 32, non-integer radius
    (20, 50, 3, 100.0, 64),     # radius beyond the diagonal: full attention
    (1, 70, 2, 3.0, 96),        # single-row grid
    (24, 40, 130, 8.0, 64),
])
def test_backward_matches_the_oracle_everywhere(gh, gw, T, r, d):
    q, k, v = workloads.make_custom(1, 2, gh, gw, T, d, dtype="f32", qk_norm=False, seed=gh * 31 + gw)
    g = torch.Generator(device="cpu").manual_seed(gh + gw)
    d_out = torch.randn(q.shape, generator=g, dtype=torch.float32)
    scale = 1 / math.sqrt(d)
    want = oracle_bwd.attn_bwd(q, k, v, d_out, gh, gw, T, r, scale)
    dev = torch.device("cuda:0")
    qd, kd, vd, gd = (t.to(dev) for t in (q, k, v, d_out))
    dq, dk, dv = (torch.full_like(qd, float("nan")) for _ in range(3))
    for _ in range(2):      # the second call finds dk, dv dirty and must start them at zero again
        clear.clear_attn_bwd_f32(qd, kd, vd, gd, dq, dk, dv, gh, gw, T, r, scale)
    torch.cuda.synchronize()
    for name, got, ref in (("dq", dq, want[0]), ("dk", dk, want[1]), ("dv", dv, want[2])):
        err = np.abs(got.cpu().double().numpy() - ref)
        assert np.isfinite(err).all(), f"{name}: non-finite"
        assert err.max() <= BWD_ATOL, f"{name}: max {err.max():.3e}"
    clear.clear_cache_clear()


def test_backward_argument_errors():
    dev = torch.device("cuda:0")
    x = torch.zeros(1, 1, 272, 64, device=dev)
    p = x.data_ptr()
    lib = clear.load()
    assert lib.clear_attn_bwd_f32(p, p, p, p, p, p, p, 1, 1, 16, 16, 16, 64, 0.0, 0.125, None) == clear.ERR_INVALID_ARG
    assert lib.clear_attn_bwd_f32(p, p, p, None, p, p, p, 1, 1, 16, 16, 16, 64, 4.0, 0.125, None) == clear.ERR_INVALID_ARG
    assert lib.clear_attn_bwd_f32(p, p, p, p, p, p + 4, p, 1, 1, 16, 16, 16, 64, 4.0, 0.125, None) == clear.ERR_MISALIGNED
    assert lib.clear_attn_bwd_f32(p, p, p, p, p, p, p, 1, 1, 16, 16, 16, 64, 4.0, float("nan"), None) == clear.ERR_INVALID_ARG


def test_backward_repeats_bit_for_bit_and_from_two_streams():
    """One writer per output element and a fixed order of summation: the same bits on every call, also when two
    streams call for the same shape at once (the library orders them: they share the row statistics)."""
    gh, gw, T, r, d = 24, 40, 130, 8.0, 64
    q, k, v = workloads.make_custom(1, 3, gh, gw, T, d, dtype="f32", qk_norm=False, seed=5)
    g = torch.Generator(device="cpu").manual_seed(6)
    d_out = torch.randn(q.shape, generator=g, dtype=torch.float32)
    scale = 1 / math.sqrt(d)
    dev = torch.device("cuda:0")
    qd, kd, vd, gd = (t.to(dev) for t in (q, k, v, d_out))
    first = [torch.full_like(qd, float("nan")) for _ in range(3)]
    clear.clear_attn_bwd_f32(qd, kd, vd, gd, *first, gh, gw, T, r, scale)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    # the second stream gets other inputs, so a mix-up of the shared statistics would show
    q2 = (qd * 1.5).contiguous()
    outs = [[torch.full_like(qd, float("nan")) for _ in range(3)] for _ in range(2)]
    for rep in range(3):
        for s, (qq, o) in zip(streams, ((qd, outs[0]), (q2, outs[1]))):
            with torch.cuda.stream(s):
                clear.clear_attn_bwd_f32(qq, kd, vd, gd, *o, gh, gw, T, r, scale, stream=s)
    torch.cuda.synchronize()
    for a, b in zip(first, outs[0]):
        assert torch.equal(a, b)
    want = oracle_bwd.attn_bwd(q * 1.5, k, v, d_out, gh, gw, T, r, scale)
    for got, ref in zip(outs[1], want):
        assert np.abs(got.cpu().double().numpy() - ref).max() <= BWD_ATOL
    clear.clear_cache_clear()


@pytest.mark.parametrize("gh,gw,T,r,d", [(16, 24, 20, 4.0, 128), (13, 19, 7, 2.5, 64), (24, 40, 130, 8.0, 128)])
def test_bf16_backward_matches_the_oracle(gh, gw, T, r, d):
    """bf16 tensors in and out, fp32 arithmetic: the error is the rounding of each gradient to bf16 (half a unit
    in the last of 8 significant bits) on top of the fp32 kernel's."""
    q, k, v = workloads.make_custom(1, 2, gh, gw, T, d, dtype="bf16", seed=gh + gw)
    g = torch.Generator(device="cpu").manual_seed(gh * gw)
    d_out = torch.randn(q.shape, generator=g, dtype=torch.float32).to(torch.bfloat16)
    scale = 1 / math.sqrt(d)
    want = oracle_bwd.attn_bwd(q, k, v, d_out, gh, gw, T, r, scale)
    dev = torch.device("cuda:0")
    qd, kd, vd, gd = (t.to(dev) for t in (q, k, v, d_out))
    dq, dk, dv = (torch.full_like(qd, float("nan")) for _ in range(3))
    clear.clear_attn_bwd_bf16(qd, kd, vd, gd, dq, dk, dv, gh, gw, T, r, scale)
    torch.cuda.synchronize()
    for name, got, ref in (("dq", dq, want[0]), ("dk", dk, want[1]), ("dv", dv, want[2])):
        err = np.abs(got.cpu().double().numpy() - ref)
        assert np.isfinite(err).all(), f"{name}: non-finite"
        assert (err <= 2.0 ** -8 * np.abs(ref) + BWD_ATOL).all(), f"{name}: max {err.max():.3e}"
    clear.clear_cache_clear()


# ----------------------------------------------------------------------------------------------
# tensor-core backward (bf16)
# ----------------------------------------------------------------------------------------------
def _tc_bound(ref):
    """P and dS enter the MMAs rounded to bf16 and every gradient is stored as bf16: errors of a few 1e-3 of the
    tensor's largest gradient were observed; the bound is 1e-2 of it."""
    return 1e-2 * np.abs(ref).max()


@pytest.mark.parametrize("gh,gw,T,r,d", [
    (16, 16, 16, 4.0, 64),       # the tiny configuration's shape
    (13, 19, 7, 2.5, 128),       # ragged patches, non-integer radius
    (24, 40, 130, 8.0, 128),     # two text tiles, the second with two rows
    (20, 50, 3, 100.0, 64),      # radius beyond the diagonal: full attention
    (33, 35, 0, 5.5, 128),       # no text
    (8, 16, 300, 3.0, 128),      # more text than image
    (1, 70, 2, 3.0, 64),         # single-row grid
])
def test_tensor_core_backward_matches_the_oracle(gh, gw, T, r, d):
    q, k, v = workloads.make_custom(1, 2, gh, gw, T, d, dtype="bf16", seed=gh + gw)
    g = torch.Generator(device="cpu").manual_seed(gh * gw)
    d_out = torch.randn(q.shape, generator=g, dtype=torch.float32).to(torch.bfloat16)
    scale = 1 / math.sqrt(d)
    want = oracle_bwd.attn_bwd(q, k, v, d_out, gh, gw, T, r, scale)
    dev = torch.device("cuda:0")
    qd, kd, vd, gd = (t.to(dev) for t in (q, k, v, d_out))
    outs = [torch.full_like(qd, float("nan")) for _ in range(3)]
    again = [torch.full_like(qd, float("nan")) for _ in range(3)]
    clear.clear_attn_bwd_bf16_tc(qd, kd, vd, gd, *outs, gh, gw, T, r, scale)
    clear.clear_attn_bwd_bf16_tc(qd, kd, vd, gd, *again, gh, gw, T, r, scale)
    torch.cuda.synchronize()
    clear.clear_cache_check()
    for name, got, rep, ref in zip(("dq", "dk", "dv"), outs, again, want):
        gn = got.cpu().double().numpy()
        assert np.isfinite(gn).all(), f"{name}: non-finite"
        assert np.abs(gn - ref).max() <= _tc_bound(ref), f"{name}: max {np.abs(gn - ref).max():.3e}"
        assert torch.equal(got, rep), f"{name}: not repeatable"
    clear.clear_cache_clear()


@pytest.mark.parametrize("name,heads", [("c1_1024px_r8", 2), ("c2_2048px_r16", 1)])
def test_tensor_core_backward_at_workload_sizes(name, heads):
    """Whole tensors against the oracle at the 1024px and 2048px shapes (fewer heads: the oracle is a CPU loop)."""
    w = workloads.WORKLOADS[name]
    q, k, v = workloads.make_inputs(w, heads=heads)
    g = torch.Generator(device="cpu").manual_seed(3)
    d_out = torch.randn(q.shape, generator=g, dtype=torch.float32).to(torch.bfloat16)
    want = oracle_bwd.attn_bwd(q, k, v, d_out, w.grid_h, w.grid_w, w.n_text, w.radius, w.scale)
    dev = torch.device("cuda:0")
    qd, kd, vd, gd = (t.to(dev) for t in (q, k, v, d_out))
    outs = [torch.full_like(qd, float("nan")) for _ in range(3)]
    clear.clear_attn_bwd_bf16_tc(qd, kd, vd, gd, *outs, w.grid_h, w.grid_w, w.n_text, w.radius, w.scale)
    torch.cuda.synchronize()
    clear.clear_cache_check()
    for nm, got, ref in zip(("dq", "dk", "dv"), outs, want):
        gn = got.cpu().double().numpy()
        assert np.isfinite(gn).all(), f"{nm}: non-finite"
        err = np.abs(gn - ref)
        assert err.max() <= _tc_bound(ref), f"{nm}: max {err.max():.3e} of {np.abs(ref).max():.3e}"
        assert err.mean() <= 1e-3 * np.abs(ref).max(), f"{nm}: mean {err.mean():.3e}"
    clear.clear_cache_clear()


@pytest.mark.parametrize("gh,gw,T,r,d,cap", [
    (4, 16, 0, 2.0, 64, None),       # one key patch, whose second half lies past the last row
    (8, 16, 40, 3.0, 128, None),     # two: the ring never reaches the stages that hold the stationary tiles
    (24, 16, 64, 30.0, 128, None),   # four: one half more than the ring of the query role has stages
    (21, 33, 129, 9.0, 128, "0"),    # no mask table: every masked patch from the half widths
    (21, 33, 129, 9.0, 64, "2"),     # a table that runs out
    (64, 72, 130, 2.0, 128, None),   # few heads: statistics in a launch of their own, 38 key tiles of a text tile in 3 parts
    (48, 50, 300, 3.0, 64, None),    # three text tiles of 22 key tiles in 2 parts
])
def test_tensor_core_backward_edges(gh, gw, T, r, d, cap, monkeypatch):
    """Ring lengths, halves outside the grid and table-free masks; the outputs start 16 but not 32 bytes off an aligned
    buffer and nothing outside them may change (bound as above)."""
    if cap is not None:
        monkeypatch.setenv("CLEAR_MAX_MASK_ENTRIES", cap)
    clear.clear_cache_clear()
    q, k, v = workloads.make_custom(1, 2, gh, gw, T, d, dtype="bf16", seed=gh + gw + d)
    g = torch.Generator(device="cpu").manual_seed(gh * gw)
    d_out = torch.randn(q.shape, generator=g, dtype=torch.float32).to(torch.bfloat16)
    scale = 1 / math.sqrt(d)
    want = oracle_bwd.attn_bwd(q, k, v, d_out, gh, gw, T, r, scale)
    dev = torch.device("cuda:0")
    n, pad = q.numel(), 8
    bufs = [torch.full((n + 2 * pad,), 7.0, dtype=torch.bfloat16, device=dev) for _ in range(3)]
    outs = [b[pad:pad + n].view(q.shape) for b in bufs]
    clear.clear_attn_bwd_bf16_tc(*(t.to(dev) for t in (q, k, v, d_out)), *outs, gh, gw, T, r, scale)
    torch.cuda.synchronize()
    clear.clear_cache_check()
    for name, buf, got, ref in zip(("dq", "dk", "dv"), bufs, outs, want):
        err = np.abs(got.cpu().double().numpy() - ref)
        assert err.max() <= _tc_bound(ref), f"{name}: max {err.max():.3e}"
        assert (buf[:pad] == 7.0).all() and (buf[pad + n:] == 7.0).all(), f"{name}: guard band"
    clear.clear_cache_clear()


@pytest.mark.parametrize("gh,gw,T,r,d", [(24, 40, 130, 8.0, 128), (13, 19, 7, 4.0, 64)])
def test_tensor_core_backward_keeps_the_centred_gradients(gh, gw, T, r, d):
    """Values with a large common part: every dP of a row has that part, and dP - delta takes it away, so delta has to be
    as good as fp32 sums make it.  What rounds then are dS and the stored gradient, each to 8 bits (2^-8 / sqrt(3) of a
    value at the start of a binade, 0.72 of that on average): 1.6e-3 twice, 2.3e-3 of the 2-norm together, and the bound
    is 2^-8.  A delta that carries the rounding of P to bf16 leaves 1.0e-2 to 1.4e-2."""
    q, k, v = workloads.make_custom(1, 2, gh, gw, T, d, dtype="bf16", seed=gh + gw)
    v = (v.float() * 0.25 + 16.0).to(torch.bfloat16)
    g = torch.Generator(device="cpu").manual_seed(gh * gw)
    d_out = torch.randn(q.shape, generator=g, dtype=torch.float32).to(torch.bfloat16)
    scale = 1 / math.sqrt(d)
    want = oracle_bwd.attn_bwd(q, k, v, d_out, gh, gw, T, r, scale)
    dev = torch.device("cuda:0")
    outs = [torch.full_like(q, float("nan"), device=dev) for _ in range(3)]
    clear.clear_attn_bwd_bf16_tc(*(t.to(dev) for t in (q, k, v, d_out)), *outs, gh, gw, T, r, scale)
    torch.cuda.synchronize()
    clear.clear_cache_check()
    for name, got, ref in zip(("dq", "dk", "dv"), outs, want):
        err = np.linalg.norm(got.cpu().double().numpy() - ref) / np.linalg.norm(ref)
        assert err <= 2.0 ** -8, f"{name}: {err:.3e}"
    clear.clear_cache_clear()


@pytest.mark.parametrize("gh,gw,T,r,d", [(24, 40, 130, 8.0, 128), (64, 72, 130, 2.0, 64)], ids=["sweeps", "launches"])
def test_a_backward_call_that_finds_the_status_word_raised_writes_nothing(gh, gw, T, r, d, monkeypatch):
    """The word is preset when the plan is made (no wait is made to expire): every block of every role leaves, the gradients
    stay untouched, the check reports it, and the call after the check runs."""
    q, k, v = workloads.make_custom(1, 2, gh, gw, T, d, dtype="bf16", seed=3)
    g = torch.Generator(device="cpu").manual_seed(4)
    d_out = torch.randn(q.shape, generator=g, dtype=torch.float32).to(torch.bfloat16)
    scale = 1 / math.sqrt(d)
    dev = torch.device("cuda:0")
    args = [t.to(dev) for t in (q, k, v, d_out)]
    outs = [torch.full_like(args[0], 7.0) for _ in range(3)]
    clear.clear_cache_clear()
    monkeypatch.setenv("CLEAR_TEST_PRESET_STATUS", "77")
    clear.clear_attn_bwd_bf16_tc(*args, *outs, gh, gw, T, r, scale)
    monkeypatch.delenv("CLEAR_TEST_PRESET_STATUS")
    torch.cuda.synchronize()
    for name, got in zip(("dq", "dk", "dv"), outs):
        assert (got == 7.0).all(), f"{name} was written"
    with pytest.raises(clear.ClearError) as e:
        clear.clear_cache_check()
    assert e.value.status == clear.ERR_DEVICE_TIMEOUT and clear.last_device_status() == 77
    clear.clear_attn_bwd_bf16_tc(*args, *outs, gh, gw, T, r, scale)
    torch.cuda.synchronize()
    clear.clear_cache_check()
    want = oracle_bwd.attn_bwd(q, k, v, d_out, gh, gw, T, r, scale)
    for name, got, ref in zip(("dq", "dk", "dv"), outs, want):
        err = np.abs(got.cpu().double().numpy() - ref)
        assert err.max() <= _tc_bound(ref), f"{name}: max {err.max():.3e}"
    clear.clear_cache_clear()


@pytest.mark.parametrize("B,H,gh,gw,T,r,d", [(1, 2, 13, 19, 7, 2.5, 64), (2, 1, 20, 50, 130, 4.0, 128), (1, 2, 64, 70, 131, 2.0, 64)])
def test_tensor_core_backward_keeps_heads_apart(B, H, gh, gw, T, r, d):
    """NaN all over the second (batch, head), the first one's last tiles ragged: the first one's gradients are the ones it has
    beside any other neighbour, bit for bit."""
    q, k, v = workloads.make_custom(B, H, gh, gw, T, d, dtype="bf16", seed=gh + gw)
    g = torch.Generator(device="cpu").manual_seed(gh * gw)
    args = [q, k, v, torch.randn(q.shape, generator=g, dtype=torch.float32).to(torch.bfloat16)]
    args = [t.to("cuda:0") for t in args]
    grads = []
    for rep in range(2):
        outs = [torch.zeros_like(args[0]) for _ in range(3)]
        clear.clear_attn_bwd_bf16_tc(*args, *outs, gh, gw, T, r, 1 / math.sqrt(d))
        grads.append([o.view(B * H, -1)[0].clone() for o in outs])
        for t in args:
            t.view(B * H, -1)[1] = float("nan")
    torch.cuda.synchronize()
    clear.clear_cache_check()
    for name, want, got in zip(("dq", "dk", "dv"), *grads):
        assert torch.isfinite(want).all() and torch.equal(want, got), name
    clear.clear_cache_clear()


def test_tensor_core_backward_argument_errors():
    dev = torch.device("cuda:0")
    x = torch.zeros(1, 1, 272, 64, device=dev, dtype=torch.bfloat16)
    p = x.data_ptr()
    lib = clear.load()
    assert lib.clear_attn_bwd_bf16_tc(p, p, p, p, p, p, p, 1, 1, 16, 16, 16, 96, 4.0, 0.125, None) == clear.ERR_UNSUPPORTED
    assert lib.clear_attn_bwd_bf16_tc(p, p, p, p, p, p, p, 1, 1, 16, 16, 16, 64, 4.0, 0.0, None) == clear.ERR_UNSUPPORTED
    assert lib.clear_attn_bwd_bf16_tc(p, p, p, p, p, p, p, 1, 1, 16, 16, 16, 64, 4.0, float("nan"), None) == clear.ERR_INVALID_ARG
    assert lib.clear_attn_bwd_bf16_tc(p, p, p, None, p, p, p, 1, 1, 16, 16, 16, 64, 4.0, 0.125, None) == clear.ERR_INVALID_ARG
    assert lib.clear_attn_bwd_bf16_tc(p, p, p, p, p, p + 4, p, 1, 1, 16, 16, 16, 64, 4.0, 0.125, None) == clear.ERR_MISALIGNED
