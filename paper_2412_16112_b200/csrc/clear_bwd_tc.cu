// Backward pass of the CLEAR attention operator on the sm_100a tensor cores (bf16 tensors, fp32 accumulation): dQ, dK,
// dV for an upstream gradient dO of  O = softmax(scale Q K^T + log M) V  (Eq. 1 under the mask of Eq. 3), the step
// through which the distillation losses of Sec. 3.3 (Eq. 4-6) reach the attention parameters.
//
// One kernel, three roles, launched one after the other; a CTA runs one work item of the forward tile schedule: a STATIONARY
// tile of 128 tokens (an 8 x 16 patch of the grid, or 128 text tokens) against the list of 128-token tiles the schedule gives
// it.  Eq. 3's mask is symmetric, so the list of key tiles a query tile sees is also the list of query tiles that see it as
// keys.
//   statistics  stationary Q_i, dO_i; streamed K_j, V_j.  S = Q K^T, dP = dO V^T; per query m' = maximum + log2(row sum), in
//               log2 units with the scale included, so that P = 2^(c S - m') is normalised, and delta = sum_j P dP, in fp32
//               from the unrounded P.  (dO . O from the forward kernel comes with the rounding of its P to bf16: where the dP
//               of a row have a common part, which dP - delta takes away, dQ and dK came out up to six times worse.)
//   query role  the same tiles: dS = P (dP - delta) as bf16 over S; dQ += dS K (dS the tensor-memory operand, K read MN-major
//               from the same shared-memory tile).
//   key role    stationary K_j, V_j; streamed Q_i, dO_i with the statistics of the queries i.  S^T = K Q^T,
//               dP^T = V dO^T; P^T and dS^T as bf16 over them; dV += P^T dO, dK += dS^T Q.
// The statistics are a first sweep of the query role over its list, unless a text tile, which sees every token, has more than
// an even share of all tiles over the SMs (few heads): then they are a launch of their own, in which the lists of the text
// tiles are cut over up to kStatParts CTAs, the last of which merges, and the other two roles run side by side behind it.
// 24 heads: 1024 px, radius 8 424 us a call in sweeps (433 in launches), 2048 px, radius 16 2288 (2332); two heads at
// 128 x 128, radius 8: 470 in sweeps, 266 in launches.
// A streamed tile is taken in two halves of 64 tokens, each with a buffer of its own in tensor memory (T1 | T2, 64 columns
// each), so the products of the next half run while the elementwise step of this one does; the accumulations of a half
// go behind them on the same pipe.  The order on the pipe is T(0), T(1), ACC(0), T(2), ACC(1), ...: a half's products
// overwrite P / dS of the half two before it only after its accumulations have read them.
// What bounds it: the MMAs, and at short lists the start and end of a block, which nothing covers (one block fills an SM:
// all 512 tensor-memory columns and 227 KB).  With both operands in shared memory, 64 columns cost 48 clocks per 16
// channels instead of 32, so the key role's tile takes 1536 clocks of products and 1024 of accumulations; measured 2900 a
// tile.  The query role has 128 tensor-memory columns to spare and keeps its stationary operands there: 1024 + 512,
// measured 2000.  The elementwise step (16 warps, 32 columns a thread) takes 700 (query) or 830 (key role) a half.
// Around the list go 4500 clocks from the block's start to its first products and 3000 behind its last ones.
// A step of the statistics sweep takes 2200 clocks a tile (1024 of products, 1024 of exponentials).
// 1024 px, radius 8, 24 heads of 128: 424 us a call; with P and dS of whole tiles in turn with the MMAs it was 873.
//   warp 0: TMA loads; warp 1: every MMA; warp 2 (key role): statistics of the streamed tiles; warps 4..19: rows.
// Every output element has one writer and a fixed order of summation.  Every wait is bounded: on expiry the CTA raises the
// plan's status word and leaves.
#include <cuda.h>
#include <cuda_bf16.h>

#include <cstring>

#include "clear_internal.hpp"
#include "ptx.cuh"

namespace clear {
namespace {

constexpr int kRowWarps = 16;
constexpr int kBwdThreads = 128 + 32 * kRowWarps;
constexpr uint32_t kBwdTmemCols = 512;   // two buffers of T1 | T2 (64 columns each), ACC1, ACC2 (128 each)
// Ring of streamed tokens: a stage holds a half (64 tokens) of both tensors of the pair and is given back after the half's
// accumulation.  With a tile of one tensor a stage (the same 160 KB) the next pair's second tile could only be asked for
// when the tile before had been used up, and came about 800 clocks late on every tile.
constexpr uint32_t kKeyStages = 5, kQueryStages = 7;   // (the query role keeps its stationary tiles in tensor memory)
constexpr uint32_t kColStages = 2;       // key role: statistics of streamed tiles
constexpr uint32_t kBwdSpinLimit = 1u << 22;
constexpr uint32_t kBwdWaitUs = 2000000;

struct BwdParams {
    const clear_work_item_t *items;
    const clear_kv_tile_t *tiles;
    const uint32_t *mask_table;
    const int32_t *half_width;
    int n_half_width;
    int grid_h, grid_w, n_text;
    int n_items, n_first, n_bh;  // the first n_first items (the longest) of every head come before all others
    long long n_tokens;
    float scale, scale_log2;   // scale, scale * log2(e)
    float2 *stats;             // [bh][token]: m', delta
    // statistics of text tiles whose lists are cut: [bh][tile][part][128] maximum, row sum, sum of p dP; finished parts [bh][tile]
    float4 *parts;
    int *part_count;
    int n_parts, n_part_slots;
    int key_waits;             // key role: the launch before it leaves the statistics
    int *status;
};
// Views of a tensor: whole tiles (patches of the image part, runs of text tokens) and half ones (patches, runs of tokens).
struct BwdViews {
    CUtensorMap img, txt, half_img, half_lin;
};
struct BwdOut {
    CUtensorMap img, txt;
};
struct BwdMaps {
    BwdViews a[2], b[2];  // stationary and streamed tensors
    BwdOut o[2];          // query role: dq, -; key role: dv, dk
};

struct BwdCtrl {
    uint64_t a_full, b_full[kQueryStages], b_empty[kQueryStages], t_full[2], p_ready[2], acc_done, col_full[kColStages],
        col_empty[kColStages], a_moved, out_ready, drain;
    alignas(16) float4 col[kColStages][64];   // key role: -m', -m', -delta, -delta of two columns of the streamed tile
    uint32_t tmem_base;
    int abort_flag, merge;
    int skip;   // 1: leave at once; 2: leave, with the first copies under way
};

__device__ __noinline__ uint32_t bwd_tick(uint32_t t0, volatile int *abort_flag, int *status, int code)
{
    const uint32_t now = (uint32_t)(ptx::globaltimer_ns() >> 10) | 1u;  // about microseconds, never 0
    if (t0 == 0) t0 = now;
    if (*abort_flag) return 0;
    if (now - t0 <= kBwdWaitUs) return t0;
    *abort_flag = 1;
    atomicCAS(status, 0, code);
    return 0;
}
// Bounded wait; false once the block has given up.
__device__ __forceinline__ bool bwd_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *status, int code)
{
    if (ptx::mbar_try_wait(bar, parity)) return true;
    uint32_t t0 = 0;
#pragma unroll 1
    for (uint32_t n = 1; !ptx::mbar_try_wait_hint(bar, parity, 20000); ++n)
        if ((n & 127u) == 0u && (t0 = bwd_tick(t0, abort_flag, status, code)) == 0u) return false;
    return true;
}
__device__ __noinline__ void bwd_drain(uint32_t bar, uint32_t parity)
{
#pragma unroll 1
    for (uint32_t it = 0; it < kBwdSpinLimit; ++it) {
        if (ptx::mbar_try_wait(bar, parity)) return;
        if (it > 64) __nanosleep(256);
    }
}

enum Role { kStats, kQuery, kStatsQuery, kKey };   // kStatsQuery: both sweeps in one CTA
// Running statistics of a row: maximum (log2 units), row sum and sum of p dP relative to it.
struct RowStat {
    float m, l, d;
    __device__ __forceinline__ void start()
    {
        m = -INFINITY;
        l = d = 0.f;
    }
    __device__ __forceinline__ void add(float m2, float l2, float d2)
    {
        const float m_new = fmaxf(m, m2), m_ref = m_new == -INFINITY ? 0.f : m_new;
        const float a = ptx::ex2(m - m_ref), b = ptx::ex2(m2 - m_ref);   // -inf: 0
        l = fmaf(b, l2, a * l);
        d = fmaf(b, d2, a * d);
        m = m_new;
    }
    // l >= 1 for every row that exists: it sees itself or the text (a NaN stays one)
    __device__ __forceinline__ float2 result() const { return l == 0.f ? make_float2(0.f, 0.f) : make_float2(m + log2f(l), d / l); }
};

template <int D, Role ROLE>
__global__ void __launch_bounds__(kBwdThreads, 1)
clear_bwd_tc_kernel(const __grid_constant__ BwdMaps maps, const __grid_constant__ BwdParams prm)
{
    constexpr bool KEY_ROLE = ROLE == kKey, STATS = ROLE == kStats || ROLE == kStatsQuery, GRAD = ROLE != kStats;
    constexpr int kHalves = D / 64;                 // 64-channel (128-byte) column blocks of a tile
    constexpr uint32_t kHalfBytes = 128 * 128;      // 128 rows x 128 B
    constexpr uint32_t kTileBytes = kHalves * kHalfBytes;   // also a stage: two tensors, 64 rows
    constexpr uint32_t kSubBytes = kTileBytes / 2, kSubHalfBytes = kHalfBytes / 2;
    constexpr uint32_t kIdescT = ptx::idesc_bf16(64, false);    // [128 rows] x [64 columns], both operands K-major
    constexpr uint32_t kIdescAcc = ptx::idesc_bf16(D, true);    // [128 rows] x [D channels], B read MN-major
    constexpr uint32_t kDescHi = ptx::smem_desc_hi_sw128(1024);
    constexpr uint32_t kStages = KEY_ROLE ? kKeyStages : kQueryStages, kFixed = KEY_ROLE ? 2 : 0;
    constexpr uint32_t kAStage = KEY_ROLE ? 0 : kStages - 2;   // where the stationary tiles land; the query role's ring gets the place back

    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t s0 = ptx::smem_u32(smem_raw), sA = s0 + kAStage * kTileBytes, sB = s0 + kFixed * kTileBytes;
    BwdCtrl *ctrl = reinterpret_cast<BwdCtrl *>(smem_raw + (kFixed + kStages) * kTileBytes);
    volatile int *abort_flag = &ctrl->abort_flag;
    const uint32_t b_a = ptx::smem_u32(&ctrl->a_full), b_full0 = ptx::smem_u32(&ctrl->b_full[0]),
                   b_empty0 = ptx::smem_u32(&ctrl->b_empty[0]), b_acc = ptx::smem_u32(&ctrl->acc_done),
                   b_moved = ptx::smem_u32(&ctrl->a_moved);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (STATS) ptx::grid_launch_dependents();
    int bh, item_id;
    if ((int)blockIdx.x < prm.n_first * prm.n_bh) {
        item_id = (int)blockIdx.x / prm.n_bh;
        bh = (int)blockIdx.x - item_id * prm.n_bh;
    } else {
        const int rest = (int)blockIdx.x - prm.n_first * prm.n_bh, per = prm.n_items - prm.n_first;
        bh = rest / per;
        item_id = prm.n_first + rest - bh * per;
    }
    const clear_work_item_t item = prm.items[item_id];
    const clear_kv_tile_t *tiles = prm.tiles + item.tile_begin;
    const int n_tiles = item.tile_count, n_iters = ROLE == kStatsQuery ? 2 * n_tiles : n_tiles;   // steps of all sweeps
    const bool is_text = item.kind == 1;

    // row of the stationary tile that a thread of the row warps works on
    const int r = (warp & 3) * 32 + lane;
    const int q_y = item.qy + (r >> 4), q_x = item.qx + (r & 15);
    const bool row_valid = is_text ? r < item.n_rows : q_y < prm.grid_h && q_x < prm.grid_w;
    const long long row_token = is_text ? (long long)item.qx + r : (long long)prm.n_text + (long long)q_y * prm.grid_w + q_x;
    // one streamed half into a stage (a half that lies past the last row or token reads as zero)
    auto load_half = [&](const clear_kv_tile_t &t, int h, uint32_t stage) {
        const bool linear = (t.flags & CLEAR_TILE_LINEAR) != 0;
        const uint32_t bar = b_full0 + 8 * stage;
        ptx::mbar_expect_tx(bar, kTileBytes);
#pragma unroll 1
        for (int j = 0; j < 2; ++j)
            ptx::tma_load_5d(sB + stage * kTileBytes + j * kSubBytes, linear ? &maps.b[j].half_lin : &maps.b[j].half_img, bar, 0,
                             linear ? t.x + 64 * h : t.x, linear ? 0 : t.y + 4 * h, 0, bh);
    };
    // once any CTA of this plan has given up, the rest of the grid leaves at once; a window that is not 1024-byte
    // aligned (never expected) cannot hold swizzled tiles
    if (tid == 0) {
        int skip = *reinterpret_cast<volatile int *>(prm.status) != 0 ? 1 : 0;
        if ((s0 & 1023u) != 0u) {
            atomicCAS(prm.status, 0, 100);
            skip = 1;
        }
        ctrl->skip = skip;
        ctrl->abort_flag = 0;
        ptx::mbar_init(b_a, 1);
        ptx::mbar_init(b_moved, kRowWarps);
        for (uint32_t i = 0; i < kStages; ++i) {
            ptx::mbar_init(b_full0 + 8 * i, 1);
            ptx::mbar_init(b_empty0 + 8 * i, 1);
        }
        for (int i = 0; i < 2; ++i) {
            ptx::mbar_init(ptx::smem_u32(&ctrl->t_full[i]), 1);
            ptx::mbar_init(ptx::smem_u32(&ctrl->p_ready[i]), kRowWarps / 2);
        }
        for (uint32_t i = 0; i < kColStages; ++i) {
            ptx::mbar_init(ptx::smem_u32(&ctrl->col_full[i]), 1);
            ptx::mbar_init(ptx::smem_u32(&ctrl->col_empty[i]), kRowWarps);
        }
        ptx::mbar_init(b_acc, 1);
        ptx::mbar_init(ptx::smem_u32(&ctrl->out_ready), kRowWarps);
        ptx::mbar_init(ptx::smem_u32(&ctrl->drain), 1);
        ptx::fence_mbar_init();
        if (skip == 0) {
            // the first copies leave before the block has met: one CTA fills an SM, so nothing else covers their way
            ptx::mbar_expect_tx(b_a, 2 * kTileBytes);
#pragma unroll 1
            for (int i = 0; i < 2; ++i)
                ptx::tma_load_5d(sA + i * kTileBytes, is_text ? &maps.a[i].txt : &maps.a[i].img, b_a, 0, item.qx, is_text ? 0 : item.qy, 0, bh);
            const clear_kv_tile_t t = tiles[0];
            load_half(t, 0, 0);
            load_half(t, 1, 1);
        }
    }
    if (ROLE == kQuery) {
        // Up to here beside the last CTAs of the statistics launch.  The key role may follow from here on: once every CTA of
        // this role has come this far, the statistics of all rows are there.
        ptx::grid_wait();
        ptx::grid_launch_dependents();
        if (tid == 0 && ctrl->skip == 0 && *reinterpret_cast<volatile int *>(prm.status) != 0) ctrl->skip = 2;
    }
    if (warp == 1) {
        ptx::tmem_alloc(ptx::smem_u32(&ctrl->tmem_base), kBwdTmemCols);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = ctrl->tmem_base, tmem_A1 = tmem + 256, tmem_A2 = tmem + 384;  // query role: q | dO in A2's place
    uint32_t n_loads = 2;   // halves that the loader has asked for
    const int skip = ctrl->skip;
    if (skip == 1) {
        if (warp == 1) ptx::tmem_dealloc(tmem, kBwdTmemCols);
        if (KEY_ROLE) ptx::grid_wait();
        return;
    }

    if (skip == 2) {
        // the statistics launch gave up: only the copies under way are left to wait for
    } else if (warp < 4) {
        if (warp == 0 && lane == 0) {
            // ================= loader ===========================================================================
            uint32_t stage = 2, par = 0;
            bool ok = true;
            int next = n_tiles > 1 ? 1 : 0;   // the list is walked once a sweep
            clear_kv_tile_t t = tiles[next];
#pragma unroll 1
            for (int it = 1; it < n_iters && ok; ++it) {
                if (++next >= n_tiles) next = 0;
                const clear_kv_tile_t t_next = tiles[next];
#pragma unroll 1
                for (int h = 0; h < 2; ++h) {
                    if (!KEY_ROLE && n_loads == kAStage) ok = bwd_wait(b_moved, 0, abort_flag, prm.status, 9);
                    ok = ok && bwd_wait(b_empty0 + 8 * stage, par ^ 1u, abort_flag, prm.status, 1);
                    if (!ok) break;
                    load_half(t, h, stage);
                    ++n_loads;
                    if (++stage == kStages) {
                        stage = 0;
                        par ^= 1u;
                    }
                }
                t = t_next;
            }
        } else if (warp == 1) {
            // ================= every MMA, all from one lane ==========================================================
            // The pipe takes about two MMAs ahead, so what this lane does between an accumulation and the next products
            // is time that the pipe stands idle, and beside 16 busy row warps every instruction of it is slow. So nothing
            // stands there: the loop goes by tiles with both halves written out, one lane walks it without votes, and the
            // waits sit behind products that are still running.
            if (ptx::elect_one()) {
                bool ok = bwd_wait(KEY_ROLE ? b_a : b_moved, 0, abort_flag, prm.status, 2);
                const uint32_t a_lo0 = ptx::smem_desc_lo(sA, 16), bk_lo0 = ptx::smem_desc_lo(sB, 16), bm_lo0 = ptx::smem_desc_lo(sB, kSubHalfBytes);
                constexpr uint32_t kTile16 = kTileBytes >> 4, kSub16 = kSubBytes >> 4;
                uint32_t next = 0, next_par = 0;
                // the next half of the streamed pair: its stage
                auto wait_half = [&]() -> uint32_t {
                    const uint32_t st = next;
                    ok = ok && bwd_wait(b_full0 + 8 * next, next_par, abort_flag, prm.status, 3);
                    if (++next == kStages) {
                        next = 0;
                        next_par ^= 1u;
                    }
                    return st;
                };
                // T1, T2 of a half: D / 16 MMAs of 16 channels each
                auto issue_t = [&](uint32_t st, int half, bool grad) {
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const uint32_t d = tmem + half * 128 + j * 64, a = a_lo0 + j * kTile16, b = bk_lo0 + st * kTile16 + j * kSub16;
                        if (!KEY_ROLE) {
                            const uint32_t a_tmem = tmem_A2 + j * (D / 2);
                            ptx::mma_ts_c<false>(d, a_tmem, ptx::make_desc(b, kDescHi), kIdescT);
#pragma unroll
                            for (int kk = 1; kk < D / 16; ++kk)
                                ptx::mma_ts_c<true>(d, a_tmem + 8 * kk, ptx::make_desc(b + (((kk >> 2) * kSubHalfBytes + (kk & 3) * 32) >> 4), kDescHi), kIdescT);
                            continue;
                        }
                        ptx::mma_ss_c<false>(d, ptx::make_desc(a, kDescHi), ptx::make_desc(b, kDescHi), kIdescT);
#pragma unroll
                        for (int kk = 1; kk < D / 16; ++kk) {
                            const uint32_t a16 = ((kk >> 2) * kHalfBytes + (kk & 3) * 32) >> 4, b16 = ((kk >> 2) * kSubHalfBytes + (kk & 3) * 32) >> 4;
                            ptx::mma_ss_c<true>(d, ptx::make_desc(a + a16, kDescHi), ptx::make_desc(b + b16, kDescHi), kIdescT);
                        }
                    }
                    ptx::tc_commit(ptx::smem_u32(&ctrl->t_full[half]));
                    if (!grad) ptx::tc_commit(b_empty0 + 8 * st);   // nothing else reads the half
                };
                auto is_grad = [&](int it) { return GRAD && (ROLE != kStatsQuery || it >= n_tiles); };
                // 4 MMAs over 16 streamed tokens each (16 rows of 128 bytes = 2048 bytes), B read MN-major; the bf16 columns
                // of the two row groups start at the groups' own fp32 columns
                auto issue_acc = [&](uint32_t st, int half, uint32_t before) {
                    const uint32_t p1 = tmem + half * 128, p2 = p1 + 64;
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        const uint32_t acc = kk > 0 ? 1u : before, col = (kk >> 1) * 32 + (kk & 1) * 8, off = st * kTile16 + kk * (2048 >> 4);
                        if (KEY_ROLE) {
                            ptx::mma_ts(tmem_A1, p1 + col, ptx::make_desc(bm_lo0 + kSub16 + off, kDescHi), kIdescAcc, acc);  // dV += P^T dO
                            ptx::mma_ts(tmem_A2, p2 + col, ptx::make_desc(bm_lo0 + off, kDescHi), kIdescAcc, acc);  // dK += dS^T Q
                        } else {
                            ptx::mma_ts(tmem_A1, p1 + col, ptx::make_desc(bm_lo0 + off, kDescHi), kIdescAcc, acc);  // dQ += dS K
                        }
                    }
                    ptx::tc_commit(b_empty0 + 8 * st);
                };
                const uint32_t b_p0 = ptx::smem_u32(&ctrl->p_ready[0]), b_p1 = ptx::smem_u32(&ctrl->p_ready[1]);
                uint32_t st0 = wait_half(), st1 = 0;
                if (ok) {
                    ptx::tc_fence_after();
                    issue_t(st0, 0, is_grad(0));
                    st1 = wait_half();
                }
#pragma unroll 1
                for (int it = 0; it < n_iters && ok; ++it) {
                    const uint32_t par = (uint32_t)it & 1u;
                    const bool more = it + 1 < n_iters, grad = is_grad(it);
                    ptx::tc_fence_after();
                    issue_t(st1, 1, grad);
                    const uint32_t st2 = more ? wait_half() : 0u;
                    // the rows have read T1, T2 of a half and put P / dS over them (statistics: only read them)
                    ok = ok && bwd_wait(b_p0, par, abort_flag, prm.status, 4);
                    if (!ok) break;
                    ptx::tc_fence_after();
                    if (grad) issue_acc(st0, 0, it > n_iters - n_tiles ? 1u : 0u);
                    if (more) issue_t(st2, 0, is_grad(it + 1));
                    const uint32_t st3 = more ? wait_half() : 0u;
                    ok = ok && bwd_wait(b_p1, par, abort_flag, prm.status, 4);
                    if (!ok) break;
                    ptx::tc_fence_after();
                    if (grad) issue_acc(st1, 1, 1u);
                    if (GRAD && !more) ptx::tc_commit(b_acc);
                    st0 = st2;
                    st1 = st3;
                }
                if (*abort_flag) {
                    // MMAs that were issued must retire before tensor memory is given back
                    ptx::tc_commit(ptx::smem_u32(&ctrl->drain));
                    bwd_drain(ptx::smem_u32(&ctrl->drain), 0);
                }
            }
        } else if (warp == 2 && KEY_ROLE) {
            // ================= statistics of the streamed tiles' columns, ahead of the row warps =====================
            // (zeros for a column that is none of the list's: P is 0 there, but P (dP - delta) is not if delta is another
            // token's NaN, of the next head or of the next grid row)
            const float2 *stats = prm.stats + (long long)bh * prm.n_tokens;
            bool ok = true;
            if (prm.key_waits) {
                // the query role leaves the statistics, and may still be at work; the rest of this CTA has started beside
                // its last ones.  If it has given up there are none, and the CTA leaves without a result.
                ptx::grid_wait();
                ok = *reinterpret_cast<volatile int *>(prm.status) == 0;
                if (!ok) *abort_flag = 1;
            }
#pragma unroll 1
            for (int i = 0; i < n_tiles && ok; ++i) {
                const uint32_t st = (uint32_t)i % kColStages, use = (uint32_t)i / kColStages;
                const clear_kv_tile_t t = tiles[i];
                float2 v[4];
                bool here[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int c = 32 * j + lane, y = t.y + (c >> 4), x = t.x + (c & 15);
                    const bool linear = (t.flags & CLEAR_TILE_LINEAR) != 0;
                    const long long tok = linear ? (long long)t.x + c : prm.n_text + (long long)y * prm.grid_w + x;
                    here[j] = linear ? c < t.n_valid : y < prm.grid_h && x < prm.grid_w;
                    v[j] = __ldcg(stats + (here[j] ? tok : 0));
                }
                ok = __all_sync(0xffffffffu, bwd_wait(ptx::smem_u32(&ctrl->col_empty[st]), (use & 1u) ^ 1u, abort_flag, prm.status, 5));
                if (!ok) break;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    float *dst = reinterpret_cast<float *>(&ctrl->col[st][16 * j + (lane >> 1)]) + (lane & 1);
                    dst[0] = here[j] ? -v[j].x : 0.f;
                    dst[2] = here[j] ? -v[j].y : 0.f;
                }
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&ctrl->col_full[st]));
            }
        }
        __syncwarp();
    } else {
        // ================= row warps: warp (g, quadrant); group g takes the halves h = g & 1 and of them the columns
        // [32 (g >> 1), +32); thread = row of the stationary tile =================
        const int g = (warp - 4) >> 2, half = g & 1, hc = g >> 1;
        const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t tmem_T1 = tmem + half * 128 + 32 * hc + lane_off, tmem_T2 = tmem_T1 + 64;
        const float c = prm.scale_log2;
        bool alive = true;
        if (!KEY_ROLE) {
            // The stationary rows go on to tensor memory, where an MMA of 64 columns takes 32 clocks instead of the 48 that
            // both operands need out of shared memory: group g moves 64 channels of q (g < 2) or of dO.  (Loaded straight
            // from global memory, a row a thread, they took 8000 clocks.)
            alive = __all_sync(0xffffffffu, bwd_wait(b_a, 0, abort_flag, prm.status, 10));
            if (alive) {
                if ((g & 1) * 64 < D) {
                    uint32_t w[32];
                    const uint8_t *src = smem_raw + (kAStage + (g >> 1)) * kTileBytes + (g & 1) * kHalfBytes + r * 128;
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const uint4 v = *reinterpret_cast<const uint4 *>(src + ((j ^ (r & 7)) << 4));
                        w[4 * j] = v.x;
                        w[4 * j + 1] = v.y;
                        w[4 * j + 2] = v.z;
                        w[4 * j + 3] = v.w;
                    }
                    ptx::tmem_st32(tmem_A2 + lane_off + (g >> 1) * (D / 2) + (g & 1) * 32, w);
                    ptx::tmem_wait_st();
                }
                ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(b_moved);
            }
        }
        // mask bits of this row for its 32 columns of a tile (bit j = column allowed; the mask is symmetric, so the row's
        // token plays the query whichever role the kernel runs in)
        auto mask_word = [&](const clear_kv_tile_t &t) -> uint32_t {
            if (!(t.flags & CLEAR_TILE_MASKED)) return 0xffffffffu;
            if (t.flags & CLEAR_TILE_LINEAR) {
                const int n = min(max(t.n_valid - 64 * half - 32 * hc, 0), 32);
                return n == 32 ? 0xffffffffu : ((1u << n) - 1u);
            }
            if (t.n_valid >= 0) return ptx::ldg_u32(prm.mask_table + ((size_t)t.n_valid * 128 + r) * 4 + 2 * half + hc);
            // no table entry (very large radius): Eq. 3 from the half widths, two grid rows a word
            uint32_t bits = 0u;
#pragma unroll 1
            for (int rr = 0; rr < 2; ++rr) {
                const int ky = t.y + 4 * half + 2 * hc + rr, ady = abs(ky - q_y);
                if (row_valid && ky < prm.grid_h && ady < prm.n_half_width) {
                    const int hw = __ldg(prm.half_width + ady);
                    const int lo = max(max(q_x - hw, 0), t.x), hi = min(min(q_x + hw, prm.grid_w - 1), t.x + 15);
                    if (lo <= hi) bits |= (((1u << (hi - lo + 1)) - 1u) << (lo - t.x)) << (16 * rr);
                }
            }
            return bits;
        };
        const uint32_t b_t = ptx::smem_u32(&ctrl->t_full[half]), b_p = ptx::smem_u32(&ctrl->p_ready[half]);
        const uint64_t c2 = ptx::pack2(c, c);
        // tile records two ahead, mask words one ahead
        clear_kv_tile_t t_next = tiles[min(1, n_tiles - 1)];
        uint32_t mw_next = mask_word(tiles[0]);
        auto next_mask = [&](int i) -> uint32_t {
            const uint32_t mw = mw_next;
            mw_next = mask_word(t_next);
            t_next = tiles[min(i + 2, n_tiles - 1)];
            return mw;
        };
        float2 row_stat = make_float2(0.f, 0.f);
        if constexpr (STATS) {
            // ---- online softmax over the thread's own columns: maximum (log2 units), row sum, sum of p dP ----
            float m = -INFINITY, l = 0.f, dl = 0.f;
#pragma unroll 1
            for (int i = 0; i < n_tiles && alive; ++i) {
                const uint32_t mw = next_mask(i);
                if (!__all_sync(0xffffffffu, bwd_wait(b_t, (uint32_t)i & 1u, abort_flag, prm.status, 12))) {
                    alive = false;
                    break;
                }
                ptx::tc_fence_after();
                uint32_t s[32], gg[32];
                ptx::tmem_ld32(tmem_T1, s);
                ptx::tmem_ld32(tmem_T2, gg);
                ptx::tmem_wait_ld();
                // nothing is written back: the next products may land as soon as these have been read
                ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(b_p);
                if (__any_sync(0xffffffffu, mw != 0xffffffffu)) {
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (!((mw >> j) & 1u)) s[j] = 0xff800000u;   // -inf
                }
                float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll
                for (int j = 0; j < 32; j += 2) {
                    mx[(j >> 1) & 1] = ptx::max3(mx[(j >> 1) & 1], __uint_as_float(s[j]), __uint_as_float(s[j + 1]));
                }
                const float m_new = fmaxf(m, fmaxf(mx[0], mx[1]) * c), m_ref = m_new == -INFINITY ? 0.f : m_new;
                const float alpha = ptx::ex2(m - m_ref);   // m = -inf: 0
                m = m_new;
                const uint64_t nm2 = ptx::pack2(-m_ref, -m_ref);
                uint64_t l2 = ptx::pack2(l * alpha, 0.f), d2 = ptx::pack2(dl * alpha, 0.f);
#pragma unroll
                for (int j = 0; j < 32; j += 2) {
                    float x0, x1;
                    ptx::unpack2(ptx::fma2(ptx::pack2(__uint_as_float(s[j]), __uint_as_float(s[j + 1])), c2, nm2), x0, x1);
                    const uint64_t p2 = ptx::pack2(ptx::ex2(x0), ptx::ex2(x1));
                    l2 = ptx::add2(l2, p2);
                    d2 = ptx::fma2(p2, ptx::pack2(__uint_as_float(gg[j]), __uint_as_float(gg[j + 1])), d2);
                }
                float a, b;
                ptx::unpack2(l2, a, b);
                l = a + b;
                ptx::unpack2(d2, a, b);
                dl = a + b;
            }
            t_next = tiles[min(1, n_tiles - 1)];
            mw_next = mask_word(tiles[0]);
            // the four threads of a row meet in tensor memory, in columns that the accumulation takes over afterwards (its
            // first MMA waits for rows that have passed the second barrier)
            ptx::tmem_st4(tmem_A1 + lane_off + 4 * g, __float_as_uint(m), __float_as_uint(l), __float_as_uint(dl), 0u);
            ptx::tmem_wait_st();
            ptx::tc_fence_before();
            ptx::named_barrier(1, 32 * kRowWarps);
            ptx::tc_fence_after();
            uint32_t part[16];
            ptx::tmem_ld16(tmem_A1 + lane_off, part);
            ptx::tmem_wait_ld();
            if constexpr (GRAD) {
                ptx::tc_fence_before();
                ptx::named_barrier(1, 32 * kRowWarps);
                ptx::tc_fence_after();
            }
            RowStat st;
            st.start();
#pragma unroll
            for (int u = 0; u < 4; ++u)
                st.add(__uint_as_float(part[4 * u]), __uint_as_float(part[4 * u + 1]), __uint_as_float(part[4 * u + 2]));
            if (g == 0) {
                if (item.partial_slot < 0) {
                    if (row_valid && alive) prm.stats[(long long)bh * prm.n_tokens + row_token] = st.result();
                } else {
                    // a part of a text tile's list: whichever CTA leaves the last part merges them, in their order
                    const int tile0 = item.partial_slot / prm.n_parts * prm.n_parts;
                    float4 *parts = prm.parts + ((long long)bh * prm.n_part_slots + tile0) * 128 + r;
                    __stcg(parts + (item.partial_slot - tile0) * 128, make_float4(st.m, st.l, st.d, 0.f));
                    __threadfence();
                    ptx::named_barrier(2, 128);   // (every warp of the group comes here, also one that has given up)
                    int *count = prm.part_count + bh * (prm.n_part_slots / prm.n_parts) + tile0 / prm.n_parts;
                    if (r == 0) ctrl->merge = *abort_flag == 0 && atomicAdd(count, 1) == prm.n_parts - 1 ? 1 : 0;
                    ptx::named_barrier(2, 128);
                    if (ctrl->merge != 0) {
                        __threadfence();
                        st.start();
                        for (int u = 0; u < prm.n_parts; ++u) {
                            const float4 x = __ldcg(parts + u * 128);
                            st.add(x.x, x.y, x.z);
                        }
                        if (row_valid) prm.stats[(long long)bh * prm.n_tokens + row_token] = st.result();
                        if (r == 0) *count = 0;   // for the next call
                    }
                }
            }
            row_stat = st.result();
        }
        if (ROLE == kQuery && row_valid) row_stat = __ldcg(prm.stats + (long long)bh * prm.n_tokens + row_token);
        const uint64_t row_nm = ptx::pack2(-row_stat.x, -row_stat.x), row_nd = ptx::pack2(-row_stat.y, -row_stat.y);
        const uint32_t it0 = ROLE == kStatsQuery ? (uint32_t)n_tiles : 0u;   // steps of the sweep before
        uint32_t col_st = 0, col_par = 0;
#pragma unroll 1
        for (int i = 0; i < n_tiles && alive && GRAD; ++i) {
            const uint32_t mw = next_mask(i);
            // warp-uniform outcome: the tcgen05.ld / st below need the whole warp
            bool got = true;
            if (KEY_ROLE) got = bwd_wait(ptx::smem_u32(&ctrl->col_full[col_st]), col_par, abort_flag, prm.status, 7);
            // kPass columns at a time.  The key role's statistics come out of shared memory, which the MMAs keep busy: 16
            // columns' worth are asked for together, the first ones before T is there, and with 32 columns at once there
            // would be no registers to hold them.
            constexpr int kPass = KEY_ROLE ? 16 : 32;
            uint64_t nm[KEY_ROLE ? kPass / 2 : 1], nd[KEY_ROLE ? kPass / 2 : 1];
            if (!KEY_ROLE) {
                nm[0] = row_nm;
                nd[0] = row_nd;
            }
            const uint32_t cols = ptx::smem_u32(&ctrl->col[col_st][32 * half + 16 * hc]);
            auto load_cols = [&](int pass) {
                if constexpr (KEY_ROLE) {
#pragma unroll
                    for (int j = 0; j < kPass / 2; ++j) ptx::lds_pairs(cols + (pass * kPass / 2 + j) * 16, nm[j], nd[j]);
                }
            };
            if (got) load_cols(0);
            got = got && bwd_wait(b_t, (it0 + (uint32_t)i) & 1u, abort_flag, prm.status, 6);
            if (!__all_sync(0xffffffffu, got)) {
                alive = false;
                break;
            }
            ptx::tc_fence_after();
#pragma unroll
            for (int pass = 0; pass < 32 / kPass; ++pass) {
                uint32_t s[kPass], gg[kPass], pk[kPass / 2], dk[kPass / 2];
                if (pass > 0) load_cols(pass);
                if constexpr (KEY_ROLE) {
                    ptx::tmem_ld16(tmem_T1 + pass * kPass, s);
                    ptx::tmem_ld16(tmem_T2 + pass * kPass, gg);
                } else {
                    ptx::tmem_ld32(tmem_T1, s);
                    ptx::tmem_ld32(tmem_T2, gg);
                }
                ptx::tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < kPass; j += 2) {
                    const int jc = KEY_ROLE ? j >> 1 : 0, bit = pass * kPass + j;
                    float x0, x1, p0, p1, d0, d1;
                    ptx::unpack2(ptx::fma2(ptx::pack2(__uint_as_float(s[j]), __uint_as_float(s[j + 1])), c2, nm[jc]), x0, x1);
                    p0 = ptx::ex2(((mw >> bit) & 1u) ? x0 : -INFINITY);
                    p1 = ptx::ex2(((mw >> (bit + 1)) & 1u) ? x1 : -INFINITY);
                    ptx::unpack2(ptx::mul2(ptx::pack2(p0, p1), ptx::add2(ptx::pack2(__uint_as_float(gg[j]), __uint_as_float(gg[j + 1])), nd[jc])), d0, d1);
                    if (KEY_ROLE) pk[j >> 1] = ptx::pack_bf16(p0, p1);
                    dk[j >> 1] = ptx::pack_bf16(d0, d1);
                }
                // a thread's bf16 columns sit at the start of its own fp32 columns, in cells that it has read by now
                if constexpr (KEY_ROLE) {
                    ptx::tmem_st8(tmem_T1 + pass * (kPass / 2), pk);
                    ptx::tmem_st8(tmem_T2 + pass * (kPass / 2), dk);
                } else {
                    ptx::tmem_st16(tmem_T1, dk);
                }
            }
            ptx::tmem_wait_st();
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                ptx::mbar_arrive(b_p);
                if (KEY_ROLE) ptx::mbar_arrive(ptx::smem_u32(&ctrl->col_empty[col_st]));
            }
            if (++col_st == kColStages) {
                col_st = 0;
                col_par ^= 1u;
            }
        }

        if constexpr (GRAD) {
        // ---- epilogue: after the last accumulation every group brings a quarter of the channels of its rows into shared
        // memory, which nothing reads any more, and a TMA store takes the tile from there (rows outside the tensor are
        // left out by its bounds).  Stored by the threads themselves, a row each, the key role's two tensors took
        // 3900 clocks. ----
        if (alive) alive = __all_sync(0xffffffffu, bwd_wait(b_acc, 0, abort_flag, prm.status, 8));
        if (alive) {
            ptx::tc_fence_after();
            auto stage_rows = [&](uint32_t tmem_acc, uint32_t tile, float factor) {
                uint8_t *dst = smem_raw + tile * kTileBytes + (D == 128 ? (g >> 1) * kHalfBytes : 0) + r * 128;
                constexpr int kChunks = D / 32;   // 16-byte chunks of a group
                const int first = g * kChunks & 7;
                uint32_t o[4 * kChunks * 2];
                if constexpr (D == 128)
                    ptx::tmem_ld32(tmem_acc + lane_off + g * (D / 4), o);
                else
                    ptx::tmem_ld16(tmem_acc + lane_off + g * (D / 4), o);
                ptx::tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < kChunks; ++j) {
                    uint32_t u[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        u[k] = ptx::pack_bf16(__uint_as_float(o[8 * j + 2 * k]) * factor, __uint_as_float(o[8 * j + 2 * k + 1]) * factor);
                    *reinterpret_cast<uint4 *>(dst + (((first + j) ^ (r & 7)) << 4)) = make_uint4(u[0], u[1], u[2], u[3]);
                }
            };
            stage_rows(tmem_A1, 0, KEY_ROLE ? 1.f : prm.scale);    // dV, or dQ
            if (KEY_ROLE) stage_rows(tmem_A2, 1, prm.scale);       // dK
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                ptx::mbar_arrive(ptx::smem_u32(&ctrl->out_ready));
                if (warp == 4 && bwd_wait(ptx::smem_u32(&ctrl->out_ready), 0, abort_flag, prm.status, 11)) {
                    ptx::fence_proxy_async_smem();
#pragma unroll 1
                    for (int i = 0; i < (KEY_ROLE ? 2 : 1); ++i)
                        ptx::tma_store_5d(is_text ? &maps.o[i].txt : &maps.o[i].img, s0 + i * kTileBytes, 0, item.qx, is_text ? 0 : item.qy, 0, bh);
                    ptx::bulk_commit_group();
                    ptx::bulk_wait_group0_read();   // the block may leave once its shared memory has been read
                }
            }
            __syncwarp();
        }
        }
    }

    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem, kBwdTmemCols);
    }
    if (tid == 0 && (skip == 2 || *abort_flag)) {
        // leave no copy in flight: whatever was issued must land before the block exits (looked at only now: the block may
        // give up after the loader has issued its last copy)
        bwd_drain(b_a, 0);
        for (uint32_t j = 0; j < kStages && j < n_loads; ++j) {
            const uint32_t idx = n_loads - 1 - j;
            bwd_drain(b_full0 + 8 * (idx % kStages), (idx / kStages) & 1u);
        }
    }
    if (KEY_ROLE) ptx::grid_wait();   // the call is over when both roles are
}

template <int D>
int launch_roles(const BwdViews &q, const BwdViews &k, const BwdViews &v, const BwdViews &g, const BwdOut &dq,
                 const BwdOut &dk, const BwdOut &dv, const BwdParams &stat_prm, const BwdParams &prm, cudaStream_t stream)
{
    constexpr size_t kSmem = 7 * (D / 64) * 16384 + sizeof(BwdCtrl);
    static_assert(kKeyStages + 2 == 7 && kQueryStages == 7 && kSmem <= 232448, "all roles take seven tiles of shared memory");
    // Each launch may start on the SMs that the one before leaves free (programmatic launches); what it waits for stands in
    // the kernel.
    auto run = [&](auto kernel, const BwdMaps &maps, const BwdParams &p, bool follows) -> int {
        CLEAR_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem));
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)p.n_items * (unsigned)p.n_bh);
        cfg.blockDim = dim3(kBwdThreads);
        cfg.dynamicSmemBytes = kSmem;
        cfg.stream = stream;
        cudaLaunchAttribute attr{};
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = follows ? 1 : 0;
        CLEAR_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, maps, p));
        return CLEAR_OK;
    };
    int rc = CLEAR_OK;
    if (prm.n_parts == 1) {
        rc = run(clear_bwd_tc_kernel<D, kStatsQuery>, BwdMaps{{q, g}, {k, v}, {dq, dq}}, prm, false);
    } else {
        rc = run(clear_bwd_tc_kernel<D, kStats>, BwdMaps{{q, g}, {k, v}, {dq, dq}}, stat_prm, false);
        if (rc == CLEAR_OK) rc = run(clear_bwd_tc_kernel<D, kQuery>, BwdMaps{{q, g}, {k, v}, {dq, dq}}, prm, true);
    }
    if (rc == CLEAR_OK) rc = run(clear_bwd_tc_kernel<D, kKey>, BwdMaps{{k, v}, {q, g}, {dv, dk}}, prm, true);
    return rc;
}

// The text tiles, which see every token, lead the list unless the grid is tiny: that many items of every head come first.
int count_first(const std::vector<clear_work_item_t> &items)
{
    size_t n = 0;
    while (n < items.size() && items[n].kind == 1) ++n;
    return n < items.size() ? (int)n : 0;
}

// Statistics of every row, to 256 bytes.
size_t row_stats_bytes(const clear_plan &p)
{
    const Shape &s = p.shape;
    const size_t rows = (size_t)s.B * s.H * ((size_t)s.n_text + (size_t)s.grid_h * s.grid_w);
    return (rows * sizeof(float2) + 255) / 256 * 256;
}

}  // namespace

int launch_bwd_tc(const clear_plan &p, const void *q, const void *k, const void *v, const void *d_out, void *dq, void *dk,
                  void *dv, float scale, cudaStream_t stream)
{
    const Shape &s = p.shape;
    if (!(scale > 0.f)) return CLEAR_ERR_UNSUPPORTED;
    if (s.head_dim != 64 && s.head_dim != 128) return CLEAR_ERR_UNSUPPORTED;
    const uint64_t gw = (uint64_t)s.grid_w, gh = (uint64_t)s.grid_h, T = (uint64_t)s.n_text;
    const uint64_t N = T + gw * gh, BH = (uint64_t)s.B * s.H, halves = (uint64_t)s.head_dim / 64;
    if (p.sch.stat_items.size() * BH > (uint64_t)INT32_MAX) return CLEAR_ERR_UNSUPPORTED;   // (no fewer than p.sch.items)
    if (!p.d_bwd_stats) {
        // behind them the partial statistics of cut text tiles and the counts of their finished parts
        const size_t slots = (size_t)BH * p.sch.n_stat_slots;
        const size_t bytes = row_stats_bytes(p) + slots * (kTileTokens * sizeof(float4) + sizeof(int));
        cudaError_t e = cudaMalloc((void **)&p.d_bwd_stats, bytes);
        if (e == cudaSuccess) e = cudaMemsetAsync(p.d_bwd_stats, 0, bytes, stream);
        if (e != cudaSuccess) {
            (void)cudaGetLastError();
            return e == cudaErrorMemoryAllocation ? CLEAR_ERR_NO_MEMORY : CLEAR_ERR_CUDA;
        }
        p.bwd_stats_bytes = bytes;
    }

    // Per tensor four views of [BH][half][rows][cols][64]: the image part in patches of 8 x 16 and of 4 x 16, runs of 128
    // tokens of the text prefix (rows past the text read as zero) and of 64 tokens of the whole sequence.
    const uint64_t row_b = (uint64_t)s.head_dim * 2;
    const uint64_t dims_img[5] = {64, gw, gh, halves, BH}, str_img[4] = {row_b, gw * row_b, 128, N * row_b};
    const uint32_t box_img[5] = {64, (uint32_t)kTileW, (uint32_t)kTileH, (uint32_t)halves, 1};
    const uint64_t dims_lin[5] = {64, N, 1, halves, BH}, dims_txt[5] = {64, T > 0 ? T : 1, 1, halves, BH};
    const uint64_t str_lin[4] = {row_b, N * row_b, 128, N * row_b};
    const uint32_t box_txt[5] = {64, (uint32_t)kTileTokens, 1, (uint32_t)halves, 1};
    const uint32_t box_himg[5] = {64, (uint32_t)kTileW, (uint32_t)kTileH / 2, (uint32_t)halves, 1};
    const uint32_t box_hlin[5] = {64, (uint32_t)kTileTokens / 2, 1, (uint32_t)halves, 1};
    BwdViews views[4];
    const void *tensors[4] = {q, k, v, d_out};
    for (int t = 0; t < 4; ++t)
        if (!encode_bf16_map(&views[t].img, static_cast<const char *>(tensors[t]) + T * row_b, 5, dims_img, str_img, box_img) ||
            !encode_bf16_map(&views[t].txt, tensors[t], 5, dims_txt, str_lin, box_txt) ||
            !encode_bf16_map(&views[t].half_img, static_cast<const char *>(tensors[t]) + T * row_b, 5, dims_img, str_img, box_himg) ||
            !encode_bf16_map(&views[t].half_lin, tensors[t], 5, dims_lin, str_lin, box_hlin))
            return CLEAR_ERR_CUDA;
    BwdOut outs[3];
    void *grads[3] = {dq, dk, dv};
    for (int t = 0; t < 3; ++t)
        if (!encode_bf16_map(&outs[t].img, static_cast<char *>(grads[t]) + T * row_b, 5, dims_img, str_img, box_img) ||
            !encode_bf16_map(&outs[t].txt, grads[t], 5, dims_txt, str_lin, box_txt))
            return CLEAR_ERR_CUDA;

    BwdParams prm{};
    prm.parts = reinterpret_cast<float4 *>(reinterpret_cast<char *>(p.d_bwd_stats) + row_stats_bytes(p));
    prm.part_count = reinterpret_cast<int *>(prm.parts + (size_t)BH * p.sch.n_stat_slots * kTileTokens);
    prm.n_parts = p.sch.n_stat_parts;
    prm.n_part_slots = p.sch.n_stat_slots;
    prm.key_waits = p.sch.n_stat_parts == 1;
    prm.items = p.d_items;
    prm.tiles = p.d_tiles;
    prm.mask_table = p.d_mask_table;
    prm.half_width = p.d_half_width;
    prm.n_half_width = (int)p.sch.half_width.size();
    prm.grid_h = s.grid_h;
    prm.grid_w = s.grid_w;
    prm.n_text = s.n_text;
    prm.n_items = (int)p.sch.items.size();
    prm.n_first = count_first(p.sch.items);
    prm.n_bh = (int)BH;
    prm.n_tokens = (long long)N;
    prm.scale = scale;
    prm.scale_log2 = scale * 1.4426950408889634f;
    prm.stats = reinterpret_cast<float2 *>(p.d_bwd_stats);
    prm.status = p.d_status;
    BwdParams stat_prm = prm;
    stat_prm.items = p.d_stat_items;
    stat_prm.n_items = (int)p.sch.stat_items.size();
    stat_prm.n_first = count_first(p.sch.stat_items);
    if (s.head_dim == 128) return launch_roles<128>(views[0], views[1], views[2], views[3], outs[0], outs[1], outs[2], stat_prm, prm, stream);
    return launch_roles<64>(views[0], views[1], views[2], views[3], outs[0], outs[1], outs[2], stat_prm, prm, stream);
}

}  // namespace clear
