// CLEAR attention forward on the sm_100a tensor cores: persistent, warp-specialised kernel.
//
// One thread block per SM takes work items from a queue (an atomic counter).  A work item is a PAIR
// of 128-query tiles -- two vertically adjacent 8 x 16 patches of the latent grid, or two tiles of
// text tokens -- and a list of steps; in each step every query tile of the pair meets one 128-key
// tile (Eq. 1 restricted by Eq. 3).  Key tiles both query tiles need are staged once.
//
// Roles (384 threads):
//   warp 0        : takes items from the queue and issues every TMA load (Q tiles, K/V ring);
//   warps 1, 2    : issue every tcgen05.mma of query tile 0 / 1: S_t = Q_t K^T and O_t += P_t V;
//   warps 4-7     : softmax and epilogue of query tile 0 (thread r owns query row r = tensor-memory
//                   lane r): P = exp2(.) on the keys Eq. 3 allows and 0 elsewhere, as bf16 into tensor
//                   memory over S, row sum; at the end of an item O / l -> bf16 -> global memory (or
//                   fp32 partial results of split text rows);
//   warps 8-11    : the same for query tile 1.
// Tensor memory (512 columns): S0 | S1 | O0 | O1, 128 columns each; P_t takes the first 64 columns of
// S_t and is the tensor-memory operand of P_t V, so that P never crosses shared memory: with both MMA
// operands in shared memory a 128 x 128 x 16 MMA reads 8 KB per 64 clocks, all a shared memory can
// deliver, and nothing else (P stores, TMA fills) fits beside it.
// Shared memory: Q0, Q1 and a ring of five key/value stages (K and V tiles take one stage each).
// Every wait is bounded: on expiry the block raises the plan's status word and leaves.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>

#include "clear_internal.hpp"
#include "ptx.cuh"

namespace clear {
namespace {

constexpr int kWsThreads = 384;   // 4 control warps + 2 x 4 softmax warps
constexpr uint32_t kRing = 5;
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kSpinLimit = 1u << 22;
constexpr uint32_t kWaitHintNs = 20000;            // one sleep inside try_wait
constexpr uint32_t kWaitLimitUs = 2000000;         // a wait that lasts 2 s has failed
constexpr float kRescaleThreshold = 8.f;  // log2 units: a reference is moved only when a row's maximum exceeds it by more
constexpr float kBumpSum = 65536.f;       // a row sum of P above this raises the row's reference
constexpr float kMaxTileSum = 0x1p64f;    // a row sum above this has its tile taken again (a NaN comes from NaN inputs only, and stays)
// Scores of a row's first tile that lie this far apart (log2 units) give the item maximum passes from the start: with less,
// normal ones would have to lie seven standard deviations above the maximum of 128 to be 64 above it.  (The least of 16 of
// them is enough to tell.)
constexpr float kWideStep = 40.f;
constexpr int kSchedDepth = 2;
// arrivals that free a queue slot: one lane of each of the 2 MMA warps, the 8 softmax warps
constexpr uint32_t kSchedReaders = 10;
// registers per thread of each role: 128 x 80 + 256 x 208 = 63488, within what the block is launched with
// (384 threads x 168); raising a warp's budget only draws on registers other warps of the block gave back
constexpr uint32_t kRegsControl = 80, kRegsSoftmax = 208;
static_assert(128 * kRegsControl + 256 * kRegsSoftmax <= 384 * 168, "a raise beyond the block's registers would wait for ever");

struct WsParams {
    const clear_pair_item_t *items;
    const clear_pair_step_t *steps;
    const int32_t *half_width;
    const uint32_t *side_words;  // [2 tiles][n_steps] (Schedule::side_words)
    int n_steps;
    const uint32_t *mask_table;  // [entry][128 query rows][4 words]: Eq. 3 per relative patch offset and border case
    int n_half_width;
    int grid_h, grid_w, n_text;
    long long n_tokens;
    int n_items, n_text_items, n_bh;
    float scale_log2;  // scale * log2(e)
    float *partial_o;  // split text rows, per (bh, slot): [D][128] un-normalised O, channel by channel
    float *partial_ml; // and [128][2]: reference (log2 units) and row sum
    int n_partial_slots;
    const __nv_bfloat16 *q, *k;
    __nv_bfloat16 *out;
    int *status;  // [0] status word of this launch, [1] queue head, [2] finished blocks, [3] status kept for the host
};

// Views of q, k, v (kMap*): patches of the image part, and runs of consecutive tokens.  Every view has five axes,
// channel (64), column or token, row, channel half, (batch, head), so one copy instruction, with one of these maps and
// its coordinates chosen at run time, brings any tile of 128 tokens and all its channels.
enum { kMapQImg = 0, kMapQTxt = 1, kMapKImg = 2, kMapKLin = 3, kMapVImg = 4, kMapVLin = 5 };
struct WsMaps {
    CUtensorMap m[6];
};

struct Ctrl {
    uint64_t q_full[2], q_empty[2];
    uint64_t kv_full[kRing], kv_empty[kRing];
    uint64_t sa_full[2], sb_full[2], sb_read[2], p_ready[2], o_full[2], o_empty[2];
    uint64_t sched_full[kSchedDepth], sched_empty[kSchedDepth];
    uint64_t turn[2], drain[2];
    int32_t sched_item[kSchedDepth];            // queue position, >= total: no more work
    int32_t sched_bh[kSchedDepth];
    clear_pair_item_t sched_rec[kSchedDepth];   // the item's record, read once from global memory
    uint32_t copies[3];   // issued by the loader: Q tiles of tile 0 and 1, K/V stages
    uint32_t tmem_base;
    int abort_flag;
    int skip;
};

// Bounded wait on an mbarrier phase.  Returns false once the block has given up.  The polling loop is a handful of
// instructions in line (each wait is one more copy of it, and the kernel's code has to stay small enough for the
// instruction caches); what happens every 128 tries -- the abort flag, the clock -- is one function.  Roles that can
// afford it (SLEEP_NS > 0) sleep between tries: a polling warp takes issue slots from the softmax warps.
__device__ __noinline__ uint32_t wait_tick(uint32_t t0, volatile int *abort_flag, int *status, int code)
{
    const uint32_t now = (uint32_t)(ptx::globaltimer_ns() >> 10) | 1u;  // about microseconds, never 0
    if (t0 == 0) t0 = now;
    if (*abort_flag) return 0;
    if (now - t0 <= kWaitLimitUs) return t0;
    *abort_flag = 1;
    atomicCAS(status, 0, code);  // the first wait that expired names the cause
    return 0;
}
template <uint32_t SLEEP_NS = 0>
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *status, int code)
{
    if (ptx::mbar_try_wait(bar, parity)) return true;
    uint32_t t0 = 0;
#pragma unroll 1
    for (uint32_t n = 1; !ptx::mbar_try_wait_hint(bar, parity, kWaitHintNs); ++n) {
        if (SLEEP_NS > 0) __nanosleep(SLEEP_NS);
        if ((n & 127u) == 0u && (t0 = wait_tick(t0, abort_flag, status, code)) == 0u) return false;
    }
    return true;
}
// One arrival for the whole warp, after every lane has got here (and its earlier writes with it).
__device__ __forceinline__ void warp_arrive(uint32_t bar, int lane)
{
    __syncwarp();
    if (lane == 0) ptx::mbar_arrive(bar);
}
// Drain: wait for a phase regardless of the abort flag (used before leaving with copies in flight).
__device__ __noinline__ void drain_bar(uint32_t bar, uint32_t parity)
{
#pragma unroll 1
    for (uint32_t it = 0; it < kSpinLimit; ++it) {
        if (ptx::mbar_try_wait(bar, parity)) return;
        if (it > 64) __nanosleep(256);
    }
}

struct ItemRef {
    int bh;
    int item;
};
// Queue position -> (batch*head, item): every text item of every head first, then the image items.
__device__ __forceinline__ ItemRef decode_item(const WsParams &prm, int g)
{
    ItemRef r;
    const int n_txt_all = prm.n_text_items * prm.n_bh;
    if (g < n_txt_all) {
        r.bh = g / prm.n_text_items;
        r.item = g - r.bh * prm.n_text_items;
    } else {
        const int n_img = prm.n_items - prm.n_text_items;
        const int g2 = g - n_txt_all;
        r.bh = g2 / n_img;
        r.item = prm.n_text_items + (g2 - r.bh * n_img);
    }
    return r;
}

__device__ __forceinline__ clear_pair_step_t load_step(const clear_pair_step_t *p)
{
    const int4 a = __ldg(reinterpret_cast<const int4 *>(p));
    const int4 b = __ldg(reinterpret_cast<const int4 *>(p) + 1);
    clear_pair_step_t s;
    s.x0 = a.x; s.y0 = a.y; s.x1 = a.z; s.y1 = a.w;
    s.flags = b.x; s.n_valid0 = b.y; s.n_valid1 = b.z; s.load_base = b.w;
    return s;
}
__device__ __forceinline__ clear_pair_item_t load_item(const clear_pair_item_t *p)
{
    const int4 a = __ldg(reinterpret_cast<const int4 *>(p));
    const int4 b = __ldg(reinterpret_cast<const int4 *>(p) + 1);
    const int4 c = __ldg(reinterpret_cast<const int4 *>(p) + 2);
    clear_pair_item_t it;
    it.kind = a.x; it.n_sides = a.y; it.qx = a.z; it.qy0 = a.w;
    it.qy1 = b.x; it.n_rows0 = b.y; it.n_rows1 = b.z; it.step_begin = b.w;
    it.step_count = c.x; it.n_loads = c.y; it.partial_slot0 = c.z; it.partial_slot1 = c.w;
    return it;
}
// Origin of the key patch of that tile (only plans without a mask table and recomputed tiles need it).
__device__ __forceinline__ int2 load_side_origin(const clear_pair_step_t *p, int side)
{
    const int4 a = __ldg(reinterpret_cast<const int4 *>(p));
    return side ? make_int2(a.z, a.w) : make_int2(a.x, a.y);
}
static_assert(sizeof(clear_pair_step_t) == 32 && sizeof(clear_pair_item_t) == 48, "table records are read as int4");

// ---- pieces of the softmax warps' work that are rare, or come once an item: functions of their own, so that their
// registers do not crowd the exponentials of the common step (with them in line the compiler had too few left to overlap
// with, and a pass over 128 scores took up to 1900 clocks instead of 1400) --------------------------------------------

// A trip count the compiler cannot see: without it these loops are unrolled whatever the source says, and most of their time
// goes into fetching instructions that run once.
__device__ __forceinline__ int opaque(int n)
{
    asm volatile("" : "+r"(n));
    return n;
}

// The row's O times alpha (O_t is at rest: P_t V of the step before is complete).
template <int D>
__device__ __noinline__ void rescale_rows(uint32_t tmem_o, float alpha)
{
#pragma unroll 1
    for (int w = 0, n = opaque(D / 16); w < n; ++w) {
        uint32_t o[16];
        ptx::tmem_ld16(tmem_o + 16 * w, o);
        ptx::tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 16; ++j) o[j] = __float_as_uint(__uint_as_float(o[j]) * alpha);
        ptx::tmem_st16(tmem_o + 16 * w, o);
    }
}

// The row's P (bf16 pairs) times alpha, a power of two.
__device__ __noinline__ void rescale_p(uint32_t tmem_p, float alpha)
{
    const __nv_bfloat162 a = __float2bfloat162_rn(alpha);
#pragma unroll 1
    for (int w = 0, n = opaque(4); w < n; ++w) {
        uint32_t p[16];
        ptx::tmem_ld16(tmem_p + 16 * w, p);
        ptx::tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            __nv_bfloat162 x = __hmul2(*reinterpret_cast<__nv_bfloat162 *>(&p[j]), a);
            p[j] = *reinterpret_cast<uint32_t *>(&x);
        }
        ptx::tmem_st16(tmem_p + 16 * w, p);
    }
}

// P of 32 keys from their scores: 2^(S c - mc) on the allowed keys and 0 elsewhere, added to the row sum (two-wide fp32
// FMA and ADD, four independent partial sums), as bf16 pairs (16 columns of tensor memory).
template <bool kMasked>
__device__ __forceinline__ void exp_chunk(const uint32_t (&sv)[32], uint32_t bits, uint64_t c2, uint64_t nmc2, uint64_t (&lsum)[2],
                                          uint32_t (&pk)[16])
{
#pragma unroll
    for (int j = 0; j < 32; j += 2) {
        const uint64_t x2 = ptx::fma2(ptx::pack2(__uint_as_float(sv[j]), __uint_as_float(sv[j + 1])), c2, nmc2);
        float x0, x1;
        ptx::unpack2(x2, x0, x1);
        if (kMasked) {
            x0 = ((bits >> j) & 1u) ? x0 : -INFINITY;
            x1 = ((bits >> (j + 1)) & 1u) ? x1 : -INFINITY;
        }
        const float p0 = ptx::ex2(x0), p1 = ptx::ex2(x1);
        lsum[(j >> 1) & 1] = ptx::add2(lsum[(j >> 1) & 1], ptx::pack2(p0, p1));
        pk[j >> 1] = ptx::pack_bf16(p0, p1);
    }
}
__device__ __forceinline__ float sum4(const uint64_t (&lsum)[2])
{
    float a0, a1, a2, a3;
    ptx::unpack2(lsum[0], a0, a1);
    ptx::unpack2(lsum[1], a2, a3);
    return (a0 + a1) + (a2 + a3);
}

struct RowState {
    float ref, l, tile_sum;   // tile_sum < 0: less that, and the row's maximum lies more than kWideStep above the least of 16 scores
};
// The largest of the 128 scores of a row that all count, and the least of 16 of them.  (Of 64 only: 0.5 % more rounding error of P
// at 512 text tokens, where the row's largest weight is then more often not a whole 1.)
struct RowTop {
    float most, least;
};
__device__ __noinline__ RowTop first_top(uint32_t tmem_s)
{
    float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY}, mn = INFINITY;
#pragma unroll 1
    for (int h = 0, n = opaque(2); h < n; ++h) {
        uint32_t sv[2][32];
        ptx::tmem_ld32(tmem_s + 64 * h, sv[0]);
        ptx::tmem_ld32(tmem_s + 64 * h + 32, sv[1]);
        ptx::tmem_wait_ld();
#pragma unroll
        for (int w = 0; w < 2; ++w)
#pragma unroll
            for (int j = 0; j < 32; j += 2) mx[(j >> 1) & 3] = ptx::max3(mx[(j >> 1) & 3], __uint_as_float(sv[w][j]), __uint_as_float(sv[w][j + 1]));
#pragma unroll
        for (int j = 0; j < 32; j += 4) mn = fminf(mn, __uint_as_float(sv[0][j]));
    }
    return RowTop{fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])), mn};
}

// A step with a maximum pass: the maximum over the allowed keys, the row's reference, then P.  The scores are read from
// tensor memory both times, 32 keys at a time (P of 32 keys takes 16 columns, so it never reaches scores still to be read).
template <int D>
__device__ __noinline__ RowState exact_step(uint32_t tmem_s, uint32_t tmem_o, uint4 mask, float c, float ref, float l, bool first)
{
    auto bits_of = [&](int w) { return w == 0 ? mask.x : w == 1 ? mask.y : w == 2 ? mask.z : mask.w; };
    float mx = -INFINITY, mn = INFINITY;
#pragma unroll 1
    for (int w = 0, n = opaque(4); w < n; ++w) {
        uint32_t sv[32];
        ptx::tmem_ld32(tmem_s + 32 * w, sv);
        const uint32_t bits = bits_of(w);
        ptx::tmem_wait_ld();
        float mx2[2] = {mx, -INFINITY};
#pragma unroll
        for (int j = 0; j < 32; j += 2)
            mx2[(j >> 1) & 1] = ptx::max3(mx2[(j >> 1) & 1], ((bits >> j) & 1u) ? __uint_as_float(sv[j]) : -INFINITY,
                                          ((bits >> (j + 1)) & 1u) ? __uint_as_float(sv[j + 1]) : -INFINITY);
        mx = fmaxf(mx2[0], mx2[1]);
#pragma unroll
        for (int j = 0; j < 32; j += 8)
            if ((bits >> j) & 1u) mn = fminf(mn, __uint_as_float(sv[j]));
    }
    const float m_new = fmaxf(ref, mx * c);
    if (first) {
        ref = m_new;
    } else {
        const bool need = m_new - ref > kRescaleThreshold;  // false for NaN (-inf minus -inf)
        if (__any_sync(0xffffffffu, need)) {
            const float alpha = need ? ptx::ex2(ref - m_new) : 1.f;
            if (need) ref = m_new;
            l *= alpha;
            rescale_rows<D>(tmem_o, alpha);
        }
    }
    const float mc = (ref == -INFINITY) ? 0.f : ref;
    const uint64_t c2 = ptx::pack2(c, c), nmc2 = ptx::pack2(-mc, -mc);
    uint64_t lsum[2] = {0ull, 0ull};
#pragma unroll 1
    for (int w = 0, n = opaque(4); w < n; ++w) {
        uint32_t sv[32], pk[16];
        ptx::tmem_ld32(tmem_s + 32 * w, sv);
        ptx::tmem_wait_ld();
        exp_chunk<true>(sv, bits_of(w), c2, nmc2, lsum, pk);
        ptx::tmem_st16(tmem_s + 16 * w, pk);
    }
    const float sum = sum4(lsum);
    return RowState{ref, l, (mx - mn) * c > kWideStep ? -sum : sum};
}

// A step whose scores lie far above the row's reference: the warp's 32 x 128 scores once more from global memory (those in
// tensor memory are gone), with warp-level MMAs and twice over -- for the rows' maxima, and for P against them.  The rows of
// an MMA lie in the lanes of a quad; reference, mask and results of row r belong to lane r, and move by shuffles.  Scores of
// one key at a time by scalar products took about a millisecond a step; the rest of the item has maximum passes, so that it
// happens once an item and warp at most, and not at all where the first tile's scores are far apart already.  24 heads at
// 1024 px, r = 8, Q times 20 or 60: 165 us a call (2.7 and 94 ms with scalar products and no memory of it; 105 us with ordinary
// scores).  The slowest measured is Q times 5, 171 us: warps of one tile with maximum passes, and others without.
template <int D>
__device__ __noinline__ RowState rescue_step(const WsParams &prm, uint32_t tmem_p, uint32_t tmem_o, uint4 mask, float c, float ref, float l,
                                             long long row0, long long q_tok, int2 org, bool linear)
{
    ptx::tmem_wait_st();
    const int lane = threadIdx.x & 31, quad = lane >> 2, sub = lane & 3;
    auto word = [&](int w) { return w == 0 ? mask.x : w == 1 ? mask.y : w == 2 ? mask.z : mask.w; };
    // Contraction channels come in an order of their own, the same for both operands: of 32 channels a lane loads the 8 from
    // 8 sub on as 16 bytes, and they serve as its four pairs of two MMAs.
    // 16 rows at a time: in the quad's lanes the rows 16 m + quad and 8 further on
    uint32_t a[D / 16][4];
    auto load_rows = [&](int m) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int tok = __shfl_sync(0xffffffffu, (int)q_tok, 16 * m + 8 * h + quad);
            const uint4 *row = reinterpret_cast<const uint4 *>(prm.q + (row0 + max(tok, 0)) * D) + sub;
#pragma unroll
            for (int kk = 0; kk < D / 32; ++kk) {
                const uint4 x = tok >= 0 ? __ldg(row + 4 * kk) : make_uint4(0u, 0u, 0u, 0u);
                a[2 * kk][h] = x.x;
                a[2 * kk][2 + h] = x.y;
                a[2 * kk + 1][h] = x.z;
                a[2 * kk + 1][2 + h] = x.w;
            }
        }
    };
    // their scores with the keys 8 n .. 8 n + 7: the lane holds the keys 8 n + 2 sub, + 1
    auto scores = [&](int n, float (&s)[4]) {
        const int key = 8 * n + quad, ky = org.y + (key >> 4), kx = org.x + (key & 15);
        const bool on = linear ? org.x + key < prm.n_tokens : ky >= 0 && ky < prm.grid_h && kx >= 0 && kx < prm.grid_w;
        const long long tok = linear ? org.x + key : prm.n_text + (long long)ky * prm.grid_w + kx;
        const uint4 *row = reinterpret_cast<const uint4 *>(prm.k + (row0 + (on ? tok : 0)) * D) + sub;
        uint4 b[D / 32];
#pragma unroll
        for (int kk = 0; kk < D / 32; ++kk) b[kk] = on ? __ldg(row + 4 * kk) : make_uint4(0u, 0u, 0u, 0u);
        s[0] = s[1] = s[2] = s[3] = 0.f;
#pragma unroll
        for (int kk = 0; kk < D / 32; ++kk) {
            const uint32_t b0[2] = {b[kk].x, b[kk].y}, b1[2] = {b[kk].z, b[kk].w};
            ptx::mma_16816_bf16(s, a[2 * kk], b0);
            ptx::mma_16816_bf16(s, a[2 * kk + 1], b1);
        }
    };
    // of the values for the two rows in the quad's lanes, the one of the lane's own row (if it is one of the 16)
    auto to_owner = [&](float v0, float v1, int src_sub) {
        const float x0 = __shfl_sync(0xffffffffu, v0, (lane & 7) * 4 + src_sub), x1 = __shfl_sync(0xffffffffu, v1, (lane & 7) * 4 + src_sub);
        return lane & 8 ? x1 : x0;
    };

    float mx = -INFINITY;
#pragma unroll 1
    for (int m = 0; m < 2; ++m) {
        load_rows(m);
        float top[2] = {-INFINITY, -INFINITY};
#pragma unroll 1
        for (int w = 0; w < 4; ++w) {
            const uint32_t bits[2] = {__shfl_sync(0xffffffffu, word(w), 16 * m + quad), __shfl_sync(0xffffffffu, word(w), 16 * m + 8 + quad)};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float s[4];
                scores(4 * w + j, s);
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if ((bits[u >> 1] >> (8 * j + 2 * sub + (u & 1))) & 1u) top[u >> 1] = fmaxf(top[u >> 1], s[u]);
            }
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            top[0] = fmaxf(top[0], __shfl_xor_sync(0xffffffffu, top[0], o));
            top[1] = fmaxf(top[1], __shfl_xor_sync(0xffffffffu, top[1], o));
        }
        const float own = to_owner(top[0], top[1], 0);
        if ((lane >> 4) == m) mx = own;
    }
    const float m_new = fmaxf(ref, mx * c);
    const bool need = m_new - ref > kRescaleThreshold;
    const float alpha = need ? ptx::ex2(ref - m_new) : 1.f;
    if (need) ref = m_new;
    l *= alpha;
    rescale_rows<D>(tmem_o, alpha);

    const float mc = (ref == -INFINITY) ? 0.f : ref;
    float sum = 0.f;
#pragma unroll 1
    for (int w = 0; w < 4; ++w) {
        uint32_t pk[16];
#pragma unroll 1
        for (int m = 0; m < 2; ++m) {
            load_rows(m);
            const uint32_t bits[2] = {__shfl_sync(0xffffffffu, word(w), 16 * m + quad), __shfl_sync(0xffffffffu, word(w), 16 * m + 8 + quad)};
            const float mc2[2] = {__shfl_sync(0xffffffffu, mc, 16 * m + quad), __shfl_sync(0xffffffffu, mc, 16 * m + 8 + quad)};
            const bool mine = (lane >> 4) == m;
            float part[2] = {0.f, 0.f};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float s[4], p[4];
                scores(4 * w + j, s);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const bool on = ((bits[u >> 1] >> (8 * j + 2 * sub + (u & 1))) & 1u) != 0u;
                    p[u] = on ? ptx::ex2(fmaf(s[u], c, -mc2[u >> 1])) : 0.f;
                    part[u >> 1] += p[u];
                }
                const float pair[2] = {__uint_as_float(ptx::pack_bf16(p[0], p[1])), __uint_as_float(ptx::pack_bf16(p[2], p[3]))};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint32_t x = __float_as_uint(to_owner(pair[0], pair[1], e));
                    pk[4 * j + e] = mine ? x : m == 0 ? 0u : pk[4 * j + e];
                }
            }
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
                part[0] += __shfl_xor_sync(0xffffffffu, part[0], o);
                part[1] += __shfl_xor_sync(0xffffffffu, part[1], o);
            }
            const float own = to_owner(part[0], part[1], 0);
            if (mine) sum += own;
        }
        ptx::tmem_st16(tmem_p + 16 * w, pk);
    }
    return RowState{ref, l, sum};
}

// End of an item for one query tile: O / l, or the partial results of split text rows, to global memory.  `first_x`: first
// token (text) or grid column, `first_y`: grid row of the tile; n_rows: rows of a text tile, -1 for a patch.  Tells the
// MMA warp (o_empty) as soon as O has been read.
template <int D>
__device__ __noinline__ void store_tile(const WsParams &prm, uint32_t tmem_o, uint32_t b_o_empty, int first_x, int first_y, int n_rows,
                                        int slot, int bh, float ref, float l)
{
    const int lane = threadIdx.x & 31, q4 = (threadIdx.x >> 5) & 3, r = q4 * 32 + lane;
    tmem_o += (uint32_t)(q4 * 32) << 16;
    if (slot >= 0) {
        // split text-query tile: un-normalised fp32 rows, channel by channel (a warp writes 32 rows of one channel as
        // 128 consecutive bytes), and per row its reference (log2 units) and its sum
        const long long slot_row = ((long long)bh * prm.n_partial_slots + slot) * 128;
        float *dst = prm.partial_o + slot_row * D + r;
#pragma unroll 1
        for (int w = 0, n = opaque(D / 16); w < n; ++w) {
            uint32_t o[16];
            ptx::tmem_ld16(tmem_o + 16 * w, o);
            ptx::tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 16; ++j) dst[(16 * w + j) * 128] = __uint_as_float(o[j]);
        }
        ptx::tc_fence_before();
        warp_arrive(b_o_empty, lane);
        prm.partial_ml[(slot_row + r) * 2] = ref;
        prm.partial_ml[(slot_row + r) * 2 + 1] = l;
        return;
    }
    // O / l as bf16, 32 channels of the thread's row at a time, in pieces of 32 bytes (a memory sector).  Once an item, so that
    // its instructions are fetched anew each time, some 16 clocks each: a short loop rather than a fast one.
    const float inv = l > 0.f ? 1.f / l : 0.f;
    const int y = first_y + (r >> 4), x = first_x + (r & 15);
    const bool on = n_rows >= 0 ? r < n_rows : (y < prm.grid_h && x < prm.grid_w);
    const long long token = n_rows >= 0 ? (long long)first_x + r : prm.n_text + (long long)y * prm.grid_w + x;
    __nv_bfloat16 *dst = prm.out + ((long long)bh * prm.n_tokens + token) * D;
    const bool wide = (reinterpret_cast<uintptr_t>(prm.out) & 31u) == 0u;  // tensors are 16-byte aligned at least
#pragma unroll 1
    for (int w = 0, n = opaque(D / 32); w < n; ++w) {
        uint32_t o[32];
        ptx::tmem_ld32(tmem_o + 32 * w, o);
        ptx::tmem_wait_ld();
        // behind the last reads the next item's first P V may start; the stores take their time
        if (w == n - 1) {
            ptx::tc_fence_before();
            warp_arrive(b_o_empty, lane);
        }
        uint32_t u[2][8];
#pragma unroll
        for (int j = 0; j < 16; ++j) u[j >> 3][j & 7] = ptx::pack_bf16(__uint_as_float(o[2 * j]) * inv, __uint_as_float(o[2 * j + 1]) * inv);
        if (on) {
            __nv_bfloat16 *to = dst + 32 * w;
            if (wide) {
                ptx::stg_u256(to, u[0]);
                ptx::stg_u256(to + 16, u[1]);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    *reinterpret_cast<uint4 *>(to + 8 * j) = make_uint4(u[j >> 1][4 * (j & 1)], u[j >> 1][4 * (j & 1) + 1], u[j >> 1][4 * (j & 1) + 2], u[j >> 1][4 * (j & 1) + 3]);
            }
        }
    }
}

// Mask words of a row that the table does not hold: a run of tokens that ends inside the tile, or (very large radius) a patch
// without an entry, Eq. 3 row by row from the half widths.  Once in many steps, so a function of its own.
__device__ __noinline__ uint4 special_mask(const WsParams &prm, const clear_pair_step_t *step, int t, bool q_valid, int q_y, int q_x)
{
    uint32_t mw[4] = {0u, 0u, 0u, 0u};
    if (__ldg(&step->flags) & CLEAR_STEP_LINEAR) {
        const int n_valid = __ldg(t ? &step->n_valid1 : &step->n_valid0);
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const int nv = min(max(n_valid - 32 * w, 0), 32);
            mw[w] = nv == 32 ? 0xffffffffu : ((1u << nv) - 1u);
        }
    } else {
        const int2 org = load_side_origin(step, t);
#pragma unroll 1
        for (int rr = 0; rr < 8; ++rr) {
            const int ky = org.y + rr;
            const int ady = abs(ky - q_y);
            uint32_t bits = 0u;
            if (q_valid && ky >= 0 && ky < prm.grid_h && ady < prm.n_half_width) {
                const int hw = __ldg(prm.half_width + ady);
                const int lo = max(max(q_x - hw, 0), org.x);
                const int hi = min(min(q_x + hw, prm.grid_w - 1), org.x + 15);
                if (lo <= hi) bits = ((1u << (hi - lo + 1)) - 1u) << (lo - org.x);
            }
            bits <<= 16 * (rr & 1);
            if ((rr >> 1) == 0) mw[0] |= bits;
            if ((rr >> 1) == 1) mw[1] |= bits;
            if ((rr >> 1) == 2) mw[2] |= bits;
            if ((rr >> 1) == 3) mw[3] |= bits;
        }
    }
    return make_uint4(mw[0], mw[1], mw[2], mw[3]);
}

// The last block of a launch to leave: the work queue goes back to zero, and a status some block raised
// moves to the word that stays until the host has read it, so that the next launch starts clean.
__device__ __forceinline__ void close_launch(int *status)
{
    atomicExch(status + 1, 0);
    atomicExch(status + 2, 0);
    const int raised = atomicExch(status, 0);
    if (raised != 0) atomicCAS(status + 3, 0, raised);
}

template <int D>
__global__ void __launch_bounds__(kWsThreads, 1)
clear_ws_kernel(const __grid_constant__ WsMaps maps, const __grid_constant__ WsParams prm)
{
    constexpr int kHalves = D / 64;                 // 64-channel (128-byte) column blocks of a tile
    constexpr uint32_t kHalfBytes = 128 * 128;      // 128 rows x 128 B
    constexpr uint32_t kTileBytes = kHalves * kHalfBytes;
    constexpr uint32_t kIdescQK = ptx::idesc_bf16(64, false);
    constexpr uint32_t kIdescPV = ptx::idesc_bf16(D, true);

    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t smem_base = ptx::smem_u32(smem_raw);
    // Q0, Q1 | ring of K/V stages | control
    const uint32_t sQ = smem_base, sRing = sQ + 2 * kTileBytes;
    constexpr uint32_t kCtrlOff = (2 + kRing) * kTileBytes;
    Ctrl *ctrl = reinterpret_cast<Ctrl *>(smem_raw + kCtrlOff);
    volatile int *abort_flag = &ctrl->abort_flag;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int total_items = prm.n_items * prm.n_bh;

    // once any block of this launch has given up, the rest of the grid leaves at once; a window that
    // is not 1024-byte aligned (never expected) cannot hold swizzled tiles
    if (tid == 0) {
        int skip = *reinterpret_cast<volatile int *>(prm.status);
        if ((smem_base & 1023u) != 0u) {
            atomicExch(prm.status, 100);
            skip = 1;
        }
        ctrl->skip = skip;
    }
    __syncthreads();
    if (ctrl->skip != 0) {
        if (tid == 0) {
            // keep the finished-block count right so that the queue is reset for the next launch
            const int done = atomicAdd(prm.status + 2, 1);
            if (done == (int)gridDim.x - 1) close_launch(prm.status);
        }
        return;
    }

    if (tid == 0) {
        ctrl->abort_flag = 0;
        for (int i = 0; i < 2; ++i) {
            ptx::mbar_init(ptx::smem_u32(&ctrl->q_full[i]), 1);
            ptx::mbar_init(ptx::smem_u32(&ctrl->q_empty[i]), 1);
            ptx::mbar_init(ptx::smem_u32(&ctrl->sa_full[i]), 1);
            ptx::mbar_init(ptx::smem_u32(&ctrl->sb_full[i]), 1);
            ptx::mbar_init(ptx::smem_u32(&ctrl->sb_read[i]), 4);  // one arrival per softmax warp of the tile
            ptx::mbar_init(ptx::smem_u32(&ctrl->p_ready[i]), 4);
            ptx::mbar_init(ptx::smem_u32(&ctrl->o_full[i]), 1);
            ptx::mbar_init(ptx::smem_u32(&ctrl->o_empty[i]), 4);
            ptx::mbar_init(ptx::smem_u32(&ctrl->turn[i]), 1);
        }
        for (uint32_t i = 0; i < kRing; ++i) {
            ptx::mbar_init(ptx::smem_u32(&ctrl->kv_full[i]), 1);
            ptx::mbar_init(ptx::smem_u32(&ctrl->kv_empty[i]), 2);  // one arrival per MMA warp
        }
        for (int i = 0; i < kSchedDepth; ++i) {
            ptx::mbar_init(ptx::smem_u32(&ctrl->sched_full[i]), 1);
            ptx::mbar_init(ptx::smem_u32(&ctrl->sched_empty[i]), kSchedReaders);
        }
        for (int i = 0; i < 2; ++i) ptx::mbar_init(ptx::smem_u32(&ctrl->drain[i]), 1);
        ptx::fence_mbar_init();
    }
    if (warp == 1) {
        ptx::tmem_alloc(ptx::smem_u32(&ctrl->tmem_base), kTmemCols);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = ctrl->tmem_base;

    if (warp < 4) {
        ptx::setmaxnreg_dec<kRegsControl>();
        if (warp == 0 && lane == 0) {
            // ================= loader: work queue + every TMA load ====================================
            uint32_t n_loads = 0;    // K/V stages filled so far by this block
            uint32_t stage = 0, stage_par = 0;  // the stage the next one goes to, parity of its fill
            const uint32_t b_full0 = ptx::smem_u32(&ctrl->kv_full[0]), b_empty0 = ptx::smem_u32(&ctrl->kv_empty[0]);
            uint32_t n_q[2] = {0, 0};
#pragma unroll 1
            for (uint32_t k = 0;; ++k) {
                const uint32_t slot = k % kSchedDepth, use = k / kSchedDepth;
                if (!wait_bar<200>(ptx::smem_u32(&ctrl->sched_empty[slot]), (use & 1u) ^ 1u, abort_flag, prm.status, 1)) break;
                const int g = atomicAdd(prm.status + 1, 1);
                ItemRef ref{0, 0};
                clear_pair_item_t item{};
                if (g < total_items) {
                    ref = decode_item(prm, g);
                    item = load_item(prm.items + ref.item);
                    ctrl->sched_rec[slot] = item;
                    ctrl->sched_bh[slot] = ref.bh;
                }
                ctrl->sched_item[slot] = g;
                ptx::mbar_arrive(ptx::smem_u32(&ctrl->sched_full[slot]));
                if (g >= total_items) break;
                bool ok = true;
#pragma unroll 1
                for (int t = 0; t < item.n_sides && ok; ++t) {
                    const uint32_t bar = ptx::smem_u32(&ctrl->q_full[t]);
                    ok = wait_bar<200>(ptx::smem_u32(&ctrl->q_empty[t]), (n_q[t] & 1u) ^ 1u, abort_flag, prm.status, 2);
                    if (!ok) break;
                    ptx::mbar_expect_tx(bar, kTileBytes);
                    const bool txt = item.kind == 1;
                    ptx::tma_load_5d(sQ + t * kTileBytes, &maps.m[txt ? kMapQTxt : kMapQImg], bar, 0,
                                     txt ? item.qx + t * 128 : item.qx, txt ? 0 : t ? item.qy1 : item.qy0, 0, ref.bh);
                    ++n_q[t];
                }
                // staging order = reading order: the K tiles of a step come before the V tiles of the step before it
                const clear_pair_step_t *steps = prm.steps + item.step_begin;
                clear_pair_step_t st = load_step(steps), st_prev = st;
                st_prev.flags = 0;
#pragma unroll 1
                for (int s = 0; s <= item.step_count && ok; ++s) {
                    // records are fetched ahead of their use, so their latency is off the critical path
                    clear_pair_step_t st_next = st;
                    if (s + 1 < item.step_count) st_next = load_step(steps + s + 1);
                    else st_next.flags = 0;
#pragma unroll 1
                    for (int i = 0; i < 4 && ok; ++i) {
                        // tile 0's, and tile 1's when it is another one
                        const int t = i & 1;
                        const bool k = i < 2;
                        const int flags = k ? st.flags : st_prev.flags;
                        if (!(t ? (flags & (CLEAR_STEP_USE1 | CLEAR_STEP_SHARED)) == CLEAR_STEP_USE1 : (flags & CLEAR_STEP_USE0) != 0)) continue;
                        ok = wait_bar<100>(b_empty0 + 8 * stage, stage_par ^ 1u, abort_flag, prm.status, 3);
                        if (!ok) break;
                        const bool linear = (flags & CLEAR_STEP_LINEAR) != 0;
                        const int x = k ? (t ? st.x1 : st.x0) : (t ? st_prev.x1 : st_prev.x0);
                        const int y = k ? (t ? st.y1 : st.y0) : (t ? st_prev.y1 : st_prev.y0);
                        const uint32_t bar = b_full0 + 8 * stage;
                        ptx::mbar_expect_tx(bar, kTileBytes);
                        ptx::tma_load_5d(sRing + stage * kTileBytes, &maps.m[(k ? kMapKImg : kMapVImg) + (linear ? 1 : 0)], bar, 0, x,
                                         linear ? 0 : y, 0, ref.bh);
                        ++n_loads;
                        if (++stage == kRing) {
                            stage = 0;
                            stage_par ^= 1u;
                        }
                    }
                    st_prev = st;
                    st = st_next;
                }
                if (!ok) break;
            }
            ctrl->copies[0] = n_q[0];
            ctrl->copies[1] = n_q[1];
            ctrl->copies[2] = n_loads;
        } else if ((warp == 1 || warp == 2) && ptx::elect_one()) {
            // ================= MMA issue: S_t = Q_t K^T, O_t += P_t V, one warp per query tile t ==============
            // S_t of a step comes in two halves of 64 keys.  The softmax warps take the second half first; P_t of the whole
            // step lies over the first half, so the second half is free as soon as its scores are in registers, and the
            // next step's is computed there while the exponentials of this one run.  What is left on the critical path of
            // a tile is P_t V and then the first half of the next Q_t K^T, over P_t (same thread, same pipe: P_t V has read
            // it by then), and meanwhile the softmax warps work on the second half.  (An MMA of 64 keys takes 48 clocks
            // where one of 128 takes 64: the tensor core works 25 % more, and waits far less.)
            // At 128 channels the two warps take turns with P_t V and the first halves, step by step: with the groups issued in
            // turn, tile 1's scores follow tile 0's by a group and its exponentials run under the other's MMAs.  Without: 1024px
            // 103 us against 99, 2048px 551 against 530.  (Passed on earlier, behind P_t V, or later, behind the second half,
            // where the pipe idles at every hand-over: 534 and 673 against 525, when it was that.)  At 64 channels, where the
            // MMAs take half, nothing is gained by keeping order: 67 x 120 in 208 us without turns, 215 with.
            // The tensor core holds about two MMAs ahead of the one it works on, some 150 clocks, and every barrier or
            // shuffle instruction of these warps spends 100 to 200 in the queue it shares with the exponentials of two
            // softmax warps: hence a warp per tile, the waits of one in the shadow of the other's MMAs (one warp for both
            // tiles: 560 us; a third one for the second halves: their MMAs get in the way of the critical ones, 552).
            // One elected lane walks the whole loop.  With the warp walking in step and a lane elected for each group, a vote
            // and two warp barriers stood between a wait's end and the first MMA (1024px: 106 us against 98.5, 2048px: 517
            // against 499, 8K: 8.40 ms against 8.24, in short runs at full clock, as the figures above).
            const int t = warp - 1;
            const int use_bit = t ? CLEAR_STEP_USE1 : CLEAR_STEP_USE0;
            constexpr uint32_t kDescHiK = ptx::smem_desc_hi_sw128(1024);  // 8-row groups are 1024 bytes apart
            const uint32_t tmem_S = tmem + t * 128, tmem_O = tmem + 256 + t * 128;
            const uint32_t b_full0 = ptx::smem_u32(&ctrl->kv_full[0]), b_empty0 = ptx::smem_u32(&ctrl->kv_empty[0]);
            const uint32_t b_p = ptx::smem_u32(&ctrl->p_ready[t]), b_read = ptx::smem_u32(&ctrl->sb_read[t]);
            constexpr bool kTurns = D == 128;
            const uint32_t b_turn = ptx::smem_u32(&ctrl->turn[t]), b_other = ptx::smem_u32(&ctrl->turn[t ^ 1]);
            const uint32_t v_lo0 = ptx::smem_desc_lo(sRing, kHalfBytes), k_lo0 = ptx::smem_desc_lo(sRing, 16);
            const uint32_t q_lo = ptx::smem_desc_lo(sQ + t * kTileBytes, 16);
            uint32_t n_it = 0;                           // items in which the query tile existed
            uint32_t p_par = 0, sb_par = 1;              // parities of the next P_t and of the next reading of the second half
            uint32_t turn_par = t ? 0u : 1u;             // tile 0 has the first turn
            uint32_t ring_stage = 0, ring_par = 0;       // next fill of the ring, in staging order
            bool ok = true;
            // A wait whose outcome is looked at once per group of MMAs.
            auto wait_lane = [&](uint32_t bar, uint32_t parity, int code) {
                if (ok) ok = wait_bar(bar, parity, abort_flag, prm.status, code);
            };
            // Both warps pass every fill of the ring in staging order and arrive once for it, after they have seen it: with
            // an MMA commit behind the MMAs that read the tile, or at once if they have no use for it.  So no phase can be
            // freed, and no warp lapped, before both have passed.
            auto take = [&]() -> uint32_t {
                const uint32_t st = ring_stage;
                wait_lane(b_full0 + 8 * st, ring_par, 4);
                const bool wrap = st == kRing - 1;
                ring_stage = wrap ? 0u : st + 1u;
                ring_par ^= wrap ? 1u : 0u;
                return st;
            };
            auto pass = [&]() {
                const uint32_t st = take();
                if (ok) ptx::mbar_arrive(b_empty0 + 8 * st);
            };
            // The K tiles, or the V tiles, of a step: this warp's one is returned, the other one (if any) passed.
            auto take_own = [&](int f) -> uint32_t {
                uint32_t own = 0;
                if (f & CLEAR_STEP_USE0) {
                    if (t == 0 || (f & CLEAR_STEP_SHARED)) own = take();
                    else pass();
                }
                if ((f & (CLEAR_STEP_USE1 | CLEAR_STEP_SHARED)) == CLEAR_STEP_USE1) {
                    if (t == 1) own = take();
                    else pass();
                }
                return own;
            };
            // S of 64 keys: 64 columns from D / 16 MMAs; the second half's keys are 64 rows, 8192 bytes, into the K tile.
            // Both operands K-major: 16 contraction channels are 32 bytes along a 128-byte row, the next 64 channels are
            // the tile's second half.
            auto issue_qk = [&](uint32_t k_st, uint32_t half) {
                const uint32_t k_lo = k_lo0 + k_st * (kTileBytes >> 4) + half * (8192 >> 4);
                ptx::mma_ss_c<false>(tmem_S + 64 * half, ptx::make_desc(q_lo, kDescHiK), ptx::make_desc(k_lo, kDescHiK), kIdescQK);
#pragma unroll
                for (int kk = 1; kk < D / 16; ++kk) {
                    const uint32_t off16 = ((kk >> 2) * kHalfBytes + (kk & 3) * 32) >> 4;
                    ptx::mma_ss_c<true>(tmem_S + 64 * half, ptx::make_desc(q_lo + off16, kDescHiK), ptx::make_desc(k_lo + off16, kDescHiK), kIdescQK);
                }
            };
            // The second half of S_t for the step whose K tile is in stage k_st, as soon as the one before has been read.
            auto issue_second_half = [&](uint32_t k_st) {
                wait_lane(b_read, sb_par, 12);
                sb_par ^= 1u;
                if (!ok) return;
                ptx::tc_fence_after();
                issue_qk(k_st, 1);
                ptx::tc_commit(ptx::smem_u32(&ctrl->sb_full[t]));
            };
#pragma unroll 1
            for (uint32_t k = 0; ok; ++k) {
                const uint32_t slot = k % kSchedDepth, use = k / kSchedDepth;
                wait_lane(ptx::smem_u32(&ctrl->sched_full[slot]), use & 1u, 5);
                if (!ok) break;
                const int g = ctrl->sched_item[slot];
                const int n_sides = ctrl->sched_rec[slot].n_sides;
                const int step_begin = ctrl->sched_rec[slot].step_begin;
                const int n = ctrl->sched_rec[slot].step_count;
                ptx::mbar_arrive(ptx::smem_u32(&ctrl->sched_empty[slot]));
                if (g >= total_items) break;
                const int *step_flags = &prm.steps[step_begin].flags;
                constexpr int kStepInts = sizeof(clear_pair_step_t) / sizeof(int);
                // the flags of the next two steps are on their way
                auto fetch_flags = [&](int s) { return s < n ? (int)ptx::ldg_u32(step_flags + s * kStepInts) : 0; };
                int pend = 0;            // flags of the step before (0: none)
                int flags = fetch_flags(0), flags_next = fetch_flags(1);
                uint32_t acc = 0;        // O_t holds something of this item
                const bool exists = t < n_sides;
                if (exists) wait_lane(ptx::smem_u32(&ctrl->q_full[t]), n_it & 1u, 6);
#pragma unroll 1
                for (int s = 0; s <= n && ok; ++s) {
                    // one step past the end: the last P_t V
                    const bool last = s == n;
                    const int flags_after = fetch_flags(s + 2);  // 0 past the end
                    const bool pv = (pend & use_bit) != 0, qk = (flags & use_bit) != 0;
                    const uint32_t k_st = take_own(flags);
                    if (qk) issue_second_half(k_st);
                    const uint32_t v_st = take_own(pend);
                    // the epilogue must have read the previous item's O_t out of tensor memory
                    if (pv && !acc) wait_lane(ptx::smem_u32(&ctrl->o_empty[t]), (n_it & 1u) ^ 1u, 8);
                    if (pv) {
                        wait_lane(b_p, p_par, 7);
                        p_par ^= 1u;
                    }
                    if (kTurns) {
                        wait_lane(b_turn, turn_par, 11);
                        turn_par ^= 1u;
                    }
                    if (!ok) break;
                    ptx::tc_fence_after();
                    if (pv) {
                        // P_t (bf16 pairs) in the first 64 columns of S_t, 16 keys = 8 columns; V MN-major, 16 keys are 16
                        // rows of 128 bytes = 2048 bytes
                        const uint32_t v_lo = v_lo0 + v_st * (kTileBytes >> 4);
                        ptx::mma_ts(tmem_O, tmem_S, ptx::make_desc(v_lo, kDescHiK), kIdescPV, acc);
#pragma unroll
                        for (int kk = 1; kk < 8; ++kk)
                            ptx::mma_ts_c<true>(tmem_O, tmem_S + kk * 8, ptx::make_desc(v_lo + kk * (2048 >> 4), kDescHiK), kIdescPV);
                    }
                    if (qk) {
                        issue_qk(k_st, 0);
                        ptx::tc_commit(ptx::smem_u32(&ctrl->sa_full[t]));
                    }
                    if (kTurns) ptx::mbar_arrive(b_other);  // the other tile's turn
                    if (qk) ptx::tc_commit(b_empty0 + 8 * k_st);
                    if (pv) ptx::tc_commit(b_empty0 + 8 * v_st);
                    // behind the item's last Q K^T the next Q_t may land; behind its last P V the output is complete
                    if (s == n - 1 && exists) ptx::tc_commit(ptx::smem_u32(&ctrl->q_empty[t]));
                    if (last && exists) ptx::tc_commit(ptx::smem_u32(&ctrl->o_full[t]));
                    if (pv) acc = 1u;
                    pend = flags;
                    flags = flags_next;
                    flags_next = flags_after;
                }
                if (exists) ++n_it;
            }
            if (*abort_flag) {
                // MMAs that were issued must retire before tensor memory is given back
                ptx::tc_commit(ptx::smem_u32(&ctrl->drain[t]));
                drain_bar(ptx::smem_u32(&ctrl->drain[t]), 0);
            }
        }
        __syncwarp();
    } else {
        // ================= softmax warps: thread r owns query row r (tensor-memory lane r) of its tile =====
        // Per step: S_t into registers, half by half, P = exp2(.) under the Eq. 3 mask as bf16 into tensor memory over
        // the first half of S_t, row sum; at the end of an item O_t / l -> bf16 -> global memory (or fp32 partial
        // results of split text rows).
        // What bounds a block: a step of both tiles takes about 3600 clocks, of which the exponentials of the two warps on a
        // scheduler are 2150 if nothing else runs and the MMAs 2560 (3050 with the copies, by a run without exponentials); the
        // rest is the chain between them, and the start and end of an item, some 7000 clocks, most of them for fetching
        // instructions that run once an item (about 16 clocks each).  So the code of an item's start and end is kept short:
        // the tiles' lists come ready from the host, the first step runs in the common loop with a reference taken beforehand,
        // and what is rare stands behind the loop (1024px 108.3 -> 103.0 us, 2048px 581 -> 552, 67 x 120 of 64 channels 230 ->
        // 209, against lists taken apart here, maximum passes in the first step and every case in line).
        ptx::setmaxnreg_inc<kRegsSoftmax>();
        const int t = (warp - 4) >> 2;  // query tile of the pair
        const int q4 = warp & 3;        // tensor-memory lane quadrant
        const int r = q4 * 32 + lane;   // query row of the tile
        const uint32_t tmem_S = tmem + ((uint32_t)(q4 * 32) << 16) + t * 128, tmem_O = tmem_S + 256;
        const float c = prm.scale_log2;
        const uint64_t c2 = ptx::pack2(c, c);
        const uint32_t b_sa = ptx::smem_u32(&ctrl->sa_full[t]), b_sb = ptx::smem_u32(&ctrl->sb_full[t]);
        const uint32_t b_p = ptx::smem_u32(&ctrl->p_ready[t]), b_read = ptx::smem_u32(&ctrl->sb_read[t]);
        // A wait that gives up leaves the warp in step: what follows runs on, on whatever there is, without waiting for or
        // telling anybody, up to the end of the item, where the warp looks.  (A vote behind every wait stood on the chain.)
        bool alive = true;
        auto wait_warp = [&](uint32_t bar, uint32_t parity, int code) {
            if (__builtin_expect(!ptx::mbar_try_wait_some(bar, parity, 128u, kWaitHintNs, alive), 0)) alive = wait_bar(bar, parity, abort_flag, prm.status, code);
            __syncwarp();
            ptx::tc_fence_after();
        };
        auto tell = [&](uint32_t bar) {
            ptx::tc_fence_before();
            __syncwarp();
            ptx::mbar_arrive_if(bar, lane == 0 && alive);
        };
        uint32_t par = 0;                  // parity of the tile's S barriers
        uint32_t o_par = 0;                // parity of the tile's results
#pragma unroll 1
        for (uint32_t k = 0;; ++k) {
            const uint32_t slot = k % kSchedDepth, use = k / kSchedDepth;
            if (alive) alive = wait_bar(ptx::smem_u32(&ctrl->sched_full[slot]), use & 1u, abort_flag, prm.status, 9);
            if (!__all_sync(0xffffffffu, alive)) break;
            if (ctrl->sched_item[slot] >= total_items) break;
            const clear_pair_item_t &item = ctrl->sched_rec[slot];   // the slot is given back at the end of the item
            if (t < item.n_sides) {
                const clear_pair_step_t *steps = prm.steps + item.step_begin;
                const int step_count = item.step_count;
                // grid position of this row's query (image tiles), and whether the row exists
                const bool is_text = item.kind == 1;
                const int q_y = (t ? item.qy1 : item.qy0) + (r >> 4), q_x = item.qx + (r & 15);
                const bool q_valid = is_text ? r < (t ? item.n_rows1 : item.n_rows0) : (q_y < prm.grid_h && q_x < prm.grid_w);

                // The steps this tile takes part in, a word each (0: none left), 32 at a time, one per lane, the 32 after them
                // fetched meanwhile; taken out of the lanes two steps ahead, and this row's mask words fetched one step ahead.
                // No latency is on the critical path, and the loads stay where they are written (left to the compiler, they
                // sank to their use).
                const uint32_t *words = prm.side_words + (size_t)t * prm.n_steps + item.step_begin + lane;
                auto fetch_words = [&](int at) { return at + lane < step_count ? ptx::ldg_u32(words + at) : 0u; };
                int at = 0;   // words taken
                uint32_t lanes = fetch_words(0), lanes_next = fetch_words(32);
                auto take_step = [&]() -> uint32_t {
                    if (__builtin_expect(at != 0 && (at & 31) == 0, 0)) {
                        lanes = lanes_next;
                        lanes_next = fetch_words(at + 32);
                    }
                    return __shfl_sync(0xffffffffu, lanes, at++ & 31);
                };
                const uint4 *mask_row = reinterpret_cast<const uint4 *>(prm.mask_table) + r;
                auto load_mask = [&](uint32_t w) -> uint4 {
                    uint4 m = make_uint4(0xffffffffu, 0xffffffffu, 0xffffffffu, 0xffffffffu);
                    if ((w & (kSideMasked | kSidePlain)) == (kSideMasked | kSidePlain)) m = ptx::ldg_u128(mask_row + ((w >> 2) & 0x3ffu) * 128u);
                    return m;
                };

                // P = 2^(S c - ref) with a reference per row that need not be the running maximum: P, the row sum and O
                // are floating-point numbers of full precision at any scale, so the reference only has to keep them
                // within range.  It is the maximum of the row's first tile; when a tile's row sum exceeds 2^16 the
                // reference is raised by a whole power of two, without a look at the maximum, and the row's P, sum and O are
                // scaled before P goes to the MMAs.  No maximum pass, then, on any other tile, and the scores die as their P is
                // formed.  A row sum beyond 2^64 means scores 64 powers of two above everything seen before; the warp then
                // computes its scores again, from global memory, before anybody has used P, and takes the rest of the item's
                // steps with maximum passes.
                float ref = -INFINITY, l = 0.f;  // reference of the row's exponents (log2 units) and row sum
                bool careful = false;            // maximum passes up to the end of the item
                bool first = true, exact = true; // this step has one
                // At 128 channels the first tile is looked at once: its own step runs against the maxima just found, and where
                // the steps behind it want maximum passes it is alone in the common loop.  1024px, Q times 20: 169 us with a
                // second look, 165 without.  At 64 channels that costs the common loop more than it saves (67 x 120: 218 us
                // with a second look, 222 without; Q times 20 355 and 351).
                constexpr bool kLookOnce = D == 128;
                uint32_t go_on = kSidePlain;     // bits that a step has to have to follow in the common loop
                uint32_t w = take_step(), w1 = take_step(), w2;
                uint4 mw = load_mask(w), mw1;    // bit j of word i = key 32 i + j allowed
                // The common steps run in a loop of their own, with what is rare outside of it.
#pragma unroll 1
                while (w != 0u) {
                    if (w & kSideRare) mw = special_mask(prm, steps + (w >> 16), t, q_valid, q_y, q_x);
                    if (first && !(w & kSideMasked)) {
                        wait_warp(b_sb, par, 10);
                        wait_warp(b_sa, par, 13);
                        const RowTop top = first_top(tmem_S);
                        ref = top.most * c;
                        careful = __any_sync(0xffffffffu, (top.most - top.least) * c > kWideStep);
                        exact = careful || __any_sync(0xffffffffu, ref == -INFINITY && q_valid);
                        if (kLookOnce && exact) {
                            exact = false;
                            go_on = 0u;
                        }
                    }
                    float tile_sum;
                    if (!exact) {
                        const float mc = (ref == -INFINITY) ? 0.f : ref;
                        const uint64_t nmc2 = ptx::pack2(-mc, -mc);
                        first = false;
                        bool over;
#pragma unroll 1
                        for (;;) {
                            // The second half comes first: its P waits in registers for the first half's scores to be read,
                            // over which P of the whole step lies.
                            uint64_t lsum[2] = {0ull, 0ull};
                            uint32_t sv[2][32], pk[2][16];
                            wait_warp(b_sb, par, 10);
                            ptx::tmem_ld32(tmem_S + 64, sv[0]);
                            ptx::tmem_ld32(tmem_S + 96, sv[1]);
                            ptx::tmem_wait_ld();
                            tell(b_read);
                            mw1 = load_mask(w1);
                            w2 = take_step();
                            if (w & kSideMasked) {
                                exp_chunk<true>(sv[0], mw.z, c2, nmc2, lsum, pk[0]);
                                exp_chunk<true>(sv[1], mw.w, c2, nmc2, lsum, pk[1]);
                            } else {
                                exp_chunk<false>(sv[0], 0u, c2, nmc2, lsum, pk[0]);
                                exp_chunk<false>(sv[1], 0u, c2, nmc2, lsum, pk[1]);
                            }
                            // Once the first half of S_t is complete, so is P_t V of the step before (same thread, same pipe,
                            // issued earlier).
                            wait_warp(b_sa, par, 13);
                            ptx::tmem_ld32(tmem_S, sv[0]);
                            ptx::tmem_ld32(tmem_S + 32, sv[1]);
                            ptx::tmem_wait_ld();
                            ptx::tmem_st16(tmem_S + 32, pk[0]);
                            ptx::tmem_st16(tmem_S + 48, pk[1]);
                            if (w & kSideMasked) {
                                exp_chunk<true>(sv[0], mw.x, c2, nmc2, lsum, pk[0]);
                                ptx::tmem_st16(tmem_S, pk[0]);
                                exp_chunk<true>(sv[1], mw.y, c2, nmc2, lsum, pk[1]);
                                ptx::tmem_st16(tmem_S + 16, pk[1]);
                            } else {
                                exp_chunk<false>(sv[0], 0u, c2, nmc2, lsum, pk[0]);
                                ptx::tmem_st16(tmem_S, pk[0]);
                                exp_chunk<false>(sv[1], 0u, c2, nmc2, lsum, pk[1]);
                                ptx::tmem_st16(tmem_S + 16, pk[1]);
                            }
                            tile_sum = sum4(lsum);
                            // P_t must be in tensor memory before the MMA thread is told
                            ptx::tmem_wait_st();
                            over = __any_sync(0xffffffffu, tile_sum > kBumpSum);
                            if (__builtin_expect(over, 0)) break;
                            tell(b_p);
                            l += tile_sum;
                            par ^= 1u;
                            w = w1;
                            w1 = w2;
                            mw = mw1;
                            if (__builtin_expect(!(w & go_on), 0)) break;
                        }
                        if (!over) {   // none left, one with a maximum pass, or one whose mask is to be worked out
                            exact = go_on == 0u;
                            go_on = kSidePlain;
                            continue;
                        }
                    } else {
                        mw1 = load_mask(w1);
                        w2 = take_step();
                        wait_warp(b_sb, par, 10);
                        wait_warp(b_sa, par, 13);
                        const RowState rs = exact_step<D>(tmem_S, tmem_O, mw, c, ref, l, first);
                        ref = rs.ref;
                        l = rs.l;
                        tile_sum = fabsf(rs.tile_sum);
                        careful = careful || __any_sync(0xffffffffu, rs.tile_sum < 0.f);
                        exact = careful || __any_sync(0xffffffffu, ref == -INFINITY && q_valid);
                        first = false;
                        tell(b_read);
                    }
                    if (!careful && __any_sync(0xffffffffu, tile_sum > kBumpSum)) {
                        if (__any_sync(0xffffffffu, tile_sum > kMaxTileSum)) {
                            careful = exact = true;
                            const int2 org = load_side_origin(steps + (w >> 16), t);
                            const long long q_tok = is_text ? (long long)item.qx + t * 128 + r : prm.n_text + (long long)q_y * prm.grid_w + q_x;
                            const RowState rs = rescue_step<D>(prm, tmem_S, tmem_O, mw, c, ref, l, (long long)ctrl->sched_bh[slot] * prm.n_tokens,
                                                               q_valid ? q_tok : -1, org, (__ldg(&steps[w >> 16].flags) & CLEAR_STEP_LINEAR) != 0);
                            ref = rs.ref;
                            l = rs.l;
                            tile_sum = rs.tile_sum;
                        } else {
                            const float bump = tile_sum > kBumpSum ? (float)((int)((__float_as_uint(tile_sum) >> 23) & 0xffu) - 127) : 0.f;
                            const float alpha = ptx::ex2(-bump);
                            rescale_rows<D>(tmem_O, alpha);   // at rest; in an item's first step nobody looks at it
                            rescale_p(tmem_S, alpha);
                            ref += bump;
                            l *= alpha;
                            tile_sum *= alpha;
                        }
                    }
                    l += tile_sum;
                    ptx::tmem_wait_st();
                    tell(b_p);
                    par ^= 1u;
                    w = w1;
                    w1 = w2;
                    mw = mw1;
                }

                // ---- epilogue: the last P_t V has retired once o_full completes; O_t / l -> global memory -----
                if (alive) alive = wait_bar(ptx::smem_u32(&ctrl->o_full[t]), o_par, abort_flag, prm.status, 14);
                if (!__all_sync(0xffffffffu, alive)) break;
                o_par ^= 1u;
                ptx::tc_fence_after();
                store_tile<D>(prm, tmem + 256 + t * 128, ptx::smem_u32(&ctrl->o_empty[t]), item.qx + (is_text ? t * 128 : 0), t ? item.qy1 : item.qy0,
                              is_text ? (t ? item.n_rows1 : item.n_rows0) : -1, t ? item.partial_slot1 : item.partial_slot0,
                              ctrl->sched_bh[slot], ref, l);
            }
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&ctrl->sched_empty[slot]));
        }
    }

    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem, kTmemCols);
    }
    if (tid == 0) {
        if (*abort_flag) {
            // leave no copy in flight: whatever was issued must land before the block exits (looked at only now: the block
            // may give up after the loader has issued its last copy)
            for (int t = 0; t < 2; ++t)
                if (ctrl->copies[t] > 0) drain_bar(ptx::smem_u32(&ctrl->q_full[t]), (ctrl->copies[t] - 1) & 1u);
            for (uint32_t j = 0, n = ctrl->copies[2]; j < kRing && j < n; ++j)
                drain_bar(ptx::smem_u32(&ctrl->kv_full[(n - 1 - j) % kRing]), ((n - 1 - j) / kRing) & 1u);
        }
        // the last block to finish puts the queue back to zero for the next launch
        const int done = atomicAdd(prm.status + 2, 1);
        if (done == (int)gridDim.x - 1) close_launch(prm.status);
    }
}

// ---- host side: tensor maps and launch ---------------------------------------------------------
// Image part of a tensor as [BH][half][grid_h][grid_w][64], runs of tokens as [BH][half][1][tokens][64]; the text
// prefix of q ends at n_text (rows past it read as zero), the token sequence of k, v at N.
int build_maps(const clear_plan &p, const void *q, const void *k, const void *v)
{
    const Shape &s = p.shape;
    const uint64_t gw = (uint64_t)s.grid_w, gh = (uint64_t)s.grid_h, T = (uint64_t)s.n_text;
    const uint64_t N = T + gw * gh, BH = (uint64_t)s.B * s.H, halves = (uint64_t)s.head_dim / 64;
    const uint64_t row_b = (uint64_t)s.head_dim * 2;
    CUtensorMap *tm = reinterpret_cast<CUtensorMap *>(p.tm_storage);
    const void *ptrs[3] = {q, k, v};
    const uint64_t dims_img[5] = {64, gw, gh, halves, BH}, str_img[4] = {row_b, gw * row_b, 128, N * row_b};
    const uint32_t box_img[5] = {64, (uint32_t)kTileW, (uint32_t)kTileH, (uint32_t)halves, 1};
    const uint64_t str_lin[4] = {row_b, N * row_b, 128, N * row_b};
    const uint32_t box_lin[5] = {64, (uint32_t)kTileTokens, 1, (uint32_t)halves, 1};
    for (int t = 0; t < 3; ++t) {
        const uint64_t dims_lin[5] = {64, t == 0 ? std::max<uint64_t>(T, 1) : N, 1, halves, BH};
        if (!encode_bf16_map(&tm[2 * t], static_cast<const char *>(ptrs[t]) + T * row_b, 5, dims_img, str_img, box_img) ||
            !encode_bf16_map(&tm[2 * t + 1], ptrs[t], 5, dims_lin, str_lin, box_lin))
            return CLEAR_ERR_CUDA;
        p.tm_ptrs[t] = ptrs[t];
    }
    p.tm_ptrs[3] = nullptr;
    p.tm_valid = true;
    return CLEAR_OK;
}

struct DeviceInfo {
    bool known = false;
    int n_sm = 0;
    bool configured[2] = {false, false};
};
DeviceInfo g_dev[64];
std::mutex g_dev_mutex;

template <int D>
int launch_variant(const clear_plan &p, const WsMaps &maps, const WsParams &prm, cudaStream_t stream)
{
    constexpr size_t kSmem = (size_t)(2 + kRing) * (D / 64) * 16384 + sizeof(Ctrl);
    static_assert(kSmem <= 232448, "shared memory of one block");
    int n_sm = 0;
    {
        std::lock_guard<std::mutex> lock(g_dev_mutex);
        if (p.device < 0 || p.device >= 64) return CLEAR_ERR_UNSUPPORTED;
        DeviceInfo &di = g_dev[p.device];
        if (!di.known) {
            CLEAR_CUDA_TRY(cudaDeviceGetAttribute(&di.n_sm, cudaDevAttrMultiProcessorCount, p.device));
            di.known = true;
        }
        if (!di.configured[D == 128]) {
            CLEAR_CUDA_TRY(cudaFuncSetAttribute(clear_ws_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem));
            di.configured[D == 128] = true;
        }
        n_sm = di.n_sm;
    }
    const long long total = (long long)prm.n_items * prm.n_bh;
    const unsigned grid = (unsigned)std::min<long long>(n_sm, total);
    clear_ws_kernel<D><<<grid, kWsThreads, kSmem, stream>>>(maps, prm);
    CLEAR_CUDA_TRY(cudaGetLastError());
    return launch_text_combine(p, prm.out, stream);
}

}  // namespace

int launch_ws(const clear_plan &p, const void *q, const void *k, const void *v, void *out, float scale, cudaStream_t stream)
{
    if (!(scale > 0.f)) return CLEAR_ERR_UNSUPPORTED;
    const long long total = (long long)p.sch.pair_items.size() * p.shape.B * p.shape.H;
    if (total <= 0 || total >= (1ll << 30)) return CLEAR_ERR_UNSUPPORTED;
    WsMaps maps;
    {
        std::lock_guard<std::mutex> lock(p.tm_mutex);
        if (!(p.tm_valid && p.tm_ptrs[0] == q && p.tm_ptrs[1] == k && p.tm_ptrs[2] == v)) {
            int rc = build_maps(p, q, k, v);
            if (rc != CLEAR_OK) {
                p.tm_valid = false;
                return rc;
            }
        }
        std::memcpy(&maps, p.tm_storage, sizeof(maps));
    }
    WsParams prm{};
    prm.items = p.d_pair_items;
    prm.steps = p.d_pair_steps;
    prm.half_width = p.d_half_width;
    prm.mask_table = p.d_mask_table;
    prm.side_words = p.d_mask_table + p.sch.mask_table.size();
    prm.n_steps = (int)p.sch.pair_steps.size();
    prm.n_half_width = (int)p.sch.half_width.size();
    prm.grid_h = p.shape.grid_h;
    prm.grid_w = p.shape.grid_w;
    prm.n_text = p.shape.n_text;
    prm.n_tokens = (long long)p.shape.n_text + (long long)p.shape.grid_h * p.shape.grid_w;
    prm.n_items = (int)p.sch.pair_items.size();
    prm.n_text_items = p.sch.n_text_pair_items;
    prm.n_bh = p.shape.B * p.shape.H;
    prm.scale_log2 = scale * 1.4426950408889634f;
    prm.partial_o = p.d_partial_o;
    prm.partial_ml = p.d_partial_ml;
    prm.n_partial_slots = p.sch.n_partial_slots;
    prm.q = static_cast<const __nv_bfloat16 *>(q);
    prm.k = static_cast<const __nv_bfloat16 *>(k);
    prm.out = static_cast<__nv_bfloat16 *>(out);
    prm.status = p.d_status;
    if (p.shape.head_dim == 128) return launch_variant<128>(p, maps, prm, stream);
    if (p.shape.head_dim == 64) return launch_variant<64>(p, maps, prm, stream);
    return CLEAR_ERR_UNSUPPORTED;
}

}  // namespace clear
