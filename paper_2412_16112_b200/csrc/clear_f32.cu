// CLEAR attention forward on the CUDA cores, fp32 arithmetic throughout, as a tiled kernel: 64 queries against 64
// keys at a time from shared memory (f32_tile.cuh).
//
// Serves fp32 tensors (where tensor-core input rounding would break a 1e-5 agreement), bf16 tensors of head sizes the
// tensor-core kernels do not take, and non-positive scales, under the windows around the query (disc, square).
//
// Up to 128 channels (padded to 64 or 128) a block is four warps with 16 whole rows each, or eight with 8
// (clear_f32_rows_kernel).  256 threads with 4 x 4 results each (clear_f32_tile_kernel) remain above, where the accumulators
// of 16 rows would not fit a warp's registers, and for bf16 tensors where blocks share an SM (launch_rows).
// What bounds it: the fp32 multiply-add units (2 x 64 x 64 x DP multiply-adds a step, DP = the head size rounded up
// to 64, 128 or 256), and in the scores the reads from shared memory beside them.  1024 px, radius 8, 24 heads of 128: 2034 us
// with 4 x 4 results a thread (shared memory at 77 % of its peak, multiply-adds at 64 %), 1734 us with whole rows (64 % and
// 70 %): about 780 for the scores and 550 for the weights times V, each of which is 525 of multiply-adds, 130 for the copies
// and 100 for the softmax, by runs without the one or the other.
// The keys are those of the union of the tile's windows and no others: rows are gathered run by
// run, 64 at a time, so a step is only ever short at the end of the list.  An 8 x 8 patch is the split that wastes
// least at the paper's radii: at r = 8 a patch walks 452 + n_text keys for windows of 193.
// Two blocks share an SM (DP <= 128, except with 8 rows to a warp): one computes while the other waits for its rows.
// A problem too small to give every SM a tile cuts the lists over a cluster of up to 8 blocks, which merge their
// partial softmax through distributed shared memory in a fixed order: no workspace, no second launch.
#include <cuda_bf16.h>
#include <math_constants.h>

#include <algorithm>
#include <cmath>

#include "clear_internal.hpp"
#include "f32_tile.cuh"

namespace clear {
namespace {

using namespace f32tile;
namespace cg = cooperative_groups;

struct F32Params {
    Geometry g;
    const void *q, *k, *v;
    void *out;
    int n_split;
    float scale;
};

template <int DP> constexpr size_t forward_smem()
{
    return 3 * (size_t)kRows * kStride<DP> * sizeof(float) + 2 * sizeof(KeyTile) + 2 * kRows * sizeof(float) + 64 * sizeof(int);
}

// Row r of the block's tile by itself (one warp).  (The code alone cost the kernel with 4 x 4 results a thread 1.6 % at 1024 px, 2.00 ->
// 2.03 ms; as a function that is not inlined, or with addresses of its own, it cost as much.)
template <typename T, int DP>
__device__ __forceinline__ void redo_row(const F32Params &p, int r)
{
    const TileRef tile = tile_of((int)(blockIdx.x / (unsigned)p.n_split), p.g);
    const KeyRuns runs = runs_of(tile, p.g);
    int qy, qx;
    const int tok = tile_token(tile, r, p.g, qy, qx);
    if (tok < 0) return;
    const long long base = (long long)tile.bh * runs.n_tokens * p.g.d;
    const T *k = static_cast<const T *>(p.k) + base, *v = static_cast<const T *>(p.v) + base;
    LaneRow<DP> q, x, o;
    q.load(static_cast<const T *>(p.q) + base + (long long)tok * p.g.d, p.g.d);
    o.zero();
    float m = -CUDART_INF_F, l = 0.f;
    for_each_seen(runs, qy, qx, [&](int t) {
        x.load(k + (long long)t * p.g.d, p.g.d);
        const float s = q.dot(x) * p.scale;
        const float m_new = fmaxf(m, s), m_ref = m_new == -CUDART_INF_F ? 0.f : m_new;
        const float alpha = expf(m - m_ref), e = expf(s - m_ref);
        l = fmaf(l, alpha, e);
#pragma unroll
        for (int c = 0; c < DP / 32; ++c) o.c[c] *= alpha;
        x.load(v + (long long)t * p.g.d, p.g.d);
        o.add(e, x);
        m = m_new;
    });
    o.store(static_cast<T *>(p.out) + base + (long long)tok * p.g.d, p.g.d, l == 0.f ? 0.f : 1.f / l);
}

// Rows of the block's tile that came out non-finite, each by a warp of its NT threads.
template <typename T, int DP, int NT>
__device__ __forceinline__ void redo_bad(const F32Params &p, const int *bad)
{
#pragma unroll 1
    for (int r = (int)threadIdx.x >> 5; r < kRows; r += NT / 32)
        if (bad[r] != 0) redo_row<T, DP>(p, r);
}

// The merge over a cluster: every block has left its un-normalised rows, references and sums in its own shared memory, and
// finishes 64 / n_split rows from everybody's, in the order of the ranks.  Marks rows that are not finite; false if there is one.
// The block stays until the cluster has met again.
template <typename T, int DP, int NT>
__device__ __forceinline__ bool merge_rows(const F32Params &p, const TileRef &tile, int part, float *sM, float *sL, float *sO, T *out, int *bad)
{
    cg::cluster_group cluster = cg::this_cluster();
    cluster.sync();
    bool all_finite = true;
    const int rows = kRows / p.n_split;
    for (int e = threadIdx.x; e < rows * (DP / 4); e += NT) {
        const int r = part * rows + e / (DP / 4), ch = e % (DP / 4) * 4;
        int qy, qx;
        const long long tok = tile_token(tile, r, p.g, qy, qx);
        float mx = -CUDART_INF_F;
        for (int c = 0; c < p.n_split; ++c) mx = fmaxf(mx, cluster.map_shared_rank(sM, c)[r]);
        if (mx == -CUDART_INF_F) mx = 0.f;
        float sum = 0.f;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int c = 0; c < p.n_split; ++c) {
            const float f = expf(cluster.map_shared_rank(sM, c)[r] - mx);
            sum = fmaf(f, cluster.map_shared_rank(sL, c)[r], sum);
            const float4 x = *reinterpret_cast<const float4 *>(cluster.map_shared_rank(sO, c) + r * kStride<DP> + ch);
            acc.x = fmaf(f, x.x, acc.x);
            acc.y = fmaf(f, x.y, acc.y);
            acc.z = fmaf(f, x.z, acc.z);
            acc.w = fmaf(f, x.w, acc.w);
        }
        const float inv = sum > 0.f ? 1.f / sum : 0.f;
        acc.x *= inv; acc.y *= inv; acc.z *= inv; acc.w *= inv;
        if (tok >= 0 && ch < p.g.d) store4(out + tok * p.g.d + ch, acc);
        if (!finite4(acc)) {
            bad[r] = 1;
            all_finite = false;
        }
    }
    return all_finite;
}

template <typename T, int DP>
__global__ void __launch_bounds__(kThreads, DP <= 128 ? 2 : 1)
clear_f32_tile_kernel(const F32Params p)
{
    extern __shared__ __align__(16) uint8_t smem[];
    float *sQ = reinterpret_cast<float *>(smem), *sK = sQ + kRows * kStride<DP>, *sV = sK + kRows * kStride<DP>;
    float *sP = sK;   // the weights take the place of the keys once the scores are in registers
    KeyTile *keys = reinterpret_cast<KeyTile *>(sV + kRows * kStride<DP>);
    float *sM = reinterpret_cast<float *>(keys + 2), *sL = sM + kRows;
    int *red = reinterpret_cast<int *>(sL + kRows);

    const int tid = threadIdx.x, ty = (tid >> 5) * 2 + ((tid >> 4) & 1), tx = tid & 15;
    const int part = (int)(blockIdx.x % (unsigned)p.n_split);   // rank in the cluster
    const TileRef tile = tile_of((int)(blockIdx.x / (unsigned)p.n_split), p.g);
    const KeyRuns runs = runs_of(tile, p.g);
    const long long base = (long long)tile.bh * runs.n_tokens * p.g.d;
    const T *q = static_cast<const T *>(p.q) + base, *k = static_cast<const T *>(p.k) + base,
            *v = static_cast<const T *>(p.v) + base;

    // this block's share of the list: whole steps of 64 keys
    const int n_steps_all = (list_length(runs, red) + kRows - 1) / kRows;
    const int per = (n_steps_all + p.n_split - 1) / p.n_split;
    const int step0 = min(part * per, n_steps_all), n_steps = min(per, n_steps_all - step0);
    KeyCursor cur;
    if (tid < kRows) {
        cur.start(runs);
        cur.advance(runs, step0 * kRows + tid);
        int qy, qx;
        keys[1].token[tid] = tile_token(tile, tid, p.g, qy, qx);
    }
    fill_key_tile(keys[0], cur, runs, n_steps > 0);
    __syncthreads();
    load_rows<T, DP>(sQ, q, keys[1].token, p.g.d);

    int q_y[4], q_x[4];
    long long q_tok[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) q_tok[i] = tile_token(tile, ty + 16 * i, p.g, q_y[i], q_x[i]);

    uint64_t o[4][DP / 64][2];
    zero_acc<DP>(o);
    float m[4], l[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        m[i] = -CUDART_INF_F;
        l[i] = 0.f;
    }

    for (int s = 0; s < n_steps; ++s) {
        const KeyTile &kt = keys[s & 1];
        load_rows<T, DP>(sK, k, kt.token, p.g.d);
        load_rows<T, DP>(sV, v, kt.token, p.g.d);
        cp_async_wait<1>();   // Q and K are here
        __syncthreads();
        if (s + 1 < n_steps) fill_key_tile(keys[(s + 1) & 1], cur, runs, true);

        float w[4][4];
        tile_dot<DP>(sQ, sK, ty, tx, w);
        __syncthreads();      // every warp is done with the keys: the weights may land on them

        // online softmax; a row's 64 scores sit in 16 lanes of one warp
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float mx = -CUDART_INF_F;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int c = tx + 16 * j;
                const bool on = kt.token[c] >= 0 && sees(runs, q_y[i], q_x[i], kt.ky[c], kt.kx[c]);
                w[i][j] = on ? w[i][j] * p.scale : -CUDART_INF_F;
                mx = fmaxf(mx, w[i][j]);
            }
            const float m_new = fmaxf(m[i], row_max16(mx));
            const float m_ref = m_new == -CUDART_INF_F ? 0.f : m_new;
            const float alpha = expf(m[i] - m_ref);   // m = -inf: 0
            m[i] = m_new;
            l[i] *= alpha;
            const uint64_t a2 = ptx::pack2(alpha, alpha);
#pragma unroll
            for (int c = 0; c < DP / 64; ++c) {
                o[i][c][0] = ptx::mul2(o[i][c][0], a2);
                o[i][c][1] = ptx::mul2(o[i][c][1], a2);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float e = expf(w[i][j] - m_ref);
                l[i] += e;
                sP[(ty + 16 * i) * kPStride + tx + 16 * j] = e;
            }
        }
        cp_async_wait<0>();
        __syncthreads();      // V has landed for everybody, and the weights are written
        tile_accumulate<DP>(sP, sV, ty, tx, o);
        __syncthreads();      // before the next rows overwrite K, V
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) l[i] = row_sum16(l[i]);

    // rows that came out non-finite are taken again, each by a warp; `bad` lies over the list lengths, which are done with
    int *bad = red;
    if (tid < kRows) bad[tid] = 0;
    __syncthreads();

    T *out = static_cast<T *>(p.out) + base;
    bool all_finite = true;
    if (p.n_split == 1) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            // a query sees itself or the text keys: l > 0 for every row that exists
            const float inv = l[i] > 0.f ? 1.f / l[i] : 0.f;
#pragma unroll
            for (int c = 0; c < DP / 64; ++c) {
                const int ch = 64 * c + 4 * tx;
                const float4 x = acc_float4(o[i][c], inv);
                if (q_tok[i] >= 0 && ch < p.g.d) store4(out + q_tok[i] * p.g.d + ch, x);
                if (!finite4(x)) {
                    bad[ty + 16 * i] = 1;
                    all_finite = false;
                }
            }
        }
        if (__syncthreads_or(!all_finite)) redo_bad<T, DP, kThreads>(p, bad);
        return;
    }

    cg::cluster_group cluster = cg::this_cluster();
    cp_async_wait<0>();
    __syncthreads();
    acc_to_rows<DP>(o, sV, ty, tx);
    if (tx == 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            sM[ty + 16 * i] = m[i];
            sL[ty + 16 * i] = l[i];
        }
    }
    all_finite = merge_rows<T, DP, kThreads>(p, tile, part, sM, sL, sV, out, bad);
    if (__syncthreads_or(!all_finite)) redo_bad<T, DP, kThreads>(p, bad);
    cluster.sync();   // nobody leaves while its rows are being read
}

// The same with a warp to R whole rows, for up to 128 channels: 16, or 8 where every block has an SM to itself (launch_rows).
// A score this far above its row's reference moves it.  The further off a reference may lie the fewer steps pay for a move (sixteen
// maxima over the lanes), but s - m is rounded at its own size, and so is the weight: with 16 the result's error against 64 bits is
// up to 5 % larger than against the maximum (keys whose scores climb by 4 to 8 a step), with 2 it is the same.  1024 px: 1739 us
// with 16, 4 or 2, 1757 with 1, 1794 with the maximum itself.
constexpr float kMaxExponent = 2.f;
template <int R> constexpr int kRowThreads = 32 * kRows / R;

// Shared memory: Q, V, then the keys, whose place the weights take once the scores are in registers (with 64 channels they are
// longer than the keys), the key lists, row values.
template <int DP, int R> constexpr size_t kRowsLists =
    (2 * kRows * kStride<DP> + std::max(kStride<DP>, kRows / R * kPairStride<R>) * kRows) * sizeof(float);
template <int DP, int R> constexpr size_t kRowsSmem = kRowsLists<DP, R> + 2 * sizeof(KeyTile) + 2 * kRows * sizeof(float) + 64 * sizeof(int);

template <typename T, int DP, int R>
__global__ void __launch_bounds__(kRowThreads<R>, R == 16 ? 2 : 1)
clear_f32_rows_kernel(const F32Params p)
{
    constexpr int C = DP / 32;
    extern __shared__ __align__(16) uint8_t smem[];
    float *sQ = reinterpret_cast<float *>(smem), *sV = sQ + kRows * kStride<DP>, *sK = sV + kRows * kStride<DP>;
    KeyTile *keys = reinterpret_cast<KeyTile *>(smem + kRowsLists<DP, R>);
    float *sM = reinterpret_cast<float *>(keys + 2), *sL = sM + kRows;
    int *red = reinterpret_cast<int *>(sL + kRows);

    const int tid = threadIdx.x, lane = tid & 31, row0 = (tid >> 5) * R;
    float *sP = sK + (tid >> 5) * kRows * kPairStride<R>;   // the warp's weights
    const int part = (int)(blockIdx.x % (unsigned)p.n_split);   // rank in the cluster
    const TileRef tile = tile_of((int)(blockIdx.x / (unsigned)p.n_split), p.g);
    const KeyRuns runs = runs_of(tile, p.g);
    const long long base = (long long)tile.bh * runs.n_tokens * p.g.d;
    const T *q = static_cast<const T *>(p.q) + base, *k = static_cast<const T *>(p.k) + base,
            *v = static_cast<const T *>(p.v) + base;

    // this block's share of the list: whole steps of 64 keys
    const int n_steps_all = (list_length<kRowThreads<R>>(runs, red) + kRows - 1) / kRows;
    const int per = (n_steps_all + p.n_split - 1) / p.n_split;
    const int step0 = min(part * per, n_steps_all), n_steps = min(per, n_steps_all - step0);
    KeyCursor cur;
    if (tid < kRows) {
        cur.start(runs);
        cur.advance(runs, step0 * kRows + tid);
        int qy, qx;
        keys[1].token[tid] = tile_token(tile, tid, p.g, qy, qx);
    }
    fill_key_tile(keys[0], cur, runs, n_steps > 0);
    __syncthreads();
    load_rows<T, DP, kRowThreads<R>>(sQ, q, keys[1].token, p.g.d);

    uint64_t o[R / 2][C];
    float m[R], l[R];   // per row its reference; of its sum the lane's share
#pragma unroll
    for (int i = 0; i < R / 2; ++i)
#pragma unroll
        for (int c = 0; c < C; ++c) o[i][c] = 0ull;
#pragma unroll
    for (int i = 0; i < R; ++i) {
        m[i] = -CUDART_INF_F;
        l[i] = 0.f;
    }

    for (int s = 0; s < n_steps; ++s) {
        const KeyTile &kt = keys[s & 1];
        load_rows<T, DP, kRowThreads<R>>(sK, k, kt.token, p.g.d);
        load_rows<T, DP, kRowThreads<R>>(sV, v, kt.token, p.g.d);
        uint32_t on[2];   // rows that see the lane's keys
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int c = lane + 32 * j;
            on[j] = kt.token[c] >= 0 ? seen_by<R>(runs, tile, p.g, row0, kt.ky[c], kt.kx[c]) : 0u;
        }
        cp_async_wait<1>();   // Q and K are here
        __syncthreads();
        if (s + 1 < n_steps) fill_key_tile(keys[(s + 1) & 1], cur, runs, true);

        float w[R][2];
        warp_dot<DP>(sQ + row0 * kStride<DP>, sK, lane, w);
        __syncthreads();      // every warp is done with the keys: the weights may land on them

        // Softmax against a reference per row that is moved only when a score lies far above it (and by the first scores that
        // a row has): no maximum over the lanes and no scaling in the common step.
        float far = -CUDART_INF_F;
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                w[i][j] = ((on[j] >> i) & 1u) ? w[i][j] * p.scale : -CUDART_INF_F;
                far = fmaxf(far, w[i][j] - m[i]);   // (-inf minus -inf is a NaN, which fmaxf passes over)
            }
        if (__any_sync(0xffffffffu, far > kMaxExponent)) {
#pragma unroll
            for (int i = 0; i < R; i += 2) {
                float alpha[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    float mx = fmaxf(w[i + u][0], w[i + u][1]);
#pragma unroll
                    for (int x = 16; x > 0; x >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, x));
                    const float m_new = fmaxf(m[i + u], mx);
                    alpha[u] = expf(m[i + u] - (m_new == -CUDART_INF_F ? 0.f : m_new));   // m = -inf: 0
                    m[i + u] = m_new;
                    l[i + u] *= alpha[u];
                }
                const uint64_t a2 = ptx::pack2(alpha[0], alpha[1]);
#pragma unroll
                for (int c = 0; c < C; ++c) o[i >> 1][c] = ptx::mul2(o[i >> 1][c], a2);
            }
        }
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int i = 0; i < R; i += 4) {
                float e[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    e[u] = expf(w[i + u][j] - (m[i + u] == -CUDART_INF_F ? 0.f : m[i + u]));
                    l[i + u] += e[u];
                }
                *reinterpret_cast<float4 *>(sP + (lane + 32 * j) * kPairStride<R> + i) = make_float4(e[0], e[1], e[2], e[3]);
            }
        cp_async_wait<0>();
        __syncthreads();      // V has landed for everybody, and the weights are written
        warp_accumulate<DP, R>(sP, sV, lane, o);
        __syncthreads();      // before the next rows overwrite K, V
    }
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int x = 16; x > 0; x >>= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], x);

    // rows that came out non-finite are taken again, each by a warp; `bad` lies over the list lengths, which are done with
    int *bad = red;
    if (tid < kRows) bad[tid] = 0;
    __syncthreads();

    T *out = static_cast<T *>(p.out) + base;
    const int ch = C * lane;
    bool all_finite = true;
    if (p.n_split == 1) {
#pragma unroll
        for (int i = 0; i < R; ++i) {
            // a query sees itself or the text keys: l > 0 for every row that exists
            const float inv = l[i] > 0.f ? 1.f / l[i] : 0.f;
            int qy, qx;
            const long long tok = tile_token(tile, row0 + i, p.g, qy, qx);
            float x[C];
            acc_row(o, i, x);
            bool fine = true;
#pragma unroll
            for (int c = 0; c < C; ++c) {
                x[c] *= inv;
                fine = fine && fabsf(x[c]) <= CUDART_MAX_NORMAL_F;
            }
            if (tok >= 0 && ch < p.g.d) store_channels(out + tok * p.g.d + ch, x);
            if (!fine) {
                bad[row0 + i] = 1;
                all_finite = false;
            }
        }
        if (__syncthreads_or(!all_finite)) redo_bad<T, DP, kRowThreads<R>>(p, bad);
        return;
    }

    cg::cluster_group cluster = cg::this_cluster();
    cp_async_wait<0>();
    __syncthreads();
#pragma unroll
    for (int i = 0; i < R; ++i) {
        float x[C];
        acc_row(o, i, x);
        store_channels(sV + (row0 + i) * kStride<DP> + ch, x);
        if (lane == 0) {
            sM[row0 + i] = m[i];
            sL[row0 + i] = l[i];
        }
    }
    all_finite = merge_rows<T, DP, kRowThreads<R>>(p, tile, part, sM, sL, sV, out, bad);
    if (__syncthreads_or(!all_finite)) redo_bad<T, DP, kRowThreads<R>>(p, bad);
    cluster.sync();   // nobody leaves while its rows are being read
}

constexpr int blocks_per_sm(int d) { return d <= 128 ? 2 : 1; }

// 16 rows to a warp read least; but a block alone on its SM, which is what the tiny configurations come to, is the chain of one
// warp, and 8 rows to each of twice as many make that shorter: 16 x 16 + 16, two heads of 64, 13.0 us against 14.3; of 128, 18.2
// against 18.5.  With more blocks than SMs: two heads at 24 x 40 + 130 36.9 against 28.7, 24 of them 180 against 148.
// bf16 rows pass through registers on their way to shared memory, with nothing else to do for the warps meanwhile: there 256 threads
// hide more of it than 128.  24 heads of 128 at 40 x 40, radius 4, 165 us with 4 x 4 results a thread, 194 with 16 rows a warp;
// at 24 x 40 + 130 344 and 371, at 1024 px, radius 8, 2400 and 2570; of 40 channels 102 and 116, 205 and 211, 1399 and 1398.
template <typename T, int DP>
int launch_rows(const F32Params &p, long long tiles, int n_sm, cudaStream_t stream)
{
    if (tiles * p.n_split <= n_sm)
        return launch_tiles(clear_f32_rows_kernel<T, DP, 8>, p, tiles, p.n_split, kRowsSmem<DP, 8>, stream, kRowThreads<8>);
    if constexpr (sizeof(T) == 2)
        return launch_tiles(clear_f32_tile_kernel<T, DP>, p, tiles, p.n_split, forward_smem<DP>(), stream);
    else
        return launch_tiles(clear_f32_rows_kernel<T, DP, 16>, p, tiles, p.n_split, kRowsSmem<DP, 16>, stream, kRowThreads<16>);
}

template <typename T>
int launch_typed(const F32Params &p, long long tiles, int n_sm, cudaStream_t stream)
{
    if (p.g.d <= 64) return launch_rows<T, 64>(p, tiles, n_sm, stream);
    if (p.g.d <= 128) return launch_rows<T, 128>(p, tiles, n_sm, stream);
    return launch_tiles(clear_f32_tile_kernel<T, 256>, p, tiles, p.n_split, forward_smem<256>(), stream);
}

}  // namespace

namespace f32tile {

Geometry geometry_of(const clear_plan &p)
{
    const Shape &s = p.shape;
    Geometry g{};
    g.half_width = p.d_half_width;
    g.n_half_width = (int)p.sch.half_width.size();
    g.grid_h = s.grid_h;
    g.grid_w = s.grid_w;
    g.n_text = s.n_text;
    g.d = s.head_dim;
    g.n_bh = s.B * s.H;
    // 8 x 8 has the smallest union of windows; a grid narrower than that in one direction takes a longer patch, so
    // that the tile's rows are not spent on cells off the grid
    g.patch_w_log = 3;
    while (g.patch_w_log > 0 && s.grid_w <= (1 << (g.patch_w_log - 1))) --g.patch_w_log;
    while (g.patch_w_log < 6 && s.grid_h <= (kRows >> (g.patch_w_log + 1)) && s.grid_w > (1 << g.patch_w_log)) ++g.patch_w_log;
    return g;
}

Extent extent_of(const clear_plan &p, const Geometry &g)
{
    const std::vector<int32_t> &hw = p.sch.half_width;
    const long long T = g.n_text, N = g.n_tokens(), R = (long long)hw.size() - 1;
    const long long n_txt = (T + kRows - 1) / kRows;
    const long long n_img = (long long)((g.grid_h + g.patch_h() - 1) / g.patch_h()) * ((g.grid_w + g.patch_w() - 1) / g.patch_w());
    // the list of an interior patch, as far as the grid has the columns and the tokens
    long long keys = T;
    for (long long dy = -R; dy < g.patch_h() + R && keys < N; ++dy) {
        const long long dist = dy < 0 ? -dy : std::max(0ll, dy - (g.patch_h() - 1));
        keys += std::min<long long>(g.grid_w, g.patch_w() + 2ll * hw[(size_t)dist]);
    }
    const long long img_steps = (std::min(keys, N) + kRows - 1) / kRows, txt_steps = (N + kRows - 1) / kRows;
    return Extent{n_txt + n_img, n_txt > 0 ? std::max(img_steps, txt_steps) : img_steps, n_txt * txt_steps + n_img * img_steps};
}

// The fewest blocks with which the longest list is no longer than an even share of all steps over the resident
// blocks, each with a step of its own: 1 where there are plenty of tiles; 8 for the tiny configuration (10 tiles of at
// most 5 steps) and for a 1024px problem of two heads, whose text tiles walk 72 steps and its patches 16.
int split_of(const Extent &e, int n_bh, int slots)
{
    int n = 1;
    while (n < 8 && e.longest > n && (e.longest + n - 1) / n > std::max(1ll, e.steps * n_bh / slots)) n *= 2;
    return n;
}

}  // namespace f32tile

int launch_f32(const clear_plan &p, const void *q, const void *k, const void *v, void *out, float scale, cudaStream_t stream)
{
    F32Params prm{};
    prm.g = geometry_of(p);
    prm.q = q;
    prm.k = k;
    prm.v = v;
    prm.out = out;
    prm.scale = scale;
    const Extent e = extent_of(p, prm.g);
    prm.n_split = split_of(e, prm.g.n_bh, p.n_sm * blocks_per_sm(prm.g.d));
    const long long tiles = e.tiles * prm.g.n_bh;
    if (p.shape.dtype == CLEAR_F32) return launch_typed<float>(prm, tiles, p.n_sm, stream);
    return launch_typed<__nv_bfloat16>(prm, tiles, p.n_sm, stream);
}

}  // namespace clear
