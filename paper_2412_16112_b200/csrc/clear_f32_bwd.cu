// Backward pass of the CLEAR attention operator on the CUDA cores, fp32 arithmetic, as tiled kernels: 64 stationary
// tokens against 64 streamed tokens at a time from shared memory (f32_tile.cuh).  Head sizes up to 128; the wider ones
// do not leave room for four row sets and keep the kernels that take one warp per token (clear_bwd.cu).
//
//   query kernel: stationary Q_i, dO_i, streamed K_j, V_j.  Sweep 1: S = Q K^T and dP = dO V^T, an online softmax of S
//       and with it delta = sum_j p dP / l (= dO . O); the three row statistics are left for the key kernel.  Sweep 2:
//       p = exp(S - m) / l, dS = p (dP - delta) scale, dQ += dS K.
//   key kernel: stationary K_j, V_j, streamed Q_i, dO_i with their statistics (the mask is symmetric, so the queries
//       that see a key are the tokens that key's own query sees).  dV += P^T dO, dK += dS^T Q.
// Two forms of both: 4 x 4 results a thread up to 64 channels (clear_f32_bwd_kernel; two blocks an SM leave 128 registers, too few
// with the mask bits of a step: the query kernel spills 48 bytes, and is 1.4 % faster all the same than with the windows asked for
// where they are used, and 4 bytes), whole rows to a warp above (clear_f32_bwd_rows_kernel, no spills).
// Bound by the fp32 multiply-add units: nine products of 64 x 64 x DP per pair of tiles.  The streamed rows go through
// a ring of three buffers, so a row set travels while the two before it are worked on; a step has two barriers in the query kernel
// and three in the key kernel.
// Every output element has one writer and a fixed order of summation (a list cut over a cluster is summed in the order
// of the ranks): results repeat bit for bit.
#include <cuda_bf16.h>
#include <math_constants.h>

#include "clear_internal.hpp"
#include "f32_tile.cuh"

namespace clear {
namespace {

using namespace f32tile;
namespace cg = cooperative_groups;

struct F32BwdParams {
    Geometry g;
    const void *q, *k, *v, *d_out;
    void *out1, *out2;   // query kernel: dq, -; key kernel: dk, dv
    float *stats;        // [bh][token][3]: m, 1 / l, delta
    int n_split;
    float scale;
};

template <int DP, int W = kRows * kPStride> struct BwdSmem {
    float a1[kRows * kStride<DP>], a2[kRows * kStride<DP>];    // stationary rows
    float ring[3][kRows * kStride<DP>];                        // streamed rows
    float w[W];                                                // weights of the accumulation
    float row[3][kRows];                                       // query kernel: this block's m, l, delta
    float col[3][3][kRows];                                    // key kernel: statistics of three streamed tiles
    KeyTile keys[3];
    int tokens[kRows];
    int red[8];
    int bad[kRows];                                            // rows that came out non-finite
};

// One streamed step after another: in step s the second row set (B2: V, or dO) of tile s is used first, then the first
// (B1: K, or Q).  Positions 2 s and 2 s + 1 of a ring of three: B2 of the next tile lands where B1 of the tile before
// was, B1 of the next tile where B2 of this one was.
template <typename T, int DP, int NT, typename Smem> struct Stream {
    Smem &sm;
    const KeyRuns &runs;
    const T *b1, *b2;
    const float *stats;   // of this (batch, head), or null
    int d, first, n_steps, n_iters;   // first step of this block's share, its steps, steps of all sweeps
    KeyCursor cur;

    __device__ __forceinline__ float *slot(int pos) const { return sm.ring[pos % 3]; }
    __device__ __forceinline__ float *b1_rows(int it) const { return slot(2 * it + 1); }
    __device__ __forceinline__ float *b2_rows(int it) const { return slot(2 * it); }
    // list of the tile of step `it`
    __device__ __forceinline__ void fill(int it)
    {
        if (it >= n_iters) return;
        if (threadIdx.x < kRows && it % n_steps == 0) {
            cur.start(runs);
            cur.advance(runs, first * kRows + (int)threadIdx.x);
        }
        fill_key_tile(sm.keys[it % 3], cur, runs, true);
        if (stats && threadIdx.x < kRows) {
            const int tok = sm.keys[it % 3].token[threadIdx.x];
#pragma unroll
            for (int u = 0; u < 3; ++u) sm.col[it % 3][u][threadIdx.x] = tok >= 0 ? __ldg(stats + 3ll * tok + u) : 0.f;
        }
    }
    __device__ __forceinline__ void load_b2(int it)
    {
        if (it < n_iters)
            load_rows<T, DP, NT>(b2_rows(it), b2, sm.keys[it % 3].token, d);
        else
            cp_async_commit();
    }
    __device__ __forceinline__ void load_b1(int it)
    {
        if (it < n_iters)
            load_rows<T, DP, NT>(b1_rows(it), b1, sm.keys[it % 3].token, d);
        else
            cp_async_commit();
    }
};

// The rows that every block of the cluster has left in its `scratch`, summed in the order of the ranks, to global memory.
template <typename T, int DP, int NT>
__device__ __forceinline__ void merge_rows(float *scratch, T *out, const F32BwdParams &p, const TileRef &tile, int part, int *bad)
{
    cg::cluster_group cluster = cg::this_cluster();
    cluster.sync();
    const int rows = kRows / p.n_split;
    for (int e = threadIdx.x; e < rows * (DP / 4); e += NT) {
        const int r = part * rows + e / (DP / 4), ch = e % (DP / 4) * 4;
        int y, x;
        const long long tok = tile_token(tile, r, p.g, y, x);
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int c = 0; c < p.n_split; ++c) {
            const float4 v = *reinterpret_cast<const float4 *>(cluster.map_shared_rank(scratch, c) + r * kStride<DP> + ch);
            a.x += v.x;
            a.y += v.y;
            a.z += v.z;
            a.w += v.w;
        }
        if (tok >= 0 && ch < p.g.d) store4(out + tok * p.g.d + ch, a);
        if (!finite4(a)) bad[r] = 1;
    }
    cluster.sync();   // nobody leaves, or reuses the rows, while they are being read
}

// Rows of an accumulator to global memory, summed over the cluster first when the list is cut.
template <typename T, int DP>
__device__ __forceinline__ void store_acc(const uint64_t (&acc)[4][DP / 64][2], float *scratch, T *out, const F32BwdParams &p,
                                          const TileRef &tile, int part, int ty, int tx, int *bad)
{
    if (p.n_split == 1) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            int y, x;
            const long long tok = tile_token(tile, ty + 16 * i, p.g, y, x);
#pragma unroll
            for (int c = 0; c < DP / 64; ++c) {
                const int ch = 64 * c + 4 * tx;
                const float4 v = acc_float4(acc[i][c], 1.f);
                if (tok >= 0 && ch < p.g.d) store4(out + tok * p.g.d + ch, v);
                if (!finite4(v)) bad[ty + 16 * i] = 1;
            }
        }
        return;
    }
    acc_to_rows<DP>(acc, scratch, ty, tx);
    merge_rows<T, DP, kThreads>(scratch, out, p, tile, part, bad);
}

// Row r of the block's tile by itself (one warp): the sums of the kernel below over the tokens that the row sees.
template <typename T, int DP, bool KEY_ROLE>
__device__ __forceinline__ void redo_row(const F32BwdParams &p, int r)
{
    const TileRef tile = tile_of((int)(blockIdx.x / (unsigned)p.n_split), p.g);
    const KeyRuns runs = runs_of(tile, p.g);
    int y, x;
    const int tok = tile_token(tile, r, p.g, y, x), d = p.g.d;
    if (tok < 0) return;
    const long long base = (long long)tile.bh * runs.n_tokens * d;
    const T *b1 = static_cast<const T *>(KEY_ROLE ? p.q : p.k) + base, *b2 = static_cast<const T *>(KEY_ROLE ? p.d_out : p.v) + base;
    const float *stats = p.stats + (long long)tile.bh * runs.n_tokens * 3;
    LaneRow<DP> a1, a2, r1, r2, o1, o2;
    a1.load(static_cast<const T *>(KEY_ROLE ? p.k : p.q) + base + (long long)tok * d, d);
    a2.load(static_cast<const T *>(KEY_ROLE ? p.v : p.d_out) + base + (long long)tok * d, d);
    o1.zero();
    o2.zero();
    for_each_seen(runs, y, x, [&](int t) {
        r1.load(b1 + (long long)t * d, d);
        r2.load(b2 + (long long)t * d, d);
        const float *st = stats + 3ll * (KEY_ROLE ? t : tok);
        const float pr = expf(a1.dot(r1) * p.scale - __ldcg(st)) * __ldcg(st + 1);
        o1.add(pr * (a2.dot(r2) - __ldcg(st + 2)) * p.scale, r1);
        if (KEY_ROLE) o2.add(pr, r2);
    });
    o1.store(static_cast<T *>(p.out1) + base + (long long)tok * d, d, 1.f);
    if (KEY_ROLE) o2.store(static_cast<T *>(p.out2) + base + (long long)tok * d, d, 1.f);
}

template <typename T, int DP, bool KEY_ROLE>
__global__ void __launch_bounds__(kThreads, 2) clear_f32_bwd_kernel(const __grid_constant__ F32BwdParams p)
{
    extern __shared__ __align__(16) uint8_t smem_raw[];
    BwdSmem<DP> &sm = *reinterpret_cast<BwdSmem<DP> *>(smem_raw);
    const int tid = threadIdx.x, ty = (tid >> 5) * 2 + ((tid >> 4) & 1), tx = tid & 15;
    const int part = (int)(blockIdx.x % (unsigned)p.n_split);
    const TileRef tile = tile_of((int)(blockIdx.x / (unsigned)p.n_split), p.g);
    const KeyRuns runs = runs_of(tile, p.g);
    const long long base = (long long)tile.bh * runs.n_tokens * p.g.d;
    const T *q = static_cast<const T *>(p.q) + base, *k = static_cast<const T *>(p.k) + base,
            *v = static_cast<const T *>(p.v) + base, *go = static_cast<const T *>(p.d_out) + base;
    float *stats = p.stats + (long long)tile.bh * runs.n_tokens * 3;

    const int n_all = (list_length(runs, sm.red) + kRows - 1) / kRows, per = (n_all + p.n_split - 1) / p.n_split;
    const int step0 = min(part * per, n_all), n_steps = min(per, n_all - step0);
    Stream<T, DP, kThreads, BwdSmem<DP>> st{sm, runs, KEY_ROLE ? q : k, KEY_ROLE ? go : v, KEY_ROLE ? stats : nullptr, p.g.d, step0, n_steps,
                     KEY_ROLE ? n_steps : 2 * n_steps};
    if (tid < kRows) {
        int y, x;
        sm.tokens[tid] = tile_token(tile, tid, p.g, y, x);
        sm.bad[tid] = 0;
    }
    st.fill(0);
    st.fill(1);
    __syncthreads();
    load_rows<T, DP>(sm.a1, KEY_ROLE ? k : q, sm.tokens, p.g.d);
    load_rows<T, DP>(sm.a2, KEY_ROLE ? v : go, sm.tokens, p.g.d);
    st.load_b2(0);
    st.load_b1(0);

    int r_y[4], r_x[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) tile_token(tile, ty + 16 * i, p.g, r_y[i], r_x[i]);
    uint64_t acc1[4][DP / 64][2], acc2[4][DP / 64][2];
    zero_acc<DP>(acc1);
    zero_acc<DP>(acc2);
    float m[4], l[4], dl[4];   // query kernel: row maximum, row sum (then its inverse), delta
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        m[i] = -CUDART_INF_F;
        l[i] = dl[i] = 0.f;
    }

    // the row statistics after sweep 1: over the row's 16 lanes, then over the cluster
    auto close_sweep1 = [&]() {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            l[i] = row_sum16(l[i]);
            dl[i] = row_sum16(dl[i]);
        }
        if (p.n_split > 1) {
            cg::cluster_group cluster = cg::this_cluster();
            if (tx == 0)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    sm.row[0][ty + 16 * i] = m[i];
                    sm.row[1][ty + 16 * i] = l[i];
                    sm.row[2][ty + 16 * i] = dl[i];
                }
            cluster.sync();
            // one of the four rows to a lane: reads from other blocks' shared memory are slow
            float mx = -CUDART_INF_F, sl = 0.f, sd = 0.f;
            if (tx < 4) {
                const int r = ty + 16 * tx;
                for (int c = 0; c < p.n_split; ++c) mx = fmaxf(mx, cluster.map_shared_rank(sm.row[0], c)[r]);
                const float m_ref = mx == -CUDART_INF_F ? 0.f : mx;
                for (int c = 0; c < p.n_split; ++c) {
                    const float f = expf(cluster.map_shared_rank(sm.row[0], c)[r] - m_ref);
                    sl = fmaf(f, cluster.map_shared_rank(sm.row[1], c)[r], sl);
                    sd = fmaf(f, cluster.map_shared_rank(sm.row[2], c)[r], sd);
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                m[i] = __shfl_sync(0xffffffffu, mx, i, 16);
                l[i] = __shfl_sync(0xffffffffu, sl, i, 16);
                dl[i] = __shfl_sync(0xffffffffu, sd, i, 16);
            }
            cluster.sync();
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            l[i] = l[i] == 0.f ? 0.f : 1.f / l[i];   // l >= 1 for every row that exists (it sees itself or the text); NaN stays
            dl[i] *= l[i];
            if (m[i] == -CUDART_INF_F) m[i] = 0.f;
            const long long tok = sm.tokens[ty + 16 * i];
            if (part == 0 && tx == 0 && tok >= 0) {
                stats[tok * 3] = m[i];
                stats[tok * 3 + 1] = l[i];
                stats[tok * 3 + 2] = dl[i];
            }
        }
    };
    if (!KEY_ROLE && n_steps == 0) close_sweep1();   // a cluster's block without a share takes part in the merges

    for (int it = 0; it < st.n_iters; ++it) {
        const bool sweep1 = !KEY_ROLE && it < n_steps;
        const KeyTile &kt = sm.keys[it % 3];
        // which of the thread's streamed tokens its rows see, while the rows are on their way: bit 4 i + j
        uint32_t on = 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = tx + 16 * j, ky = kt.ky[c], kx = kt.kx[c];
            const bool here = kt.token[c] >= 0;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (here && sees(runs, r_y[i], r_x[i], ky, kx)) on |= 1u << (4 * i + j);
        }
        cp_async_wait<1>();   // the stationary rows and B2 of this step are here
        __syncthreads();      // ... for everybody, and B1 of the step before is free
        st.load_b2(it + 1);
        float g[4][4], s[4][4];
        tile_dot<DP>(sm.a2, st.b2_rows(it), ty, tx, g);
        if (!KEY_ROLE) {
            cp_async_wait<1>();
            __syncthreads();  // B1 is here, B2 is free
            st.load_b1(it + 1);
            st.fill(it + 2);
        } else {
            cp_async_wait<1>();
            __syncthreads();
        }
        tile_dot<DP>(sm.a1, st.b1_rows(it), ty, tx, s);

        if (sweep1) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float mx = -CUDART_INF_F;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const bool here = (on >> (4 * i + j)) & 1u;
                    s[i][j] = here ? s[i][j] * p.scale : -CUDART_INF_F;
                    g[i][j] = here ? g[i][j] : 0.f;   // (its weight is 0, but it may be no number)
                    mx = fmaxf(mx, s[i][j]);
                }
                const float m_new = fmaxf(m[i], row_max16(mx)), m_ref = m_new == -CUDART_INF_F ? 0.f : m_new;
                const float alpha = expf(m[i] - m_ref);   // m = -inf: 0
                m[i] = m_new;
                l[i] *= alpha;
                dl[i] *= alpha;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float e = expf(s[i][j] - m_ref);
                    l[i] += e;
                    dl[i] = fmaf(e, g[i][j], dl[i]);
                }
            }
            if (it + 1 == n_steps) close_sweep1();
            continue;
        }

        // P and dS in place of S and dP
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int c = tx + 16 * j;
                const bool here = (on >> (4 * i + j)) & 1u;
                const float mm = KEY_ROLE ? sm.col[it % 3][0][c] : m[i], il = KEY_ROLE ? sm.col[it % 3][1][c] : l[i],
                            de = KEY_ROLE ? sm.col[it % 3][2][c] : dl[i];
                const float pr = here ? expf(s[i][j] * p.scale - mm) * il : 0.f;
                s[i][j] = pr;
                g[i][j] = here ? pr * (g[i][j] - de) * p.scale : 0.f;
            }
        if (KEY_ROLE) {
            // dV += P^T dO; a row of weights is written and read by one warp
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) sm.w[(ty + 16 * i) * kPStride + tx + 16 * j] = s[i][j];
            __syncwarp();
            tile_accumulate<DP>(sm.w, st.b2_rows(it), ty, tx, acc2);
            __syncthreads();   // B2 is free
            st.load_b1(it + 1);
            st.fill(it + 2);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) sm.w[(ty + 16 * i) * kPStride + tx + 16 * j] = g[i][j];
        __syncwarp();
        tile_accumulate<DP>(sm.w, st.b1_rows(it), ty, tx, acc1);   // dQ += dS K, or dK += dS^T Q
        __syncwarp();
    }
    cp_async_wait<0>();
    __syncthreads();
    store_acc<T, DP>(acc1, sm.ring[0], static_cast<T *>(p.out1) + base, p, tile, part, ty, tx, sm.bad);
    if (KEY_ROLE) store_acc<T, DP>(acc2, sm.ring[1], static_cast<T *>(p.out2) + base, p, tile, part, ty, tx, sm.bad);
    __syncthreads();
#pragma unroll 1
    for (int r = tid >> 5; r < kRows; r += kThreads / 32)
        if (sm.bad[r] != 0) redo_row<T, DP, KEY_ROLE>(p, r);
}

// The same with a warp to 8 whole rows (warp_dot), for 65 to 128 channels: less shared memory is read for the products, and in the
// first sweep lanes exchange nothing in a step without a new maximum.  24 heads of 128 at
// 24 x 40 + 130, radius 8: 1211 us, 1357 with 4 x 4 results a thread.  At 64 channels, where the products are half as long and
// two blocks share an SM, 801 against 672 (and 704 with 16 rows to a warp of 128 threads, at 128 channels 1681).
// A row's reference is its running maximum: against one that may lie 16 below (1201 us) weights were rounded at 2^-21, 14 % more error
// of the gradients where keys climb, and delta's sum of weights times dP left fp32's range where dP was 10^7 times smaller.
constexpr int kWarpRows = 8, kRowThreads = 32 * kRows / kWarpRows;

template <int DP> using RowsSmem = BwdSmem<DP, kRows / kWarpRows * kRows * kPairStride<kWarpRows>>;

template <typename T, int DP, bool KEY_ROLE>
__global__ void __launch_bounds__(kRowThreads, 1) clear_f32_bwd_rows_kernel(const __grid_constant__ F32BwdParams p)
{
    constexpr int C = DP / 32;
    extern __shared__ __align__(16) uint8_t smem_raw[];
    RowsSmem<DP> &sm = *reinterpret_cast<RowsSmem<DP> *>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, row0 = (tid >> 5) * kWarpRows;
    float *w = sm.w + (tid >> 5) * kRows * kPairStride<kWarpRows>;   // the warp's weights
    const int part = (int)(blockIdx.x % (unsigned)p.n_split);
    const TileRef tile = tile_of((int)(blockIdx.x / (unsigned)p.n_split), p.g);
    const KeyRuns runs = runs_of(tile, p.g);
    const long long base = (long long)tile.bh * runs.n_tokens * p.g.d;
    const T *q = static_cast<const T *>(p.q) + base, *k = static_cast<const T *>(p.k) + base,
            *v = static_cast<const T *>(p.v) + base, *go = static_cast<const T *>(p.d_out) + base;
    float *stats = p.stats + (long long)tile.bh * runs.n_tokens * 3;

    const int n_all = (list_length<kRowThreads>(runs, sm.red) + kRows - 1) / kRows, per = (n_all + p.n_split - 1) / p.n_split;
    const int step0 = min(part * per, n_all), n_steps = min(per, n_all - step0);
    Stream<T, DP, kRowThreads, RowsSmem<DP>> st{sm, runs, KEY_ROLE ? q : k, KEY_ROLE ? go : v, KEY_ROLE ? stats : nullptr, p.g.d, step0,
                                                n_steps, KEY_ROLE ? n_steps : 2 * n_steps};
    if (tid < kRows) {
        int y, x;
        sm.tokens[tid] = tile_token(tile, tid, p.g, y, x);
        sm.bad[tid] = 0;
    }
    st.fill(0);
    st.fill(1);
    __syncthreads();
    load_rows<T, DP, kRowThreads>(sm.a1, KEY_ROLE ? k : q, sm.tokens, p.g.d);
    load_rows<T, DP, kRowThreads>(sm.a2, KEY_ROLE ? v : go, sm.tokens, p.g.d);
    st.load_b2(0);
    st.load_b1(0);

    uint64_t acc1[kWarpRows / 2][C], acc2[kWarpRows / 2][C];
#pragma unroll
    for (int i = 0; i < kWarpRows / 2; ++i)
#pragma unroll
        for (int c = 0; c < C; ++c) acc1[i][c] = acc2[i][c] = 0ull;
    // query kernel: row reference, row sum (then its inverse), delta; in sweep 1 the lane's share of the two sums
    float m[kWarpRows], l[kWarpRows], dl[kWarpRows];
#pragma unroll
    for (int i = 0; i < kWarpRows; ++i) {
        m[i] = -CUDART_INF_F;
        l[i] = dl[i] = 0.f;
    }

    // the row statistics after sweep 1: over the lanes, then over the cluster
    auto close_sweep1 = [&]() {
#pragma unroll
        for (int i = 0; i < kWarpRows; ++i)
#pragma unroll
            for (int x = 16; x > 0; x >>= 1) {
                l[i] += __shfl_xor_sync(0xffffffffu, l[i], x);
                dl[i] += __shfl_xor_sync(0xffffffffu, dl[i], x);
            }
        if (p.n_split > 1) {
            cg::cluster_group cluster = cg::this_cluster();
            if (lane == 0)
#pragma unroll
                for (int i = 0; i < kWarpRows; ++i) {
                    sm.row[0][row0 + i] = m[i];
                    sm.row[1][row0 + i] = l[i];
                    sm.row[2][row0 + i] = dl[i];
                }
            cluster.sync();
            // a row to a lane: reads from other blocks' shared memory are slow
            float mx = -CUDART_INF_F, sl = 0.f, sd = 0.f;
            if (lane < kWarpRows) {
                const int r = row0 + lane;
                for (int c = 0; c < p.n_split; ++c) mx = fmaxf(mx, cluster.map_shared_rank(sm.row[0], c)[r]);
                const float m_ref = mx == -CUDART_INF_F ? 0.f : mx;
                for (int c = 0; c < p.n_split; ++c) {
                    const float f = expf(cluster.map_shared_rank(sm.row[0], c)[r] - m_ref);
                    sl = fmaf(f, cluster.map_shared_rank(sm.row[1], c)[r], sl);
                    sd = fmaf(f, cluster.map_shared_rank(sm.row[2], c)[r], sd);
                }
            }
#pragma unroll
            for (int i = 0; i < kWarpRows; ++i) {
                m[i] = __shfl_sync(0xffffffffu, mx, i);
                l[i] = __shfl_sync(0xffffffffu, sl, i);
                dl[i] = __shfl_sync(0xffffffffu, sd, i);
            }
            cluster.sync();
        }
#pragma unroll
        for (int i = 0; i < kWarpRows; ++i) {
            l[i] = l[i] == 0.f ? 0.f : 1.f / l[i];   // l > 0 for every row that exists (it sees itself or the text); NaN stays
            dl[i] *= l[i];
            if (m[i] == -CUDART_INF_F) m[i] = 0.f;
            const long long tok = sm.tokens[row0 + i];
            if (part == 0 && lane == 0 && tok >= 0) {
                stats[tok * 3] = m[i];
                stats[tok * 3 + 1] = l[i];
                stats[tok * 3 + 2] = dl[i];
            }
        }
    };
    if (!KEY_ROLE && n_steps == 0) close_sweep1();   // a cluster's block without a share takes part in the merges

    auto put_weights = [&](const float (&x)[kWarpRows][2]) {
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int i = 0; i < kWarpRows; i += 4)
                *reinterpret_cast<float4 *>(w + (lane + 32 * j) * kPairStride<kWarpRows> + i) = make_float4(x[i][j], x[i + 1][j], x[i + 2][j], x[i + 3][j]);
        __syncwarp();
    };
    for (int it = 0; it < st.n_iters; ++it) {
        const bool sweep1 = !KEY_ROLE && it < n_steps;
        const KeyTile &kt = sm.keys[it % 3];
        cp_async_wait<1>();   // the stationary rows and B2 of this step are here
        __syncthreads();      // ... for everybody, and B1 of the step before is free
        st.load_b2(it + 1);
        uint32_t on[2];       // rows that see the lane's tokens
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int c = lane + 32 * j;
            on[j] = kt.token[c] >= 0 ? seen_by<kWarpRows>(runs, tile, p.g, row0, kt.ky[c], kt.kx[c]) : 0u;
        }
        float g[kWarpRows][2], s[kWarpRows][2];
        warp_dot<DP>(sm.a2 + row0 * kStride<DP>, st.b2_rows(it), lane, g);
        cp_async_wait<1>();
        __syncthreads();      // B1 is here; in the query kernel B2 is free
        if (!KEY_ROLE) {
            st.load_b1(it + 1);
            st.fill(it + 2);
        }
        warp_dot<DP>(sm.a1 + row0 * kStride<DP>, st.b1_rows(it), lane, s);

        if (sweep1) {
            bool higher = false;   // than the row's reference
#pragma unroll
            for (int i = 0; i < kWarpRows; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const bool here = (on[j] >> i) & 1u;
                    s[i][j] = here ? s[i][j] * p.scale : -CUDART_INF_F;
                    g[i][j] = here ? g[i][j] : 0.f;   // (its weight is 0, but it may be no number)
                    higher = higher || s[i][j] > m[i];
                }
            if (__any_sync(0xffffffffu, higher)) {
#pragma unroll
                for (int i = 0; i < kWarpRows; ++i) {
                    float mx = fmaxf(s[i][0], s[i][1]);
#pragma unroll
                    for (int x = 16; x > 0; x >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, x));
                    const float m_new = fmaxf(m[i], mx);
                    const float alpha = expf(m[i] - (m_new == -CUDART_INF_F ? 0.f : m_new));   // m = -inf: 0
                    m[i] = m_new;
                    l[i] *= alpha;
                    dl[i] *= alpha;
                }
            }
#pragma unroll
            for (int i = 0; i < kWarpRows; ++i) {
                const float m_ref = m[i] == -CUDART_INF_F ? 0.f : m[i];
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const float e = expf(s[i][j] - m_ref);
                    l[i] += e;
                    dl[i] = fmaf(e, g[i][j], dl[i]);
                }
            }
            if (it + 1 == n_steps) close_sweep1();
            continue;
        }

        // P and dS in place of S and dP
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int c = lane + 32 * j;
            const float cm = KEY_ROLE ? sm.col[it % 3][0][c] : 0.f, cl = KEY_ROLE ? sm.col[it % 3][1][c] : 0.f,
                        cd = KEY_ROLE ? sm.col[it % 3][2][c] : 0.f;
#pragma unroll
            for (int i = 0; i < kWarpRows; ++i) {
                const bool here = (on[j] >> i) & 1u;
                const float pr = here ? expf(s[i][j] * p.scale - (KEY_ROLE ? cm : m[i])) * (KEY_ROLE ? cl : l[i]) : 0.f;
                s[i][j] = pr;
                g[i][j] = here ? pr * (g[i][j] - (KEY_ROLE ? cd : dl[i])) * p.scale : 0.f;
            }
        }
        if (KEY_ROLE) {
            put_weights(s);    // dV += P^T dO; a warp writes and reads its own weights
            warp_accumulate<DP, kWarpRows>(w, st.b2_rows(it), lane, acc2);
            __syncthreads();   // B2 is free
            st.load_b1(it + 1);
            st.fill(it + 2);
        }
        put_weights(g);
        warp_accumulate<DP, kWarpRows>(w, st.b1_rows(it), lane, acc1);   // dQ += dS K, or dK += dS^T Q
        __syncwarp();
    }
    cp_async_wait<0>();
    __syncthreads();
    auto store = [&](const uint64_t (&acc)[kWarpRows / 2][C], float *scratch, T *out) {
        const int ch = C * lane;
#pragma unroll
        for (int i = 0; i < kWarpRows; ++i) {
            float x[C];
            acc_row(acc, i, x);
            if (p.n_split > 1) {
                store_channels(scratch + (row0 + i) * kStride<DP> + ch, x);
                continue;
            }
            const long long tok = sm.tokens[row0 + i];
            if (tok >= 0 && ch < p.g.d) store_channels(out + tok * p.g.d + ch, x);
            bool fine = true;
#pragma unroll
            for (int c = 0; c < C; ++c) fine = fine && fabsf(x[c]) <= CUDART_MAX_NORMAL_F;
            if (!fine) sm.bad[row0 + i] = 1;
        }
        if (p.n_split > 1) merge_rows<T, DP, kRowThreads>(scratch, out, p, tile, part, sm.bad);
    };
    store(acc1, sm.ring[0], static_cast<T *>(p.out1) + base);
    if (KEY_ROLE) store(acc2, sm.ring[1], static_cast<T *>(p.out2) + base);
    __syncthreads();
#pragma unroll 1
    for (int r = tid >> 5; r < kRows; r += kRowThreads / 32)
        if (sm.bad[r] != 0) redo_row<T, DP, KEY_ROLE>(p, r);
}

template <typename T, int DP>
int launch_dp(F32BwdParams p, void *dq, void *dk, void *dv, long long tiles, cudaStream_t stream)
{
    p.out1 = dq;
    if constexpr (DP == 64) {
        const int rc = launch_tiles(clear_f32_bwd_kernel<T, DP, false>, p, tiles, p.n_split, sizeof(BwdSmem<DP>), stream);
        if (rc != CLEAR_OK) return rc;
        p.out1 = dk;
        p.out2 = dv;
        return launch_tiles(clear_f32_bwd_kernel<T, DP, true>, p, tiles, p.n_split, sizeof(BwdSmem<DP>), stream);
    } else {
        const int rc = launch_tiles(clear_f32_bwd_rows_kernel<T, DP, false>, p, tiles, p.n_split, sizeof(RowsSmem<DP>), stream, kRowThreads);
        if (rc != CLEAR_OK) return rc;
        p.out1 = dk;
        p.out2 = dv;
        return launch_tiles(clear_f32_bwd_rows_kernel<T, DP, true>, p, tiles, p.n_split, sizeof(RowsSmem<DP>), stream, kRowThreads);
    }
}

}  // namespace

int launch_f32_bwd(const clear_plan &p, const void *q, const void *k, const void *v, const void *d_out, void *dq, void *dk,
                   void *dv, float scale, cudaStream_t stream)
{
    const int rc = ensure_bwd_stats(p);
    if (rc != CLEAR_OK) return rc;
    F32BwdParams prm{};
    prm.g = geometry_of(p);
    prm.q = q;
    prm.k = k;
    prm.v = v;
    prm.d_out = d_out;
    prm.stats = p.d_bwd_stats;
    prm.scale = scale;
    const Extent e = extent_of(p, prm.g);
    prm.n_split = split_of(e, prm.g.n_bh, p.n_sm * (prm.g.d <= 64 ? 2 : 1));
    const long long tiles = e.tiles * prm.g.n_bh;
    if (p.shape.dtype == CLEAR_F32)
        return prm.g.d <= 64 ? launch_dp<float, 64>(prm, dq, dk, dv, tiles, stream) : launch_dp<float, 128>(prm, dq, dk, dv, tiles, stream);
    return prm.g.d <= 64 ? launch_dp<__nv_bfloat16, 64>(prm, dq, dk, dv, tiles, stream)
                         : launch_dp<__nv_bfloat16, 128>(prm, dq, dk, dv, tiles, stream);
}

}  // namespace clear
