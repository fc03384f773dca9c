// Building blocks of the fp32 tile kernels (forward and backward pass on the CUDA cores): a block works on a tile of 64 tokens
// (an 8 x 8 patch of the grid, longer and flatter on grids narrower than 8, or 64 consecutive text tokens) against the tokens
// its queries can see, 64 at a time.  Two ways to share the work: 4 x 4 results a thread, of 256, or whole rows to a warp
// (warp_dot below), 8 of 256 threads or 16 of 128.
//
// 4 x 4 results: thread (ty, tx), 16 x 16, owns the rows ty + 16 i (i < 4) of the tile; one warp holds two values of ty with all
// their tx, so everything that is exchanged along a row stays inside a warp.
//   product of two row sets (tile_dot):    4 x 4 results a thread, both operands as float4 along the channels, even
//       and odd channels summed apart in the two halves of a packed fp32 pair (fma.rn.f32x2): no operand is ever
//       repacked.  Rows are padded to DP + 4 floats, so the 16 rows a warp reads at one channel lie 16 bytes apart
//       modulo 128: 4 shared-memory wavefronts per float4 of the streamed rows, 2 per float4 of the thread's own,
//       24 per 16 clocks of multiply-adds.
//   accumulation (tile_accumulate): row weights (64 x 64, in shared memory) times the streamed rows; a thread owns
//       4 rows x DP / 16 channels, pairs of channels in packed arithmetic.
#pragma once

#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math_constants.h>

#include <cstdint>

#include "clear_internal.hpp"
#include "ptx.cuh"

namespace clear {
namespace f32tile {

constexpr int kThreads = 256;
constexpr int kRows = 64;        // tokens of a tile, and of a streamed tile
constexpr int kPStride = 68;     // floats between rows of the 64 x 64 weight matrix

template <int DP> constexpr int kStride = DP + 4;   // floats between rows of 64 x DP

// Tokens the queries of one tile can see, in order: the text tokens, then for every grid row within reach the run of
// columns [x0 - w, x1 + w] with w the half width at the row's distance from the patch.  (The half widths do not grow
// with the distance, so this is the union of the windows of the patch's queries: no token is listed that none of
// them needs.)  A text query sees all tokens: one run.
struct KeyRuns {
    const int32_t *half_width;
    int n_half_width, grid_h, grid_w, n_text, n_tokens;
    int y0, y1, x0, x1;   // patch of the queries, clipped to the grid (image tiles)
    bool text;

    __device__ __forceinline__ int first_row() const { return text ? 0 : max(0, y0 - (n_half_width - 1)); }
    __device__ __forceinline__ int end_row() const { return text ? 0 : min(grid_h, y1 + n_half_width); }
    // run of grid row y: first column and length
    __device__ __forceinline__ int run(int y, int &x_first) const
    {
        const int dist = max(0, max(y0 - y, y - y1));
        const int w = __ldg(half_width + dist);
        x_first = max(x0 - w, 0);
        return min(x1 + w, grid_w - 1) - x_first + 1;
    }
    __device__ __forceinline__ int head_length() const { return text ? n_tokens : n_text; }
};

// Walks the list of KeyRuns: one position, moved forward only.
struct KeyCursor {
    int row, off, len, x_first;   // row == first_row - 1: inside the leading run of tokens
    __device__ __forceinline__ void start(const KeyRuns &k)
    {
        row = k.first_row() - 1;
        off = 0;
        len = k.head_length();
        x_first = 0;
        advance(k, 0);   // an empty leading run is left at once
    }
    __device__ __forceinline__ void advance(const KeyRuns &k, int n)
    {
        off += n;
        while (off >= len && row < k.end_row()) {
            off -= len;
            ++row;
            len = row < k.end_row() ? k.run(row, x_first) : 0;
        }
    }
    // token at the position, or -1 past the end; ky, kx: its grid cell (ky = -1: a token every query of the tile sees)
    __device__ __forceinline__ int token(const KeyRuns &k, int &ky, int &kx) const
    {
        ky = -1;
        kx = 0;
        if (row < k.first_row()) return off < len ? off : -1;
        if (row >= k.end_row()) return -1;
        ky = row;
        kx = x_first + off;
        return k.n_text + row * k.grid_w + kx;
    }
};

// Number of tokens in the list (every one of the block's NT threads gets it; `red` is 8 ints of shared memory).
template <int NT = kThreads>
__device__ __forceinline__ int list_length(const KeyRuns &k, int *red)
{
    int n = 0, xf;
    for (int y = k.first_row() + (int)threadIdx.x; y < k.end_row(); y += NT) n += k.run(y, xf);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = n;
    __syncthreads();
    int sum = k.head_length();
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) sum += red[w];
    return sum;
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, bool valid)
{
    const int n = valid ? 16 : 0;   // 0 source bytes: the 16 bytes are filled with zeros
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// 64 rows of d channels into shared memory as fp32 (row stride DP + 4), zeros for absent rows (token < 0) and for the
// channels d .. DP - 1.  fp32 rows travel asynchronously (one commit group), bf16 rows through registers.
template <typename T, int DP, int NT = kThreads>
__device__ __forceinline__ void load_rows(float *dst, const T *__restrict__ base, const int *tokens, int d)
{
    constexpr int kChunks = DP / 4;              // float4 of a row
    constexpr int kRowsPerPass = NT / kChunks;   // of 256 threads: DP = 64, 128, 256: 16, 8, 4
    const int chunk = threadIdx.x % kChunks, r0 = threadIdx.x / kChunks;
#pragma unroll
    for (int i = 0; i < kRows / kRowsPerPass; ++i) {
        const int r = r0 + i * kRowsPerPass;
        const int tok = tokens[r];
        const bool valid = tok >= 0 && chunk * 4 < d;
        float *to = dst + r * kStride<DP> + chunk * 4;
        const T *src = base + (valid ? (long long)tok * d + chunk * 4 : 0);
        if constexpr (sizeof(T) == 4) {
            cp_async16(ptx::smem_u32(to), src, valid);
        } else {
            uint2 u = make_uint2(0u, 0u);
            if (valid) u = *reinterpret_cast<const uint2 *>(src);
            *reinterpret_cast<float4 *>(to) = make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u),
                                                          __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xffff0000u));
        }
    }
    cp_async_commit();
}

// s[i][j] = sum over channels of A[ty + 16 i] . B[tx + 16 j]
template <int DP>
__device__ __forceinline__ void tile_dot(const float *A, const float *B, int ty, int tx, float (&s)[4][4])
{
    uint64_t acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
    const float *a0 = A + ty * kStride<DP>, *b0 = B + tx * kStride<DP>;
#pragma unroll 4
    for (int c = 0; c < DP; c += 4) {
        ulonglong2 a[4], b[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const ulonglong2 *>(a0 + i * 16 * kStride<DP> + c);
#pragma unroll
        for (int j = 0; j < 4; ++j) b[j] = *reinterpret_cast<const ulonglong2 *>(b0 + j * 16 * kStride<DP> + c);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                acc[i][j] = ptx::fma2(a[i].x, b[j].x, acc[i][j]);
                acc[i][j] = ptx::fma2(a[i].y, b[j].y, acc[i][j]);
            }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float lo, hi;
            ptx::unpack2(acc[i][j], lo, hi);
            s[i][j] = lo + hi;
        }
}

// acc[i][c] (+)= sum over the 64 streamed rows j of W[ty + 16 i][j] * B[j][channels]; the thread's channels are
// 64 c + 4 tx + (0..3), two packed pairs each.
template <int DP>
__device__ __forceinline__ void tile_accumulate(const float *W, const float *B, int ty, int tx, uint64_t (&acc)[4][DP / 64][2])
{
    const float *w0 = W + ty * kPStride, *b0 = B + tx * 4;
#pragma unroll 2
    for (int j = 0; j < kRows; j += 4) {
        float4 w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = *reinterpret_cast<const float4 *>(w0 + i * 16 * kPStride + j);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            ulonglong2 b[DP / 64];
#pragma unroll
            for (int c = 0; c < DP / 64; ++c)
                b[c] = *reinterpret_cast<const ulonglong2 *>(b0 + (j + u) * kStride<DP> + 64 * c);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float p = u == 0 ? w[i].x : u == 1 ? w[i].y : u == 2 ? w[i].z : w[i].w;
                const uint64_t p2 = ptx::pack2(p, p);
#pragma unroll
                for (int c = 0; c < DP / 64; ++c) {
                    acc[i][c][0] = ptx::fma2(p2, b[c].x, acc[i][c][0]);
                    acc[i][c][1] = ptx::fma2(p2, b[c].y, acc[i][c][1]);
                }
            }
        }
    }
}

template <int DP>
__device__ __forceinline__ void zero_acc(uint64_t (&acc)[4][DP / 64][2])
{
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c < DP / 64; ++c) acc[i][c][0] = acc[i][c][1] = 0ull;
}

// Accumulator rows as plain fp32 rows in shared memory (stride DP + 4).
template <int DP>
__device__ __forceinline__ void acc_to_rows(const uint64_t (&acc)[4][DP / 64][2], float *dst, int ty, int tx)
{
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c < DP / 64; ++c) {
            ulonglong2 v;
            v.x = acc[i][c][0];
            v.y = acc[i][c][1];
            *reinterpret_cast<ulonglong2 *>(dst + (ty + 16 * i) * kStride<DP> + 64 * c + 4 * tx) = v;
        }
}

__device__ __forceinline__ float row_max16(float x)
{
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
}
__device__ __forceinline__ float row_sum16(float x)
{
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// ---- a warp to R whole rows (DP <= 128) --------------------------------------------------------------------------------
// Shared memory serves 16-byte reads eight lanes at a time, and lanes in different eights share nothing unless all 32 read one
// address: so a warp's own rows are read by all its lanes at once (1 wavefront a read) and the streamed rows by a lane each (4).
// 16 own rows x 2 streamed ones a lane take 24 wavefronts per 64 packed multiply-adds a lane (32 clocks), 8 own rows 16 per 32;
// 4 x 4 results a thread, with 2 x 16 threads a warp, take 24 per 32.
template <int R> constexpr int kPairStride = R + 4;   // floats between the streamed rows of a warp's weights [64][R]: no conflicts

// s[i][j] = sum over channels of A[i] . B[lane + 32 j], even and odd channels apart as in tile_dot
template <int DP, int R>
__device__ __forceinline__ void warp_dot(const float *A, const float *B, int lane, float (&s)[R][2])
{
    uint64_t acc[R][2];
#pragma unroll
    for (int i = 0; i < R; ++i) acc[i][0] = acc[i][1] = 0ull;
    const float *b0 = B + lane * kStride<DP>;
    constexpr int kUnroll = R == 16 ? 2 : 4;   // what the registers hold
#pragma unroll kUnroll
    for (int c = 0; c < DP; c += 4) {
        const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(b0 + c), y = *reinterpret_cast<const ulonglong2 *>(b0 + 32 * kStride<DP> + c);
#pragma unroll
        for (int i0 = 0; i0 < R; i0 += 4) {   // four rows at a time: eight chains side by side
            ulonglong2 a[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const ulonglong2 *>(A + (i0 + i) * kStride<DP> + c);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                acc[i0 + i][0] = ptx::fma2(a[i].x, x.x, acc[i0 + i][0]);
                acc[i0 + i][1] = ptx::fma2(a[i].x, y.x, acc[i0 + i][1]);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                acc[i0 + i][0] = ptx::fma2(a[i].y, x.y, acc[i0 + i][0]);
                acc[i0 + i][1] = ptx::fma2(a[i].y, y.y, acc[i0 + i][1]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            float lo, hi;
            ptx::unpack2(acc[i][j], lo, hi);
            s[i][j] = lo + hi;
        }
}

// acc[k][c]: rows 2 k, 2 k + 1 of the warp (a packed pair) of channel DP / 32 lane + c; += sum over the 64 streamed rows j of
// W[j][rows] * B[j][channels]
template <int DP, int R>
__device__ __forceinline__ void warp_accumulate(const float *W, const float *B, int lane, uint64_t (&acc)[R / 2][DP / 32])
{
    constexpr int C = DP / 32;
    const float *b0 = B + lane * C;
#pragma unroll 8
    for (int j = 0; j < kRows; ++j) {
        float b[C];
        if constexpr (C == 4) {
            const float4 v = *reinterpret_cast<const float4 *>(b0 + j * kStride<DP>);
            b[0] = v.x; b[1] = v.y; b[2] = v.z; b[3] = v.w;
        } else {
            const float2 v = *reinterpret_cast<const float2 *>(b0 + j * kStride<DP>);
            b[0] = v.x; b[1] = v.y;
        }
        uint64_t b2[C];
#pragma unroll
        for (int c = 0; c < C; ++c) b2[c] = ptx::pack2(b[c], b[c]);
#pragma unroll
        for (int k = 0; k < R / 2; k += 2) {
            const ulonglong2 w = *reinterpret_cast<const ulonglong2 *>(W + j * kPairStride<R> + 2 * k);
#pragma unroll
            for (int c = 0; c < C; ++c) {
                acc[k][c] = ptx::fma2(w.x, b2[c], acc[k][c]);
                acc[k + 1][c] = ptx::fma2(w.y, b2[c], acc[k + 1][c]);
            }
        }
    }
}

// Row i of the warp's accumulators, the lane's channels.
template <int R2, int C>
__device__ __forceinline__ void acc_row(const uint64_t (&acc)[R2][C], int i, float (&x)[C])
{
#pragma unroll
    for (int c = 0; c < C; ++c) {
        float lo, hi;
        ptx::unpack2(acc[i >> 1][c], lo, hi);
        x[c] = (i & 1) ? hi : lo;
    }
}

__device__ __forceinline__ void store4(float *p, float4 v) { *reinterpret_cast<float4 *>(p) = v; }
__device__ __forceinline__ void store4(__nv_bfloat16 *p, float4 v)
{
    uint2 u;
    u.x = ptx::pack_bf16(v.x, v.y);
    u.y = ptx::pack_bf16(v.z, v.w);
    *reinterpret_cast<uint2 *>(p) = u;
}
__device__ __forceinline__ void store_channels(float *p, const float (&x)[4]) { store4(p, make_float4(x[0], x[1], x[2], x[3])); }
__device__ __forceinline__ void store_channels(__nv_bfloat16 *p, const float (&x)[4]) { store4(p, make_float4(x[0], x[1], x[2], x[3])); }
__device__ __forceinline__ void store_channels(float *p, const float (&x)[2]) { *reinterpret_cast<float2 *>(p) = make_float2(x[0], x[1]); }
__device__ __forceinline__ void store_channels(__nv_bfloat16 *p, const float (&x)[2]) { *reinterpret_cast<uint32_t *>(p) = ptx::pack_bf16(x[0], x[1]); }
__device__ __forceinline__ float4 acc_float4(const uint64_t (&a)[2], float f)
{
    float4 v;
    ptx::unpack2(a[0], v.x, v.y);
    ptx::unpack2(a[1], v.z, v.w);
    v.x *= f; v.y *= f; v.z *= f; v.w *= f;
    return v;
}

// The problem as the kernels see it.  patch_w_log: the patch is (64 >> patch_w_log) rows by (1 << patch_w_log) columns.
struct Geometry {
    const int32_t *half_width;
    int n_half_width, grid_h, grid_w, n_text, d, n_bh, patch_w_log;
    __host__ __device__ int patch_w() const { return 1 << patch_w_log; }
    __host__ __device__ int patch_h() const { return kRows >> patch_w_log; }
    __host__ __device__ int n_tokens() const { return n_text + grid_h * grid_w; }
};

// Where a block works: its tile of 64 tokens and its (batch, head).  Tiles are numbered text tiles of every head first
// (their lists are the longest), then the patches.
struct TileRef {
    bool text;
    int bh, first;      // text: first token
    int y, x;           // patch: top left cell
};
__device__ __forceinline__ TileRef tile_of(int id, const Geometry &g)
{
    TileRef t{};
    const int n_txt = (g.n_text + kRows - 1) / kRows;
    t.text = id < n_txt * g.n_bh;
    if (t.text) {
        t.bh = id / n_txt;
        t.first = (id - t.bh * n_txt) * kRows;
    } else {
        const int ntx = (g.grid_w + g.patch_w() - 1) >> g.patch_w_log, nty = (g.grid_h + g.patch_h() - 1) / g.patch_h();
        id -= n_txt * g.n_bh;
        t.bh = id / (ntx * nty);
        id -= t.bh * ntx * nty;
        t.y = id / ntx * g.patch_h();
        t.x = id % ntx * g.patch_w();
    }
    return t;
}
// Token of row r of the tile, or -1; qy, qx its cell.
__device__ __forceinline__ int tile_token(const TileRef &t, int r, const Geometry &g, int &qy, int &qx)
{
    qy = t.y + (r >> g.patch_w_log);
    qx = t.x + (r & (g.patch_w() - 1));
    if (t.text) return t.first + r < g.n_text ? t.first + r : -1;
    return qy < g.grid_h && qx < g.grid_w ? g.n_text + qy * g.grid_w + qx : -1;
}
__device__ __forceinline__ KeyRuns runs_of(const TileRef &t, const Geometry &g)
{
    KeyRuns k;
    k.half_width = g.half_width;
    k.n_half_width = g.n_half_width;
    k.grid_h = g.grid_h;
    k.grid_w = g.grid_w;
    k.n_text = g.n_text;
    k.n_tokens = g.n_tokens();
    k.y0 = t.y;
    k.y1 = min(t.y + g.patch_h(), g.grid_h) - 1;
    k.x0 = t.x;
    k.x1 = min(t.x + g.patch_w(), g.grid_w) - 1;
    k.text = t.text;
    return k;
}

// Does the query at (qy, qx) see the streamed token?  (Eq. 3 as half widths; ky = -1: every query of the tile does.)
__device__ __forceinline__ bool sees(const KeyRuns &k, int qy, int qx, int ky, int kx)
{
    if (k.text || ky < 0) return true;
    const int dy = abs(ky - qy);
    return dy < k.n_half_width && abs(kx - qx) <= __ldg(k.half_width + dy);
}

// Which of the R (8 or 16) rows of the tile from `row0` on see the token at (ky, kx), one bit each.
template <int R>
__device__ __forceinline__ uint32_t seen_by(const KeyRuns &k, const TileRef &t, const Geometry &g, int row0, int ky, int kx)
{
    if (k.text || ky < 0) return (1u << R) - 1u;
    const int w_log = min(g.patch_w_log, R == 16 ? 4 : 3), width = 1 << w_log;   // of the R rows, so many lie in one row of the patch
    const int x0 = t.x + (row0 & (g.patch_w() - 1));
    int dy = ky - (t.y + (row0 >> g.patch_w_log));
    uint32_t bits = 0u;
#pragma unroll 2
    for (int b = 0; b < R; b += width, --dy) {
        const int dist = abs(dy);
        if (dist >= k.n_half_width) continue;
        const int w = __ldg(k.half_width + dist), lo = max(kx - w - x0, 0), hi = min(kx + w - x0, width - 1);
        if (lo <= hi) bits |= ((2u << hi) - (1u << lo)) << b;
    }
    return bits;
}

// The list of one streamed tile in shared memory, filled by the first 64 threads a tile ahead.
struct KeyTile {
    int token[kRows], ky[kRows], kx[kRows];
};
__device__ __forceinline__ void fill_key_tile(KeyTile &t, KeyCursor &cur, const KeyRuns &k, bool in_range)
{
    if (threadIdx.x < kRows) {
        int ky = -1, kx = 0;
        const int tok = in_range ? cur.token(k, ky, kx) : -1;
        t.token[threadIdx.x] = tok;
        t.ky[threadIdx.x] = ky;
        t.kx[threadIdx.x] = kx;
        cur.advance(k, kRows);
    }
}

// ---- rows taken by themselves --------------------------------------------------------------------------------------
// A weight of 0 hides a streamed row from a query that does not see it, unless the row holds a NaN or an infinity.  So the
// rows of a tile that come out non-finite are taken again, a warp a row over the tokens that the row sees and no others:
// non-finite values reach the rows that see them, and nobody pays for the rest.
__device__ __forceinline__ bool finite4(float4 v)
{
    return fabsf(v.x) <= CUDART_MAX_NORMAL_F && fabsf(v.y) <= CUDART_MAX_NORMAL_F && fabsf(v.z) <= CUDART_MAX_NORMAL_F &&
           fabsf(v.w) <= CUDART_MAX_NORMAL_F;
}
__device__ __forceinline__ float as_float(float x) { return x; }
__device__ __forceinline__ float as_float(__nv_bfloat16 x) { return __bfloat162float(x); }
__device__ __forceinline__ void put(float *p, float x) { *p = x; }
__device__ __forceinline__ void put(__nv_bfloat16 *p, float x) { *p = __float2bfloat16_rn(x); }

// A lane's channels of a row: lane, lane + 32, ...
template <int DP> struct LaneRow {
    float c[DP / 32];
    template <typename T> __device__ __forceinline__ void load(const T *row, int d)
    {
#pragma unroll
        for (int t = 0; t < DP / 32; ++t) {
            const int e = (int)(threadIdx.x & 31) + 32 * t;
            c[t] = e < d ? as_float(row[e]) : 0.f;
        }
    }
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int t = 0; t < DP / 32; ++t) c[t] = 0.f;
    }
    __device__ __forceinline__ void add(float f, const LaneRow &o)
    {
#pragma unroll
        for (int t = 0; t < DP / 32; ++t) c[t] = fmaf(f, o.c[t], c[t]);
    }
    __device__ __forceinline__ float dot(const LaneRow &o) const
    {
        float x = 0.f;
#pragma unroll
        for (int t = 0; t < DP / 32; ++t) x = fmaf(c[t], o.c[t], x);
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) x += __shfl_xor_sync(0xffffffffu, x, s);
        return x;
    }
    template <typename T> __device__ __forceinline__ void store(T *row, int d, float f) const
    {
#pragma unroll
        for (int t = 0; t < DP / 32; ++t) {
            const int e = (int)(threadIdx.x & 31) + 32 * t;
            if (e < d) put(row + e, c[t] * f);
        }
    }
};
// body(token) for every token that the query at (qy, qx) sees, in order.
template <typename Body> __device__ __forceinline__ void for_each_seen(const KeyRuns &k, int qy, int qx, Body &&body)
{
#pragma unroll 1
    for (int t = 0; t < k.head_length(); ++t) body(t);
    if (k.text) return;
#pragma unroll 1
    for (int y = max(0, qy - (k.n_half_width - 1)); y < min(k.grid_h, qy + k.n_half_width); ++y) {
        const int w = __ldg(k.half_width + abs(y - qy));
#pragma unroll 1
        for (int x = max(qx - w, 0); x <= min(qx + w, k.grid_w - 1); ++x) body(k.n_text + y * k.grid_w + x);
    }
}

// ---- host side ---------------------------------------------------------------------------------------------------
// Tiles of one (batch, head), steps of 64 tokens of the longest list and of all lists together.
struct Extent {
    long long tiles, longest, steps;
};
Geometry geometry_of(const clear_plan &p);
Extent extent_of(const clear_plan &p, const Geometry &g);
// Blocks a list is cut over (1, 2, 4 or 8), given the blocks the device holds at once.
int split_of(const Extent &e, int n_bh, int slots);

template <typename Kernel, typename Params>
int launch_tiles(Kernel kernel, const Params &prm, long long tiles, int n_split, size_t smem, cudaStream_t stream, int threads = kThreads)
{
    if (tiles * n_split > INT32_MAX) return CLEAR_ERR_UNSUPPORTED;
    // set again on every call: a table lookup in the runtime, per device, without a lock of our own
    CLEAR_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(tiles * n_split));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)n_split;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = n_split > 1 ? 1 : 0;
    CLEAR_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, prm));
    return CLEAR_OK;
}

}  // namespace f32tile
}  // namespace clear
