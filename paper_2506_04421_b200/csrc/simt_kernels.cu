// Plain SIMT kernels for HMAR's Markovian masked attention: the fp32 debug build, the path of head dimensions 32 and 128,
// and the bf16 fall-back used while debugging the tensor-core kernels.  All arithmetic is fp32 FMA; inputs and outputs
// are float or bf16.
//
// A block of 128 threads owns a tile of up to 64 rows of ONE scale, so all of its rows see the same contiguous range of
// the other operand (mask: paper Sec. 4.1, Fig. attn-mask) and no element needs a mask but the ragged end of that range
// (calls of small scales: one warp, 16 rows; see tile_height).
// It walks the range 64 rows at a time, as small dense products from shared memory with 8 x 4 results per thread: 12
// 16-byte shared-memory loads feed 128 FMAs, which leaves the FMA pipe as the bound (a warp's loads take half of the
// shared-memory cycles its FMAs last).  One row per thread pair, an operand of every FMA from shared memory, was bound
// by those loads: B2 H16 L680 D64, forward + backward, 954 us, against 70 us of FMAs.
// Blocks are ordered tile by tile over all heads, the tiles of the last (largest) scale first, so that the costly blocks
// start first and spread over the SMs (head by head, an SM could get three of them and another none).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "hmar_common.h"
#include "launchers.h"

namespace hmar {
namespace {

// A tile has TR rows on either side, 64 or 16, and 2 TR threads: thread t has rows 8 (t / 16) .. + 7 and columns
// t % 16 + 16 j, j < TR / 16, of a TR x TR product.
constexpr int DELTA_THREADS = 128;

__device__ __forceinline__ void from_f(float* p, float x) { *p = x; }
__device__ __forceinline__ void from_f(__nv_bfloat16* p, float x) { *p = __float2bfloat16_rn(x); }

// Four consecutive elements as float.
__device__ __forceinline__ float4 load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
    const uint2 v = *reinterpret_cast<const uint2*>(p);
    return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16),
                       __uint_as_float(v.y & 0xffff0000u));
}

// Rows in shared memory are padded by four floats: 16-byte loads of eight consecutive rows then hit 32 distinct banks.
template <int D, int TR> struct RowTile { float v[TR][D + 4]; };
template <int TR> struct SquareTile { float v[TR][TR + 4]; };

// dst rows [0, TR) = src rows [0, n) as float; the rest zeros.
template <typename T, int D, int TR>
__device__ __forceinline__ void stage(RowTile<D, TR>& dst, const T* src, int n) {
#pragma unroll 8
    for (int idx = threadIdx.x; idx < TR * (D / 4); idx += 2 * TR) {
        const int r = idx / (D / 4), c = idx % (D / 4) * 4;
        *reinterpret_cast<float4*>(&dst.v[r][c]) = r < n ? load4(src + (size_t)r * D + c) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// acc[i][j] = sum_d a[r0 + i][d] b[tx + 16 j][d].  Sums of eight products are added up: one chain over all of d doubles
// the rounding error of large logits (LSE at |logits| = 30, D = 64: 1.1e-5 against 0.6e-5), and an addition per eight
// FMAs costs less than that.
template <int D, int TR>
__device__ __forceinline__ void product_nt(const RowTile<D, TR>& a, const RowTile<D, TR>& b, int r0, int tx, float (&acc)[8][TR / 16]) {
    constexpr int J = TR / 16;
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < J; ++j) acc[i][j] = 0.f;
    // two chunks of d per round for D = 128 (bf16, 32 heads of L = 680: forward 190 -> 132 us, backward 558 -> 542); D = 64 is
    // the same either way, and D = 32 1 % slower
    constexpr int UNROLL = D == 128 ? 2 : 1;
#pragma unroll UNROLL
    for (int d = 0; d < D; d += 8) {
        float4 b0[J], b1[J];
#pragma unroll
        for (int j = 0; j < J; ++j) {
            b0[j] = *reinterpret_cast<const float4*>(&b.v[tx + 16 * j][d]);
            b1[j] = *reinterpret_cast<const float4*>(&b.v[tx + 16 * j][d + 4]);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float4 a0 = *reinterpret_cast<const float4*>(&a.v[r0 + i][d]);
            const float4 a1 = *reinterpret_cast<const float4*>(&a.v[r0 + i][d + 4]);
#pragma unroll
            for (int j = 0; j < J; ++j) {
                float t = fmaf(a0.w, b0[j].w, fmaf(a0.z, b0[j].z, fmaf(a0.y, b0[j].y, a0.x * b0[j].x)));
                t = fmaf(a1.w, b1[j].w, fmaf(a1.z, b1[j].z, fmaf(a1.y, b1[j].y, fmaf(a1.x, b1[j].x, t))));
                acc[i][j] += t;
            }
        }
    }
}

// A thread's columns of a [TR x D] result: D / 16 of them, in groups of W consecutive ones that are 16 W apart.
template <int D> struct Cols {
    static constexpr int W = D >= 64 ? 4 : 2, GROUPS = D / (16 * W), N = D / 16;
};

// acc[i][.] += sum_k p[r0 + i][k] b[k][columns of the thread], k < n (a multiple of 4)
template <int D, int TR>
__device__ __forceinline__ void product_nn(const SquareTile<TR>& p, const RowTile<D, TR>& b, int r0, int tx, int n, float (&acc)[8][Cols<D>::N]) {
    constexpr int W = Cols<D>::W, G = Cols<D>::GROUPS;
#pragma unroll 2
    for (int k = 0; k < n; k += 4) {
        float4 pv[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) pv[i] = *reinterpret_cast<const float4*>(&p.v[r0 + i][k]);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
#pragma unroll
            for (int g = 0; g < G; ++g) {
                float bv[W];
                const float* src = &b.v[k + kk][g * 16 * W + tx * W];
                if (W == 4) {
                    const float4 x = *reinterpret_cast<const float4*>(src);
                    bv[0] = x.x; bv[1] = x.y; bv[W - 2] = x.z; bv[W - 1] = x.w;
                } else {
                    const float2 x = *reinterpret_cast<const float2*>(src);
                    bv[0] = x.x; bv[1] = x.y;
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float w = kk == 0 ? pv[i].x : kk == 1 ? pv[i].y : kk == 2 ? pv[i].z : pv[i].w;
#pragma unroll
                    for (int e = 0; e < W; ++e) acc[i][g * W + e] = fmaf(w, bv[e], acc[i][g * W + e]);
                }
            }
        }
    }
}

// dst[r][d] = acc * mul for the thread's rows below n
template <typename T, int D>
__device__ __forceinline__ void store_rows(T* dst, const float (&acc)[8][Cols<D>::N], const float (&mul)[8], int r0, int tx, int n) {
    constexpr int W = Cols<D>::W, G = Cols<D>::GROUPS;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        if (r0 + i >= n) break;
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
            for (int e = 0; e < W; ++e) from_f(dst + (size_t)(r0 + i) * D + g * 16 * W + tx * W + e, acc[i][g * W + e] * mul[i]);
    }
}

// Tile number `t` of a head: rows [row0, row0 + n) of scale s.  Tiles of the last scale come first.
struct TileRows { int s, row0, n; };
template <int TR>
__device__ __forceinline__ TileRows tile_rows(const ScaleTable& st, int t) {
    int s = st.n_scales - 1;
    while (true) {
        const int rows = st.start[s + 1] - st.start[s], tiles = (rows + TR - 1) / TR;
        if (t < tiles || s == 0) return {s, st.start[s] + t * TR, min(TR, rows - t * TR)};
        t -= tiles;
        --s;
    }
}

// ---------------------------------------------------------------------------------------------
// Forward and inference step.  The keys are rows [lo, hi) of one sequence, or (inference step: st has one scale, the
// queries) n0 rows of the previous scale followed by n1 of the current one.
template <int D, int TR> struct FwdSmem { RowTile<D, TR> q, k, v; SquareTile<TR> p; };

template <typename T, int D, int TR>
__global__ void __launch_bounds__(2 * TR)
simt_fwd_kernel(const T* __restrict__ q, const T* __restrict__ k0, const T* __restrict__ v0,
                const T* __restrict__ k1, const T* __restrict__ v1,
                T* __restrict__ out, float* __restrict__ lse,
                const __grid_constant__ ScaleTable st, int n_heads, int n_q, int n0, int n1, int dense, float scale) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FwdSmem<D, TR>& sm = *reinterpret_cast<FwdSmem<D, TR>*>(smem_raw);
    constexpr int J = TR / 16;
    const int bh = blockIdx.x % n_heads;
    const TileRows tile = tile_rows<TR>(st, blockIdx.x / n_heads);
    const int tx = threadIdx.x & 15, r0 = (threadIdx.x >> 4) * 8;
    const bool live = (threadIdx.x >> 5) * 16 < tile.n;     // the warp has rows of the tile
    const int lo = dense ? 0 : st.start[first_key_scale(st.window, tile.s)];
    const int hi = dense ? n0 + n1 : st.start[last_key_scale(st.window, tile.s) + 1];
    const T* kh = k0 + (size_t)bh * n0 * D;
    const T* vh = v0 + (size_t)bh * n0 * D;

    stage(sm.q, q + ((size_t)bh * n_q + tile.row0) * D, tile.n);
    float o[8][Cols<D>::N], m[8], l[8];                     // l: this thread's columns only, summed over the row at the end
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        m[i] = -INFINITY;
        l[i] = 0.f;
#pragma unroll
        for (int e = 0; e < Cols<D>::N; ++e) o[i][e] = 0.f;
    }
    for (int t = lo; t < hi;) {
        // the tile does not cross from one segment into the other
        const bool second = dense && t >= n0;
        const int n = min(TR, (dense && !second ? n0 : hi) - t);
        const T* ks = second ? k1 + ((size_t)bh * n1 + (t - n0)) * D : kh + (size_t)t * D;
        const T* vs = second ? v1 + ((size_t)bh * n1 + (t - n0)) * D : vh + (size_t)t * D;
        __syncthreads();
        stage(sm.k, ks, n);
        stage(sm.v, vs, n);
        __syncthreads();
        if (live) {
            float s[8][J];
            product_nt(sm.q, sm.k, r0, tx, s);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                float mx = -INFINITY;
#pragma unroll
                for (int j = 0; j < J; ++j) {
                    s[i][j] = tx + 16 * j < n ? s[i][j] * scale : -INFINITY;
                    mx = fmaxf(mx, s[i][j]);
                }
#pragma unroll
                for (int w = 8; w > 0; w >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, w));
                const float m_new = fmaxf(m[i], mx), corr = expf(m[i] - m_new);      // exp(-inf) = 0 on the first tile
                m[i] = m_new;
                l[i] *= corr;
#pragma unroll
                for (int e = 0; e < Cols<D>::N; ++e) o[i][e] *= corr;
#pragma unroll
                for (int j = 0; j < J; ++j) {
                    const float p = expf(s[i][j] - m_new);
                    l[i] += p;
                    sm.p.v[r0 + i][tx + 16 * j] = p;
                }
            }
            __syncwarp();                     // a row of P is written and read by the same 16 lanes
            product_nn(sm.p, sm.v, r0, tx, (n + 3) & ~3, o);
        }
        t += n;
    }
    if (!live) return;
    float inv[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
#pragma unroll
        for (int w = 8; w > 0; w >>= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], w);
        inv[i] = 1.f / l[i];
        if (lse != nullptr && tx == 0 && r0 + i < tile.n) lse[(size_t)bh * n_q + tile.row0 + r0 + i] = m[i] + logf(l[i]);
    }
    store_rows<T, D>(out + ((size_t)bh * n_q + tile.row0) * D, o, inv, r0, tx, tile.n);
}

// ---------------------------------------------------------------------------------------------
// delta_i = sum_d dO_id * O_id, in the very order in which product_nt sums a dot product: where a query has a single key,
// O is that key's V and dP - delta is exactly zero.  D / 8 threads per row, eight products each.
template <typename T, int D>
__global__ void __launch_bounds__(DELTA_THREADS)
simt_delta_kernel(const T* __restrict__ out, const T* __restrict__ dout, float* __restrict__ delta,
                  size_t n_rows) {
    constexpr int PARTS = D / 8;
    const size_t row = ((size_t)blockIdx.x * DELTA_THREADS + threadIdx.x) / PARTS;
    const int part = threadIdx.x % PARTS;
    float t = 0.f;
    if (row < n_rows) {
        const T* a = dout + row * D + part * 8;
        const T* b = out + row * D + part * 8;
        const float4 a0 = load4(a), a1 = load4(a + 4), b0 = load4(b), b1 = load4(b + 4);
        t = fmaf(a0.w, b0.w, fmaf(a0.z, b0.z, fmaf(a0.y, b0.y, a0.x * b0.x)));
        t = fmaf(a1.w, b1.w, fmaf(a1.z, b1.z, fmaf(a1.y, b1.y, fmaf(a1.x, b1.x, t))));
    }
    float acc = 0.f;
#pragma unroll
    for (int c = 0; c < PARTS; ++c) acc += __shfl_sync(0xffffffffu, t, c, PARTS);
    if (row < n_rows && part == 0) delta[row] = acc;
}

// ---------------------------------------------------------------------------------------------
// Backward: a tile's first block owns it as a key tile (dK, dV over the queries that see it), its second as a query tile
// (dQ over its keys); one launch, so that both kinds fill the chip together.  Each result has one owner that
// adds in a fixed order: the gradients are bit-reproducible.
template <int D, int TR> struct BwdSmem { RowTile<D, TR> a, b, x, y; SquareTile<TR> p; float lse[TR], delta[TR]; };

template <typename T, int D, int TR>
__global__ void __launch_bounds__(2 * TR)
simt_bwd_kernel(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v,
                const T* __restrict__ dout, const float* __restrict__ lse, const float* __restrict__ delta,
                T* __restrict__ dq, T* __restrict__ dk, T* __restrict__ dv,
                const __grid_constant__ ScaleTable st, int n_heads, int L, float scale) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    BwdSmem<D, TR>& sm = *reinterpret_cast<BwdSmem<D, TR>*>(smem_raw);
    constexpr int J = TR / 16;
    const int unit = blockIdx.x / n_heads;
    const size_t head = (size_t)(blockIdx.x - unit * n_heads) * L;
    const bool keys = (unit & 1) == 0;                      // the block owns a key tile
    const TileRows tile = tile_rows<TR>(st, unit >> 1);
    const int tx = threadIdx.x & 15, r0 = (threadIdx.x >> 4) * 8;
    const bool live = (threadIdx.x >> 5) * 16 < tile.n;     // the warp has rows of the tile
    // Own rows a, b against partner rows x, y: keys own K, V and walk Q, dO; queries own Q, dO and walk K, V.
    const T* own_a = keys ? k : q;
    const T* own_b = keys ? v : dout;
    const T* far_x = keys ? q : k;
    const T* far_y = keys ? dout : v;
    // (under HMAR_WINDOW_PREV the keys of the last scale have no queries: lo = hi, and zeros are stored)
    const int lo = st.start[keys ? first_query_scale(st.window, tile.s) : first_key_scale(st.window, tile.s)];
    const int hi = st.start[(keys ? last_query_scale(st.window, tile.s, st.n_scales) : last_key_scale(st.window, tile.s)) + 1];

    stage(sm.a, own_a + (head + tile.row0) * D, tile.n);
    stage(sm.b, own_b + (head + tile.row0) * D, tile.n);
    float row_lse[8], row_delta[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const bool in = !keys && r0 + i < tile.n;
        row_lse[i] = in ? lse[head + tile.row0 + r0 + i] : 0.f;
        row_delta[i] = in ? delta[head + tile.row0 + r0 + i] : 0.f;
    }
    constexpr int N = Cols<D>::N;
    float acc1[8][N], acc2[8][N];                           // dK and dV, or dQ and nothing
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int e = 0; e < N; ++e) acc1[i][e] = acc2[i][e] = 0.f;

    for (int t = lo; t < hi; t += TR) {
        const int n = min(TR, hi - t);
        __syncthreads();
        stage(sm.x, far_x + (head + t) * D, n);
        stage(sm.y, far_y + (head + t) * D, n);
        if (keys && threadIdx.x < TR) {
            sm.lse[threadIdx.x] = threadIdx.x < n ? lse[head + t + threadIdx.x] : 0.f;
            sm.delta[threadIdx.x] = threadIdx.x < n ? delta[head + t + threadIdx.x] : 0.f;
        }
        __syncthreads();
        if (!live) continue;
        float s[8][J], dp[8][J];
        product_nt(sm.a, sm.x, r0, tx, s);
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const int c = tx + 16 * j;
                s[i][j] = c < n ? expf(s[i][j] * scale - (keys ? sm.lse[c] : row_lse[i])) : 0.f;
            }
        if (keys) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < J; ++j) sm.p.v[r0 + i][tx + 16 * j] = s[i][j];
            __syncwarp();                     // a row of P is written and read by the same 16 lanes
            product_nn(sm.p, sm.y, r0, tx, (n + 3) & ~3, acc2);
            __syncwarp();
        }
        product_nt(sm.b, sm.y, r0, tx, dp);
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const int c = tx + 16 * j;
                sm.p.v[r0 + i][c] = s[i][j] * (dp[i][j] - (keys ? sm.delta[c] : row_delta[i]));
            }
        __syncwarp();
        product_nn(sm.p, sm.x, r0, tx, (n + 3) & ~3, acc1);
    }
    if (!live) return;
    float mul[8], one[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) { mul[i] = scale; one[i] = 1.f; }
    store_rows<T, D>((keys ? dk : dq) + (head + tile.row0) * D, acc1, mul, r0, tx, tile.n);
    if (keys) store_rows<T, D>(dv + (head + tile.row0) * D, acc2, one, r0, tx, tile.n);
}

}  // namespace

// ---------------------------------------------------------------------------------------------
// Launchers

static int count_tiles(const ScaleTable& st, int tile) {
    int n = 0;
    for (int s = 0; s < st.n_scales; ++s) n += (st.start[s + 1] - st.start[s] + tile - 1) / tile;
    return n;
}

// Height of a call's tiles.  A block of 64 rows of which a scale fills one to sixteen spends its time on rows that are not
// there, and its 53 to 153 KB of shared memory keep an SM at one to four blocks; a block of 16 rows is one warp in 14 to 34 KB.
// us with 64 and 16 rows: fp32 forward + backward of sides (1, 2), 960 heads 152 and 39, of (1, 2, 3, 4) 312 and 80; bf16
// D = 128 (1, 2, 3), 256 heads 256 and 45; fp32 step 1 -> 2, 1536 heads 41 and 12.  At 17 to 36 rows the many products
// per load of a high tile count for more until the chip is full: (1, 2, 4, 6) 4 heads 28.7 and 39, 64 heads 41 and 39, 512
// heads 207 and 115; (5, 6) 64 heads 37 and 43, 512 heads 155 and 127.  Beyond that the high tiles win at any number of heads
// ((7, 8), 512 heads 252 and 319).
static int tile_height(const ScaleTable& st, int BH, int n_prev) {
    int rows = n_prev;                  // inference step: the previous scale, walked as far as the current one
    for (int s = 0; s < st.n_scales; ++s) rows = std::max(rows, st.start[s + 1] - st.start[s]);
    return rows <= 16 || (rows <= 36 && (long long)count_tiles(st, 64) * BH >= 512) ? 16 : 64;
}

template <typename T, int D, int TR>
static cudaError_t simt_fwd_tiles(const T* q, const T* k0, const T* v0, const T* k1, const T* v1, T* out, float* lse, int BH,
                                const ScaleTable& st, int n_q, int n0, int n1, int dense, float scale, cudaStream_t stream) {
    static SmemOptIn opt_in;
    const cudaError_t e = opt_in((const void*)simt_fwd_kernel<T, D, TR>, sizeof(FwdSmem<D, TR>));
    if (e != cudaSuccess) return e;
    simt_fwd_kernel<T, D, TR><<<(unsigned)count_tiles(st, TR) * BH, 2 * TR, sizeof(FwdSmem<D, TR>), stream>>>(q, k0, v0, k1, v1, out, lse, st, BH,
                                                                                                           n_q, n0, n1, dense, scale);
    count_launch(1);
    return cudaGetLastError();
}

template <typename T, int D>
static cudaError_t simt_fwd_any(const T* q, const T* k0, const T* v0, const T* k1, const T* v1, T* out, float* lse, int BH,
                                const ScaleTable& st, int n_q, int n0, int n1, int dense, float scale, cudaStream_t stream) {
    return tile_height(st, BH, dense ? n0 : 0) == 16 ? simt_fwd_tiles<T, D, 16>(q, k0, v0, k1, v1, out, lse, BH, st, n_q, n0, n1, dense, scale, stream)
                                                     : simt_fwd_tiles<T, D, 64>(q, k0, v0, k1, v1, out, lse, BH, st, n_q, n0, n1, dense, scale, stream);
}

template <typename T, int D>
static cudaError_t simt_fwd_d(const T* q, const T* k, const T* v, T* out, float* lse, int BH,
                              const ScaleTable& st, float scale, cudaStream_t stream) {
    const int L = st.start[st.n_scales];
    return simt_fwd_any<T, D>(q, k, v, nullptr, nullptr, out, lse, BH, st, L, L, 0, 0, scale, stream);
}

template <typename T, int D>
static cudaError_t simt_scale_step_d(const T* q, const T* k_prev, const T* v_prev, const T* k_cur, const T* v_cur,
                                     T* out, float* lse, int BH, int n_prev, int n_cur, float scale,
                                     cudaStream_t stream) {
    ScaleTable st{};
    st.n_scales = 1;
    st.start[1] = n_cur;
    if (n_prev > 0)
        return simt_fwd_any<T, D>(q, k_prev, v_prev, k_cur, v_cur, out, lse, BH, st, n_cur, n_prev, n_cur, 1, scale, stream);
    return simt_fwd_any<T, D>(q, k_cur, v_cur, nullptr, nullptr, out, lse, BH, st, n_cur, n_cur, 0, 1, scale, stream);
}

template <typename T, int D, int TR>
static cudaError_t simt_bwd_tiles(const T* q, const T* k, const T* v, const float* lse, const T* dout, T* dq, T* dk, T* dv,
                                  const float* delta, int BH, const ScaleTable& st, float scale, cudaStream_t stream) {
    static SmemOptIn opt_in;
    const cudaError_t e = opt_in((const void*)simt_bwd_kernel<T, D, TR>, sizeof(BwdSmem<D, TR>));
    if (e != cudaSuccess) return e;
    simt_bwd_kernel<T, D, TR><<<2u * count_tiles(st, TR) * BH, 2 * TR, sizeof(BwdSmem<D, TR>), stream>>>(q, k, v, dout, lse, delta, dq, dk, dv, st, BH,
                                                                                                      st.start[st.n_scales], scale);
    return cudaGetLastError();
}

template <typename T, int D>
static cudaError_t simt_bwd_d(const T* q, const T* k, const T* v, const T* out, const float* lse, const T* dout,
                              T* dq, T* dk, T* dv, float* delta, int BH, const ScaleTable& st, float scale,
                              cudaStream_t stream) {
    const size_t n_rows = (size_t)BH * st.start[st.n_scales];
    constexpr int ROWS = DELTA_THREADS / (D / 8);
    simt_delta_kernel<T, D><<<(unsigned)((n_rows + ROWS - 1) / ROWS), DELTA_THREADS, 0, stream>>>(out, dout, delta, n_rows);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess)
        e = tile_height(st, BH, 0) == 16 ? simt_bwd_tiles<T, D, 16>(q, k, v, lse, dout, dq, dk, dv, delta, BH, st, scale, stream)
                                         : simt_bwd_tiles<T, D, 64>(q, k, v, lse, dout, dq, dk, dv, delta, BH, st, scale, stream);
    if (e == cudaSuccess) count_launch(2);
    return e;
}

// The public launchers pick the instantiation for the head dimension (32, 64 or 128; checked by the caller).
#define HMAR_BY_D(call32, call64, call128) (D == 32 ? (call32) : (D == 128 ? (call128) : (call64)))

template <typename T>
cudaError_t simt_fwd(const T* q, const T* k, const T* v, T* out, float* lse, int BH, int D,
                     const ScaleTable& st, float scale, cudaStream_t stream) {
    return HMAR_BY_D((simt_fwd_d<T, 32>(q, k, v, out, lse, BH, st, scale, stream)), (simt_fwd_d<T, 64>(q, k, v, out, lse, BH, st, scale, stream)),
                     (simt_fwd_d<T, 128>(q, k, v, out, lse, BH, st, scale, stream)));
}

template <typename T>
cudaError_t simt_scale_step(const T* q, const T* k_prev, const T* v_prev, const T* k_cur, const T* v_cur,
                            T* out, float* lse, int BH, int D, int n_prev, int n_cur, float scale,
                            cudaStream_t stream) {
    return HMAR_BY_D((simt_scale_step_d<T, 32>(q, k_prev, v_prev, k_cur, v_cur, out, lse, BH, n_prev, n_cur, scale, stream)),
                     (simt_scale_step_d<T, 64>(q, k_prev, v_prev, k_cur, v_cur, out, lse, BH, n_prev, n_cur, scale, stream)),
                     (simt_scale_step_d<T, 128>(q, k_prev, v_prev, k_cur, v_cur, out, lse, BH, n_prev, n_cur, scale, stream)));
}

template <typename T>
cudaError_t simt_bwd(const T* q, const T* k, const T* v, const T* out, const float* lse, const T* dout,
                     T* dq, T* dk, T* dv, float* delta, int BH, int D, const ScaleTable& st, float scale,
                     cudaStream_t stream) {
    return HMAR_BY_D((simt_bwd_d<T, 32>(q, k, v, out, lse, dout, dq, dk, dv, delta, BH, st, scale, stream)),
                     (simt_bwd_d<T, 64>(q, k, v, out, lse, dout, dq, dk, dv, delta, BH, st, scale, stream)),
                     (simt_bwd_d<T, 128>(q, k, v, out, lse, dout, dq, dk, dv, delta, BH, st, scale, stream)));
}

#define INSTANTIATE(T)                                                                                        \
    template cudaError_t simt_fwd<T>(const T*, const T*, const T*, T*, float*, int, int, const ScaleTable&,   \
                                     float, cudaStream_t);                                                    \
    template cudaError_t simt_scale_step<T>(const T*, const T*, const T*, const T*, const T*, T*, float*,     \
                                            int, int, int, int, float, cudaStream_t);                         \
    template cudaError_t simt_bwd<T>(const T*, const T*, const T*, const T*, const float*, const T*, T*,      \
                                     T*, T*, float*, int, int, const ScaleTable&, float, cudaStream_t);
INSTANTIATE(float)
INSTANTIATE(__nv_bfloat16)

}  // namespace hmar
