// Learned predictor of the block sensor maxima: three 3x3 convolutions (cin -> H -> H -> 1, ReLU
// after the first two, zero padding), trained with a mean-square loss and Adam.  Not part of the
// paper: it lets a dynamic regrid (Sec. 5.2) refine ahead of the flow, with the Knudsen sensor as
// the judge of its flags.
//
// Precision: weights, biases and activations are stored in BF16; every product is accumulated in
// FP32; the master copy of the parameters, their gradients and the Adam moments are FP32, as are
// the gradients of the activations and the network output.  The layers are small (at most 16 x 16
// x 9 weights), so each kernel keeps its weights in shared memory and works on a staged tile of
// pixels; sums over pixels are added in a fixed order, so a training step is deterministic.
//
// A training step of 16 x 64 x 64 pixels (1.1 GFLOP, 16 us at the FP32 rate) takes 106 us in an
// epoch, 780 us before the kernels were tiled (the weight gradients took 960 us of 1080 us of
// serialised kernel time, now 30 us of 84) and 144 us while each step gathered its minibatch in two
// launches and the host waited for its loss.  The launches overlap their starts with the end of the
// one before (launch_pdl).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <new>
#include <vector>

#include "../../include/lbm.h"
#include "lbm_internal.h"

namespace lbm {
namespace net {
namespace {

using bf16 = __nv_bfloat16;
constexpr int NT = 256;           // threads of the pixel kernels
constexpr int MAX_CIN = 8;

struct Norm {
    float shift[MAX_CIN], scale[MAX_CIN];
};

// The layers' kernels work on tiles of TILE_X x TILE_Y pixels of one batch item, staged with their
// one-pixel border in shared memory.  A thread takes four neighbouring pixels of a row and four of
// the output channels: for one input channel and window row it reads six pixels (a 16- and an 8-byte
// load) and three weight vectors for 48 multiply-adds, so that the multiply-adds, not the
// shared-memory reads, bound the loop.  The sums run over channel, row and column of the window in
// that order.
constexpr int TILE_X = 32, TILE_Y = 4, PX = 4;
constexpr int TILE_QUADS = TILE_X / PX;  // pixel groups of a row
constexpr int ROW_PITCH = 36;            // staged row: TILE_X + 2 pixels, 16-byte multiples

struct Tiling {
    int H, W, tiles_x, tiles_y;
    __host__ __device__ Tiling(int h, int w, int th)
        : H(h), W(w), tiles_x((w + TILE_X - 1) / TILE_X), tiles_y((h + th - 1) / th) {}
    __host__ __device__ long long tiles(int B) const { return (long long)B * tiles_x * tiles_y; }
    __device__ void origin(long long t, int th, int &b, int &y0, int &x0) const {
        x0 = (int)(t % tiles_x) * TILE_X;
        y0 = (int)((t / tiles_x) % tiles_y) * th;
        b = (int)(t / ((long long)tiles_x * tiles_y));
    }
};

__device__ __forceinline__ float to_float(float v) { return v; }
__device__ __forceinline__ float to_float(bf16 v) { return __bfloat162float(v); }

// Two neighbouring pixels as loaded.
template <class T>
struct Two;
template <>
struct Two<float> {
    using V = float2;
    static __device__ __forceinline__ float2 widen(V v) { return v; }
};
template <>
struct Two<bf16> {
    using V = __nv_bfloat162;
    static __device__ __forceinline__ float2 widen(V v) { return __bfloat1622float2(v); }
};
template <class T>
__device__ __forceinline__ bool pairs_aligned(const T *p, int W) {
    return W % 2 == 0 && reinterpret_cast<uintptr_t>(p) % (2 * sizeof(T)) == 0;
}

// Copy columns x0 .. x0 + TILE_X of rows y0 .. y0 + RW of C planes of batch item b to shared memory,
// zero outside the image: pixel (c, y0 + r, x0 + col) at xs[c * pitch_c + r * pitch_r + col].
// Every thread issues all its loads (two pixels each where rows are aligned for it) before it
// stores any: one round of memory latency a tile.
template <int C, int RW, int THREADS, class T, class Map>
__device__ __forceinline__ void stage_rows(const T *__restrict__ in, int b, int y0, int x0,
                                           const Tiling &g, float *xs, int pitch_c, int pitch_r,
                                           Map &&map) {
    using V = typename Two<T>::V;
    constexpr int UNITS = C * RW * (TILE_X / 2), N = (UNITS + THREADS - 1) / THREADS;
    const bool aligned = pairs_aligned(in, g.W);
    V v[N];
#pragma unroll
    for (int n = 0; n < N; ++n) {
        const int k = n * THREADS + threadIdx.x;
        const int row = k / (TILE_X / 2), c = row / RW, y = y0 + row % RW;
        const int x = x0 + k % (TILE_X / 2) * 2;
        const T *p = in + (((size_t)b * C + c) * g.H + y) * g.W + x;
        const bool rows = k < UNITS && y >= 0 && y < g.H;
        v[n] = V();
        if (aligned) {
            if (rows && x < g.W) v[n] = *reinterpret_cast<const V *>(p);
        } else {
            if (rows && x < g.W) v[n].x = p[0];
            if (rows && x + 1 < g.W) v[n].y = p[1];
        }
    }
#pragma unroll
    for (int n = 0; n < N; ++n) {
        const int k = n * THREADS + threadIdx.x;
        if (k >= UNITS) break;
        const int row = k / (TILE_X / 2), c = row / RW, y = y0 + row % RW;
        const int col = k % (TILE_X / 2) * 2, x = x0 + col;
        const bool in_rows = y >= 0 && y < g.H;
        const float2 f = Two<T>::widen(v[n]);
        float *q = xs + c * pitch_c + row % RW * pitch_r + col;
        q[0] = in_rows && x < g.W ? map(c, f.x) : 0.f;
        q[1] = in_rows && x + 1 < g.W ? map(c, f.y) : 0.f;
    }
}

// The same with a border of one pixel: rows y0 - 1 .. y0 + ROWS, columns x0 - 1 .. x0 + TILE_X,
// pixel (c, y0 + r - 1, x0 + col - 1) at xs[c * pitch_c + r * ROW_PITCH + col].
template <int C, int ROWS, int THREADS, class T, class Map>
__device__ __forceinline__ void stage_window(const T *__restrict__ in, int b, int y0, int x0,
                                             const Tiling &g, float *xs, int pitch_c, Map &&map) {
    constexpr int RW = ROWS + 2, EDGE = C * RW * 2, N = (EDGE + THREADS - 1) / THREADS;
    T e[N];
#pragma unroll
    for (int n = 0; n < N; ++n) {  // the border columns
        const int k = n * THREADS + threadIdx.x;
        const int row = k / 2, c = row / RW, y = y0 + row % RW - 1;
        const int x = k % 2 ? x0 + TILE_X : x0 - 1;
        e[n] = T(0.f);
        if (k < EDGE && y >= 0 && y < g.H && x >= 0 && x < g.W)
            e[n] = in[(((size_t)b * C + c) * g.H + y) * g.W + x];
    }
    stage_rows<C, RW, THREADS>(in, b, y0 - 1, x0, g, xs + 1, pitch_c, ROW_PITCH, map);
#pragma unroll
    for (int n = 0; n < N; ++n) {
        const int k = n * THREADS + threadIdx.x;
        if (k >= EDGE) break;
        const int row = k / 2, c = row / RW, y = y0 + row % RW - 1;
        const int x = k % 2 ? x0 + TILE_X : x0 - 1;
        const bool in_image = y >= 0 && y < g.H && x >= 0 && x < g.W;
        xs[c * pitch_c + row % RW * ROW_PITCH + (k % 2 ? TILE_X + 1 : 0)] =
            in_image ? map(c, to_float(e[n])) : 0.f;
    }
}

// A layer's weights as its kernel reads them, FP32 [channel][tap][4-vectors of channels]: copied
// to shared memory by 16-byte loads, all in flight at once.
template <int FLOATS, int THREADS>
__device__ __forceinline__ void stage_weights(const float *__restrict__ w, float *ws) {
    constexpr int UNITS = FLOATS / 4, N = (UNITS + THREADS - 1) / THREADS;
    static_assert(FLOATS % 4 == 0, "whole vectors");
    float4 v[N];
#pragma unroll
    for (int n = 0; n < N; ++n) {
        const int k = n * THREADS + threadIdx.x;
        if (k < UNITS) v[n] = reinterpret_cast<const float4 *>(w)[k];
    }
#pragma unroll
    for (int n = 0; n < N; ++n) {
        const int k = n * THREADS + threadIdx.x;
        if (k < UNITS) reinterpret_cast<float4 *>(ws)[k] = v[n];
    }
}

__device__ __forceinline__ void fma_quad(const float4 w, float v, float (&acc)[4]) {
    acc[0] = fmaf(w.x, v, acc[0]);
    acc[1] = fmaf(w.y, v, acc[1]);
    acc[2] = fmaf(w.z, v, acc[2]);
    acc[3] = fmaf(w.w, v, acc[3]);
}

// Six staged pixels from column `col` (a multiple of 4) of a row.
__device__ __forceinline__ void load_six(const float *row, int col, float (&v)[6]) {
    const float4 p = *reinterpret_cast<const float4 *>(row + col);
    const float2 q = *reinterpret_cast<const float2 *>(row + col + 4);
    v[0] = p.x, v[1] = p.y, v[2] = p.z, v[3] = p.w, v[4] = q.x, v[5] = q.y;
}

// Store up to four neighbouring BF16 / FP32 values of a row (one vector store where `vec`).
__device__ __forceinline__ void store_px(bf16 *p, const float (&v)[PX], int n, bool vec) {
    if (vec) {
        __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]), b = __floats2bfloat162_rn(v[2], v[3]);
        uint2 u;
        u.x = *reinterpret_cast<unsigned *>(&a);
        u.y = *reinterpret_cast<unsigned *>(&b);
        *reinterpret_cast<uint2 *>(p) = u;
        return;
    }
#pragma unroll
    for (int k = 0; k < PX; ++k)
        if (k < n) p[k] = __float2bfloat16_rn(v[k]);
}
__device__ __forceinline__ void store_px(float *p, const float (&v)[PX], int n, bool vec) {
    if (vec) {
        *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
        return;
    }
#pragma unroll
    for (int k = 0; k < PX; ++k)
        if (k < n) p[k] = v[k];
}

// Where the items of a minibatch lie in the training set: item b is row idx[b] of nrows, or row b
// without idx.  An index outside the set sets *bad and reads row 0.
struct Rows {
    const int *idx;
    long long nrows;
    int *bad;
    __device__ __forceinline__ int of(int b) const {
        if (!idx) return b;
        const int r = idx[b];
        if (r >= 0 && r < nrows) return r;
        *bad = 1;
        return 0;
    }
};

// out[b, o, y, x] = relu(bias[o] + sum_{c,i,j} W[o, c, i, j] in[b, c, y+i-1, x+j-1]).  FIRST: the
// input is the caller's FP32 field, normalised and rounded to BF16 as it is staged (and kept in x0,
// which the weight gradient reads); else BF16 activations.  2 x TILE_Y x COUT threads.  At 16 x 64
// x 64, 16 -> 16 channels: 28.2 -> 12.1 us against one pixel a thread; 4 -> 16 with the
// normalisation: 10.0 + 5.4 -> 6.7 us.  FIRST takes its items where `rows` says, so a minibatch needs
// no gather of its own.
template <int CIN, int COUT, bool FIRST>
__global__ void __launch_bounds__(TILE_QUADS *TILE_Y *(COUT / 4))
    k_conv_relu(const void *__restrict__ in, const Norm nm, bf16 *__restrict__ x0_out,
                const float *__restrict__ W, const bf16 *__restrict__ bias, const Tiling g,
                bf16 *__restrict__ out, const Rows rows) {
    constexpr int THREADS = TILE_QUADS * TILE_Y * (COUT / 4);
    in = pdl_wait(in);
    W = pdl_order(W);
    bias = pdl_order(bias);
    constexpr int PITCH = (TILE_Y + 2) * ROW_PITCH;
    __shared__ __align__(16) float ws[CIN * 9 * COUT];
    __shared__ __align__(16) float xs[CIN * PITCH];
    int b, y0, x0;
    g.origin(blockIdx.x, TILE_Y, b, y0, x0);
    stage_weights<CIN * 9 * COUT, THREADS>(W, ws);  // [c][tap][o]
    if constexpr (FIRST) {
        stage_window<CIN, TILE_Y, THREADS>(
            static_cast<const float *>(in), rows.of(b), y0, x0, g, xs, PITCH,
            [&](int c, float v) {
                return __bfloat162float(__float2bfloat16_rn((v - nm.shift[c]) * nm.scale[c]));
            });
    } else {
        stage_window<CIN, TILE_Y, THREADS>(static_cast<const bf16 *>(in), b, y0, x0, g, xs, PITCH,
                                           [](int, float v) { return v; });
    }
    __syncthreads();
    const int xq = threadIdx.x % TILE_QUADS, row = (threadIdx.x / TILE_QUADS) % TILE_Y;
    const int o0 = threadIdx.x / (TILE_QUADS * TILE_Y) * 4;
    float acc[PX][4];
#pragma unroll
    for (int p = 0; p < PX; ++p)
#pragma unroll
        for (int o = 0; o < 4; ++o) acc[p][o] = __bfloat162float(bias[o0 + o]);
#pragma unroll 2
    for (int c = 0; c < CIN; ++c)
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            float v[6];
            load_six(xs + c * PITCH + (row + i) * ROW_PITCH, xq * PX, v);
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const float4 w = *reinterpret_cast<const float4 *>(ws + (c * 9 + i * 3 + j) * COUT + o0);
#pragma unroll
                for (int p = 0; p < PX; ++p) fma_quad(w, v[p + j], acc[p]);
            }
        }
    const int x = x0 + xq * PX, y = y0 + row, left = g.W - x;
    if (y >= g.H || left <= 0) return;
    const bool vec = left >= PX && g.W % PX == 0;
#pragma unroll
    for (int o = 0; o < 4; ++o) {
        float v[PX];
#pragma unroll
        for (int p = 0; p < PX; ++p) v[p] = fmaxf(acc[p][o], 0.f);
        store_px(out + (((size_t)b * COUT + o0 + o) * g.H + y) * g.W + x, v, left, vec);
    }
    if constexpr (FIRST) {  // this tile's part of the normalised input, exact in BF16
        for (int c = o0 / 4; c < CIN; c += COUT / 4) {
            float v[6];
            load_six(xs + c * PITCH + (row + 1) * ROW_PITCH, xq * PX, v);
            const float u[PX] = {v[1], v[2], v[3], v[4]};
            store_px(x0_out + (((size_t)b * CIN + c) * g.H + y) * g.W + x, u, left, vec);
        }
    }
}

// The output layer y[b, y, x] = bias + sum W[0, c, i, j] in[b, c, y+i-1, x+j-1], each of the
// OUT_GROUPS warps of a tile taking a group of the input channels, whose sums are added in order.
// GRAD: also dy = 2 (y - t) / n and the CTA's sum of (y - t)^2; a CTA walks tiles in a fixed
// order, so the sums are deterministic.
constexpr int OUT_GROUPS = 4;
constexpr int OUT_THREADS = TILE_QUADS * TILE_Y * OUT_GROUPS;
constexpr int LOSS_SLOTS = 1024;  // steps queued at most before the host reads their losses
constexpr int LOSS_PARTS = 512;  // CTAs of the output layer at most, one partial sum each

template <int CIN, bool GRAD>
__global__ void __launch_bounds__(OUT_THREADS)
    k_conv_out(const bf16 *__restrict__ in, const bf16 *__restrict__ W, const bf16 *__restrict__ bias,
               const Tiling g, long long tiles, float *__restrict__ out, const float *__restrict__ t,
               float two_n, float *__restrict__ dy, double *__restrict__ loss_part, const Rows rows) {
    in = pdl_wait(in);
    W = pdl_order(W);
    bias = pdl_order(bias);
    static_assert(CIN % OUT_GROUPS == 0 && OUT_THREADS == TILE_X * TILE_Y, "unsupported layer shape");
    constexpr int PITCH = (TILE_Y + 2) * ROW_PITCH, CPT = CIN / OUT_GROUPS;
    __shared__ __align__(16) float xs[CIN * PITCH];
    __shared__ __align__(16) float part[OUT_GROUPS][TILE_Y][TILE_X];
    __shared__ float ws[CIN * 9];
    __shared__ double sh[OUT_THREADS / 32];
    for (int k = threadIdx.x; k < CIN * 9; k += OUT_THREADS) ws[k] = __bfloat162float(W[k]);
    const float b0 = __bfloat162float(bias[0]);
    const int xq = threadIdx.x % TILE_QUADS, row = (threadIdx.x / TILE_QUADS) % TILE_Y;
    const int grp = threadIdx.x / (TILE_QUADS * TILE_Y);
    const int px = threadIdx.x % TILE_X, py = threadIdx.x / TILE_X;  // the pixel this thread ends
    double loss = 0.0;
    for (long long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        int b, y0, x0;
        g.origin(tile, TILE_Y, b, y0, x0);
        __syncthreads();  // the last tile's window and sums have been read
        stage_window<CIN, TILE_Y, OUT_THREADS>(in, b, y0, x0, g, xs, PITCH,
                                               [](int, float v) { return v; });
        __syncthreads();
        float acc[PX] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int cc = 0; cc < CPT; ++cc) {
            const int c = grp * CPT + cc;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                float v[6];
                load_six(xs + c * PITCH + (row + i) * ROW_PITCH, xq * PX, v);
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    const float w = ws[c * 9 + i * 3 + j];
#pragma unroll
                    for (int p = 0; p < PX; ++p) acc[p] = fmaf(w, v[p + j], acc[p]);
                }
            }
        }
        *reinterpret_cast<float4 *>(&part[grp][row][xq * PX]) =
            make_float4(acc[0], acc[1], acc[2], acc[3]);
        __syncthreads();
        const int x = x0 + px, y = y0 + py;
        if (x < g.W && y < g.H) {
            float v = b0;
#pragma unroll
            for (int k = 0; k < OUT_GROUPS; ++k) v += part[k][py][px];
            const size_t at = ((size_t)b * g.H + y) * g.W + x;
            out[at] = v;
            if (GRAD) {
                const float d = v - t[((size_t)rows.of(b) * g.H + y) * g.W + x];
                dy[at] = two_n * d;
                loss += (double)d * (double)d;
            }
        }
    }
    if (GRAD) {
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, off);
        if (threadIdx.x % 32 == 0) sh[threadIdx.x / 32] = loss;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
            for (int k = 0; k < OUT_THREADS / 32; ++k) s += sh[k];
            loss_part[blockIdx.x] = s;
        }
    }
}

// dA[b, c, y, x] = (A > 0) * sum_{o,i,j} W[o, c, i, j] dO[b, o, y-i+1, x-j+1]: the forward tiling
// with the window walked backwards and the input channels as outputs.  16 -> 16 channels at 16 x 64
// x 64: 29.2 -> 13.9 us.
template <int CIN, int COUT>
__global__ void __launch_bounds__(TILE_QUADS *TILE_Y *(CIN / 4))
    k_conv_bwd_data(const float *__restrict__ dO, const float *__restrict__ W,
                    const bf16 *__restrict__ A, const Tiling g, float *__restrict__ dA) {
    dO = pdl_wait(dO);
    W = pdl_order(W);
    A = pdl_order(A);
    constexpr int THREADS = TILE_QUADS * TILE_Y * (CIN / 4);
    constexpr int PITCH = (TILE_Y + 2) * ROW_PITCH;
    __shared__ __align__(16) float ws[COUT * 9 * CIN];
    __shared__ __align__(16) float xs[COUT * PITCH];
    int b, y0, x0;
    g.origin(blockIdx.x, TILE_Y, b, y0, x0);
    stage_weights<COUT * 9 * CIN, THREADS>(W, ws);  // [o][tap][c]
    stage_window<COUT, TILE_Y, THREADS>(dO, b, y0, x0, g, xs, PITCH, [](int, float v) { return v; });
    __syncthreads();
    const int xq = threadIdx.x % TILE_QUADS, row = (threadIdx.x / TILE_QUADS) % TILE_Y;
    const int c0 = threadIdx.x / (TILE_QUADS * TILE_Y) * 4;
    float acc[PX][4];
#pragma unroll
    for (int p = 0; p < PX; ++p)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[p][c] = 0.f;
#pragma unroll 2
    for (int o = 0; o < COUT; ++o)
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            float v[6];
            load_six(xs + o * PITCH + (row + 2 - i) * ROW_PITCH, xq * PX, v);
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const float4 w = *reinterpret_cast<const float4 *>(ws + (o * 9 + i * 3 + j) * CIN + c0);
#pragma unroll
                for (int p = 0; p < PX; ++p) fma_quad(w, v[p + 2 - j], acc[p]);
            }
        }
    const int x = x0 + xq * PX, y = y0 + row, left = g.W - x;
    if (y >= g.H || left <= 0) return;
    const bool vec = left >= PX && g.W % PX == 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const size_t at = (((size_t)b * CIN + c0 + c) * g.H + y) * g.W + x;
        float v[PX];
#pragma unroll
        for (int p = 0; p < PX; ++p)
            v[p] = p < left && __bfloat162float(A[at + p]) > 0.f ? acc[p][c] : 0.f;
        store_px(dA + at, v, left, vec);
    }
}

__device__ __forceinline__ float warp_sum(float s) {
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    return s;
}

// Weight and bias gradients of one layer,
//     gW[o, c, i, j] = sum_{b,y,x} dO[b, o, y, x] A[b, c, y+i-1, x+j-1],   gb[o] = sum dO[b, o],
// as partial sums of one CTA each: the CTA walks tiles of TILE_X x WG_ROWS pixels (every
// `ctas`-th), staged in shared memory.  A thread keeps the 9 taps of one input channel and (where
// there are four) four output channels in registers and takes every STREAMS-th pixel group: 4 + 6
// staged vectors for 144 multiply-adds.  The CTA's streams are added in order, and k_net_reduce
// adds the CTAs' sums in order: deterministic.  With one CTA an (out, in) channel pair, every
// thread of which loaded 9 + 1 values for 9 multiply-adds and in 16 to 256 CTAs of one wave, the
// three layers took 320 us each at 16 x 64 x 64; all three together now take 30.5 us.
constexpr int WG_THREADS = 256, WG_ROWS = 8, WG_MAX_CTAS = 304;
constexpr int WG_PITCH_A = (WG_ROWS + 2) * ROW_PITCH + 4;  // conflict-free across channels
constexpr int WG_PITCH_O = WG_ROWS * TILE_X;

__host__ __device__ constexpr int wg_smem_floats(int cin, int cout) {
    const int tile = cin * WG_PITCH_A + cout * WG_PITCH_O;
    const int red = WG_THREADS * 9 * (cout >= 4 ? 4 : 1);
    return tile > red ? tile : red;
}

template <int CIN, int COUT>
__device__ void conv_bwd_weight(const float *__restrict__ dO, const bf16 *__restrict__ A,
                                const Tiling &g, long long tiles, int cta, int ctas, float *sm,
                                float *__restrict__ part) {
    constexpr int OPT = COUT >= 4 ? 4 : 1, COMB = COUT / OPT * CIN, STREAMS = WG_THREADS / COMB;
    constexpr int QUADS = WG_ROWS * TILE_QUADS, NW = COUT * CIN * 9;
    float *xa = sm, *xo = sm + CIN * WG_PITCH_A;
    const int stream = threadIdx.x / COMB, comb = threadIdx.x % COMB;
    const int c = comb % CIN, o0 = comb / CIN * OPT;
    float acc[OPT][9], bsum = 0.f;
#pragma unroll
    for (int o = 0; o < OPT; ++o)
#pragma unroll
        for (int k = 0; k < 9; ++k) acc[o][k] = 0.f;
    for (long long tile = cta; tile < tiles; tile += ctas) {
        int b, y0, x0;
        g.origin(tile, WG_ROWS, b, y0, x0);
        __syncthreads();
        stage_window<CIN, WG_ROWS, WG_THREADS>(A, b, y0, x0, g, xa, WG_PITCH_A,
                                               [](int, float v) { return v; });
        stage_rows<COUT, WG_ROWS, WG_THREADS>(dO, b, y0, x0, g, xo, WG_PITCH_O, TILE_X,
                                              [](int, float v) { return v; });
        __syncthreads();
        if (stream < STREAMS)
            for (int q = stream; q < QUADS; q += STREAMS) {
                const int r = q / TILE_QUADS, col = q % TILE_QUADS * PX, left = g.W - x0 - col;
                if (y0 + r >= g.H || left <= 0) continue;
                float4 d[OPT];
#pragma unroll
                for (int o = 0; o < OPT; ++o)
                    d[o] = *reinterpret_cast<const float4 *>(xo + (o0 + o) * WG_PITCH_O + r * TILE_X + col);
                const int px = left < PX ? left : PX;  // fewer where the image's edge cuts the group
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    float v[6];
                    load_six(xa + c * WG_PITCH_A + (r + i) * ROW_PITCH, col, v);
                    const auto add = [&](int p, float (&dp)[OPT]) {
#pragma unroll
                        for (int j = 0; j < 3; ++j)
#pragma unroll
                            for (int o = 0; o < OPT; ++o)
                                acc[o][i * 3 + j] = fmaf(dp[o], v[p + j], acc[o][i * 3 + j]);
                    };
                    float dp[PX][OPT];
#pragma unroll
                    for (int o = 0; o < OPT; ++o)
                        dp[0][o] = d[o].x, dp[1][o] = d[o].y, dp[2][o] = d[o].z, dp[3][o] = d[o].w;
                    if (px == PX) {
#pragma unroll
                        for (int p = 0; p < PX; ++p) add(p, dp[p]);
                    } else {
#pragma unroll
                        for (int p = 0; p < PX - 1; ++p)
                            if (p < px) add(p, dp[p]);
                    }
                }
            }
        // biases: a warp sums the tile of an output channel
        for (int o = threadIdx.x / 32; o < COUT; o += WG_THREADS / 32) {
            float s = 0.f;
#pragma unroll
            for (int k = 0; k < WG_PITCH_O / 32; ++k) s += xo[o * WG_PITCH_O + k * 32 + threadIdx.x % 32];
            // lane l keeps the sum of output channel warp + 8 l
            s = warp_sum(s);
            if (threadIdx.x % 32 == o / (WG_THREADS / 32)) bsum += s;
        }
    }
    __syncthreads();
#pragma unroll
    for (int o = 0; o < OPT; ++o)
#pragma unroll
        for (int k = 0; k < 9; ++k) sm[(o * 9 + k) * WG_THREADS + threadIdx.x] = acc[o][k];
    __syncthreads();
    float *p = part + (size_t)cta * (NW + COUT);
    for (int e = threadIdx.x; e < NW; e += WG_THREADS) {
        const int o = e / (CIN * 9), cc = e / 9 % CIN, tap = e % 9;
        const int from = (o % OPT * 9 + tap) * WG_THREADS + o / OPT * CIN + cc;
        float s = 0.f;
        for (int k = 0; k < STREAMS; ++k) s += sm[from + k * COMB];
        p[e] = s;
    }
    const int ob = threadIdx.x / 32 + threadIdx.x % 32 * (WG_THREADS / 32);
    if (ob < COUT) p[NW + ob] = bsum;
}

// The weight gradients of the three layers in one launch: layer 2 (the most work) first.
struct WgradArgs {
    const float *dy, *dz2, *dz1;
    const bf16 *a2, *a1, *x0;
    float *part[3];  // layers 1, 2, 3
    int ctas[3];
    long long tiles;
};
template <int CI, int HD>
__global__ void __launch_bounds__(WG_THREADS) k_wgrad(WgradArgs a, const Tiling g) {
    extern __shared__ __align__(16) float sm[];
    a.dy = pdl_wait(a.dy);
    a.dz2 = pdl_order(a.dz2);
    a.dz1 = pdl_order(a.dz1);
    a.a2 = pdl_order(a.a2);
    a.a1 = pdl_order(a.a1);
    a.x0 = pdl_order(a.x0);
    int k = blockIdx.x;
    if (k < a.ctas[1]) {
        conv_bwd_weight<HD, HD>(a.dz2, a.a1, g, a.tiles, k, a.ctas[1], sm, a.part[1]);
    } else if ((k -= a.ctas[1]) < a.ctas[0]) {
        conv_bwd_weight<CI, HD>(a.dz1, a.x0, g, a.tiles, k, a.ctas[0], sm, a.part[0]);
    } else {
        conv_bwd_weight<HD, 1>(a.dy, a.a2, g, a.tiles, k - a.ctas[0], a.ctas[2], sm, a.part[2]);
    }
}

// Where a parameter's BF16 value goes in FP32 for the kernels: the weights of layers 1 and 2 as
// [c][tap][o] for the forward pass, those of layers 2 and 3 as [o][tap][c] for the input gradients.
struct Layout {
    int cin, hid, off[6];
    float *fwd, *bwd;  // layer 1 then 2; layer 2 then 3
};
__device__ __forceinline__ void put_param(const Layout &l, int k, bf16 b, bf16 *theta_b) {
    theta_b[k] = b;
    const float v = __bfloat162float(b);
    const int n1 = l.cin * 9 * l.hid, n2 = l.hid * 9 * l.hid;
    if (k < l.off[1]) {
        const int o = k / (l.cin * 9), r = k % (l.cin * 9);
        l.fwd[r * l.hid + o] = v;
    } else if (k >= l.off[2] && k < l.off[3]) {
        const int q = k - l.off[2], o = q / (l.hid * 9), c = q / 9 % l.hid, tap = q % 9;
        l.fwd[n1 + (c * 9 + tap) * l.hid + o] = v;
        l.bwd[(o * 9 + tap) * l.hid + c] = v;
    } else if (k >= l.off[4] && k < l.off[5]) {
        const int q = k - l.off[4], c = q / 9, tap = q % 9;
        l.bwd[n2 + tap * l.hid + c] = v;
    }
}

struct AdamArgs {
    bool on;
    float lr, b1, b2, eps, bc1, bc2;
    float *theta, *m, *v;
    bf16 *theta_b;
    Layout layout;
};
__device__ __forceinline__ void adam_one(const AdamArgs &a, int k, float gk) {
    const float mk = a.b1 * a.m[k] + (1.f - a.b1) * gk;
    const float vk = a.b2 * a.v[k] + (1.f - a.b2) * gk * gk;
    a.m[k] = mk;
    a.v[k] = vk;
    const float th = a.theta[k] - a.lr * (mk / a.bc1) / (sqrtf(vk / a.bc2) + a.eps);
    a.theta[k] = th;
    put_param(a.layout, k, __float2bfloat16_rn(th), a.theta_b);
}

// Gradients from the CTAs' partial sums, one parameter a lane and a slice of the CTAs a warp, and
// (a.on) the Adam update of the parameter; the last CTA adds up the loss.
struct ReduceArgs {
    const float *part[3];
    int ctas[3], count[3];  // partial sums and parameters of each layer
    const double *loss_part;
    int loss_parts;
    long long n;
    double *loss;
    float *grad;
    int nparam;
};
constexpr int RED_PARAMS = 32, RED_SLICES = 16;
__global__ void __launch_bounds__(RED_PARAMS *RED_SLICES)
    k_net_reduce(ReduceArgs r, const AdamArgs a) {
    r.loss_part = pdl_wait(r.loss_part);
    __shared__ float sh[RED_SLICES][RED_PARAMS];
    __shared__ double shl[RED_SLICES];
    const int lane = threadIdx.x % RED_PARAMS, slice = threadIdx.x / RED_PARAMS;
    if (blockIdx.x == gridDim.x - 1) {
        double s = threadIdx.x < r.loss_parts ? r.loss_part[threadIdx.x] : 0.0;
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        if (lane == 0) shl[slice] = s;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int k = 0; k < RED_SLICES; ++k) t += shl[k];
            *r.loss = t / (double)r.n;
        }
        return;
    }
    const int p = blockIdx.x * RED_PARAMS + lane;
    float s = 0.f;
    if (p < r.nparam) {
        int l = 0, q = p;
        while (q >= r.count[l]) q -= r.count[l++];
        const float *src = pdl_order(r.part[l]) + q;
        const size_t pitch = r.count[l];
        const int per = (r.ctas[l] + RED_SLICES - 1) / RED_SLICES, k0 = slice * per;
        const int k1 = min(k0 + per, r.ctas[l]);
#pragma unroll 8
        for (int k = k0; k < k1; ++k) s += src[k * pitch];
    }
    sh[slice][lane] = s;
    __syncthreads();
    if (slice == 0 && p < r.nparam) {
        float t = 0.f;
#pragma unroll
        for (int k = 0; k < RED_SLICES; ++k) t += sh[k][lane];
        r.grad[p] = t;
        if (a.on) adam_one(a, p, t);
    }
}

__global__ void k_adam(const AdamArgs a, const float *__restrict__ g, int n) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) adam_one(a, k, g[k]);
}

__global__ void k_to_bf16(const float *__restrict__ in, int n, const Layout l,
                          bf16 *__restrict__ out) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) put_param(l, k, __float2bfloat16_rn(in[k]), out);
}

__global__ void k_log_targets(const double *__restrict__ kmax, long long n, float offset,
                              float floor_k, float *__restrict__ t) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const double K = kmax[k];
    if (K != K) {  // a NaN maximum stays visible in the targets
        t[k] = __int_as_float(0x7fc00000);
        return;
    }
    t[k] = (float)(log10(K > (double)floor_k ? K : (double)floor_k)) - offset;
}

__global__ void k_to_maxima(const float *__restrict__ y, long long n, float offset,
                            double *__restrict__ out) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    out[k] = exp10((double)y[k] + (double)offset);
}

// Residual form: targets are the change of log10 K over the horizon, predictions are added to
// the log of the maximum now.  NaN in either maximum gives NaN.
__global__ void k_log_residual(const double *__restrict__ next, const double *__restrict__ now,
                               long long n, float floor_k, float *__restrict__ t) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const double a = next[k], b = now[k], f = (double)floor_k;
    if (a != a || b != b) {
        t[k] = __int_as_float(0x7fc00000);
        return;
    }
    t[k] = (float)(log10(a > f ? a : f) - log10(b > f ? b : f));
}

__global__ void k_to_maxima_residual(const float *__restrict__ y, const double *__restrict__ now,
                                     long long n, float floor_k, double *__restrict__ out) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const double b = now[k], f = (double)floor_k;
    out[k] = (b != b) ? b : exp10((double)y[k] + log10(b > f ? b : f));
}

// Fraction of equal flags, counted by one CTA of 1024 threads (the flag arrays of a regrid hold a
// few thousand blocks).
constexpr int JUDGE_THREADS = 1024;

__device__ __forceinline__ double cta_agreement(const int8_t *a, const int8_t *b, int n,
                                                int *red) {
    int c = 0;
    for (int k = threadIdx.x; k < n; k += JUDGE_THREADS) c += a[k] == b[k];
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) c += __shfl_xor_sync(0xffffffffu, c, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x < 32) {
        c = red[threadIdx.x];
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) c += __shfl_xor_sync(0xffffffffu, c, off);
        if (threadIdx.x == 0) red[0] = c;
    }
    __syncthreads();
    const double r = n > 0 ? (double)red[0] / (double)n : 1.0;
    __syncthreads();  // red is reused by the caller
    return r;
}

__global__ void __launch_bounds__(JUDGE_THREADS)
    k_flags_agreement(const int8_t *a, const int8_t *b, int n, double *out) {
    __shared__ int red[JUDGE_THREADS / 32];
    const double r = cta_agreement(a, b, n, red);
    if (threadIdx.x == 0) *out = r;
}

// The judge and fallback of a predicted regrid: the agreement of the previous regrid's predicted
// flags with the exact flags now decides the flags used now -- the prediction for the next
// interval if it reached min_agree (or if there is no previous prediction), else the exact flags.
__global__ void __launch_bounds__(JUDGE_THREADS)
    k_judge_select(const int8_t *pred_prev, const int8_t *exact_now, const int8_t *pred_next,
                   int n, double min_agree, int8_t *used, double *agree_out, int *fell_out) {
    __shared__ int red[JUDGE_THREADS / 32];
    double r = __longlong_as_double(0x7ff8000000000000ll);  // no previous prediction: NaN
    if (pred_prev) r = cta_agreement(pred_prev, exact_now, n, red);
    const bool exact = pred_prev && !(r >= min_agree);
    for (int k = threadIdx.x; k < n; k += JUDGE_THREADS) used[k] = exact ? exact_now[k] : pred_next[k];
    if (threadIdx.x == 0) {
        if (agree_out) *agree_out = r;
        if (fell_out) *fell_out = exact ? 1 : 0;
    }
}

// dst row k = src row idx[k] (rows of `words` 32-bit words)
__global__ void k_gather_rows(const uint32_t *__restrict__ src, size_t words,
                              const int *__restrict__ idx, int count, long long nrows,
                              uint32_t *__restrict__ dst, int *bad) {
    const size_t total = words * (size_t)count;
    for (size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x; k < total;
         k += (size_t)gridDim.x * blockDim.x) {
        const size_t row = k / words, w = k % words;
        const int r = idx[row];
        if (r < 0 || r >= nrows) {  // an index outside the source: flagged, nothing read
            if (w == 0) atomicOr(bad, 1);
            continue;
        }
        dst[k] = src[(size_t)r * words + w];
    }
}

inline unsigned grid_for(long long n, int t) { return (unsigned)((n + t - 1) / t); }

#define NETCK(call, what)                                          \
    do {                                                           \
        cudaError_t e_ = (call);                                   \
        if (e_ != cudaSuccess) return lbm::report_cuda_error(e_, what); \
    } while (0)

}  // namespace
}  // namespace net
}  // namespace lbm

struct lbm_net_s {
    int cin = 0, hid = 0, nparam = 0;
    int off[6] = {0, 0, 0, 0, 0, 0};  // W1, b1, W2, b2, W3, b3 in the flat parameter vector
    float *theta = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;
    __nv_bfloat16 *theta_b = nullptr;
    float *w_fwd = nullptr, *w_bwd = nullptr;  // the weights in FP32 as the kernels read them
    lbm::net::Norm norm;
    long long t = 0;  // Adam steps taken
    cudaStream_t stream = nullptr;
    long long cap = 0;  // positions (batch x h x w) the activation buffers hold
    __nv_bfloat16 *x0 = nullptr, *a1 = nullptr, *a2 = nullptr;
    float *y = nullptr, *dy = nullptr, *dz1 = nullptr, *dz2 = nullptr;
    double *loss_part = nullptr;
    // pinned host memory and its device address: the losses of up to LOSS_SLOTS steps, an error word
    double *loss_host = nullptr, *loss_dev = nullptr;
    float *wpart[3] = {nullptr, nullptr, nullptr};  // partial weight gradients of the layers
    long long last_pos = 0;  // positions of the last forward / backward call (0: none yet)
};

namespace {

using namespace lbm::net;

Layout layout_of(const lbm_net *n) {
    Layout l = {n->cin, n->hid, {}, n->w_fwd, n->w_bwd};
    for (int k = 0; k < 6; ++k) l.off[k] = n->off[k];
    return l;
}

void free_acts(lbm_net *n) {
    cudaFree(n->x0);
    cudaFree(n->a1);
    cudaFree(n->a2);
    cudaFree(n->y);
    cudaFree(n->dy);
    cudaFree(n->dz1);
    cudaFree(n->dz2);
    n->x0 = n->a1 = n->a2 = nullptr;
    n->y = n->dy = n->dz1 = n->dz2 = nullptr;
    n->cap = 0;
}

int ensure_acts(lbm_net *n, long long pos) {
    if (pos <= n->cap) return LBM_OK;
    free_acts(n);
    const size_t P = (size_t)pos;
    cudaError_t e = lbm::dev_alloc(&n->x0, P * n->cin * sizeof(__nv_bfloat16));
    if (e == cudaSuccess) e = lbm::dev_alloc(&n->a1, P * n->hid * sizeof(__nv_bfloat16));
    if (e == cudaSuccess) e = lbm::dev_alloc(&n->a2, P * n->hid * sizeof(__nv_bfloat16));
    if (e == cudaSuccess) e = lbm::dev_alloc(&n->y, P * sizeof(float));
    if (e == cudaSuccess) e = lbm::dev_alloc(&n->dy, P * sizeof(float));
    if (e == cudaSuccess) e = lbm::dev_alloc(&n->dz1, P * n->hid * sizeof(float));
    if (e == cudaSuccess) e = lbm::dev_alloc(&n->dz2, P * n->hid * sizeof(float));
    if (e != cudaSuccess) {
        free_acts(n);
        return lbm::report_cuda_error(e, "cudaMalloc(network activations)");
    }
    n->cap = pos;
    return LBM_OK;
}

#define NET_DISPATCH(cin, hid, CALL)                                      \
    do {                                                                  \
        if ((cin) == 3 && (hid) == 16) {                                  \
            constexpr int CI = 3, HD = 16;                                \
            CALL;                                                         \
        } else if ((cin) == 4 && (hid) == 16) {                           \
            constexpr int CI = 4, HD = 16;                                \
            CALL;                                                         \
        } else if ((cin) == 3 && (hid) == 8) {                            \
            constexpr int CI = 3, HD = 8;                                 \
            CALL;                                                         \
        } else if ((cin) == 4 && (hid) == 8) {                            \
            constexpr int CI = 4, HD = 8;                                 \
            CALL;                                                         \
        } else {                                                          \
            return lbm::report_error(LBM_EINVAL, "unsupported network shape"); \
        }                                                                 \
    } while (0)

int out_ctas(long long tiles) { return (int)(tiles < LOSS_PARTS ? tiles : LOSS_PARTS); }

// The three layers; GRAD: also dL/dy and the loss's partial sums for `target`.
template <int CI, int HD, bool GRAD>
int forward_layers(lbm_net *n, const float *x, int B, int H, int W, float *y_out,
                   const float *target, const Rows &rows) {
    const __nv_bfloat16 *tb = n->theta_b;
    cudaStream_t s = n->stream;
    const Tiling g(H, W, TILE_Y);
    const long long tiles = g.tiles(B);
    if (tiles > 0x7fffffffLL) return lbm::report_error(LBM_EINVAL, "network input too large");
    const unsigned nt = TILE_QUADS * TILE_Y * (HD / 4);
    const float two_n = (float)(2.0 / (double)((long long)B * H * W));
    NETCK(lbm::launch_pdl(k_conv_relu<CI, HD, true>, (unsigned)tiles, nt, 0, s, x, n->norm, n->x0,
                          n->w_fwd, tb + n->off[1], g, n->a1, rows),
          "network forward");
    NETCK(lbm::launch_pdl(k_conv_relu<HD, HD, false>, (unsigned)tiles, nt, 0, s, n->a1, n->norm,
                          nullptr, n->w_fwd + CI * 9 * HD, tb + n->off[3], g, n->a2, Rows{}),
          "network forward");
    NETCK(lbm::launch_pdl(k_conv_out<HD, GRAD>, out_ctas(tiles), OUT_THREADS, 0, s, n->a2,
                          tb + n->off[4], tb + n->off[5], g, tiles, y_out, target, two_n, n->dy,
                          n->loss_part, rows),
          "network forward");
    return LBM_OK;
}

template <int CI, int HD>
int run_forward(lbm_net *n, const float *x, int B, int H, int W, float *y_out) {
    return forward_layers<CI, HD, false>(n, x, B, H, W, y_out, nullptr, Rows{});
}

template <int CI, int HD>
int run_backward(lbm_net *n, const float *x, const float *target, int B, int H, int W,
                 const AdamArgs &adam, const Rows &rows, int slot) {
    int st = forward_layers<CI, HD, true>(n, x, B, H, W, n->y, target, rows);
    if (st != LBM_OK) return st;
    cudaStream_t s = n->stream;
    const Tiling g(H, W, TILE_Y), gw(H, W, WG_ROWS);
    const unsigned tiles = (unsigned)g.tiles(B), nt = TILE_QUADS * TILE_Y * (HD / 4);
    NETCK(lbm::launch_pdl(k_conv_bwd_data<HD, 1>, tiles, nt, 0, s, n->dy, n->w_bwd + HD * 9 * HD,
                          n->a2, g, n->dz2),
          "network backward");
    NETCK(lbm::launch_pdl(k_conv_bwd_data<HD, HD>, tiles, nt, 0, s, n->dz2, n->w_bwd, n->a1, g,
                          n->dz1),
          "network backward");
    WgradArgs a = {n->dy, n->dz2, n->dz1, n->a2, n->a1, n->x0, {}, {}, gw.tiles(B)};
    ReduceArgs r = {};
    for (int l = 0; l < 3; ++l) {
        a.part[l] = n->wpart[l];
        r.part[l] = n->wpart[l];
        a.ctas[l] = r.ctas[l] = (int)(a.tiles < WG_MAX_CTAS ? a.tiles : WG_MAX_CTAS);
        r.count[l] = (l == 2 ? n->nparam : n->off[2 * l + 2]) - n->off[2 * l];
    }
    constexpr int smem = sizeof(float) * wg_smem_floats(HD, HD);
    static_assert(smem <= 48 * 1024 && wg_smem_floats(CI, HD) <= wg_smem_floats(HD, HD) &&
                      wg_smem_floats(HD, 1) <= wg_smem_floats(HD, HD),
                  "shared memory of the weight gradients");
    NETCK(lbm::launch_pdl(k_wgrad<CI, HD>, a.ctas[0] + a.ctas[1] + a.ctas[2], WG_THREADS, smem, s, a, gw),
          "network backward");
    r.loss_part = n->loss_part;
    r.loss_parts = out_ctas(g.tiles(B));
    r.n = (long long)B * H * W;
    r.loss = n->loss_dev + slot;
    r.grad = n->grad;
    r.nparam = n->nparam;
    NETCK(lbm::launch_pdl(k_net_reduce, (n->nparam + RED_PARAMS - 1) / RED_PARAMS + 1,
                          RED_PARAMS * RED_SLICES, 0, s, r, adam),
          "network backward");
    return LBM_OK;
}

#define CHECK_NET(n)                                                             \
    do {                                                                         \
        lbm::clear_error();                                                      \
        if (!(n)) return lbm::report_error(LBM_EINVAL, "NULL network handle");   \
    } while (0)

int check_shape(int B, int H, int W) {
    if (B < 1 || H < 1 || W < 1 || (long long)B * H * W > (1LL << 30))
        return lbm::report_error(LBM_EINVAL, "batch, h, w must be >= 1 (and their product <= 2^30)");
    return LBM_OK;
}

}  // namespace

extern "C" {

LBM_API lbm_net *lbm_net_create(int cin, int hidden) {
    lbm::clear_error();
    if (!((cin == 3 || cin == 4) && (hidden == 8 || hidden == 16))) {
        lbm::report_error(LBM_EINVAL, "lbm_net_create: cin must be 3 or 4, hidden 8 or 16");
        return nullptr;
    }
    lbm_net *n = new (std::nothrow) lbm_net_s();
    if (!n) {
        lbm::report_error(LBM_ENOMEM, "lbm_net_create: out of host memory");
        return nullptr;
    }
    n->cin = cin;
    n->hid = hidden;
    const int sizes[6] = {hidden * cin * 9, hidden, hidden * hidden * 9, hidden, hidden * 9, 1};
    int o = 0;
    for (int k = 0; k < 6; ++k) {
        n->off[k] = o;
        o += sizes[k];
    }
    n->nparam = o;
    for (int c = 0; c < MAX_CIN; ++c) {
        n->norm.shift[c] = 0.f;
        n->norm.scale[c] = 1.f;
    }
    cudaError_t e = lbm::dev_alloc(&n->theta, sizeof(float) * o);
    if (e == cudaSuccess) e = lbm::dev_alloc(&n->grad, sizeof(float) * o);
    if (e == cudaSuccess) e = lbm::dev_alloc(&n->m, sizeof(float) * o);
    if (e == cudaSuccess) e = lbm::dev_alloc(&n->v, sizeof(float) * o);
    if (e == cudaSuccess) e = lbm::dev_alloc(&n->theta_b, sizeof(__nv_bfloat16) * o);
    if (e == cudaSuccess) e = lbm::dev_alloc(&n->loss_part, sizeof(double) * LOSS_PARTS);
    if (e == cudaSuccess)
        e = cudaHostAlloc((void **)&n->loss_host, sizeof(double) * (LOSS_SLOTS + 1),
                          cudaHostAllocMapped);
    if (e == cudaSuccess) e = cudaHostGetDevicePointer((void **)&n->loss_dev, n->loss_host, 0);
    for (int l = 0; l < 3 && e == cudaSuccess; ++l)
        e = lbm::dev_alloc(&n->wpart[l],
                           sizeof(float) * WG_MAX_CTAS * (size_t)(sizes[2 * l] + sizes[2 * l + 1]));
    const size_t fwd = sizeof(float) * (sizes[0] + sizes[2]), bwd = sizeof(float) * (sizes[2] + sizes[4]);
    if (e == cudaSuccess) e = lbm::dev_alloc(&n->w_fwd, fwd);
    if (e == cudaSuccess) e = lbm::dev_alloc(&n->w_bwd, bwd);
    if (e == cudaSuccess) e = cudaMemset(n->w_fwd, 0, fwd);
    if (e == cudaSuccess) e = cudaMemset(n->w_bwd, 0, bwd);
    if (e == cudaSuccess) e = cudaMemset(n->theta, 0, sizeof(float) * o);
    if (e == cudaSuccess) e = cudaMemset(n->grad, 0, sizeof(float) * o);
    if (e == cudaSuccess) e = cudaMemset(n->m, 0, sizeof(float) * o);
    if (e == cudaSuccess) e = cudaMemset(n->v, 0, sizeof(float) * o);
    if (e == cudaSuccess) e = cudaMemset(n->theta_b, 0, sizeof(__nv_bfloat16) * o);
    if (e != cudaSuccess) {
        lbm::report_cuda_error(e, "lbm_net_create");
        lbm_net_destroy(n);
        return nullptr;
    }
    return n;
}

LBM_API void lbm_net_destroy(lbm_net *n) {
    if (!n) return;
    free_acts(n);
    cudaFree(n->theta);
    cudaFree(n->grad);
    cudaFree(n->m);
    cudaFree(n->v);
    cudaFree(n->theta_b);
    cudaFree(n->loss_part);
    if (n->loss_host) cudaFreeHost(n->loss_host);
    for (float *p : n->wpart) cudaFree(p);
    cudaFree(n->w_fwd);
    cudaFree(n->w_bwd);
    delete n;
}

LBM_API int lbm_net_set_stream(lbm_net *n, void *stream) {
    CHECK_NET(n);
    n->stream = (cudaStream_t)stream;
    return LBM_OK;
}

LBM_API int lbm_net_param_count(lbm_net *n) {
    CHECK_NET(n);
    return n->nparam;
}

LBM_API int lbm_net_set_normalisation(lbm_net *n, const float *shift, const float *scale) {
    CHECK_NET(n);
    if (!shift || !scale) return lbm::report_error(LBM_EINVAL, "NULL shift or scale");
    for (int c = 0; c < n->cin; ++c) {
        n->norm.shift[c] = shift[c];
        n->norm.scale[c] = scale[c];
    }
    return LBM_OK;
}

LBM_API int lbm_net_set_params(lbm_net *n, const float *host) {
    CHECK_NET(n);
    if (!host) return lbm::report_error(LBM_EINVAL, "NULL parameters");
    NETCK(cudaMemcpyAsync(n->theta, host, sizeof(float) * n->nparam, cudaMemcpyHostToDevice,
                          n->stream),
          "parameters upload");
    k_to_bf16<<<grid_for(n->nparam, NT), NT, 0, n->stream>>>(n->theta, n->nparam, layout_of(n),
                                                             n->theta_b);
    NETCK(cudaMemsetAsync(n->m, 0, sizeof(float) * n->nparam, n->stream), "memset");
    NETCK(cudaMemsetAsync(n->v, 0, sizeof(float) * n->nparam, n->stream), "memset");
    n->t = 0;
    NETCK(cudaStreamSynchronize(n->stream), "lbm_net_set_params");
    return LBM_OK;
}

LBM_API int lbm_net_get_params(lbm_net *n, float *host) {
    CHECK_NET(n);
    if (!host) return lbm::report_error(LBM_EINVAL, "NULL output");
    NETCK(cudaMemcpyAsync(host, n->theta, sizeof(float) * n->nparam, cudaMemcpyDeviceToHost,
                          n->stream),
          "parameters download");
    NETCK(cudaStreamSynchronize(n->stream), "lbm_net_get_params");
    return LBM_OK;
}

LBM_API int lbm_net_get_grads(lbm_net *n, float *host) {
    CHECK_NET(n);
    if (!host) return lbm::report_error(LBM_EINVAL, "NULL output");
    NETCK(cudaMemcpyAsync(host, n->grad, sizeof(float) * n->nparam, cudaMemcpyDeviceToHost,
                          n->stream),
          "gradients download");
    NETCK(cudaStreamSynchronize(n->stream), "lbm_net_get_grads");
    return LBM_OK;
}

LBM_API int lbm_net_set_grads(lbm_net *n, const float *host) {
    CHECK_NET(n);
    if (!host) return lbm::report_error(LBM_EINVAL, "NULL gradients");
    NETCK(cudaMemcpyAsync(n->grad, host, sizeof(float) * n->nparam, cudaMemcpyHostToDevice,
                          n->stream),
          "gradients upload");
    NETCK(cudaStreamSynchronize(n->stream), "lbm_net_set_grads");
    return LBM_OK;
}

LBM_API int lbm_net_forward(lbm_net *n, const float *x_dev, int batch, int h, int w,
                            float *y_dev) {
    CHECK_NET(n);
    if (!x_dev || !y_dev) return lbm::report_error(LBM_EINVAL, "NULL input or output");
    int st = check_shape(batch, h, w);
    if (st != LBM_OK) return st;
    st = ensure_acts(n, (long long)batch * h * w);
    if (st != LBM_OK) return st;
    NET_DISPATCH(n->cin, n->hid, (st = run_forward<CI, HD>(n, x_dev, batch, h, w, y_dev)));
    if (st == LBM_OK) n->last_pos = (long long)batch * h * w;
    return st;
}

static int backward(lbm_net *n, const float *x_dev, const float *target_dev, int batch, int h, int w,
                    const AdamArgs &adam, const Rows &rows = Rows{}, int slot = 0) {
    if (!x_dev || !target_dev) return lbm::report_error(LBM_EINVAL, "NULL input or target");
    int st = check_shape(batch, h, w);
    if (st != LBM_OK) return st;
    st = ensure_acts(n, (long long)batch * h * w);
    if (st != LBM_OK) return st;
    NET_DISPATCH(n->cin, n->hid,
                 (st = run_backward<CI, HD>(n, x_dev, target_dev, batch, h, w, adam, rows, slot)));
    if (st != LBM_OK) return st;
    n->last_pos = (long long)batch * h * w;
    return LBM_OK;
}

static int read_loss(lbm_net *n, double *loss_host, const char *what) {
    if (!loss_host) return LBM_OK;
    NETCK(cudaStreamSynchronize(n->stream), what);
    *loss_host = *static_cast<volatile double *>(n->loss_host);  // written by k_net_reduce
    return LBM_OK;
}

// The Adam step that follows step n->t, or LBM_EINVAL.
static int adam_args(const lbm_net *n, float lr, float beta1, float beta2, float eps, AdamArgs *a) {
    if (!(lr >= 0.f) || !(beta1 >= 0.f && beta1 < 1.f) || !(beta2 >= 0.f && beta2 < 1.f) ||
        !(eps > 0.f))
        return lbm::report_error(LBM_EINVAL, "Adam needs lr >= 0, beta in [0, 1), eps > 0");
    const double t = (double)(n->t + 1);
    *a = {true, lr, beta1, beta2, eps, (float)(1.0 - pow((double)beta1, t)),
          (float)(1.0 - pow((double)beta2, t)), n->theta, n->m, n->v, n->theta_b, layout_of(n)};
    return LBM_OK;
}

LBM_API int lbm_net_backward(lbm_net *n, const float *x_dev, const float *target_dev, int batch,
                             int h, int w, double *loss_host) {
    CHECK_NET(n);
    const int st = backward(n, x_dev, target_dev, batch, h, w, AdamArgs{});
    return st != LBM_OK ? st : read_loss(n, loss_host, "lbm_net_backward");
}

LBM_API int lbm_net_get_buffer(lbm_net *n, int which, void *out_host, size_t bytes) {
    CHECK_NET(n);
    if (!out_host) return lbm::report_error(LBM_EINVAL, "NULL output");
    const size_t P = (size_t)n->last_pos;
    const void *src = nullptr;
    size_t need = 0;
    switch (which) {
        case LBM_NET_BUF_PARAMS_BF16:
            src = n->theta_b;
            need = (size_t)n->nparam * sizeof(__nv_bfloat16);
            break;
        case LBM_NET_BUF_X0: src = n->x0; need = P * n->cin * sizeof(__nv_bfloat16); break;
        case LBM_NET_BUF_A1: src = n->a1; need = P * n->hid * sizeof(__nv_bfloat16); break;
        case LBM_NET_BUF_A2: src = n->a2; need = P * n->hid * sizeof(__nv_bfloat16); break;
        case LBM_NET_BUF_Y: src = n->y; need = P * sizeof(float); break;
        case LBM_NET_BUF_DY: src = n->dy; need = P * sizeof(float); break;
        case LBM_NET_BUF_DZ2: src = n->dz2; need = P * n->hid * sizeof(float); break;
        case LBM_NET_BUF_DZ1: src = n->dz1; need = P * n->hid * sizeof(float); break;
        default: return lbm::report_error(LBM_EINVAL, "unknown network buffer");
    }
    if (which != LBM_NET_BUF_PARAMS_BF16 && n->last_pos == 0)
        return lbm::report_error(LBM_ESTATE, "no forward or backward pass yet");
    if (bytes != need) return lbm::report_error(LBM_EINVAL, "bytes must equal the buffer's size");
    NETCK(cudaMemcpyAsync(out_host, src, need, cudaMemcpyDeviceToHost, n->stream),
          "buffer download");
    NETCK(cudaStreamSynchronize(n->stream), "lbm_net_get_buffer");
    return LBM_OK;
}

LBM_API int lbm_net_adam(lbm_net *n, float lr, float beta1, float beta2, float eps) {
    CHECK_NET(n);
    AdamArgs a;
    const int st = adam_args(n, lr, beta1, beta2, eps, &a);
    if (st != LBM_OK) return st;
    n->t += 1;
    k_adam<<<grid_for(n->nparam, NT), NT, 0, n->stream>>>(a, n->grad, n->nparam);
    NETCK(cudaGetLastError(), "lbm_net_adam");
    return LBM_OK;
}

LBM_API int lbm_net_train_step(lbm_net *n, const float *x_dev, const float *target_dev, int batch,
                               int h, int w, float lr, double *loss_host) {
    CHECK_NET(n);
    AdamArgs a = {};
    // a rate that lbm_net_adam refuses: the gradients are left as lbm_net_backward leaves them
    const bool ok = lr >= 0.f;
    int st = ok ? adam_args(n, lr, 0.9f, 0.999f, 1e-8f, &a) : LBM_OK;
    if (st == LBM_OK) st = backward(n, x_dev, target_dev, batch, h, w, a);
    if (st != LBM_OK) return st;
    if (!ok) return lbm_net_adam(n, lr, 0.9f, 0.999f, 1e-8f);
    n->t += 1;
    return read_loss(n, loss_host, "lbm_net_train_step");
}

LBM_API int lbm_net_train_epoch(lbm_net *n, const float *x_dev, const float *target_dev,
                                long long nrows, const int *idx_dev, int steps, int batch, int h,
                                int w, float lr, double *losses_host) {
    CHECK_NET(n);
    if (!idx_dev || steps < 0 || nrows < 1)
        return lbm::report_error(LBM_EINVAL, "need indices, steps >= 0 and nrows >= 1");
    // the steps are queued one behind the other; the host waits once, or where the slots are full
    volatile int *bad = reinterpret_cast<int *>(n->loss_host + LOSS_SLOTS);
    *bad = 0;
    int st = LBM_OK;
    for (int from = 0; from < steps && st == LBM_OK; from += LOSS_SLOTS) {
        const int count = steps - from < LOSS_SLOTS ? steps - from : LOSS_SLOTS;
        for (int k = 0; k < count && st == LBM_OK; ++k) {
            const Rows rows = {idx_dev + (size_t)(from + k) * batch, nrows,
                               reinterpret_cast<int *>(n->loss_dev + LOSS_SLOTS)};
            AdamArgs a;
            st = adam_args(n, lr, 0.9f, 0.999f, 1e-8f, &a);
            if (st == LBM_OK) st = backward(n, x_dev, target_dev, batch, h, w, a, rows, k);
            if (st == LBM_OK) n->t += 1;
        }
        NETCK(cudaStreamSynchronize(n->stream), "lbm_net_train_epoch");
        if (st == LBM_OK && losses_host)
            for (int k = 0; k < count; ++k)
                losses_host[from + k] = static_cast<volatile double *>(n->loss_host)[k];
    }
    if (st == LBM_OK && *bad)
        return lbm::report_error(LBM_EINVAL, "minibatch index outside the training set");
    return st;
}

LBM_API int lbm_net_log_targets(const double *kmax_dev, long long n, float offset, float floor_k,
                                float *t_dev, void *stream) {
    lbm::clear_error();
    if (!kmax_dev || !t_dev || n < 0 || !(floor_k > 0.f))
        return lbm::report_error(LBM_EINVAL, "lbm_net_log_targets: bad arguments");
    if (n == 0) return LBM_OK;
    k_log_targets<<<grid_for(n, NT), NT, 0, (cudaStream_t)stream>>>(kmax_dev, n, offset, floor_k,
                                                                     t_dev);
    NETCK(cudaGetLastError(), "lbm_net_log_targets");
    return LBM_OK;
}

LBM_API int lbm_flags_agreement(const int8_t *a_dev, const int8_t *b_dev, int n, double *out_dev,
                                void *stream) {
    lbm::clear_error();
    if (n < 0 || (n > 0 && (!a_dev || !b_dev)) || !out_dev)
        return lbm::report_error(LBM_EINVAL, "lbm_flags_agreement: bad arguments");
    k_flags_agreement<<<1, JUDGE_THREADS, 0, (cudaStream_t)stream>>>(a_dev, b_dev, n, out_dev);
    NETCK(cudaGetLastError(), "lbm_flags_agreement");
    return LBM_OK;
}

LBM_API int lbm_flags_judge_select(const int8_t *pred_prev_dev, const int8_t *exact_now_dev,
                                   const int8_t *pred_next_dev, int n, double min_agreement,
                                   int8_t *used_dev, double *agreement_dev, int *fell_back_dev,
                                   void *stream) {
    lbm::clear_error();
    if (n < 0 || (n > 0 && (!exact_now_dev || !pred_next_dev || !used_dev)) ||
        !(min_agreement >= 0.0 && min_agreement <= 1.0))
        return lbm::report_error(LBM_EINVAL, "lbm_flags_judge_select: bad arguments");
    k_judge_select<<<1, JUDGE_THREADS, 0, (cudaStream_t)stream>>>(
        pred_prev_dev, exact_now_dev, pred_next_dev, n, min_agreement, used_dev, agreement_dev,
        fell_back_dev);
    NETCK(cudaGetLastError(), "lbm_flags_judge_select");
    return LBM_OK;
}

LBM_API int lbm_gather_rows(const void *src_dev, long long nrows, size_t row_bytes,
                            const int *idx_dev, int count, void *dst_dev, int *bad_dev,
                            void *stream) {
    lbm::clear_error();
    if (nrows < 0 || count < 0 || row_bytes % 4 != 0 ||
        (count > 0 && (!src_dev || !idx_dev || !dst_dev || !bad_dev)))
        return lbm::report_error(LBM_EINVAL, "lbm_gather_rows: bad arguments (rows of a multiple "
                                             "of 4 bytes)");
    if (count == 0 || row_bytes == 0) return LBM_OK;
    const size_t words = row_bytes / 4;
    long long total = (long long)words * count;
    unsigned g = grid_for(total, NT);
    if (g > 4096) g = 4096;
    k_gather_rows<<<g, NT, 0, (cudaStream_t)stream>>>(static_cast<const uint32_t *>(src_dev), words,
                                                       idx_dev, count, nrows,
                                                       static_cast<uint32_t *>(dst_dev), bad_dev);
    NETCK(cudaGetLastError(), "lbm_gather_rows");
    return LBM_OK;
}

LBM_API int lbm_net_log_residual(const double *kmax_next_dev, const double *kmax_now_dev,
                                 long long n, float floor_k, float *t_dev, void *stream) {
    lbm::clear_error();
    if (!kmax_next_dev || !kmax_now_dev || !t_dev || n < 0 || !(floor_k > 0.f))
        return lbm::report_error(LBM_EINVAL, "lbm_net_log_residual: bad arguments");
    if (n == 0) return LBM_OK;
    k_log_residual<<<grid_for(n, NT), NT, 0, (cudaStream_t)stream>>>(kmax_next_dev, kmax_now_dev, n,
                                                                      floor_k, t_dev);
    NETCK(cudaGetLastError(), "lbm_net_log_residual");
    return LBM_OK;
}

LBM_API int lbm_net_to_maxima_residual(const float *y_dev, const double *kmax_now_dev, long long n,
                                       float floor_k, double *kmax_dev, void *stream) {
    lbm::clear_error();
    if (!y_dev || !kmax_now_dev || !kmax_dev || n < 0 || !(floor_k > 0.f))
        return lbm::report_error(LBM_EINVAL, "lbm_net_to_maxima_residual: bad arguments");
    if (n == 0) return LBM_OK;
    k_to_maxima_residual<<<grid_for(n, NT), NT, 0, (cudaStream_t)stream>>>(y_dev, kmax_now_dev, n,
                                                                            floor_k, kmax_dev);
    NETCK(cudaGetLastError(), "lbm_net_to_maxima_residual");
    return LBM_OK;
}

LBM_API int lbm_net_to_maxima(const float *y_dev, long long n, float offset, double *kmax_dev,
                              void *stream) {
    lbm::clear_error();
    if (!y_dev || !kmax_dev || n < 0)
        return lbm::report_error(LBM_EINVAL, "lbm_net_to_maxima: bad arguments");
    if (n == 0) return LBM_OK;
    k_to_maxima<<<grid_for(n, NT), NT, 0, (cudaStream_t)stream>>>(y_dev, n, offset, kmax_dev);
    NETCK(cudaGetLastError(), "lbm_net_to_maxima");
    return LBM_OK;
}

}  // extern "C"
