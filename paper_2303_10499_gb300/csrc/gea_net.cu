// gea_net.cu -- the learned pressure-correction network: a convolutional
// multigrid-style U-Net (4 levels, 16 base channels) with its forward pass,
// energy loss, backward pass and Adam update, all on the GPU.
//
// The 3x3 layers with 16-64 channels run on the tensor cores (gea_conv.cu):
// forward, and the data gradient as the same correlation with the taps
// mirrored and the channel roles swapped. The first layer (one input
// channel), the 1x1 output layer, the weight gradients (FP32 gradients times
// bfloat16 inputs, summed over all pixels) and the elementwise parts run on
// the CUDA cores in FP32.
// Every reduction is deterministic: per-block partial sums added in a fixed
// order.
#include "../../include/gea.h"
#include "../../include/gea_net.h"

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <vector>

cudaError_t gea_conv3x3_launch(int n, int h, int w, int cin, int cout, int mode, int flags, const uint16_t *x0,
                               const uint16_t *x1, const uint16_t *wt, const float *bias, void *y, int *status,
                               cudaStream_t st);

namespace gea_net_impl {

enum { SRC_X = 0, SRC_PREV = 1, SRC_POOL = 2, SRC_UPADD = 3 };

// cin, cout, kernel size, activation, input kind, input layer a (the layer
// read, averaged or prolonged), skip layer b (UPADD), level
struct LayerDef {
    int cin, cout, k, act, kind, a, b, level;
};

constexpr int L = GEA_NET_LAYERS;
constexpr LayerDef kL[L] = {
    {1, 16, 3, 1, SRC_X, -1, -1, 0},     // e0a
    {16, 16, 3, 1, SRC_PREV, 0, -1, 0},  // e0b
    {16, 32, 3, 1, SRC_POOL, 1, -1, 1},  // e1a
    {32, 32, 3, 1, SRC_PREV, 2, -1, 1},  // e1b
    {32, 64, 3, 1, SRC_POOL, 3, -1, 2},  // e2a
    {64, 64, 3, 1, SRC_PREV, 4, -1, 2},  // e2b
    {64, 64, 3, 1, SRC_POOL, 5, -1, 3},  // e3a
    {64, 64, 3, 1, SRC_PREV, 6, -1, 3},  // e3b
    {64, 64, 3, 1, SRC_UPADD, 7, 5, 2},  // d2a
    {64, 32, 3, 1, SRC_PREV, 8, -1, 2},  // d2b
    {32, 32, 3, 1, SRC_UPADD, 9, 3, 1},  // d1a
    {32, 16, 3, 1, SRC_PREV, 10, -1, 1}, // d1b
    {16, 16, 3, 1, SRC_UPADD, 11, 1, 0}, // d0a
    {16, 16, 3, 1, SRC_PREV, 12, -1, 0}, // d0b
    {16, 1, 1, 0, SRC_PREV, 13, -1, 0},  // out
};
constexpr int kOut = L - 1;
constexpr int kThreads = 256;
constexpr int kWgPix = 64;       // pixels of a weight-gradient row segment at most
constexpr int kWgChain = 256;    // terms of one thread's running weight-gradient sum at most (k_wgrad)

__device__ __forceinline__ float bf2f(uint16_t u) { return __uint_as_float((uint32_t)u << 16); }
__device__ __forceinline__ uint16_t f2bf(float f)
{
    __nv_bfloat16 h = __float2bfloat16_rn(f);
    return *reinterpret_cast<uint16_t *>(&h);
}
__device__ __forceinline__ float round_bf(float f) { return bf2f(f2bf(f)); }

// ---- per-sample sums (deterministic: block partials, then a fixed-order sum) ----

// part[b * gridDim.x + blk] = sum over the block's share of sample b of v^2
// (sq) or v. A thread takes four consecutive values at a time (per is a
// multiple of 64) into four FP64 sums, which it adds in a fixed order, with
// one 16-byte load when x is 16-byte aligned (vec); v^2 of an FP32 value is
// exact in FP64, so fma(v, v, s) adds it with the one rounding of the sum.
__global__ void k_sample_partials(const float *x, long long per, int sq, int vec, double *part)
{
    __shared__ double red[kThreads];
    const int b = blockIdx.y;
    const float *xs = x + (size_t)b * per;
    const long long n4 = per / 4;
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
    for (long long i = blockIdx.x * (long long)kThreads + threadIdx.x; i < n4; i += (long long)gridDim.x * kThreads) {
        float4 v;
        if (vec) {
            v = __ldg(reinterpret_cast<const float4 *>(xs) + i);
        } else {
            v.x = __ldg(&xs[4 * i]); v.y = __ldg(&xs[4 * i + 1]);
            v.z = __ldg(&xs[4 * i + 2]); v.w = __ldg(&xs[4 * i + 3]);
        }
        if (sq) {
            s0 = fma((double)v.x, (double)v.x, s0);
            s1 = fma((double)v.y, (double)v.y, s1);
            s2 = fma((double)v.z, (double)v.z, s2);
            s3 = fma((double)v.w, (double)v.w, s3);
        } else {
            s0 += v.x; s1 += v.y; s2 += v.z; s3 += v.w;
        }
    }
    red[threadIdx.x] = (s0 + s1) + (s2 + s3);
    __syncthreads();
    for (int o = kThreads / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[(size_t)b * gridDim.x + blockIdx.x] = red[0];
}

// out[b] = scale(sum of the nblk partials of sample b); mode 0: sqrt(s / per)
// (rms), 1: s / per (mean). One block per sample: thread t adds partials
// t, t + kThreads, ..., then a fixed-order tree.
__global__ void k_sample_finish(const double *part, int nblk, long long per, int mode, float *out)
{
    __shared__ double red[kThreads];
    const int b = blockIdx.x;
    double s = 0.0;
    for (int i = threadIdx.x; i < nblk; i += kThreads) s += part[(size_t)b * nblk + i];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = kThreads / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[b] = mode == 0 ? (float)sqrt(red[0] / (double)per) : (float)(red[0] / (double)per);
}

// x = r / rms per sample (0 if rms = 0), FP32 and bfloat16
__global__ void k_prep(const float *r, const float *rms, long long per, long long total, float *xh, uint16_t *xb)
{
    const long long i = blockIdx.x * (long long)kThreads + threadIdx.x;
    if (i >= total) return;
    const float s = rms[i / per];
    const float v = s > 0.0f ? r[i] / s : 0.0f;
    xh[i] = v;
    xb[i] = f2bf(v);
}

// ---- first layer (1 input channel) and output layer (1x1) on the CUDA cores ----

// Pixels of one row per thread in the first layer (w is a multiple of 8):
// each weight read from shared memory serves kFirstPix multiply-adds.
constexpr int kFirstPix = 4;

__global__ void __launch_bounds__(kThreads) k_conv_first(int n, int h, int w, const uint16_t *x, const float *wt,
                                                         const float *bias, int relu, uint16_t *y)
{
    __shared__ float sw[16 * 9], sb[16];
    for (int e = threadIdx.x; e < 16 * 9; e += kThreads) sw[e] = round_bf(wt[e]);
    if (threadIdx.x < 16) sb[threadIdx.x] = bias[threadIdx.x];
    __syncthreads();
    const long long p0 = (blockIdx.x * (long long)kThreads + threadIdx.x) * kFirstPix;
    if (p0 >= (long long)n * h * w) return;
    const int j0 = (int)(p0 % w);
    const int i = (int)((p0 / w) % h);
    const long long base = p0 - ((long long)i * w + j0);
    // input rows i-1..i+1, columns j0-1..j0+kFirstPix (zero outside the image)
    float xv[3][kFirstPix + 2];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const int ii = i + r - 1;
#pragma unroll
        for (int c = 0; c < kFirstPix + 2; ++c) {
            const int jj = j0 + c - 1;
            xv[r][c] = (ii >= 0 && ii < h && jj >= 0 && jj < w) ? bf2f(x[base + (long long)ii * w + jj]) : 0.0f;
        }
    }
    // per output: the bias, then the taps in row-major order, one FMA each
    uint32_t u[kFirstPix][8];
#pragma unroll
    for (int c = 0; c < 16; c += 2) {
        float o[2][kFirstPix];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
#pragma unroll
            for (int px = 0; px < kFirstPix; ++px) o[k][px] = sb[c + k];
#pragma unroll
            for (int t = 0; t < 9; ++t) {
                const float wv = sw[(c + k) * 9 + t];
#pragma unroll
                for (int px = 0; px < kFirstPix; ++px) o[k][px] = fmaf(wv, xv[t / 3][px + t % 3], o[k][px]);
            }
#pragma unroll
            for (int px = 0; px < kFirstPix; ++px)
                if (relu) o[k][px] = fmaxf(o[k][px], 0.0f);
        }
#pragma unroll
        for (int px = 0; px < kFirstPix; ++px)
            u[px][c / 2] = (uint32_t)f2bf(o[0][px]) | ((uint32_t)f2bf(o[1][px]) << 16);
    }
    uint4 *dst = reinterpret_cast<uint4 *>(y + p0 * 16);
#pragma unroll
    for (int px = 0; px < kFirstPix; ++px) {
        dst[2 * px] = make_uint4(u[px][0], u[px][1], u[px][2], u[px][3]);
        dst[2 * px + 1] = make_uint4(u[px][4], u[px][5], u[px][6], u[px][7]);
    }
}

__global__ void k_conv_out(long long npix, const uint16_t *x, const float *wt, const float *bias, float *y)
{
    const long long p = blockIdx.x * (long long)kThreads + threadIdx.x;
    if (p >= npix) return;
    const uint4 *src = reinterpret_cast<const uint4 *>(x + p * 16);
    const uint4 a = src[0], b = src[1];
    const uint32_t u[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    float s = bias[0];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        s = fmaf(round_bf(wt[2 * c]), bf2f((uint16_t)(u[c] & 0xFFFFu)), s);
        s = fmaf(round_bf(wt[2 * c + 1]), bf2f((uint16_t)(u[c] >> 16)), s);
    }
    y[p] = s;
}

// Output layer backward: g13[p][c] = dy[p] w[c]; block partials of
// dW[c] = sum dy x[p][c] and db = sum dy (17 per block).
__global__ void k_out_backward(long long npix, const float *dy, const uint16_t *x, const float *wt, float *g13,
                               float *part)
{
    __shared__ float red[17][kThreads];
    const long long p = blockIdx.x * (long long)kThreads + threadIdx.x;
    float v[17];
#pragma unroll
    for (int c = 0; c < 17; ++c) v[c] = 0.0f;
    if (p < npix) {
        const float d = dy[p];
#pragma unroll
        for (int c = 0; c < 16; ++c) {
            g13[p * 16 + c] = d * round_bf(wt[c]);
            v[c] = d * bf2f(x[p * 16 + c]);
        }
        v[16] = d;
    }
#pragma unroll
    for (int c = 0; c < 17; ++c) red[c][threadIdx.x] = v[c];
    __syncthreads();
    for (int o = kThreads / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o)
#pragma unroll
            for (int c = 0; c < 17; ++c) red[c][threadIdx.x] += red[c][threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x < 17) part[(size_t)blockIdx.x * 17 + threadIdx.x] = red[threadIdx.x][0];
}

// out[j] = sum over s < ns of part[s * stride + j], one block per output: thread
// t adds partials t, t + kThreads, ..., then a fixed-order tree
__global__ void k_sum_partials(const float *part, int ns, int stride, float *out)
{
    __shared__ float red[kThreads];
    const int j = blockIdx.x;
    float s = 0.0f;
#pragma unroll 4
    for (int i = threadIdx.x; i < ns; i += kThreads) s += part[(size_t)i * stride + j];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = kThreads / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[j] = red[0];
}

// ---- backward elementwise parts ----

// Four values a thread (channel counts are multiples of 16): one 16-byte
// access of FP32 data, 8 bytes of bfloat16.
__device__ __forceinline__ uint2 pack4(float4 v)
{
    return make_uint2((uint32_t)f2bf(v.x) | ((uint32_t)f2bf(v.y) << 16),
                      (uint32_t)f2bf(v.z) | ((uint32_t)f2bf(v.w) << 16));
}
__device__ __forceinline__ float4 unpack4(uint2 u)
{
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u), __uint_as_float(u.y << 16),
                       __uint_as_float(u.y & 0xFFFF0000u));
}

// g *= (act > 0) when relu; gb = bfloat16(g) (may be null)
__global__ void k_mask(long long quads, float4 *g, const uint2 *act, int relu, uint2 *gb)
{
    const long long i = blockIdx.x * (long long)kThreads + threadIdx.x;
    if (i >= quads) return;
    float4 v = g[i];
    if (relu) {
        const float4 a = unpack4(act[i]);
        if (!(a.x > 0.0f)) v.x = 0.0f;
        if (!(a.y > 0.0f)) v.y = 0.0f;
        if (!(a.z > 0.0f)) v.z = 0.0f;
        if (!(a.w > 0.0f)) v.w = 0.0f;
        g[i] = v;
    }
    if (gb) gb[i] = pack4(v);
}

// the gradient of a 2x2 average: dst (n x 2h x 2w x 4 c4) += gin(n x h x w x 4 c4) / 4
__global__ void k_pool_backward(int n, int h, int w, int c4, float4 *dst, const float4 *gin)
{
    const long long i = blockIdx.x * (long long)kThreads + threadIdx.x;
    const long long tot = (long long)n * 4 * h * w * c4;
    if (i >= tot) return;
    const int ch = (int)(i % c4);
    const long long pix = i / c4;
    const int W2 = 2 * w, H2 = 2 * h;
    const int x = (int)(pix % W2), y = (int)((pix / W2) % H2);
    const long long b = pix / ((long long)W2 * H2);
    const float4 s = gin[(((size_t)b * h + y / 2) * w + x / 2) * c4 + ch];
    float4 d = dst[i];
    d.x += 0.25f * s.x;
    d.y += 0.25f * s.y;
    d.z += 0.25f * s.z;
    d.w += 0.25f * s.w;
    dst[i] = d;
}

// the gradient of a nearest-neighbour prolongation: dst (n x h/2 x w/2 x 4 c4)
// = sum of the 2x2 children in gin (n x h x w x 4 c4)
__global__ void k_up_backward(int n, int h, int w, int c4, float4 *dst, const float4 *gin)
{
    const int hc = h / 2, wc = w / 2;
    const long long i = blockIdx.x * (long long)kThreads + threadIdx.x;
    const long long tot = (long long)n * hc * wc * c4;
    if (i >= tot) return;
    const int ch = (int)(i % c4);
    const long long pix = i / c4;
    const int x = (int)(pix % wc), y = (int)((pix / wc) % hc);
    const long long b = pix / ((long long)wc * hc);
    const float4 *g = gin + (((size_t)b * h + 2 * y) * w + 2 * x) * c4 + ch;
    const float4 p = g[0], q = g[c4], r = g[(size_t)w * c4], s = g[(size_t)w * c4 + c4];
    dst[i] = make_float4((p.x + q.x) + (r.x + s.x), (p.y + q.y) + (r.y + s.y), (p.z + q.z) + (r.z + s.z),
                         (p.w + q.w) + (r.w + s.w));
}

// The input of a layer that reads an average (POOL: x0 n x 2h x 2w x 4 c4) or a
// sum with a prolonged coarser tensor (x1 n x h/2 x w/2), in bfloat16, formed
// as the forward pass forms it.
template <int MODE>
__global__ void k_form_input(int n, int h, int w, int c4, const uint2 *x0, const uint2 *x1, uint2 *out)
{
    const long long i = blockIdx.x * (long long)kThreads + threadIdx.x;
    const long long tot = (long long)n * h * w * c4;
    if (i >= tot) return;
    const int ch = (int)(i % c4);
    const long long pix = i / c4;
    const int x = (int)(pix % w), y = (int)((pix / w) % h);
    const long long b = pix / ((long long)w * h);
    if (MODE == GEA_CONV_POOL) {
        const size_t W2 = (size_t)2 * w * c4;
        const uint2 *s = x0 + ((size_t)b * 2 * h + 2 * y) * W2 + (size_t)2 * x * c4 + ch;
        const float4 p = unpack4(s[0]), q = unpack4(s[c4]), r = unpack4(s[W2]), t = unpack4(s[W2 + c4]);
        out[i] = pack4(make_float4(0.25f * ((p.x + q.x) + (r.x + t.x)), 0.25f * ((p.y + q.y) + (r.y + t.y)),
                                   0.25f * ((p.z + q.z) + (r.z + t.z)), 0.25f * ((p.w + q.w) + (r.w + t.w))));
    } else {
        const float4 p = unpack4(x0[i]);
        const float4 q = unpack4(x1[(((size_t)b * (h / 2) + y / 2) * (w / 2) + x / 2) * c4 + ch]);
        out[i] = pack4(make_float4(p.x + q.x, p.y + q.y, p.z + q.z, p.w + q.w));
    }
}

// ---- weight gradients (FP32, CUDA cores) ----

//
// dW[tap][co][ci] = sum over pixels p of g[p][co] x[p + off(tap)][ci], db = sum g.
//
// Bound: FP32 FMA issue (2 x 9 x cin x cout flops per pixel; 23 GFLOP for a
// batch of 8 x 256 x 256, 0.3 ms at the FP32 rate). A thread keeps a 4 x 4
// block of (co, ci) for the three taps of one row offset in registers and
// walks along a row with a sliding window of three input pixels: per pixel
// one 16-byte read of g and one 8-byte read of x from shared memory feed 48
// FMAs. Rows arrive by 16-byte asynchronous copies one row ahead, each input
// row once per block for its three uses. Against one accumulator per thread
// and tap with two shared-memory reads per FMA, a layer of that batch went
// from 461 to 73 us (16 -> 16 channels, full size) and from 490 to 44 us
// (64 -> 64, a quarter of the size), 33 TFLOP/s; with the sums over the blocks
// in parallel and first gradients written in place the backward pass went
// from 6.46 to 1.2 ms.
//
// A thread's running sums end after kWgChain terms, so that a larger batch
// does not lose bits: sums of equal terms, the worst case, are off by 2.4e-6 at
// 12 x 256 x 256 and 3.2e-6 at 64 x 512 x 512 (running through all of a
// block's items 4.1e-6 and 7.0e-5; one accumulator per thread and tap with
// 128-pixel partial sums 2.9e-6 and 1.4e-5). Of 64 / 128 / 256 / 512 terms, 256 is
// the longest that is no further off at any size than those partial sums. The
// split is by launches: the sums added to the block's partial inside the
// kernel took 1 to 2 % more at 8 x 256 x 256, where one launch holds all items
// (1300 us before and 1292 after; 4 x 1024 x 1024: 6763 -> 7284).

struct WgArgs {
    int n, h, w;            // the layer's size
    const uint16_t *x;      // its input, n x h x w x cin
    const float *g;         // masked output gradient, n x h x w x cout
    float *part;            // [block][tap][cout][cin]
    float *partb;           // [block][cout]
    int strips, pt;         // row segments per row and their pixels
    int rb, chunks;         // rows of a work item and items per column of segments
    int items;              // n x strips x chunks
    int first, last, add;   // the launch's items; add: to the partials of the launches before
};

// First pixel, rows and sample of item t.
__device__ __forceinline__ void wg_item(const WgArgs &a, int t, int &b, int &x0, int &y0, int &y1)
{
    const int c = t % a.chunks, s = (t / a.chunks) % a.strips;
    b = t / (a.chunks * a.strips);
    x0 = s * a.pt;
    y0 = c * a.rb;
    y1 = min(y0 + a.rb, a.h);
}

__device__ __forceinline__ void cp_async16(void *dst, const void *src, bool valid)
{
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(valid ? 16 : 0));
}

// Threads: 3 row offsets x cout/4 x cin/4 blocks of outputs x GR groups that
// split a segment's pixels (so that small layers fill a block).
template <int CIN, int COUT, int GR>
struct WgShape {
    static constexpr int TI = CIN / 4, TC = COUT / 4, OUT = 3 * TI * TC, THREADS = OUT * GR;
    static constexpr int GF = kWgPix * COUT;               // floats of a gradient row
    static constexpr int XH = (kWgPix + 2) * CIN;          // bfloat16s of an input row
    static constexpr int STAGE = 2 * GF * 4 + 4 * XH * 2;  // bytes: two gradient rows, four input rows
    static constexpr int RED = (GR - 1) * OUT * 52 * 4;    // bytes of the groups' sums
    static constexpr int SMEM = STAGE > RED ? STAGE : RED;
};

template <int CIN, int COUT, int GR>
__global__ void __launch_bounds__(WgShape<CIN, COUT, GR>::THREADS, 768 / WgShape<CIN, COUT, GR>::THREADS) k_wgrad(WgArgs a)
{
    using S = WgShape<CIN, COUT, GR>;
    extern __shared__ __align__(16) unsigned char wsm[];
    float *gs = reinterpret_cast<float *>(wsm);                              // [2][kWgPix][COUT]
    uint16_t *xs = reinterpret_cast<uint16_t *>(wsm + 2 * S::GF * 4);        // [4][kWgPix + 2][CIN]
    const int tid = threadIdx.x;
    const int ci = (tid % S::TI) * 4, co = (tid / S::TI % S::TC) * 4;
    const int dy = tid / (S::TI * S::TC) % 3, gr = tid / S::OUT;
    const bool bias = dy == 1 && ci == 0;
    const int pg = (a.pt + GR - 1) / GR, p0 = gr * pg, p1 = min(p0 + pg, a.pt);
    float acc[3][4][4], accb[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int t = 0; t < 3; ++t)
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[t][c][i] = 0.0f;
    for (int t = a.first + blockIdx.x; t < a.last; t += gridDim.x) {
        int b, x0, y0, y1;
        wg_item(a, t, b, x0, y0, y1);
        // input row y into slot (y - y0 + 1) & 3, pixels x0 - 1 .. x0 + pt, zero outside the image
        auto load_x = [&](int y) {
            uint16_t *dst = xs + ((y - y0 + 1) & 3) * S::XH;
            const bool yin = y >= 0 && y < a.h;
            for (int e = tid; e < (a.pt + 2) * (CIN / 8); e += S::THREADS) {
                const int p = e / (CIN / 8), c = e % (CIN / 8) * 8, xx = x0 - 1 + p;
                const bool in = yin && xx >= 0 && xx < a.w;
                cp_async16(dst + p * CIN + c, in ? a.x + (((size_t)b * a.h + y) * a.w + xx) * CIN + c : a.x, in);
            }
        };
        auto load_g = [&](int y) {
            float *dst = gs + ((y - y0) & 1) * S::GF;
            for (int e = tid; e < a.pt * (COUT / 4); e += S::THREADS) {
                const int p = e / (COUT / 4), c = e % (COUT / 4) * 4;
                const bool in = x0 + p < a.w;
                cp_async16(dst + p * COUT + c, in ? a.g + (((size_t)b * a.h + y) * a.w + x0 + p) * COUT + c : a.g, in);
            }
        };
        load_x(y0 - 1);
        load_x(y0);
        load_x(y0 + 1);
        load_g(y0);
        asm volatile("cp.async.commit_group;");
        for (int y = y0; y < y1; ++y) {
            if (y + 1 < y1) {
                load_x(y + 2);
                load_g(y + 1);
            }
            asm volatile("cp.async.commit_group;");
            asm volatile("cp.async.wait_group 1;");
            __syncthreads();
            const float *gp = gs + ((y - y0) & 1) * S::GF + co;
            const uint16_t *xp = xs + ((y - y0 + dy) & 3) * S::XH + ci;
            auto ldx = [&](int p) { return unpack4(*reinterpret_cast<const uint2 *>(xp + p * CIN)); };
            float4 xl = ldx(min(p0, a.pt)), xc = ldx(min(p0, a.pt) + 1);
#pragma unroll 3
            for (int p = p0; p < p1; ++p) {
                const float4 xr = ldx(p + 2);
                const float4 gv = *reinterpret_cast<const float4 *>(gp + p * COUT);
                const float g4[4] = {gv.x, gv.y, gv.z, gv.w};
                const float xv[3][4] = {{xl.x, xl.y, xl.z, xl.w}, {xc.x, xc.y, xc.z, xc.w}, {xr.x, xr.y, xr.z, xr.w}};
#pragma unroll
                for (int k = 0; k < 3; ++k)
#pragma unroll
                    for (int c = 0; c < 4; ++c)
#pragma unroll
                        for (int i = 0; i < 4; ++i) acc[k][c][i] = fmaf(g4[c], xv[k][i], acc[k][c][i]);
                if (bias) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) accb[c] += g4[c];
                }
                xl = xc;
                xc = xr;
            }
            __syncthreads();
        }
    }
    // the groups' sums in group order, then the block's partials
    asm volatile("cp.async.wait_group 0;");
    if (GR > 1) {
        float *red = reinterpret_cast<float *>(wsm);
        const int o = tid % S::OUT;
        __syncthreads();
        if (gr > 0) {
            float *r = red + (size_t)(gr - 1) * 52 * S::OUT + o;
#pragma unroll
            for (int k = 0; k < 48; ++k) r[k * S::OUT] = acc[k / 16][k / 4 % 4][k % 4];
#pragma unroll
            for (int c = 0; c < 4; ++c) r[(48 + c) * S::OUT] = accb[c];
        }
        __syncthreads();
        if (gr > 0) return;
        for (int q = 0; q < GR - 1; ++q) {
            const float *r = red + (size_t)q * 52 * S::OUT + o;
#pragma unroll
            for (int k = 0; k < 48; ++k) acc[k / 16][k / 4 % 4][k % 4] += r[k * S::OUT];
#pragma unroll
            for (int c = 0; c < 4; ++c) accb[c] += r[(48 + c) * S::OUT];
        }
    }
    float *out = a.part + (size_t)blockIdx.x * 9 * CIN * COUT;
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            float4 *p = reinterpret_cast<float4 *>(out + ((size_t)(dy * 3 + k) * COUT + co + c) * CIN + ci);
            const float4 u = a.add ? *p : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            *p = make_float4(u.x + acc[k][c][0], u.y + acc[k][c][1], u.z + acc[k][c][2], u.w + acc[k][c][3]);
        }
    if (bias)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            float *p = a.partb + (size_t)blockIdx.x * COUT + co + c;
            *p = (a.add ? *p : 0.0f) + accb[c];
        }
}

// The first layer (one input channel, 16 outputs): a thread keeps the 9 taps
// of four outputs for one pixel column of a segment and walks down its rows
// with a 3 x 3 window of the input; the 64 columns of a block are added in a
// fixed order (lanes, then warps).
__global__ void __launch_bounds__(kThreads) k_wgrad_first(WgArgs a)
{
    __shared__ float red[kThreads / 32][160];
    const int cg = threadIdx.x & 3, px = threadIdx.x >> 2;
    float acc[40];   // 9 taps x 4 outputs, then db
#pragma unroll
    for (int k = 0; k < 40; ++k) acc[k] = 0.0f;
    for (int t = a.first + blockIdx.x; t < a.last; t += gridDim.x) {
        int b, x0, y0, y1;
        wg_item(a, t, b, x0, y0, y1);
        const int xx = x0 + px;
        if (px >= a.pt || xx >= a.w) continue;
        auto row = [&](int y, float (&v)[3]) {
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const int c = xx + d - 1;
                v[d] = (y >= 0 && y < a.h && c >= 0 && c < a.w) ? bf2f(a.x[((size_t)b * a.h + y) * a.w + c]) : 0.0f;
            }
        };
        float v[3][3];
        row(y0 - 1, v[0]);
        row(y0, v[1]);
#pragma unroll 3
        for (int y = y0; y < y1; ++y) {
            row(y + 1, v[2]);
            const float4 gv =
                *reinterpret_cast<const float4 *>(a.g + (((size_t)b * a.h + y) * a.w + xx) * 16 + 4 * cg);
            const float g4[4] = {gv.x, gv.y, gv.z, gv.w};
#pragma unroll
            for (int k = 0; k < 9; ++k)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[4 * k + c] = fmaf(g4[c], v[k / 3][k % 3], acc[4 * k + c]);
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[36 + c] += g4[c];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                v[0][d] = v[1][d];
                v[1][d] = v[2][d];
            }
        }
    }
#pragma unroll
    for (int k = 0; k < 40; ++k)
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
    if ((threadIdx.x & 31) < 4)
#pragma unroll
        for (int k = 0; k < 40; ++k) red[threadIdx.x / 32][k / 4 * 16 + 4 * cg + k % 4] = acc[k];
    __syncthreads();
    const int j = threadIdx.x;
    if (j < 160) {
        float s = 0.0f;
        for (int q = 0; q < kThreads / 32; ++q) s += red[q][j];
        float *p = j < 144 ? a.part + (size_t)blockIdx.x * 144 + j : a.partb + (size_t)blockIdx.x * 16 + j - 144;
        *p = (a.add ? *p : 0.0f) + s;
    }
}

// dW[co][tap][ci] (parameter order) and db from the block partials: 32 outputs
// x 8 lanes per block; lane q adds partials q, q + 8, ..., the lanes are added
// in order.
__global__ void k_wgrad_reduce(const float *part, const float *partb, int ns, int cin, int cout, float *dw, float *db)
{
    __shared__ float red[8][32];
    const int nout = cin * cout, nw = 9 * nout;
    const int j = blockIdx.x * 32 + threadIdx.x, q = threadIdx.y;
    float s = 0.0f;
    if (j < nw + cout) {
        const float *p = j < nw ? part + j : partb + (j - nw);
        const size_t stride = j < nw ? nw : cout;
#pragma unroll 8
        for (int i = q; i < ns; i += 8) s += p[i * stride];
    }
    red[q][threadIdx.x] = s;
    __syncthreads();
    if (q || j >= nw + cout) return;
    s = 0.0f;
#pragma unroll
    for (int k = 0; k < 8; ++k) s += red[k][threadIdx.x];
    if (j < nw) {
        const int tap = j / nout, r = j % nout, co = r / cin, ci = r % cin;
        dw[((size_t)co * 9 + tap) * cin + ci] = s;
    } else {
        db[j - nw] = s;
    }
}

// ---- parameters: bfloat16 weight copies and Adam ----

// wf[co][t][ci] = bf16(W[co][t][ci]); wb[ci][t][co] = bf16(W[co][8 - t][ci])
__global__ void k_pack(const float *W, int cin, int cout, uint16_t *wf, uint16_t *wb)
{
    const int j = blockIdx.x * kThreads + threadIdx.x;
    if (j >= cout * 9 * cin) return;
    const int ci = j % cin, t = (j / cin) % 9, co = j / (9 * cin);
    const uint16_t v = f2bf(W[j]);
    wf[j] = v;
    wb[((size_t)ci * 9 + (8 - t)) * cout + co] = v;
}

__global__ void k_adam(long long np, float *th, float *m, float *v, const float *g, float lr, float b1, float b2,
                       float c1, float c2, float eps)
{
    const long long i = blockIdx.x * (long long)kThreads + threadIdx.x;
    if (i >= np) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    th[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// ---- energy loss ----

// q = A y / mean(c); per pixel loss 0.5 y q - y x and gradient (q - x) / (h w n);
// block partials of the loss (double) per sample
__global__ void k_energy(int n, int h, int w, const float *y, const float *x, const float *c, const float *ax,
                         const float *az, const float *cmean, float *dy, double *part)
{
    __shared__ double red[kThreads];
    const int b = blockIdx.y;
    const long long per = (long long)h * w;
    double s = 0.0;
    for (long long i = blockIdx.x * (long long)kThreads + threadIdx.x; i < per; i += (long long)gridDim.x * kThreads) {
        const int col = (int)(i % w), row = (int)(i / w);
        const float *ys = y + (size_t)b * per;
        const float yc = ys[i];
        const float *axs = ax + (size_t)b * h * (w + 1);
        const float *azs = az + (size_t)b * (h + 1) * w;
        float q = c[(size_t)b * per + i] * yc;
        if (col > 0) q += axs[(size_t)row * (w + 1) + col] * (yc - ys[i - 1]);
        if (col + 1 < w) q += axs[(size_t)row * (w + 1) + col + 1] * (yc - ys[i + 1]);
        if (row > 0) q += azs[(size_t)row * w + col] * (yc - ys[i - w]);
        if (row + 1 < h) q += azs[(size_t)(row + 1) * w + col] * (yc - ys[i + w]);
        q /= cmean[b];
        const float xv = x[(size_t)b * per + i];
        dy[(size_t)b * per + i] = (q - xv) / (float)((double)per * n);
        s += 0.5 * (double)yc * q - (double)yc * xv;
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = kThreads / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[(size_t)b * gridDim.x + blockIdx.x] = red[0];
}

// mean over the samples of each one's loss sum / per; one block
__global__ void k_energy_finish(const double *part, int nblk, int n, long long per, double *out)
{
    __shared__ double red[kThreads];
    double s = 0.0;
    for (int i = threadIdx.x; i < n * nblk; i += kThreads) s += part[i];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = kThreads / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = red[0] / (double)per / n;
}

inline unsigned blocks(long long cnt) { return (unsigned)((cnt + kThreads - 1) / kThreads); }

// Weight-gradient kernel of a layer: its function, threads and shared memory.
struct WgKernel {
    void (*f)(WgArgs);
    int threads, smem, groups;   // groups: of a segment's pixels, each summed by threads of its own
};
template <int CIN, int COUT, int GR>
constexpr WgKernel wg_of()
{
    return WgKernel{k_wgrad<CIN, COUT, GR>, WgShape<CIN, COUT, GR>::THREADS, WgShape<CIN, COUT, GR>::SMEM, GR};
}
// Pixel groups: a block of 192 threads (48 or 96 per group) keeps several
// blocks on an SM; from 32 x 32 on one group fills it. Backward pass at
// 8 x 256 x 256, us: 16 x 16 with 1, 2, 4 groups 1622, 1301, 1295; 16 x 32 and
// 32 x 16 with 1, 2, 4 1292, 1295, 1285; 32 x 32 with 1, 2 1295, 1290 (12 x 256 x 256:
// 1757, 1797); 32 x 64 and 64 x 32 with 1, 2 1295, 1301.
inline WgKernel wg_kernel(int cin, int cout)
{
    switch (cin * 100 + cout) {
    case 1616: return wg_of<16, 16, 4>();
    case 1632: return wg_of<16, 32, 2>();
    case 3216: return wg_of<32, 16, 2>();
    case 3232: return wg_of<32, 32, 1>();
    case 3264: return wg_of<32, 64, 1>();
    case 6432: return wg_of<64, 32, 1>();
    case 6464: return wg_of<64, 64, 1>();
    default: return WgKernel{k_wgrad_first, kThreads, 0, kWgPix};
    }
}

}  // namespace gea_net_impl

using namespace gea_net_impl;

struct gea_net {
    int nmax = 0, hmax = 0, wmax = 0, relu = 0;
    cudaStream_t st = nullptr;
    long long np = 0;
    long long offw[L], offb[L];
    float *theta = nullptr, *m = nullptr, *v = nullptr, *grad = nullptr, *dy = nullptr;
    uint16_t *wf[L] = {}, *wb[L] = {};
    uint16_t *act[L] = {};
    float *gact[L] = {};
    uint16_t *gbf = nullptr, *xbf = nullptr;
    float *gin = nullptr, *xh = nullptr, *rms = nullptr, *cmean = nullptr;
    float *part = nullptr, *partb = nullptr;
    int wg_blocks[L] = {};   // resident blocks of each layer's weight-gradient kernel
    double *dpart = nullptr, *loss = nullptr;
    int *status = nullptr;
    int n = 0, h = 0, w = 0;
    const float *last_y = nullptr;
    int t = 0;
    bool have_fwd = false;
    std::vector<void *> allocs;
};

namespace {

constexpr int kSampleBlocks = 64;
// blocks per sample of the per-sample sums of the forward pass (a read of
// the whole input, as wide as the GPU)
constexpr int kStatBlocks = 608;

long long count_params(long long *offw, long long *offb)
{
    long long o = 0;
    for (int l = 0; l < L; ++l) {
        if (offw) offw[l] = o;
        o += (long long)kL[l].cout * kL[l].k * kL[l].k * kL[l].cin;
        if (offb) offb[l] = o;
        o += kL[l].cout;
    }
    return o;
}

template <class T>
T *take(gea_net *net, size_t count, bool &ok)
{
    void *p = nullptr;
    if (!ok) return nullptr;
    if (cudaMalloc(&p, count * sizeof(T) + 16) != cudaSuccess) {
        cudaGetLastError();
        ok = false;
        return nullptr;
    }
    net->allocs.push_back(p);
    return static_cast<T *>(p);
}

long long level_pix(int n, int h, int w, int lev) { return (long long)n * (h >> lev) * (w >> lev); }

int pack_all(gea_net *net)
{
    for (int l = 1; l < kOut; ++l) {
        const int cnt = kL[l].cout * 9 * kL[l].cin;
        k_pack<<<blocks(cnt), kThreads, 0, net->st>>>(net->theta + net->offw[l], kL[l].cin, kL[l].cout, net->wf[l],
                                                      net->wb[l]);
    }
    return cudaGetLastError() == cudaSuccess ? GEA_OK : GEA_ERR_CUDA;
}

// per-sample reduction of x (n samples of `per` values) into out[b]
void sample_stat(gea_net *net, const float *x, int n, long long per, int mode, float *out)
{
    // one pass of the threads over a small sample, several over a large one
    const int nb = (int)std::min<long long>(kStatBlocks, (per / 4 + kThreads - 1) / kThreads);
    dim3 g(nb, n);
    const int vec = (reinterpret_cast<uintptr_t>(x) & 15u) == 0;
    k_sample_partials<<<g, kThreads, 0, net->st>>>(x, per, mode == 0 ? 1 : 0, vec, net->dpart);
    k_sample_finish<<<n, kThreads, 0, net->st>>>(net->dpart, nb, per, mode, out);
}

int forward(gea_net *net, int n, int h, int w, const float *r, float *y)
{
    cudaStream_t st = net->st;
    const long long per = (long long)h * w, tot = per * n;
    sample_stat(net, r, n, per, 0, net->rms);
    k_prep<<<blocks(tot), kThreads, 0, st>>>(r, net->rms, per, tot, net->xh, net->xbf);
    k_conv_first<<<blocks(tot / kFirstPix), kThreads, 0, st>>>(n, h, w, net->xbf, net->theta + net->offw[0],
                                                   net->theta + net->offb[0], net->relu && kL[0].act, net->act[0]);
    for (int l = 1; l < kOut; ++l) {
        const LayerDef &d = kL[l];
        const int hl = h >> d.level, wl = w >> d.level;
        const uint16_t *x0 = nullptr, *x1 = nullptr;
        int mode = GEA_CONV_PLAIN;
        if (d.kind == SRC_PREV) x0 = net->act[d.a];
        else if (d.kind == SRC_POOL) { x0 = net->act[d.a]; mode = GEA_CONV_POOL; }
        else { x0 = net->act[d.b]; x1 = net->act[d.a]; mode = GEA_CONV_UPADD; }
        const int flags = (net->relu && d.act) ? GEA_CONV_RELU : 0;
        if (gea_conv3x3_launch(n, hl, wl, d.cin, d.cout, mode, flags, x0, x1, net->wf[l], net->theta + net->offb[l],
                               net->act[l], net->status, st) != cudaSuccess)
            return GEA_ERR_CUDA;
    }
    k_conv_out<<<blocks(tot), kThreads, 0, st>>>(tot, net->act[kOut - 1], net->theta + net->offw[kOut],
                                                 net->theta + net->offb[kOut], y);
    if (cudaGetLastError() != cudaSuccess) return GEA_ERR_CUDA;
    net->n = n; net->h = h; net->w = w;
    net->last_y = y;
    net->have_fwd = true;
    return GEA_OK;
}

// Weight gradient of a layer into block partials, on at most `slots` resident
// blocks: row segments of at most kWgPix pixels, and as many rows per work item as
// make the longest block's rows fewest, within a thread's kWgChain terms. An
// item counts one row more than it has, for its first rows' loads, which nothing
// overlaps (8 x 256 x 256: 1295 us, without it 1351, with two rows 1295; its two
// extra input rows cost loads only). Items
// beyond those terms go to further launches, which add to the same partials.
// Returns the number of partials.
int wgrad(WgArgs &a, const WgKernel &k, int n, int h, int w, int slots, cudaStream_t st)
{
    a.n = n; a.h = h; a.w = w;
    a.strips = (w + kWgPix - 1) / kWgPix;
    a.pt = (w + a.strips - 1) / a.strips;
    const int pg = (a.pt + k.groups - 1) / k.groups;   // pixels of a row that one thread walks
    long long best = -1;
    for (int rb = 1; rb <= std::min(h, kWgChain / pg); ++rb) {
        const int chunks = (h + rb - 1) / rb;
        const long long items = (long long)n * a.strips * chunks;
        const long long cost = (items + slots - 1) / slots * (rb + 1);
        if (best < 0 || cost < best) {
            best = cost;
            a.rb = rb;
            a.chunks = chunks;
            a.items = (int)items;
        }
    }
    const int ns = std::min(a.items, slots), step = ns * (kWgChain / (a.rb * pg));
    for (a.first = 0, a.add = 0; a.first < a.items; a.first = a.last, a.add = 1) {
        a.last = std::min(a.first + step, a.items);
        k.f<<<std::min(ns, a.last - a.first), k.threads, k.smem, st>>>(a);
    }
    return ns;
}

int backward(gea_net *net, const float *dy, float *grad)
{
    cudaStream_t st = net->st;
    const int n = net->n, h = net->h, w = net->w;
    const long long tot = (long long)n * h * w;
    // output layer
    {
        const unsigned nb = blocks(tot);
        k_out_backward<<<nb, kThreads, 0, st>>>(tot, dy, net->act[kOut - 1], net->theta + net->offw[kOut],
                                                net->gact[kOut - 1], net->part);
        k_sum_partials<<<17, kThreads, 0, st>>>(net->part, (int)nb, 17, grad + net->offw[kOut]);
    }
    for (int l = kOut - 1; l >= 0; --l) {
        const LayerDef &d = kL[l];
        const int hl = h >> d.level, wl = w >> d.level;
        const long long pix = level_pix(n, h, w, d.level), quads = pix * d.cout / 4;
        const int relu = net->relu && d.act;
        if (relu || l > 0)
            k_mask<<<blocks(quads), kThreads, 0, st>>>(quads, reinterpret_cast<float4 *>(net->gact[l]),
                                                       reinterpret_cast<const uint2 *>(net->act[l]), relu,
                                                       l > 0 ? reinterpret_cast<uint2 *>(net->gbf) : nullptr);
        // the layer's input: an averaged or summed one is formed again, in the
        // buffer that the data gradient overwrites afterwards
        WgArgs a{};
        uint2 *xin = reinterpret_cast<uint2 *>(net->gin);
        const int c4 = d.cin / 4;
        if (d.kind == SRC_X) a.x = net->xbf;
        else if (d.kind == SRC_PREV) a.x = net->act[d.a];
        else {
            a.x = reinterpret_cast<const uint16_t *>(xin);
            if (d.kind == SRC_POOL)
                k_form_input<GEA_CONV_POOL><<<blocks(pix * c4), kThreads, 0, st>>>(
                    n, hl, wl, c4, reinterpret_cast<const uint2 *>(net->act[d.a]), nullptr, xin);
            else
                k_form_input<GEA_CONV_UPADD><<<blocks(pix * c4), kThreads, 0, st>>>(
                    n, hl, wl, c4, reinterpret_cast<const uint2 *>(net->act[d.b]),
                    reinterpret_cast<const uint2 *>(net->act[d.a]), xin);
        }
        a.g = net->gact[l];
        a.part = net->part; a.partb = net->partb;
        const int ns = wgrad(a, wg_kernel(d.cin, d.cout), n, hl, wl, net->wg_blocks[l], st);
        k_wgrad_reduce<<<(9 * d.cin * d.cout + d.cout + 31) / 32, dim3(32, 8), 0, st>>>(
            net->part, net->partb, ns, d.cin, d.cout, grad + net->offw[l], grad + net->offb[l]);
        if (l == 0) break;
        // data gradient on the tensor cores: correlation of bf16(g) with the
        // mirrored, transposed weights. A tensor's first gradient is written
        // in place (the layers run last to first: a skip tensor's comes from
        // the way up), the averaging's is added to it.
        float *dst = d.kind == SRC_POOL ? net->gin : net->gact[d.kind == SRC_UPADD ? d.b : d.a];
        if (gea_conv3x3_launch(n, hl, wl, d.cout, d.cin, GEA_CONV_PLAIN, GEA_CONV_OUT_F32, net->gbf, nullptr,
                               net->wb[l], nullptr, dst, net->status, st) != cudaSuccess)
            return GEA_ERR_CUDA;
        const float4 *dst4 = reinterpret_cast<const float4 *>(dst);
        float4 *ga = reinterpret_cast<float4 *>(net->gact[d.a]);
        if (d.kind == SRC_POOL)
            k_pool_backward<<<blocks(pix * c4 * 4), kThreads, 0, st>>>(n, hl, wl, c4, ga, dst4);
        else if (d.kind == SRC_UPADD)
            k_up_backward<<<blocks(pix * c4 / 4), kThreads, 0, st>>>(n, hl, wl, c4, ga, dst4);
    }
    return cudaGetLastError() == cudaSuccess ? GEA_OK : GEA_ERR_CUDA;
}

int energy(gea_net *net, const float *c, const float *ax, const float *az, float *dy, float *loss)
{
    if (!net->have_fwd) return GEA_ERR_STATE;
    cudaStream_t st = net->st;
    const int n = net->n, h = net->h, w = net->w;
    const long long per = (long long)h * w;
    sample_stat(net, c, n, per, 1, net->cmean);
    dim3 g(kSampleBlocks, n);
    k_energy<<<g, kThreads, 0, st>>>(n, h, w, net->last_y, net->xh, c, ax, az, net->cmean, dy, net->dpart);
    k_energy_finish<<<1, kThreads, 0, st>>>(net->dpart, kSampleBlocks, n, per, net->loss);
    double hl = 0.0;
    if (cudaMemcpyAsync(&hl, net->loss, sizeof(double), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return GEA_ERR_CUDA;
    if (loss) *loss = (float)hl;
    return GEA_OK;
}

int adam(gea_net *net, const float *grad, float lr)
{
    net->t += 1;
    const double b1 = 0.9, b2 = 0.999;
    const float c1 = (float)(1.0 - pow(b1, net->t)), c2 = (float)(1.0 - pow(b2, net->t));
    k_adam<<<blocks(net->np), kThreads, 0, net->st>>>(net->np, net->theta, net->m, net->v, grad, lr, (float)b1,
                                                      (float)b2, c1, c2, 1e-8f);
    if (cudaGetLastError() != cudaSuccess) return GEA_ERR_CUDA;
    return pack_all(net);
}

bool shape_ok(const gea_net *net, int n, int h, int w)
{
    // every buffer is sized by the total pixel count (and the per-sample
    // arrays by n_max)
    return n >= 1 && n <= net->nmax && h >= 8 && w >= 8 && h % 8 == 0 && w % 8 == 0 &&
           (long long)n * h * w <= (long long)net->nmax * net->hmax * net->wmax;
}

}  // namespace

int gea_net_launches();

int gea_net_run(gea_net *net, cudaStream_t st, int n, int h, int w, const float *r, float *y)
{
    if (!net || !shape_ok(net, n, h, w)) return -1;
    cudaStream_t old = net->st;
    net->st = st;
    const int rc = forward(net, n, h, w, r, y);
    net->st = old;
    return rc ? -1 : gea_net_launches();
}

// per-sample statistics (2), input scaling, first layer, 13 tensor-core
// layers, output layer
int gea_net_launches() { return 2 + 1 + 1 + (kOut - 1) + 1; }

bool gea_net_fits(const gea_net *net, int n, int h, int w) { return net && shape_ok(net, n, h, w); }

extern "C" {

int64_t gea_net_param_count(void) { return count_params(nullptr, nullptr); }

int gea_net_layout(int32_t *desc)
{
    if (!desc) return GEA_ERR_INVAL;
    for (int l = 0; l < L; ++l) {
        const LayerDef &d = kL[l];
        const int32_t v[6] = {d.cin, d.cout, d.k, d.act, d.kind, d.level};
        for (int j = 0; j < 6; ++j) desc[6 * l + j] = v[j];
    }
    return GEA_OK;
}

int gea_net_create(int32_t n_max, int32_t h_max, int32_t w_max, int32_t flags, gea_net **out)
{
    if (!out) return GEA_ERR_INVAL;
    *out = nullptr;
    if (n_max < 1 || h_max < 8 || w_max < 8 || h_max % 8 || w_max % 8 || (flags & ~GEA_NET_RELU) ||
        (long long)n_max * h_max * w_max > (1LL << 31) / 64)
        return GEA_ERR_INVAL;
    gea_net *net = new gea_net();
    net->nmax = n_max; net->hmax = h_max; net->wmax = w_max;
    net->relu = (flags & GEA_NET_RELU) ? 1 : 0;
    net->np = count_params(net->offw, net->offb);
    bool ok = true;
    net->theta = take<float>(net, net->np, ok);
    net->m = take<float>(net, net->np, ok);
    net->v = take<float>(net, net->np, ok);
    net->grad = take<float>(net, net->np, ok);
    const long long pix = (long long)n_max * h_max * w_max;
    net->dy = take<float>(net, pix, ok);
    for (int l = 0; l < L; ++l) {
        const long long lp = level_pix(n_max, h_max, w_max, kL[l].level);
        if (l < kOut) {
            net->act[l] = take<uint16_t>(net, lp * kL[l].cout, ok);
            net->gact[l] = take<float>(net, lp * kL[l].cout, ok);
        }
        if (l >= 1 && l < kOut) {
            net->wf[l] = take<uint16_t>(net, (size_t)kL[l].cout * 9 * kL[l].cin, ok);
            net->wb[l] = take<uint16_t>(net, (size_t)kL[l].cout * 9 * kL[l].cin, ok);
        }
    }
    net->gbf = take<uint16_t>(net, pix * 16, ok);
    net->gin = take<float>(net, pix * 16, ok);
    net->xbf = take<uint16_t>(net, pix, ok);
    net->xh = take<float>(net, pix, ok);
    net->rms = take<float>(net, n_max, ok);
    net->cmean = take<float>(net, n_max, ok);
    // block partials of the weight gradients: one set per resident block
    int dev = 0, sms = 0;
    long long pcount = 17 * ((pix + kThreads - 1) / kThreads), bcount = 0;
    ok = ok && cudaGetDevice(&dev) == cudaSuccess &&
         cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess;
    for (int l = 0; l < kOut && ok; ++l) {
        const WgKernel k = wg_kernel(kL[l].cin, kL[l].cout);
        int per_sm = 0;
        ok = cudaFuncSetAttribute(k.f, cudaFuncAttributeMaxDynamicSharedMemorySize, k.smem) == cudaSuccess &&
             cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k.f, k.threads, k.smem) == cudaSuccess && per_sm > 0;
        net->wg_blocks[l] = per_sm * sms;
        pcount = std::max(pcount, (long long)net->wg_blocks[l] * 9 * kL[l].cin * kL[l].cout);
        bcount = std::max(bcount, (long long)net->wg_blocks[l] * kL[l].cout);
    }
    net->part = take<float>(net, pcount, ok);
    net->partb = take<float>(net, bcount, ok);
    net->dpart = take<double>(net, (size_t)n_max * (kStatBlocks > kSampleBlocks ? kStatBlocks : kSampleBlocks), ok);
    net->loss = take<double>(net, 1, ok);
    net->status = take<int>(net, 1, ok);
    if (!ok) {
        gea_net_destroy(net);
        return GEA_ERR_NOMEM;
    }
    if (cudaMemset(net->theta, 0, net->np * sizeof(float)) != cudaSuccess ||
        cudaMemset(net->m, 0, net->np * sizeof(float)) != cudaSuccess ||
        cudaMemset(net->v, 0, net->np * sizeof(float)) != cudaSuccess ||
        cudaMemset(net->status, 0, sizeof(int)) != cudaSuccess || pack_all(net) != GEA_OK ||
        cudaDeviceSynchronize() != cudaSuccess) {
        gea_net_destroy(net);
        return GEA_ERR_CUDA;
    }
    *out = net;
    return GEA_OK;
}

int gea_net_set_stream(gea_net *net, void *stream)
{
    if (!net) return GEA_ERR_INVAL;
    net->st = (cudaStream_t)stream;
    return GEA_OK;
}

int gea_net_set_params(gea_net *net, const float *theta, int32_t mem)
{
    if (!net || !theta || (mem != GEA_MEM_HOST && mem != GEA_MEM_DEVICE)) return GEA_ERR_INVAL;
    if (cudaMemcpyAsync(net->theta, theta, net->np * sizeof(float), cudaMemcpyDefault, net->st) != cudaSuccess ||
        cudaMemsetAsync(net->m, 0, net->np * sizeof(float), net->st) != cudaSuccess ||
        cudaMemsetAsync(net->v, 0, net->np * sizeof(float), net->st) != cudaSuccess)
        return GEA_ERR_CUDA;
    net->t = 0;
    int rc = pack_all(net);
    if (rc) return rc;
    return cudaStreamSynchronize(net->st) == cudaSuccess ? GEA_OK : GEA_ERR_CUDA;
}

int gea_net_get_params(gea_net *net, float *theta, int32_t mem)
{
    if (!net || !theta || (mem != GEA_MEM_HOST && mem != GEA_MEM_DEVICE)) return GEA_ERR_INVAL;
    if (cudaMemcpyAsync(theta, net->theta, net->np * sizeof(float), cudaMemcpyDefault, net->st) != cudaSuccess ||
        cudaStreamSynchronize(net->st) != cudaSuccess)
        return GEA_ERR_CUDA;
    return GEA_OK;
}

int gea_net_forward(gea_net *net, int32_t n, int32_t h, int32_t w, const float *r, float *y)
{
    if (!net || !r || !y || !shape_ok(net, n, h, w)) return GEA_ERR_INVAL;
    return forward(net, n, h, w, r, y);
}

int gea_net_energy(gea_net *net, const float *c, const float *ax, const float *az, float *dy, float *loss)
{
    if (!net || !c || !ax || !az || !dy) return GEA_ERR_INVAL;
    return energy(net, c, ax, az, dy, loss);
}

int gea_net_backward(gea_net *net, const float *dy, float *grad)
{
    if (!net || !dy || !grad) return GEA_ERR_INVAL;
    if (!net->have_fwd) return GEA_ERR_STATE;
    return backward(net, dy, grad);
}

int gea_net_adam(gea_net *net, const float *grad, float lr)
{
    if (!net || !grad || !(lr >= 0.0f)) return GEA_ERR_INVAL;
    return adam(net, grad, lr);
}

int gea_net_train_step(gea_net *net, int32_t n, int32_t h, int32_t w, const float *r, const float *c,
                       const float *ax, const float *az, float lr, float *loss)
{
    if (!net || !r || !c || !ax || !az || !shape_ok(net, n, h, w) || !(lr >= 0.0f)) return GEA_ERR_INVAL;
    // the network's own output buffer: the gradient buffer's first n h w values
    // are free until the backward pass (which reads dy, not y)
    float *y = net->gin;
    int rc = forward(net, n, h, w, r, y);
    if (!rc) rc = energy(net, c, ax, az, net->dy, loss);
    if (!rc) rc = backward(net, net->dy, net->grad);
    if (!rc) rc = adam(net, net->grad, lr);
    return rc;
}

void gea_net_destroy(gea_net *net)
{
    if (!net) return;
    if (net->st) cudaStreamSynchronize(net->st);
    else cudaDeviceSynchronize();
    for (void *p : net->allocs) cudaFree(p);
    delete net;
}

}  // extern "C"
