// Warm-start network: forward, backward and Adam kernels (BF16 operands, FP32 accumulation).
//
// Architecture (the same flat parameter layout as the FP64 reference in the tests):
//   block l = 0..3: h <- silu(rmsnorm(conv3x3(h; W_l, b_l, dilation 2^l); g_l)), 2 -> C -> C -> C -> C
//   head:           y <- conv3x3(h; W_4, b_4), C -> 2: predicted (u, v) / k^2
// Layouts: features, prediction and their gradients NCHW (2 channels).  The 32-channel conv inputs and
// the gradients that are convolution operands in BF16, 32 channels of a pixel together (64 bytes), so
// that a tile's im2col operand is 16-byte copies; pre-normalisation outputs z in FP32, four channels of
// a pixel together in blocks of 128 pixels (zoff), so that a thread per pixel reads and writes whole
// lines.  Weights are kept in FP32 (Adam's master copy) with BF16 copies for the convolutions.
// The convolutions from 32 channels (forward, data and weight gradients; of the head the
// weight gradient) are implicit GEMMs on the
// tensor cores, with the bias, the normalisation, its backward and the sums of the bias and gain
// gradients in their epilogues; the 2 -> 32 convolution, the head and the data gradients around the two
// 2-channel ends run on the FP32 pipes.  Every reduction runs in a fixed order (per-CTA partials, one pass).
#include <cuda_bf16.h>

#include <cmath>
#include <cstring>
#include <new>
#include <string>

#include "common.cuh"
#include "ot_ipm.h"
#include "tc05.cuh"

namespace ot {
namespace {

constexpr int kLayers = 5;
constexpr int kMaxBatch = 4096;
constexpr int kDil[kLayers] = {1, 2, 4, 8, 1};
constexpr float kEps = 1e-5f;
constexpr int kPix = 128;     // pixels of a tile
constexpr int kThr = 4 * kPix;   // a thread for 8 of a pixel's 32 channels: row tid % 128, channels 8 (tid / 128) ..

struct Layer {
    int cin, cout, dil;
    bool norm;
    int64_t W, b, g;   // offsets in the flat parameter array
};

__device__ __forceinline__ float silu_f(float t) { return t / (1.f + __expf(-t)); }

// float4 index of channels 4 q .. 4 q + 3 of pixel p in a z buffer
__device__ __forceinline__ int64_t zoff(int64_t p, int q) { return ((p >> 7) * 8 + q) * 128 + (p & 127); }

// Programmatic dependent launch: a kernel launched with it may start before the one ahead has ended;
// everything that kernel (or an earlier one) wrote is read after pdl_wait.
__device__ __forceinline__ void pdl_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ void st_bf16x8(__nv_bfloat16 *dst, const float (&v)[8]) {
    uint32_t w[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const uint32_t lo = __bfloat16_as_ushort(__float2bfloat16(v[2 * e]));
        const uint32_t hi = __bfloat16_as_ushort(__float2bfloat16(v[2 * e + 1]));
        w[e] = lo | (hi << 16);
    }
    *(uint4 *)dst = make_uint4(w[0], w[1], w[2], w[3]);
}

__device__ __forceinline__ void st_z8(float *zb, int64_t p, int q, const float (&v)[8]) {
    ((float4 *)zb)[zoff(p, 2 * q)] = make_float4(v[0], v[1], v[2], v[3]);
    ((float4 *)zb)[zoff(p, 2 * q + 1)] = make_float4(v[4], v[5], v[6], v[7]);
}

// Eight of a pixel's pre-normalisation values, the sum of all 32 squares given: stored, normalised (h =
// silu(g z / r), r = sqrt(mean_c z^2 + eps)) and stored in BF16.  Two divisions and an exponential per
// value: a thread for all 32 took longer over them than over the convolution, on a chip that its
// pixels fill with one warp per scheduler.
__device__ __forceinline__ void norm_fwd8(int64_t p, int q, float ss, const float (&z)[8], const float *g,
                                          float *__restrict__ zb, float *__restrict__ r,
                                          __nv_bfloat16 *__restrict__ h) {
    const float rr = sqrtf(ss / 32 + kEps);
    if (q == 0) r[p] = rr;
    st_z8(zb, p, q, z);
    float o[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) o[c] = silu_f(g[8 * q + c] * z[c] / rr);
    st_bf16x8(h + p * 32 + 8 * q, o);
}

// dh -> dz of eight of a pixel's channels through silu and the RMS normalisation (called by all threads
// of the CTA; others' pixels with valid = false); dgl: the part of the gain's gradient.  The pixel's dot
// product runs through its four threads in the order of the channels (sdot[4][128]): dz is rounded to BF16,
// and other orders turn roundings over that three layers' gradients then carry (four partial sums added:
// 1e-5 of the gradient at 21x21 x 5).
__device__ __forceinline__ void norm_bwd8(bool valid, int64_t p, int row, int q, float (&dh)[8],
                                          const float *__restrict__ zb, const float *__restrict__ r, const float *g,
                                          float (&dgl)[8], float (*sdot)[kPix]) {
    float rr = 1.f;
    float xh[8] = {};
    if (valid) {
        rr = r[p];
        const float4 a = ((const float4 *)zb)[zoff(p, 2 * q)], b = ((const float4 *)zb)[zoff(p, 2 * q + 1)];
        xh[0] = a.x; xh[1] = a.y; xh[2] = a.z; xh[3] = a.w;
        xh[4] = b.x; xh[5] = b.y; xh[6] = b.z; xh[7] = b.w;
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        xh[c] = xh[c] / rr;
        const float yn = g[8 * q + c] * xh[c];
        const float s = 1.f / (1.f + __expf(-yn));
        const float dyn = dh[c] * (s + yn * s * (1.f - s));
        dgl[c] = dyn * xh[c];
        dh[c] = dyn * g[8 * q + c];
    }
    for (int k = 0; k < 4; ++k) {
        if (q == k) {
            float d = k ? sdot[k - 1][row] : 0.f;
#pragma unroll
            for (int c = 0; c < 8; ++c) d += dh[c] * xh[c];
            sdot[k][row] = d;
        }
        __syncthreads();
    }
    const float dot = sdot[3][row] / 32;
#pragma unroll
    for (int c = 0; c < 8; ++c) dh[c] = (dh[c] - xh[c] * dot) / rr;
}

// Per-CTA sums over the pixels of dgl and dz: lane l of a warp holds column (l / 2) of its 16 (8 gains, 8
// biases), by 16 shuffles per tile (each step halves what a lane keeps).
struct GradSums {
    float s = 0.f;
    __device__ __forceinline__ void add(const float (&dgl)[8], const float (&dz)[8], int lane) {
        float v[16];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            v[c] = dgl[c];
            v[8 + c] = dz[c];
        }
#pragma unroll
        for (int half = 8; half > 0; half >>= 1) {
            const bool up = lane & (2 * half);
#pragma unroll
            for (int i = 0; i < half; ++i) {
                const float send = up ? v[i] : v[i + half], keep = up ? v[i + half] : v[i];
                v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * half);
            }
        }
        s += v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
    }
    // the 16 warps' sums through sh to row[0 .. 63] (32 gains, 32 biases)
    __device__ __forceinline__ void store(float (*sh)[16], float *row, int lane, int warp) {
        if (!(lane & 1)) sh[warp][lane >> 1] = s;
        __syncthreads();
        if (threadIdx.x < 64) {
            const int c = threadIdx.x & 31, w = 4 * (c >> 3), j = (c & 7) + (threadIdx.x >> 5) * 8;
            row[threadIdx.x] = ((sh[w][j] + sh[w + 1][j]) + sh[w + 2][j]) + sh[w + 3][j];
        }
    }
};
constexpr int kSumRow = 80;   // one CTA's row: 32 gains, 32 biases, 2 biases of the head

// First block: features x (FP32, rounded to BF16 as the convolution's operand and kept for the weight
// gradient), 2 -> 32 convolution, normalisation.
__global__ void __launch_bounds__(kThr)
block0_kernel(int B, int H, int Wd, int dil, const float *__restrict__ x, const __nv_bfloat16 *__restrict__ w,
              const float *__restrict__ bias, const float *__restrict__ g, __nv_bfloat16 *__restrict__ xb,
              float *__restrict__ zb, float *__restrict__ r, __nv_bfloat16 *__restrict__ h) {
    __shared__ __align__(16) float ws[18 * 32];   // [c][t][o]
    __shared__ float sz[kPix][33], sg[32];
    pdl_start();
    for (int q = threadIdx.x; q < 18 * 32; q += kThr) {
        const int o = q % 32, ct = q / 32;
        ws[q] = __bfloat162float(w[o * 18 + ct]);
    }
    if (threadIdx.x < 32) sg[threadIdx.x] = g[threadIdx.x];
    __syncthreads();
    const int HW = H * Wd, row = threadIdx.x & (kPix - 1), q = threadIdx.x / kPix;
    const int64_t p = (int64_t)blockIdx.x * kPix + row;
    const bool valid = p < (int64_t)B * HW;
    float acc[8];
    if (valid) {
        const int b = (int)(p / HW), yx = (int)(p % HW), y = yx / Wd, xx0 = yx % Wd;
#pragma unroll
        for (int o = 0; o < 8; ++o) acc[o] = bias[8 * q + o];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const float *src = x + ((int64_t)b * 2 + c) * HW;
            if (q == c) xb[((int64_t)b * 2 + c) * HW + yx] = __float2bfloat16(src[yx]);
#pragma unroll
            for (int t = 0; t < 9; ++t) {
                const int yy = y + (t / 3 - 1) * dil, xx = xx0 + (t % 3 - 1) * dil;
                const float v = (yy >= 0 && yy < H && xx >= 0 && xx < Wd)
                                    ? __bfloat162float(__float2bfloat16(src[yy * Wd + xx])) : 0.f;
                const float4 *wr = (const float4 *)(ws + (c * 9 + t) * 32 + 8 * q);
                const float4 wa = wr[0], wc = wr[1];
                acc[0] += v * wa.x; acc[1] += v * wa.y; acc[2] += v * wa.z; acc[3] += v * wa.w;
                acc[4] += v * wc.x; acc[5] += v * wc.y; acc[6] += v * wc.z; acc[7] += v * wc.w;
            }
        }
#pragma unroll
        for (int o = 0; o < 8; ++o) sz[row][8 * q + o] = acc[o];
    }
    __syncthreads();
    if (!valid) return;
    float ss = 0.f;
#pragma unroll
    for (int c = 0; c < 32; ++c) ss += sz[row][c] * sz[row][c];
    norm_fwd8(p, q, ss, acc, sg, zb, r, h);
}

// Head: y[o] = bias[o] + sum_{c, t} W[o, c, t] h[pixel + offset_t, c], a thread per pixel, channels outermost.
// Its last bits decide BF16 roundings throughout the backward pass, so the sum keeps one FP32 chain in
// this order (as MMAs with eight partial sums it gave gradients up to 5e-5 apart).  A
// pixel's channels lie together: nine 16-byte loads for eight channels, the next nine already in flight.
// Latency-bound, a chain of 288 multiply-adds per output; 64x64 x 16: 35 -> 11.6 us (as MMAs 12).
constexpr int kHdThr = 64;
__global__ void __launch_bounds__(kHdThr)
head_kernel(int B, int H, int Wd, int dil, const __nv_bfloat16 *__restrict__ h, const __nv_bfloat16 *__restrict__ w,
            const float *__restrict__ bias, float *__restrict__ out, float *__restrict__ out2) {
    __shared__ __align__(16) float2 ws[32 * 9];   // [c][t] of both outputs
    pdl_start();
    for (int q = threadIdx.x; q < 32 * 9; q += kHdThr)
        ws[q] = make_float2(__bfloat162float(w[q]), __bfloat162float(w[32 * 9 + q]));
    __syncthreads();
    pdl_wait();
    const int HW = H * Wd;
    const int64_t p = (int64_t)blockIdx.x * kHdThr + threadIdx.x;
    if (p >= (int64_t)B * HW) return;
    const int yx = (int)(p % HW), y = yx / Wd, x = yx % Wd;
    const __nv_bfloat16 *src = h + p * 32;
    int off[9];
    unsigned in = 0;
#pragma unroll
    for (int t = 0; t < 9; ++t) {
        const int dy = (t / 3 - 1) * dil, dx = (t % 3 - 1) * dil;
        off[t] = (dy * Wd + dx) * 32;
        if (y + dy >= 0 && y + dy < H && x + dx >= 0 && x + dx < Wd) in |= 1u << t;
    }
    uint4 nxt[9], cur[9];
    auto load = [&](int c0) {
#pragma unroll
        for (int t = 0; t < 9; ++t)
            nxt[t] = in >> t & 1 ? *(const uint4 *)(src + off[t] + c0) : make_uint4(0u, 0u, 0u, 0u);
    };
    float a0 = bias[0], a1 = bias[1];
    load(0);
#pragma unroll 1
    for (int c0 = 0; c0 < 32; c0 += 8) {
#pragma unroll
        for (int t = 0; t < 9; ++t) cur[t] = nxt[t];
        if (c0 < 24) load(c0 + 8);
#pragma unroll
        for (int e = 0; e < 8; ++e)
#pragma unroll
            for (int t = 0; t < 9; ++t) {
                const uint32_t u = e < 2 ? cur[t].x : e < 4 ? cur[t].y : e < 6 ? cur[t].z : cur[t].w;
                const float v = __uint_as_float(e & 1 ? u & 0xffff0000u : u << 16);
                const float2 wv = ws[(c0 + e) * 9 + t];
                a0 += v * wv.x;
                a1 += v * wv.y;
            }
    }
    const int64_t at = (p / HW) * 2 * HW + yx;
    out[at] = a0;
    out[at + HW] = a1;
    if (out2) {
        out2[at] = a0;
        out2[at + HW] = a1;
    }
}

// Head's data gradient dh[c] = sum_{o, t} W[o, c, t] dy[o, y - oy_t, x - ox_t], then the last block's
// normalisation backward: dz in BF16, row sums of dg, db and of dy (the head's bias).  CTAs take tiles
// gridDim.x apart.
__global__ void __launch_bounds__(kThr, 2)
head_bwd_kernel(int B, int H, int Wd, const float *__restrict__ dy, const __nv_bfloat16 *__restrict__ w,
                const float *__restrict__ g, const float *__restrict__ zb, const float *__restrict__ r,
                __nv_bfloat16 *__restrict__ dzb, float *__restrict__ part) {
    __shared__ __align__(16) float ws[18 * 32];   // [o][t][c]
    __shared__ float sg[32], sh[16][16], sdot[4][kPix];
    __shared__ float shb[4][2];
    pdl_start();
    for (int q = threadIdx.x; q < 18 * 32; q += kThr) {
        const int c = q % 32, ot = q / 32, o = ot / 9, t = ot % 9;
        ws[q] = __bfloat162float(w[(o * 32 + c) * 9 + t]);
    }
    if (threadIdx.x < 32) sg[threadIdx.x] = g[threadIdx.x];
    __syncthreads();
    const int HW = H * Wd, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int row = threadIdx.x & (kPix - 1), q = threadIdx.x / kPix;
    const int64_t P = (int64_t)B * HW;
    GradSums sums;
    float sy[2] = {0.f, 0.f};
    for (int64_t t0 = (int64_t)blockIdx.x * kPix; t0 < P; t0 += (int64_t)gridDim.x * kPix) {
        const int64_t p = t0 + row;
        const bool valid = p < P;
        float acc[8] = {}, dgl[8];
        if (valid) {
            const int b = (int)(p / HW), yx = (int)(p % HW), y = yx / Wd, x = yx % Wd;
#pragma unroll
            for (int o = 0; o < 2; ++o) {
                const float *src = dy + ((int64_t)b * 2 + o) * HW;
                sy[o] += src[yx];
#pragma unroll
                for (int t = 0; t < 9; ++t) {
                    const int yy = y - (t / 3 - 1), xx = x - (t % 3 - 1);
                    if (yy < 0 || yy >= H || xx < 0 || xx >= Wd) continue;
                    const float v = src[yy * Wd + xx];
                    const float4 *wr = (const float4 *)(ws + (o * 9 + t) * 32 + 8 * q);
                    const float4 wa = wr[0], wc = wr[1];
                    acc[0] += v * wa.x; acc[1] += v * wa.y; acc[2] += v * wa.z; acc[3] += v * wa.w;
                    acc[4] += v * wc.x; acc[5] += v * wc.y; acc[6] += v * wc.z; acc[7] += v * wc.w;
                }
            }
        }
        norm_bwd8(valid, p, row, q, acc, zb, r, sg, dgl, sdot);
        if (valid) st_bf16x8(dzb + p * 32 + 8 * q, acc);
        sums.add(dgl, acc, lane);
        __syncthreads();   // sdot
    }
    if (q == 0) {
#pragma unroll
        for (int o = 0; o < 2; ++o) {
#pragma unroll
            for (int k = 16; k > 0; k >>= 1) sy[o] += __shfl_xor_sync(0xffffffffu, sy[o], k);
            if (lane == 0) shb[warp][o] = sy[o];
        }
    }
    float *prow = part + (int64_t)blockIdx.x * kSumRow;
    sums.store(sh, prow, lane, warp);
    if (threadIdx.x < 2)
        prow[64 + threadIdx.x] = ((shb[0][threadIdx.x] + shb[1][threadIdx.x]) + shb[2][threadIdx.x]) + shb[3][threadIdx.x];
}

// din[b, c, y, x] = sum_{o, t} W[o, c, t] dz[o, y - oy_t, x - ox_t] of the first convolution (dz in FP32
// z layout)
__global__ void __launch_bounds__(kPix)
block0_bwd_data_kernel(int B, int H, int Wd, int dil, const float *__restrict__ dz,
                       const __nv_bfloat16 *__restrict__ w, float *__restrict__ din) {
    __shared__ float ws[32 * 9 * 2];   // [o][t][c]
    for (int q = threadIdx.x; q < 32 * 9 * 2; q += blockDim.x) {
        const int c = q % 2, ot = q / 2, o = ot / 9, t = ot % 9;
        ws[q] = __bfloat162float(w[(o * 2 + c) * 9 + t]);
    }
    __syncthreads();
    const int HW = H * Wd;
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= (int64_t)B * HW) return;
    const int b = (int)(p / HW), yx = (int)(p % HW), y = yx / Wd, x = yx % Wd;
    float acc[2] = {0.f, 0.f};
    for (int q = 0; q < 8; ++q)
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            const int yy = y - (t / 3 - 1) * dil, xx = x - (t % 3 - 1) * dil;
            if (yy < 0 || yy >= H || xx < 0 || xx >= Wd) continue;
            const float4 v = ((const float4 *)dz)[zoff((int64_t)b * HW + yy * Wd + xx, q)];
            const float d[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float *wr = ws + ((4 * q + e) * 9 + t) * 2;
                acc[0] += d[e] * wr[0];
                acc[1] += d[e] * wr[1];
            }
        }
#pragma unroll
    for (int c = 0; c < 2; ++c) din[((int64_t)b * 2 + c) * HW + yx] = acc[c];
}

// Per-CTA partials of the first convolution's weight gradient over kW0 pixels: lane = output channel,
// warp w the (channel, tap) pairs w, w + 8, w + 16 of 18; dz (FP32) and the shifted features staged in
// shared memory, read four pixels at a time.  part[cta 576 + ct 32 + o].
constexpr int kW0 = 128;
__global__ void __launch_bounds__(256)
block0_wgrad_kernel(int B, int H, int Wd, int dil, const __nv_bfloat16 *__restrict__ xb,
                    const float *__restrict__ dz, float *__restrict__ part) {
    __shared__ __align__(16) float sd[32][kW0 + 4];
    __shared__ __align__(16) float sx[18][kW0];
    const int HW = H * Wd, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t P = (int64_t)B * HW, p0 = (int64_t)blockIdx.x * kW0;
    pdl_start();
    pdl_wait();
    for (int q = threadIdx.x; q < kW0 * 8; q += 256) {
        const int i = q & (kW0 - 1), c4 = q / kW0;
        const float4 v = p0 + i < P ? ((const float4 *)dz)[zoff(p0 + i, c4)] : make_float4(0.f, 0.f, 0.f, 0.f);
        sd[4 * c4][i] = v.x; sd[4 * c4 + 1][i] = v.y; sd[4 * c4 + 2][i] = v.z; sd[4 * c4 + 3][i] = v.w;
    }
    {
        const int i = threadIdx.x & (kW0 - 1), c = threadIdx.x / kW0;   // 256 threads: 128 pixels, 2 channels
        const int64_t p = p0 + i;
        const bool valid = p < P;
        const int b = valid ? (int)(p / HW) : 0, yx = valid ? (int)(p % HW) : 0, y = yx / Wd, x = yx % Wd;
        const __nv_bfloat16 *src = xb + ((int64_t)b * 2 + c) * HW;
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            const int yy = y + (t / 3 - 1) * dil, xx = x + (t % 3 - 1) * dil;
            sx[9 * c + t][i] = (valid && yy >= 0 && yy < H && xx >= 0 && xx < Wd) ? __bfloat162float(src[yy * Wd + xx]) : 0.f;
        }
    }
    __syncthreads();
    float acc[3] = {0.f, 0.f, 0.f};
    const int ct0 = warp, ct1 = warp + 8, ct2 = warp + 16 < 18 ? warp + 16 : 0;
#pragma unroll 4
    for (int i = 0; i < kW0; i += 4) {
        const float4 d = *(const float4 *)&sd[lane][i];
        const float4 a = *(const float4 *)&sx[ct0][i], b = *(const float4 *)&sx[ct1][i], e = *(const float4 *)&sx[ct2][i];
        acc[0] += d.x * a.x; acc[1] += d.x * b.x; acc[2] += d.x * e.x;
        acc[0] += d.y * a.y; acc[1] += d.y * b.y; acc[2] += d.y * e.y;
        acc[0] += d.z * a.z; acc[1] += d.z * b.z; acc[2] += d.z * e.z;
        acc[0] += d.w * a.w; acc[1] += d.w * b.w; acc[2] += d.w * e.w;
    }
    float *row = part + (int64_t)blockIdx.x * 576;
    row[ct0 * 32 + lane] = acc[0];
    row[ct1 * 32 + lane] = acc[1];
    if (warp + 16 < 18) row[(warp + 16) * 32 + lane] = acc[2];
}

// ---- the convolutions from 32 channels on the tensor cores (implicit GEMM)
// BF16 operands in shared memory, FP32 accumulators in tensor memory, one elected thread issuing
// the MMAs.  No swizzle: core matrices of 8 rows x 8 BF16 (16 bytes), element (row, k) of an R-row
// operand in core matrix (row / 8, k / 8) at byte ((k / 8)(R / 8) + row / 8) 128, its row row % 8 at
// 16-byte steps.  A tile's im2col operand has 128 pixels as rows and k = 32 tap + channel (288):
//   conv:   D[pixel, o] = sum_k A[pixel, k] Wop[o, k], both K-major: M = 128, N = 32, K = 288
//           (18 MMAs).  The data gradient is the same product over the output gradient with
//           the taps mirrored.
//   wgrad:  D[k, o] = sum_pixel A[pixel, k] dz[pixel, o]: the same A read MN-major (channels contiguous,
//           pixels as depth), dz likewise: M = 128 at rows 0, 128 and 160 of the 288, K = 128 pixels
//           (8 MMAs each), read back and added in FP32 registers tile by tile.
// The operand is copied by the CTA's threads, 16 bytes of a neighbour pixel at a time (36 copies per
// pixel, zero-filled outside the image): with one channel plane after another it took 288 two-byte
// loads per pixel and bound both kernels.  Device times at 64x64 x 16 (65,536 pixels), before -> now: convolution
// and normalisation 26.5 + 8 -> 15.0 us, data gradient and normalisation backward 26.5 + 25 -> 18.7, weight
// gradient 95 -> 13.6 (head: 49 -> 11.9), sums of the partials 381 -> 12.  At these
// sizes neither memory (12 MB per convolution) nor the tensor cores bound them but one tile's chain of copies,
// MMAs, read-back and epilogue, twice (512 tiles on 304 resident CTAs).
constexpr int kCvM = 128, kCvK = 9 * 32;
constexpr int kCvAbytes = kCvM * kCvK * 2;     // 73,728
constexpr int kCvSlot = 32 * kCvK;             // elements of one layer's weight operand
constexpr int kWgStride = kCvK * 32;           // one CTA's partial of a weight gradient

constexpr int kCvSmem = kCvAbytes + 32 * kCvK * 2 + 32;
template <int N>
constexpr int wg_smem() { return kCvAbytes + kCvM * N * 2 + 32; }

// byte offset of element (row, k) in an operand of R rows
__host__ __device__ __forceinline__ int cv_off(int row, int k, int R) {
    return ((k >> 3) * (R >> 3) + (row >> 3)) * 128 + (row & 7) * 16 + (k & 7) * 2;
}

__device__ __forceinline__ void copy16(uint32_t dst, const void *src, bool in) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" :: "r"(dst), "l"(src), "r"(in ? 16 : 0) : "memory");
}

// A tile's im2col operand at sA (zeros outside the image and beyond the last pixel) and, where dz is given,
// its dz operand at sB.  A warp copies the 64 bytes of 8 pixels at once: 16 bytes of pixel lane % 8 by each
// lane, so that 8 lanes fill a core matrix.
__device__ __forceinline__ void gather_tile(uint32_t sA, int64_t p0, int64_t P, int H, int Wd, int dil,
                                            const __nv_bfloat16 *__restrict__ in, uint32_t sB,
                                            const __nv_bfloat16 *__restrict__ dz) {
    const int HW = H * Wd, row = (threadIdx.x >> 5) * 8 + (threadIdx.x & 7), q = (threadIdx.x >> 3) & 3;
    const int64_t pix = p0 + row;
    const bool valid = pix < P;
    const int yx = valid ? (int)(pix % HW) : 0, y = yx / Wd, x = yx % Wd;
#pragma unroll
    for (int t = 0; t < 9; ++t) {
        const int dy = (t / 3 - 1) * dil, dx = (t % 3 - 1) * dil;
        const bool ok = valid && y + dy >= 0 && y + dy < H && x + dx >= 0 && x + dx < Wd;
        copy16(sA + cv_off(row, t * 32 + q * 8, kCvM), ok ? in + (pix + dy * Wd + dx) * 32 + q * 8 : in, ok);
    }
    if (dz) copy16(sB + cv_off(row, q * 8, kCvM), valid ? dz + pix * 32 + q * 8 : dz, valid);
}

__device__ __forceinline__ void record_gave_up(int *err) {
    *(volatile int *)err = 1;
    __threadfence_system();
}

__device__ __forceinline__ void copies_visible() {   // to the MMAs (async proxy), before a barrier
    asm volatile("cp.async.wait_all;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Where parameter j of a layer goes among the convolution operands: BF16 copy and, for a layer with 32
// inputs, its places in the forward operand (Wop[o, 32 t + c] = W[o, c, t]) and the mirrored one of the
// data gradient (Wop'[c, 32 t + o] = W[o, c, 8 - t]); operand (layer l, mirrored f) at wop + (2 (l - 1) + f)
// kCvSlot.
struct WopMap { int64_t off[3]; };   // W offsets of layers 1 .. 3

__device__ __forceinline__ void place_param(int64_t j, float v, const WopMap &mp, __nv_bfloat16 *__restrict__ wb,
                                            __nv_bfloat16 *__restrict__ wop) {
    const __nv_bfloat16 b = __float2bfloat16(v);
    wb[j] = b;
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        const int64_t e = j - mp.off[l];
        if (e < 0 || e >= 32 * 288) continue;
        const int o = (int)(e / 288), c = (int)(e % 288) / 9, t = (int)(e % 9);
        wop[(int64_t)(2 * l) * kCvSlot + cv_off(o, t * 32 + c, 32) / 2] = b;
        wop[(int64_t)(2 * l + 1) * kCvSlot + cv_off(c, (8 - t) * 32 + o, 32) / 2] = b;
    }
}

__global__ void place_kernel(int64_t n, WopMap mp, const float *__restrict__ w, __nv_bfloat16 *__restrict__ wb,
                             __nv_bfloat16 *__restrict__ wop) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x)
        place_param(j, w[j], mp, wb, wop);
}

struct ConvIo {
    const float *bias, *gain;     // forward: this layer's; data gradient: gain of the block before
    float *z, *r;                 // forward: written; data gradient: the block before's, read
    __nv_bfloat16 *h;             // forward: the next layer's input; data gradient: dz in BF16 (or NULL)
    float *dz32;                  // data gradient: dz in FP32, z layout (or NULL)
    float *part;                  // data gradient: rows of kSumRow
};
enum { CV_BLOCK, CV_GRAD };

// A 3x3 convolution from 32 channels over `in` and what follows it on the same pixel.  Persistent CTAs
// of 512 threads take 128-pixel tiles gridDim.x apart; all copy the operand, thread 0 issues the 18 MMAs
// and commits them to an mbarrier, and warp w reads channels 8 (w / 4) .. + 7 of accumulator lanes
// 32 (w % 4) .. + 31 (its pixels) back.  The wait is bounded: a CTA in which it gives up records that in
// *err, waits once more for its MMAs and stops.
template <int MODE>
__global__ void __launch_bounds__(kThr, 2)
conv_tc_kernel(int B, int H, int Wd, int dil, const __nv_bfloat16 *__restrict__ in,
               const __nv_bfloat16 *__restrict__ wop, ConvIo io, int *__restrict__ err) {
    constexpr int N = 32, Bbytes = N * kCvK * 2;
    constexpr uint32_t idesc = tc_idesc(kCvM, N);
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ float sh[16][16], sdot[4][kPix], sg[32], sbias[32];
    unsigned char *sB = smem + kCvAbytes;
    uint64_t *mb = (uint64_t *)(sB + Bbytes);
    uint32_t *tslot = (uint32_t *)(mb + 1);
    const int HW = H * Wd;
    const int64_t P = (int64_t)B * HW, ntiles = (P + kCvM - 1) / kCvM;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, row = threadIdx.x & (kPix - 1), q = threadIdx.x / kPix;
    const uint32_t a0 = tc_smem_u32(smem), b0 = tc_smem_u32(sB), mbar = tc_smem_u32(mb);
    pdl_start();
    if (warp == 0) tc_alloc(tslot, 32);
    if (threadIdx.x == 0) {
        tc_mbar_init(mbar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    pdl_wait();
    gather_tile(a0, (int64_t)blockIdx.x * kCvM, P, H, Wd, dil, in, 0, nullptr);
    for (int e = threadIdx.x; e < Bbytes / 16; e += kThr) copy16(b0 + 16 * e, (const uint4 *)wop + e, true);
    if (threadIdx.x < 32) {
        if (MODE != CV_GRAD) sbias[threadIdx.x] = io.bias[threadIdx.x];
        sg[threadIdx.x] = io.gain[threadIdx.x];
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot, trow = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    GradSums sums;
    int it = 0;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++it) {
        const int64_t pix = tile * kCvM + row;
        const bool valid = pix < P;
        if (it > 0) gather_tile(a0, tile * kCvM, P, H, Wd, dil, in, 0, nullptr);
        copies_visible();
        tc_fence_before();
        __syncthreads();
        if (threadIdx.x == 0) {
            tc_fence_after();
            const uint32_t lboA = (kCvM / 8) * 128, lboB = (N / 8) * 128;
#pragma unroll
            for (int ks = 0; ks < kCvK / 16; ++ks)
                tc_mma(tmem, tc_desc(a0 + ks * 2 * lboA, lboA), tc_desc(b0 + ks * 2 * lboB, lboB), idesc, ks > 0);
            tc_commit(mbar);
        }
        const bool done = tc_wait(mbar, (uint32_t)(it & 1));
        if (__syncthreads_or(!done)) {
            if (threadIdx.x == 0) {
                record_gave_up(err);
                tc_wait(mbar, (uint32_t)(it & 1));   // its MMAs read this CTA's shared memory
            }
            break;
        }
        tc_fence_after();
        if constexpr (MODE == CV_BLOCK) {
            float z[8], ss = 0.f;
            {
                float v[32];
                tc_ld32(trow, v);
#pragma unroll
                for (int c = 0; c < 32; ++c) {
                    const float t = sbias[c] + v[c];
                    ss += t * t;
                }
            }
            tc_ld8(trow + 8 * q, z);
#pragma unroll
            for (int c = 0; c < 8; ++c) z[c] = sbias[8 * q + c] + z[c];
            if (valid) norm_fwd8(pix, q, ss, z, sg, io.z, io.r, io.h);
        } else {
            float v[8], dgl[8];
            tc_ld8(trow + 8 * q, v);
            if (!valid) {
#pragma unroll
                for (int c = 0; c < 8; ++c) v[c] = 0.f;
            }
            norm_bwd8(valid, pix, row, q, v, io.z, io.r, sg, dgl, sdot);
            if (valid) {
                if (io.h) st_bf16x8(io.h + pix * 32 + 8 * q, v);
                if (io.dz32) st_z8(io.dz32, pix, q, v);
            }
            sums.add(dgl, v, lane);
        }
        tc_fence_before();
    }
    if constexpr (MODE == CV_GRAD) sums.store(sh, io.part + (int64_t)blockIdx.x * kSumRow, lane, warp);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tc_dealloc(tmem, 32);
}

// Partial weight gradients of a convolution from 32 channels over this CTA's 128-pixel tiles:
// part[cta kWgStride + k N' + o] = sum_pixel in[pixel + offset_t, c] dz[pixel, o], k = 32 t + c, N' = 32.
// HEAD: dz is the head's output gradient, NCHW FP32 with 2 channels, as three BF16 pieces each (their sum
// is the FP32 value), N = 16 columns of which 6 are used and added: N' = 2; relative L2 error of the head's
// weight gradient against FP64 from the same inputs, 64x64 x 16: 3.7e-7 with FP32 FMAs and a
// tree, 1.7e-7 so.  Same waits and clean-up as
// conv_tc_kernel.
template <bool HEAD>
__global__ void __launch_bounds__(kThr, 2)
conv_wgrad_tc_kernel(int B, int H, int Wd, int dil, const __nv_bfloat16 *__restrict__ in,
                     const __nv_bfloat16 *__restrict__ dz, const float *__restrict__ dy, float *__restrict__ part,
                     int *__restrict__ err) {
    constexpr int N = HEAD ? 16 : 32, Bbytes = kCvM * N * 2;
    // both operands MN-major (bits 15 and 16)
    constexpr uint32_t idesc = tc_idesc(kCvM, N) | (1u << 15) | (1u << 16);
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char *sB = smem + kCvAbytes;
    uint64_t *mb = (uint64_t *)(sB + Bbytes);
    uint32_t *tslot = (uint32_t *)(mb + 1);
    const int HW = H * Wd;
    const int64_t P = (int64_t)B * HW, ntiles = (P + kCvM - 1) / kCvM;
    const int warp = threadIdx.x >> 5, row = threadIdx.x & (kPix - 1), q = threadIdx.x / kPix;
    const uint32_t a0 = tc_smem_u32(smem), b0 = tc_smem_u32(sB), mbar = tc_smem_u32(mb);
    pdl_start();
    if (warp == 0) tc_alloc(tslot, 128);
    if (threadIdx.x == 0) {
        tc_mbar_init(mbar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    pdl_wait();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot, trow = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    float acc[3][HEAD ? 2 : 8] = {};   // this thread's row of each third, its columns, summed over the tiles
    int it = 0;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++it) {
        gather_tile(a0, tile * kCvM, P, H, Wd, dil, in, b0, HEAD ? nullptr : dz);
        if (HEAD && q == 0) {
            const int64_t pix = tile * kCvM + row;
            uint32_t w[4] = {0u, 0u, 0u, 0u};   // columns 3 o + piece
            if (pix < P) {
                unsigned short e[6];
#pragma unroll
                for (int o = 0; o < 2; ++o) {
                    float v = dy[((pix / HW) * 2 + o) * HW + pix % HW];
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        const __nv_bfloat16 b = __float2bfloat16(v);
                        e[3 * o + k] = __bfloat16_as_ushort(b);
                        v = isfinite(v) ? v - __bfloat162float(b) : 0.f;
                    }
                }
                w[0] = e[0] | ((uint32_t)e[1] << 16);
                w[1] = e[2] | ((uint32_t)e[3] << 16);
                w[2] = e[4] | ((uint32_t)e[5] << 16);
            }
            *(uint4 *)(sB + cv_off(row, 0, kCvM)) = make_uint4(w[0], w[1], w[2], w[3]);
            *(uint4 *)(sB + cv_off(row, 8, kCvM)) = make_uint4(0u, 0u, 0u, 0u);
        }
        copies_visible();
        tc_fence_before();
        __syncthreads();
        if (threadIdx.x == 0) {
            tc_fence_after();
            // depth (pixels): core matrices 128 bytes apart; channels: (128 / 8) 128
            const uint32_t sbo = (kCvM / 8) * 128;
#pragma unroll
            for (int mt = 0; mt < 3; ++mt) {
                const uint32_t am = a0 + (mt == 0 ? 0 : mt == 1 ? 16 : 20) * sbo;
#pragma unroll
                for (int ks = 0; ks < kCvM / 16; ++ks)
                    tc_mma(tmem + (uint32_t)(mt * 32), tc_desc2(am + ks * 256, 128, sbo),
                                 tc_desc2(b0 + ks * 256, 128, sbo), idesc, ks > 0);
            }
            tc_commit(mbar);
        }
        const bool done = tc_wait(mbar, (uint32_t)(it & 1));
        if (__syncthreads_or(!done)) {
            if (threadIdx.x == 0) {
                record_gave_up(err);
                tc_wait(mbar, (uint32_t)(it & 1));
            }
            break;
        }
        tc_fence_after();
        if (!HEAD || q == 0) {
#pragma unroll
            for (int mt = 0; mt < 3; ++mt) {
                if (mt == 2 && (warp & 3) < 3) break;   // rows 160 .. 255 are in the first two
                float v[8];
                tc_ld8(trow + mt * 32 + 8 * q, v);
                if constexpr (HEAD) {
                    acc[mt][0] += (v[2] + v[1]) + v[0];
                    acc[mt][1] += (v[5] + v[4]) + v[3];
                } else {
#pragma unroll
                    for (int o = 0; o < 8; ++o) acc[mt][o] += v[o];
                }
            }
        }
        tc_fence_before();
    }
    float *prow = part + (int64_t)blockIdx.x * kWgStride;
    if (!HEAD || q == 0) {
#pragma unroll
        for (int mt = 0; mt < 3; ++mt) {
            if (mt == 2 && (warp & 3) < 3) break;
            const int k = (mt == 2 ? 160 : mt * 128) + row;
            if constexpr (HEAD) {
                *(float2 *)(prow + k * 2) = make_float2(acc[mt][0], acc[mt][1]);
            } else {
                *(float4 *)(prow + k * 32 + 8 * q) = make_float4(acc[mt][0], acc[mt][1], acc[mt][2], acc[mt][3]);
                *(float4 *)(prow + k * 32 + 8 * q + 4) = make_float4(acc[mt][4], acc[mt][5], acc[mt][6], acc[mt][7]);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tc_dealloc(tmem, 128);
}

// Sums of the per-CTA partials into the gradient, all layers in one launch (nine launches of one thread per
// column before).  Segment: `count` columns of
// `rows` partial rows; column j goes to grad[dst + ...] by kind.  A CTA takes 32 columns of one segment,
// its 8 warps every eighth row each, added in a fixed order.
enum { SEG_PLAIN, SEG_W32, SEG_HEAD, SEG_W0 };
struct Segment { const float *src; int rows, stride, count, kind; int64_t dst; int first; };
constexpr int kMaxSeg = 16;
struct Segments { Segment s[kMaxSeg]; int n; };

__global__ void __launch_bounds__(256)
grad_reduce_kernel(Segments S, float *__restrict__ grad) {
    __shared__ float sh[8][32];
    int k = 0;
    while (k + 1 < S.n && (int)blockIdx.x >= S.s[k + 1].first) ++k;
    const Segment g = S.s[k];
    pdl_wait();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, j = ((int)blockIdx.x - g.first) * 32 + lane;
    float a = 0.f;
    if (j < g.count) {
#pragma unroll 8
        for (int q = warp; q < g.rows; q += 8) a += g.src[(int64_t)q * g.stride + j];
    }
    sh[warp][lane] = a;
    __syncthreads();
    if (warp == 0 && j < g.count) {
        a = sh[0][lane];
#pragma unroll
        for (int w = 1; w < 8; ++w) a += sh[w][lane];
        int64_t at = g.dst + j;
        if (g.kind == SEG_W32) {          // j = (32 t + c) 32 + o
            const int o = j & 31, c = (j >> 5) & 31, t = j >> 10;
            at = g.dst + (o * 32 + c) * 9 + t;
        } else if (g.kind == SEG_HEAD) {  // j = (32 t + c) 2 + o
            const int o = j & 1, c = (j >> 1) & 31, t = j >> 6;
            at = g.dst + (o * 32 + c) * 9 + t;
        } else if (g.kind == SEG_W0) {    // j = (9 c + t) 32 + o
            at = g.dst + (j & 31) * 18 + (j >> 5);
        }
        grad[at] = a;
    }
}

// gauge-invariant loss per image: t = mean((yu-u)-(yv-v))/2, r = residuals, dy = r / (B npix), lpart[b] =
// sum r^2.  The sums are FP64, whose pipe takes 64 clocks per warp instruction: a cluster of eight CTAs
// per image spreads them over eight SMs (64x64 x 16: 17 -> 11.8 us).
constexpr int kLossCl = 8, kLossThr = 256;

__device__ __forceinline__ void cluster_barrier() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// sum over the cluster of every thread's v, the same in all (sh: this CTA's kLossThr / 32 + kLossCl doubles)
__device__ __forceinline__ double cluster_sum(double v, double *sh, int rank) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double *all = sh + kLossThr / 32;
    for (int k = 16; k > 0; k >>= 1) v += __shfl_xor_sync(0xffffffffu, v, k);
    if (lane == 0) sh[warp] = v;
    __syncthreads();
    if (threadIdx.x < kLossCl) {
        v = 0.0;
        for (int w = 0; w < kLossThr / 32; ++w) v += sh[w];
        uint32_t dst;   // CTA threadIdx.x's all[rank]
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                     : "=r"(dst) : "r"((uint32_t)__cvta_generic_to_shared(all + rank)), "r"(threadIdx.x));
        asm volatile("st.shared::cluster.f64 [%0], %1;" :: "r"(dst), "d"(v) : "memory");
    }
    cluster_barrier();
    v = 0.0;
    for (int c = 0; c < kLossCl; ++c) v += all[c];
    return v;
}

__global__ void __cluster_dims__(kLossCl, 1, 1) __launch_bounds__(kLossThr)
loss_kernel(int B, int64_t HW, const float *__restrict__ y, const float *__restrict__ tgt,
            float *__restrict__ dy, float *__restrict__ lpart) {
    __shared__ double sh[2][kLossThr / 32 + kLossCl];
    const int b = blockIdx.x / kLossCl, rank = blockIdx.x % kLossCl;
    const float *yu = y + (int64_t)b * 2 * HW, *yv = yu + HW;
    const float *tu = tgt + (int64_t)b * 2 * HW, *tv = tu + HW;
    const int64_t q0 = rank * kLossThr + threadIdx.x, step = kLossCl * kLossThr;
    cluster_barrier();   // all CTAs have started: their shared memory may be written
    double s = 0.0;
    for (int64_t q = q0; q < HW; q += step) s += (double)(yu[q] - tu[q]) - (double)(yv[q] - tv[q]);
    const float t = (float)(cluster_sum(s, sh[0], rank) / (2.0 * (double)HW));
    double l = 0.0;
    const float inv = 1.f / (float)((double)B * (double)HW);
    float *du = dy + (int64_t)b * 2 * HW, *dv = du + HW;
    for (int64_t q = q0; q < HW; q += step) {
        const float ru = (yu[q] - tu[q]) - t, rv = (yv[q] - tv[q]) + t;
        du[q] = ru * inv;
        dv[q] = rv * inv;
        l += (double)ru * ru + (double)rv * rv;
    }
    l = cluster_sum(l, sh[1], rank);
    if (rank == 0 && threadIdx.x == 0) lpart[b] = (float)l;
}

__global__ void adam_kernel(int64_t n, WopMap mp, const float *__restrict__ grad, float *__restrict__ w,
                            float *__restrict__ m, float *__restrict__ v, __nv_bfloat16 *__restrict__ wb,
                            __nv_bfloat16 *__restrict__ wop, float lr, float b1, float b2, float eps, float c1,
                            float c2) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
        const float g = grad[j];
        const float mj = b1 * m[j] + (1.f - b1) * g;
        const float vj = b2 * v[j] + (1.f - b2) * g * g;
        m[j] = mj;
        v[j] = vj;
        const float wj = w[j] - lr * (mj / c1) / (sqrtf(vj / c2) + eps);
        w[j] = wj;
        place_param(j, wj, mp, wb, wop);
    }
}

inline unsigned blocks_for(int64_t n, int t) { return (unsigned)std::max<int64_t>(1, (n + t - 1) / t); }

}  // namespace
}  // namespace ot

using namespace ot;

struct ot_cnn {
    int ch = 32;
    Layer L[kLayers];
    int64_t nparam = 0;
    cudaStream_t st = nullptr;
    float *w = nullptr, *m = nullptr, *v = nullptr;   // FP32 master weights and Adam moments
    __nv_bfloat16 *wb = nullptr;                      // BF16 copy
    __nv_bfloat16 *wop = nullptr;   // tensor-core weight operands of layers 1-3 (forward, mirrored)
    // pinned host memory that the kernels write, read after a synchronisation (a copy into pageable memory
    // took longer than a small image's kernels): flag of a tensor-core wait that gave up, loss per image
    int *derr = nullptr;
    float *lpart = nullptr;
    int sms = 1;
    // activations of the last forward (B, k); buffers for whole tiles of 128 pixels
    int B = 0, k = 0;
    int64_t cap_pix = 0, cap_grad = 0;   // pixels that the two allocations are for
    unsigned char *acts = nullptr, *grads = nullptr;
    __nv_bfloat16 *h[kLayers] = {};   // conv inputs: h[0] = the features (NCHW), else 32 per pixel
    float *z[kLayers] = {};           // conv outputs (z[4] = prediction, NCHW; else the z layout)
    float *r[kLayers] = {};           // RMS of the normalised blocks
    __nv_bfloat16 *gb[2] = {};        // BF16 gradients of two blocks in turn
    float *g0 = nullptr;              // FP32 gradient of the first block's output (z layout)
    float *part = nullptr;            // per-CTA partials of the gradients
    std::string err;
};

namespace {

thread_local std::string g_cnn_err;

int cnn_fail(ot_cnn *c, int code, const std::string &msg) {
    if (c) c->err = msg;
    g_cnn_err = msg;
    return code;
}

void layout(ot_cnn *c) {
    int64_t off = 0;
    int cin = 2;
    for (int l = 0; l < kLayers; ++l) {
        Layer &y = c->L[l];
        y.cin = cin;
        y.cout = l < kLayers - 1 ? c->ch : 2;
        y.dil = kDil[l];
        y.norm = l < kLayers - 1;
        y.W = off;
        off += (int64_t)y.cout * y.cin * 9;
        y.b = off;
        off += y.cout;
        y.g = -1;
        if (y.norm) {
            y.g = off;
            off += y.cout;
        }
        cin = y.cout;
    }
    c->nparam = off;
}

// the activations and everything that says there are some: no forward to take a loss or a gradient of
void free_acts(ot_cnn *c) {
    if (c->acts) cudaFree(c->acts);
    c->acts = nullptr;
    c->cap_pix = 0;
    c->B = c->k = 0;
    for (int l = 0; l < kLayers; ++l) {
        c->h[l] = nullptr;
        c->z[l] = nullptr;
        c->r[l] = nullptr;
    }
}

// cudaMalloc whose failure is reported here and not by the next launch's check too
bool dev_malloc(void **p, int64_t bytes) {
    if (cudaMalloc(p, (size_t)bytes) == cudaSuccess) return true;
    *p = nullptr;
    cudaGetLastError();
    return false;
}

// CTAs of the tensor-core kernels and of the head's backward: two per SM at most
int64_t tc_ctas(const ot_cnn *c, int64_t pix) { return std::min<int64_t>((pix + kCvM - 1) / kCvM, 2LL * c->sms); }

// activations of a forward pass, one allocation (each buffer whole tiles of 128 pixels)
int ensure_acts(ot_cnn *c, int B, int k) {
    const int64_t pix = (int64_t)B * k * k;
    if (pix > c->cap_pix) {
        free_acts(c);
        const int64_t tp = (pix + kCvM - 1) / kCvM * kCvM;
        int64_t per = 0;   // bytes per pixel
        for (int l = 0; l < kLayers; ++l) per += 2 * c->L[l].cin + 4 * c->L[l].cout + 4;
        if (!dev_malloc((void **)&c->acts, per * tp))
            return cnn_fail(c, OT_ERR_OOM, "ot_cnn: activation allocation failed");
        unsigned char *p = c->acts;
        for (int l = 0; l < kLayers; ++l) {
            c->h[l] = (__nv_bfloat16 *)p;
            p += 2 * c->L[l].cin * tp;
            c->z[l] = (float *)p;
            p += 4 * c->L[l].cout * tp;
            c->r[l] = (float *)p;
            p += 4 * tp;
        }
        c->cap_pix = pix;
    }
    c->B = B;
    c->k = k;
    return OT_OK;
}

// of a backward pass: FP32 and BF16 gradients, sum rows of four blocks, weight-gradient partials of layers
// 1 .. 4 and of the first
int ensure_grads(ot_cnn *c) {
    const int64_t pix = (int64_t)c->B * c->k * c->k;
    if (pix > c->cap_grad) {
        if (c->grads) cudaFree(c->grads);
        c->grads = nullptr;
        c->cap_grad = 0;
        const int64_t tp = (pix + kCvM - 1) / kCvM * kCvM, ctas = tc_ctas(c, pix);
        const int64_t parts = 4 * ctas * (kSumRow + kWgStride) + (pix + kW0 - 1) / kW0 * 576;
        if (!dev_malloc((void **)&c->grads, 4 * parts + tp * c->ch * (4 + 2 + 2)))
            return cnn_fail(c, OT_ERR_OOM, "ot_cnn: gradient allocation failed");
        c->g0 = (float *)c->grads;
        c->gb[0] = (__nv_bfloat16 *)(c->g0 + tp * c->ch);
        c->gb[1] = c->gb[0] + tp * c->ch;
        c->part = (float *)(c->gb[1] + tp * c->ch);
        c->cap_grad = pix;
    }
    return OT_OK;
}

WopMap wop_map(const ot_cnn *c) {
    WopMap m;
    for (int l = 0; l < 3; ++l) m.off[l] = c->L[l + 1].W;
    return m;
}

// BF16 copies and convolution operands of all parameters
int place_params(ot_cnn *c) {
    place_kernel<<<blocks_for(c->nparam, 256), 256, 0, c->st>>>(c->nparam, wop_map(c), c->w, c->wb, c->wop);
    if (cudaGetLastError() != cudaSuccess) return cnn_fail(c, OT_ERR_CUDA, "ot_cnn: launch failed");
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return OT_OK;
}

// weight operand of layer l = 1 .. 3, forward or mirrored
const __nv_bfloat16 *wop_of(const ot_cnn *c, int l, int mirrored) {
    return c->wop + (int64_t)(2 * (l - 1) + mirrored) * kCvSlot;
}

// a tensor-core kernel's wait that gave up (bounded waits; the flag is read after a synchronisation)
int check_tc(ot_cnn *c, const char *where) {
    if (cudaStreamSynchronize(c->st) != cudaSuccess)
        return cnn_fail(c, OT_ERR_CUDA, std::string(where) + ": synchronisation failed");
    if (*(volatile int *)c->derr) return cnn_fail(c, OT_ERR_TIMEOUT, std::string(where) + ": a tensor-core wait gave up");
    return OT_OK;
}

// launch with programmatic dependence on the kernel ahead (which has pdl_start, this one pdl_wait)
template <class... P, class... A>
void launch_pdl(void (*f)(P...), unsigned grid, int threads, int smem, cudaStream_t st, A... args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, f, P(args)...);
}

#define CNN_LAUNCHED(c)                                                                   \
    do {                                                                                  \
        cudaError_t e_ = cudaGetLastError();                                              \
        if (e_ != cudaSuccess) return cnn_fail(c, OT_ERR_CUDA, cudaGetErrorString(e_));   \
        g_launches.fetch_add(1, std::memory_order_relaxed);                               \
    } while (0)

}  // namespace

extern "C" {

int64_t ot_cnn_param_count(int32_t channels) {
    if (channels != 32) return -1;
    ot_cnn c;
    c.ch = channels;
    layout(&c);
    return c.nparam;
}

int ot_cnn_create(int32_t channels, const float *params, void *stream, ot_cnn_t **out) {
    if (!out) return cnn_fail(nullptr, OT_ERR_ARG, "ot_cnn_create: out is NULL");
    *out = nullptr;
    if (channels != 32) return cnn_fail(nullptr, OT_ERR_UNSUPPORTED, "ot_cnn_create: only 32 channels are built");
    if (!params) return cnn_fail(nullptr, OT_ERR_ARG, "ot_cnn_create: params is NULL");
    ot_cnn *c = new (std::nothrow) ot_cnn();
    if (!c) return cnn_fail(nullptr, OT_ERR_OOM, "ot_cnn_create: host allocation failed");
    c->ch = channels;
    layout(c);
    c->st = (cudaStream_t)stream;
    const size_t nb = sizeof(float) * c->nparam;
    if (cudaMalloc((void **)&c->w, nb) != cudaSuccess || cudaMalloc((void **)&c->m, nb) != cudaSuccess ||
        cudaMalloc((void **)&c->v, nb) != cudaSuccess ||
        cudaMalloc((void **)&c->wb, sizeof(__nv_bfloat16) * c->nparam) != cudaSuccess ||
        cudaMalloc((void **)&c->wop, sizeof(__nv_bfloat16) * 6 * kCvSlot) != cudaSuccess ||
        cudaHostAlloc((void **)&c->derr, 64 + sizeof(float) * kMaxBatch, cudaHostAllocDefault) != cudaSuccess) {
        ot_cnn_destroy(c);
        return cnn_fail(nullptr, OT_ERR_OOM, "ot_cnn_create: weight allocation failed");
    }
    cudaMemcpyAsync(c->w, params, nb, cudaMemcpyHostToDevice, c->st);
    cudaMemsetAsync(c->m, 0, nb, c->st);
    cudaMemsetAsync(c->v, 0, nb, c->st);
    *c->derr = 0;
    c->lpart = (float *)((unsigned char *)c->derr + 64);
    {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaFuncSetAttribute(conv_tc_kernel<CV_BLOCK>, cudaFuncAttributeMaxDynamicSharedMemorySize, kCvSmem) != cudaSuccess ||
            cudaFuncSetAttribute(conv_tc_kernel<CV_GRAD>, cudaFuncAttributeMaxDynamicSharedMemorySize, kCvSmem) != cudaSuccess ||
            cudaFuncSetAttribute(conv_wgrad_tc_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, wg_smem<32>()) != cudaSuccess ||
            cudaFuncSetAttribute(conv_wgrad_tc_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, wg_smem<16>()) != cudaSuccess) {
            ot_cnn_destroy(c);
            return cnn_fail(nullptr, OT_ERR_CUDA, "ot_cnn_create: device query failed");
        }
    }
    int rc = place_params(c);
    if (rc == OT_OK && cudaStreamSynchronize(c->st) != cudaSuccess) rc = cnn_fail(c, OT_ERR_CUDA, "ot_cnn_create: copy failed");
    if (rc != OT_OK) {
        ot_cnn_destroy(c);
        return rc;
    }
    *out = c;
    return OT_OK;
}

int ot_cnn_get_params(ot_cnn_t *c, float *params, int64_t cap) {
    if (!c || !params) return cnn_fail(c, OT_ERR_ARG, "ot_cnn_get_params: NULL argument");
    if (cap < c->nparam) return cnn_fail(c, OT_ERR_BUF_TOO_SMALL, "ot_cnn_get_params: buffer too small");
    if (cudaMemcpyAsync(params, c->w, sizeof(float) * c->nparam, cudaMemcpyDeviceToHost, c->st) != cudaSuccess ||
        cudaStreamSynchronize(c->st) != cudaSuccess)
        return cnn_fail(c, OT_ERR_CUDA, "ot_cnn_get_params: copy failed");
    return OT_OK;
}

int ot_cnn_forward(ot_cnn_t *c, int32_t batch, int32_t k, const float *x, float *y) {
    if (!c || !x || batch <= 0 || k <= 0 || batch > kMaxBatch) return cnn_fail(c, OT_ERR_ARG, "ot_cnn_forward: bad argument");
    int rc = ensure_acts(c, batch, k);
    if (rc != OT_OK) return rc;
    const int64_t pix = (int64_t)batch * k * k;
    cudaStream_t st = c->st;
    const unsigned grid = (unsigned)tc_ctas(c, pix);
    block0_kernel<<<blocks_for(pix, kPix), kThr, 0, st>>>(batch, k, k, c->L[0].dil, x, c->wb + c->L[0].W, c->w + c->L[0].b,
                                                          c->w + c->L[0].g, c->h[0], c->z[0], c->r[0], c->h[1]);
    CNN_LAUNCHED(c);
    for (int l = 1; l < kLayers; ++l) {
        const Layer &Ly = c->L[l];
        if (Ly.norm) {
            ConvIo io{};
            io.bias = c->w + Ly.b;
            io.gain = c->w + Ly.g;
            io.z = c->z[l];
            io.r = c->r[l];
            io.h = c->h[l + 1];
            launch_pdl(conv_tc_kernel<CV_BLOCK>, grid, kThr, kCvSmem, st, batch, k, k, Ly.dil, c->h[l], wop_of(c, l, 0), io,
                       c->derr);
        } else {
            launch_pdl(head_kernel, blocks_for(pix, kHdThr), kHdThr, 0, st, batch, k, k, Ly.dil, c->h[l], c->wb + Ly.W,
                       c->w + Ly.b, c->z[l], y);
        }
        CNN_LAUNCHED(c);
    }
    return check_tc(c, "ot_cnn_forward");
}

int ot_cnn_loss(ot_cnn_t *c, const float *target, float *dy, float *loss) {
    if (!c || !target || !dy || !loss || c->B <= 0) return cnn_fail(c, OT_ERR_ARG, "ot_cnn_loss: bad argument");
    const int64_t HW = (int64_t)c->k * c->k;
    loss_kernel<<<c->B * kLossCl, kLossThr, 0, c->st>>>(c->B, HW, c->z[kLayers - 1], target, dy, c->lpart);
    CNN_LAUNCHED(c);
    if (cudaStreamSynchronize(c->st) != cudaSuccess) return cnn_fail(c, OT_ERR_CUDA, "ot_cnn_loss: synchronisation failed");
    double s = 0.0;
    for (int b = 0; b < c->B; ++b) s += ((volatile float *)c->lpart)[b];
    *loss = (float)(s / (2.0 * (double)c->B * (double)HW));
    return OT_OK;
}

int ot_cnn_backward(ot_cnn_t *c, const float *dy, float *grad, float *dx) {
    if (!c || !dy || !grad || c->B <= 0) return cnn_fail(c, OT_ERR_ARG, "ot_cnn_backward: bad argument");
    int rc = ensure_grads(c);
    if (rc != OT_OK) return rc;
    const int B = c->B, k = c->k;
    const int64_t pix = (int64_t)B * k * k, ctas = tc_ctas(c, pix), n0 = (pix + kW0 - 1) / kW0;
    cudaStream_t st = c->st;
    const unsigned grid = (unsigned)ctas;
    // partials: sum rows of blocks 0 .. 3, weight gradients of layers 1 .. 4, the first layer's
    float *sums = c->part, *wpart = sums + 4 * ctas * kSumRow, *w0part = wpart + 4 * ctas * kWgStride;
    Segments S{};
    int first = 0;
    auto segment = [&](const float *src, int64_t rows, int stride, int count, int kind, int64_t dst) {
        S.s[S.n++] = Segment{src, (int)rows, stride, count, kind, dst, first};
        first += (count + 31) / 32;
    };
    const Layer &head = c->L[kLayers - 1];
    // the head and the last block's normalisation, then layers 3 .. 1: weight gradient, and data
    // gradient with the normalisation of the block before
    head_bwd_kernel<<<grid, kThr, 0, st>>>(B, k, k, dy, c->wb + head.W, c->w + c->L[3].g, c->z[3], c->r[3], c->gb[1],
                                           sums + 3 * ctas * kSumRow);
    CNN_LAUNCHED(c);
    launch_pdl(conv_wgrad_tc_kernel<true>, grid, kThr, wg_smem<16>(), st, B, k, k, head.dil, c->h[4], nullptr, dy,
               wpart + 3 * ctas * kWgStride, c->derr);
    CNN_LAUNCHED(c);
    segment(wpart + 3 * ctas * kWgStride, ctas, kWgStride, 576, SEG_HEAD, head.W);
    segment(sums + 3 * ctas * kSumRow + 64, ctas, kSumRow, 2, SEG_PLAIN, head.b);
    for (int l = kLayers - 2; l >= 0; --l) {
        const Layer &Ly = c->L[l];
        segment(sums + l * ctas * kSumRow, ctas, kSumRow, 32, SEG_PLAIN, Ly.g);
        segment(sums + l * ctas * kSumRow + 32, ctas, kSumRow, 32, SEG_PLAIN, Ly.b);
        if (l == 0) break;
        const __nv_bfloat16 *dz = c->gb[l & 1];
        float *wp = wpart + (l - 1) * ctas * kWgStride;
        launch_pdl(conv_wgrad_tc_kernel<false>, grid, kThr, wg_smem<32>(), st, B, k, k, Ly.dil, c->h[l], dz, nullptr, wp,
                   c->derr);
        CNN_LAUNCHED(c);
        segment(wp, ctas, kWgStride, kWgStride, SEG_W32, Ly.W);
        ConvIo io{};
        io.gain = c->w + c->L[l - 1].g;
        io.z = c->z[l - 1];
        io.r = c->r[l - 1];
        io.h = l > 1 ? c->gb[(l - 1) & 1] : nullptr;
        io.dz32 = l > 1 ? nullptr : c->g0;
        io.part = sums + (l - 1) * ctas * kSumRow;
        launch_pdl(conv_tc_kernel<CV_GRAD>, grid, kThr, kCvSmem, st, B, k, k, Ly.dil, dz, wop_of(c, l, 1), io, c->derr);
        CNN_LAUNCHED(c);
    }
    launch_pdl(block0_wgrad_kernel, (unsigned)n0, 256, 0, st, B, k, k, c->L[0].dil, c->h[0], c->g0, w0part);
    CNN_LAUNCHED(c);
    segment(w0part, n0, 576, 576, SEG_W0, c->L[0].W);
    if (dx) {
        block0_bwd_data_kernel<<<blocks_for(pix, kPix), kPix, 0, st>>>(B, k, k, c->L[0].dil, c->g0, c->wb + c->L[0].W, dx);
        CNN_LAUNCHED(c);
    }
    launch_pdl(grad_reduce_kernel, (unsigned)first, 256, 0, st, S, grad);
    CNN_LAUNCHED(c);
    return check_tc(c, "ot_cnn_backward");
}

int ot_cnn_adam(ot_cnn_t *c, const float *grad, float lr, float beta1, float beta2, float eps, int32_t step) {
    if (!c || !grad || step < 1) return cnn_fail(c, OT_ERR_ARG, "ot_cnn_adam: bad argument");
    const float c1 = 1.f - std::pow(beta1, (float)step), c2 = 1.f - std::pow(beta2, (float)step);
    adam_kernel<<<blocks_for(c->nparam, 256), 256, 0, c->st>>>(c->nparam, wop_map(c), grad, c->w, c->m, c->v, c->wb,
                                                               c->wop, lr, beta1, beta2, eps, c1, c2);
    CNN_LAUNCHED(c);
    return OT_OK;
}

const char *ot_cnn_last_error(const ot_cnn_t *c) { return c ? c->err.c_str() : g_cnn_err.c_str(); }

void ot_cnn_destroy(ot_cnn_t *c) {
    if (!c) return;
    free_acts(c);
    for (void *p : {(void *)c->w, (void *)c->m, (void *)c->v, (void *)c->wb, (void *)c->wop, (void *)c->grads})
        if (p) cudaFree(p);
    if (c->derr) cudaFreeHost(c->derr);
    delete c;
}

}  // extern "C"
