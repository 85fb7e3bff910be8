// Small convolutional network for the learned warm start of the solver.
//
// Four 3x3 convolution layers (zero padding): C_in -> 32 -> 32 -> 32 -> C_out,
// ReLU after the first three.  Weights are kept as FP32 master copies for the
// optimiser and used as BF16 in every product; all sums accumulate in FP32.
// Activations are FP32, layout [N][C][H][W].
//
// Kernels: direct convolution in FP32 for the forward pass and the input
// gradient (the same convolution with transposed, flipped weights and the ReLU
// of the layer below applied to its result), the weight / bias gradients
// (partial sums per block in registers, then one reduction), a mean-squared-
// error loss with its gradient, and Adam.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <cstdint>
#include <string>
#include <vector>

#include "../../include/mf.h"
#include "mf_internal.cuh"

namespace mf {

// two FP32 fused multiply-adds in one instruction (each rounded as fmaf)
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ void unpack2(uint64_t v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
// global -> shared copy of one float; zero where !in
__device__ __forceinline__ void copy_f32(float *dst, const float *src, bool in) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(in ? 4 : 0) : "memory");
}

// Direct 3x3 convolution.  A thread computes PX pixels of a row times CO output
// channels, channels in pairs (one two-wide FMA per pair, pixel and tap), so
// that a weight read from shared memory (a broadcast) serves PX pixels and an
// input CO channels.  A warp covers 32 columns and PX rows; the block's warps
// are CG channel groups times NWARP / CG row groups.  The input tile comes in
// chunks of CK channels, the next one copied asynchronously under the
// arithmetic; the weights stay in shared memory as FP32 [ci][tap][co].
// Per output: the bias, then fmaf over ci and tap in ascending order.
//   TRANS: the input gradient: weight of (out o, in i, tap k) = w[i][o][8 - k].
//   MASK:  zero where act <= 0 (the ReLU of the layer whose output gradient
//          this is).
// Bound by FP32 FMAs.  A thread per pixel with all 32 channels and a scalar
// weight read per FMA took 573 us for 32 -> 32 channels on 8 x 256 x 256 pixels
// (17 TFLOP/s), this 210 us (46 TFLOP/s; the FMA pipe is 70% busy).
template <int CIN, int COUT>
struct ConvCfg {
    static constexpr int CG = COUT == 32 ? 2 : 1;         // channel groups
    static constexpr int CO = COUT / CG;                  // channels per thread
    static constexpr int PX = COUT == 32 ? 4 : 8;         // pixels per thread
    static constexpr int NWARP = COUT == 32 ? 8 : 4;
    static constexpr int TH = PX * (NWARP / CG);          // tile height (width 32)
    static constexpr int CK = CIN == 32 ? 8 : CIN == 10 ? 5 : CIN;  // input channels per chunk
    static constexpr int NC = CIN / CK;
    static constexpr int XS = 36;                         // row stride of the staged tile
    static constexpr int WS = COUT == 10 ? 12 : COUT == 6 ? 8 : COUT;  // channel stride of the weights
    static constexpr size_t chunk = (size_t)CK * (TH + 2) * XS;
    static constexpr size_t smem = ((size_t)CIN * 9 * WS + (NC > 1 ? 2 : 1) * chunk) * 4;
    static_assert(CIN % CK == 0 && COUT % CG == 0 && CO % 2 == 0, "channel split");
};

template <int CIN, int COUT, bool RELU, bool TRANS, bool MASK>
__global__ void __launch_bounds__(ConvCfg<CIN, COUT>::NWARP * 32, 2)
conv3x3_kernel(const float *__restrict__ x, const __nv_bfloat16 *__restrict__ w, const float *__restrict__ b,
               const float *__restrict__ act, float *__restrict__ y, int H, int W) {
    using C = ConvCfg<CIN, COUT>;
    constexpr int NT = C::NWARP * 32, PX = C::PX, P2 = C::CO / 2, XS = C::XS, WS = C::WS, CK = C::CK, TH = C::TH;
    extern __shared__ __align__(16) float sm[];
    float *s_w = sm;                        // [CIN][9][WS]
    float *s_x = sm + CIN * 9 * WS;         // [1 or 2][CK][TH + 2][XS]
    const int n = blockIdx.z, ox = blockIdx.x * 32, oy = blockIdx.y * TH;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float *xn = x + (size_t)n * CIN * H * W;
    const int gx = ox + lane - 1;
    const bool xin = gx >= 0 && gx < W, xin2 = gx + 32 < W;
    auto stage = [&](int c) {
        float *dst = s_x + (c & 1) * C::chunk;
        const float *src = xn + (size_t)c * CK * H * W;
        // a row of 34 per warp and step: the index arithmetic is the warp's, not
        // a thread's (it would run on the FMA pipes)
        for (int row = warp; row < CK * (TH + 2); row += C::NWARP) {
            const int ci = row / (TH + 2), gy = oy + row % (TH + 2) - 1;
            const bool yin = gy >= 0 && gy < H;
            const float *sr = src + ((size_t)ci * H + (yin ? gy : 0)) * W;
            copy_f32(dst + row * XS + lane, xin ? sr + gx : src, yin && xin);
            if (lane < 2) copy_f32(dst + row * XS + 32 + lane, xin2 ? sr + gx + 32 : src, yin && xin2);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    stage(0);
    for (int i = tid; i < CIN * 9 * WS; i += NT) {
        const int co = i % WS, k = (i / WS) % 9, ci = i / (9 * WS);
        float v = 0.f;
        if (co < COUT) v = __bfloat162float(TRANS ? w[((size_t)ci * COUT + co) * 9 + 8 - k] : w[((size_t)co * CIN + ci) * 9 + k]);
        s_w[i] = v;
    }
    const int co0 = (warp % C::CG) * C::CO;
    const int xl = (lane % (32 / PX)) * PX, yl = (warp / C::CG) * PX + lane / (32 / PX);
    uint64_t acc[PX][P2];
#pragma unroll
    for (int j = 0; j < P2; ++j) {
        const uint64_t b2 = TRANS ? 0ull : pack2(b[co0 + 2 * j], b[co0 + 2 * j + 1]);
#pragma unroll
        for (int p = 0; p < PX; ++p) acc[p][j] = b2;
    }
#pragma unroll 1
    for (int c = 0; c < C::NC; ++c) {
        if (c + 1 < C::NC) {
            stage(c + 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const float *xt = s_x + (c & 1) * C::chunk + yl * XS + xl;
        const float *wt = s_w + c * CK * 9 * WS + co0;
#pragma unroll 1
        for (int ci = 0; ci < CK; ++ci) {
#pragma unroll
            for (int ky = 0; ky < 3; ++ky) {
                uint64_t xd[PX + 2];  // (x, x) pairs
                const float *xr = xt + (ci * (TH + 2) + ky) * XS;
#pragma unroll
                for (int q = 0; q < PX; q += 4) {
                    const float4 v = *(const float4 *)(xr + q);
                    xd[q] = pack2(v.x, v.x);
                    xd[q + 1] = pack2(v.y, v.y);
                    xd[q + 2] = pack2(v.z, v.z);
                    xd[q + 3] = pack2(v.w, v.w);
                }
                const float2 e = *(const float2 *)(xr + PX);
                xd[PX] = pack2(e.x, e.x);
                xd[PX + 1] = pack2(e.y, e.y);
#pragma unroll
                for (int kx = 0; kx < 3; ++kx) {
                    uint64_t w2[P2];
                    const float *wr = wt + (ci * 9 + ky * 3 + kx) * WS;
#pragma unroll
                    for (int j = 0; j + 1 < P2; j += 2) {
                        const ulonglong2 v = *(const ulonglong2 *)(wr + 2 * j);
                        w2[j] = v.x;
                        w2[j + 1] = v.y;
                    }
                    if (P2 & 1) w2[P2 - 1] = *(const uint64_t *)(wr + 2 * (P2 - 1));
#pragma unroll
                    for (int p = 0; p < PX; ++p)
#pragma unroll
                        for (int j = 0; j < P2; ++j) acc[p][j] = fma2(w2[j], xd[p + kx], acc[p][j]);
                }
            }
        }
        __syncthreads();  // the chunk after next reuses this buffer
    }
    const int py = oy + yl, px = ox + xl;
    if (py >= H) return;
    const size_t out0 = ((size_t)(n * COUT + co0) * H + py) * W + px;
    const bool vec = W % 4 == 0 && px + PX <= W && (((uintptr_t)y | (uintptr_t)act) & 15) == 0;
#pragma unroll
    for (int j = 0; j < P2; ++j) {
        float v[2][PX];
#pragma unroll
        for (int p = 0; p < PX; ++p) {
            unpack2(acc[p][j], v[0][p], v[1][p]);
            if (RELU) {
                v[0][p] = fmaxf(v[0][p], 0.f);
                v[1][p] = fmaxf(v[1][p], 0.f);
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const size_t o = out0 + (size_t)(2 * j + h) * H * W;
            if (vec) {
#pragma unroll
                for (int p = 0; p < PX; p += 4) {
                    if (MASK) {
                        const float4 a = *(const float4 *)(act + o + p);
                        if (!(a.x > 0.f)) v[h][p] = 0.f;
                        if (!(a.y > 0.f)) v[h][p + 1] = 0.f;
                        if (!(a.z > 0.f)) v[h][p + 2] = 0.f;
                        if (!(a.w > 0.f)) v[h][p + 3] = 0.f;
                    }
                    *(float4 *)(y + o + p) = make_float4(v[h][p], v[h][p + 1], v[h][p + 2], v[h][p + 3]);
                }
            } else {
#pragma unroll
                for (int p = 0; p < PX; ++p)
                    if (px + p < W) y[o + p] = MASK && !(act[o + p] > 0.f) ? 0.f : v[h][p];
            }
        }
    }
}

// Weight and bias gradients of a layer:
//   dW[co][ci][k] = sum over pixels of dy[co][p] * x[ci][p + off(k)],  db[co] = sum of dy[co][p].
// A thread holds 4 output channels x 1 input channel x 9 taps, each sum split
// over even and odd columns (two-wide FMAs on pixel pairs): 7 vector reads from
// shared memory per 72 FMAs.  Lanes are input channels; with few of them the
// lanes also split the tile's rows, with few output channels the warps do.  A
// block walks 16x16 tiles and keeps its sums in registers; its partial sums go
// to part[block * RGW + row group][..], summed by wgrad_reduce_kernel.
// Bound by FP32 FMAs.  One thread per weight walking a tile with scalar reads
// and an atomic add per weight and tile took 1298 us for 32 -> 32 channels on
// 8 x 256 x 256 pixels, this 291 us.
template <int CIN, int COUT>
struct WgradCfg {
    static constexpr int LC = CIN <= 8 ? 8 : CIN <= 16 ? 16 : 32;  // lanes over input channels
    static constexpr int RGL = 32 / LC;                            // row groups within a warp
    static constexpr int Q = (COUT + 3) / 4;                       // quads of output channels
    static constexpr int RGW = Q >= 8 ? 1 : Q >= 3 ? 2 : 4;        // row groups over warps
    static constexpr int RG = RGL * RGW, RR = 16 / RG;             // row groups, rows of one
    static constexpr int NT = 32 * Q * RGW;
    static constexpr int XP = 364;                                 // plane stride of x (18 rows of 20)
    static constexpr int DG = RR * 16 + 4, DP = RG * DG;           // row group and plane stride of dy
    static constexpr int K = COUT * CIN * 9 + COUT;                // sums of one layer
    static constexpr size_t smem = (size_t)(LC * XP + Q * 4 * DP) * 4;
};

template <int CIN, int COUT>
__global__ void __launch_bounds__(WgradCfg<CIN, COUT>::NT, 2)
conv3x3_wgrad_kernel(const float *__restrict__ x, const float *__restrict__ dy, float *__restrict__ part, int N, int H,
                     int W) {
    using C = WgradCfg<CIN, COUT>;
    constexpr int NT = C::NT;
    extern __shared__ __align__(16) float sm[];
    float *s_x = sm;                   // [LC][18][20], plane stride XP
    float *s_d = sm + C::LC * C::XP;   // [4 Q][RG][RR][16], strides DP, DG
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int q = warp % C::Q, rgw = warp / C::Q, ci = lane % C::LC, rg = rgw * C::RGL + lane / C::LC;
    for (int i = tid; i < C::LC * C::XP + C::Q * 4 * C::DP; i += NT) sm[i] = 0.f;  // unused channels and padding
    const int tx = (W + 15) / 16, ty = (H + 15) / 16, tiles = tx * ty * N;
    uint64_t acc[4][9];
    float db[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int k = 0; k < 9; ++k) acc[c][k] = 0ull;
    for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int n = t / (tx * ty), oy = (t / tx) % ty * 16, ox = t % tx * 16;
        const float *xn = x + (size_t)n * CIN * H * W;
        const float *dn = dy + (size_t)n * COUT * H * W;
        __syncthreads();  // the previous tile has been used
        // two rows per warp and step, a half-warp each
        const int hl = lane & 15, hr = lane >> 4;
        const int gx = ox + hl - 1;
        const bool xin = gx >= 0 && gx < W, xin2 = gx + 16 < W, din = ox + hl < W;
        for (int row = 2 * warp; row < CIN * 18; row += NT / 16) {
            const int c = row / 18, r = row % 18 + hr, gy = oy + r - 1;  // (18 is even: one channel per step)
            const bool yin = gy >= 0 && gy < H;
            const float *sr = xn + ((size_t)c * H + (yin ? gy : 0)) * W;
            float *dst = s_x + c * C::XP + r * 20;
            copy_f32(dst + hl, xin ? sr + gx : xn, yin && xin);
            if (hl < 2) copy_f32(dst + 16 + hl, xin2 ? sr + gx + 16 : xn, yin && xin2);
        }
        for (int row = 2 * warp; row < COUT * 16; row += NT / 16) {
            const int c = row / 16, r = row % 16 + hr, gy = oy + r;
            const bool in = gy < H && din;
            copy_f32(s_d + c * C::DP + (r / C::RR) * C::DG + (r % C::RR) * 16 + hl,
                     in ? dn + ((size_t)c * H + gy) * W + ox + hl : dn, in);
        }
        asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        const float *xp = s_x + ci * C::XP + rg * C::RR * 20;
        const float *dp = s_d + q * 4 * C::DP + rg * C::DG;
#pragma unroll 1
        for (int r = 0; r < C::RR; ++r) {
#pragma unroll 1
            for (int p = 0; p < 16; p += 4) {
                uint64_t d[4][2];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const ulonglong2 v = *(const ulonglong2 *)(dp + c * C::DP + r * 16 + p);
                    d[c][0] = v.x;
                    d[c][1] = v.y;
                }
#pragma unroll
                for (int ky = 0; ky < 3; ++ky) {
                    const float *xr = xp + (r + ky) * 20 + p;
                    const float4 v = *(const float4 *)xr;
                    const float2 e = *(const float2 *)(xr + 4);
                    // pixel pairs (0,1), (2,3) shifted by kx
                    const uint64_t x0 = pack2(v.x, v.y), x1 = pack2(v.y, v.z), x2 = pack2(v.z, v.w), x3 = pack2(v.w, e.x),
                                   x4 = pack2(e.x, e.y);
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        acc[c][ky * 3] = fma2(d[c][0], x0, acc[c][ky * 3]);
                        acc[c][ky * 3 + 1] = fma2(d[c][0], x1, acc[c][ky * 3 + 1]);
                        acc[c][ky * 3 + 2] = fma2(d[c][0], x2, acc[c][ky * 3 + 2]);
                    }
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        acc[c][ky * 3] = fma2(d[c][1], x2, acc[c][ky * 3]);
                        acc[c][ky * 3 + 1] = fma2(d[c][1], x3, acc[c][ky * 3 + 1]);
                        acc[c][ky * 3 + 2] = fma2(d[c][1], x4, acc[c][ky * 3 + 2]);
                    }
                }
            }
        }
        // bias: the lanes of a row group share its pixels
        for (int p = ci; p < C::RR * 16; p += C::LC)
#pragma unroll
            for (int c = 0; c < 4; ++c) db[c] += dp[c * C::DP + p];
    }
    float *out = part + (size_t)(blockIdx.x * C::RGW + rgw) * C::K;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int co = q * 4 + c;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            float lo, hi;
            unpack2(acc[c][k], lo, hi);
            float v = lo + hi;
#pragma unroll
            for (int o = C::LC; o < 32; o *= 2) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane < C::LC && ci < CIN && co < COUT) out[(co * CIN + ci) * 9 + k] = v;
        }
        float v = db[c];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0 && co < COUT) out[COUT * CIN * 9 + co] = v;
    }
}

// g[e] += sum over the partial sums part[0 .. rows)[e], in float64 (a warp per
// 32 sums and slice of the rows, four loads in flight); g holds a layer's weight
// gradients followed by its bias gradients
__global__ void __launch_bounds__(512) wgrad_reduce_kernel(const float *__restrict__ part, int rows, int K, float *g) {
    __shared__ double s[16][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, e = blockIdx.x * 32 + lane;
    double v = 0;
    if (e < K) {
        int r = warp;
        for (; r + 48 < rows; r += 64) {
            const float a = part[(size_t)r * K + e], b = part[(size_t)(r + 16) * K + e];
            const float c = part[(size_t)(r + 32) * K + e], d = part[(size_t)(r + 48) * K + e];
            v += ((double)a + b) + ((double)c + d);
        }
        for (; r < rows; r += 16) v += (double)part[(size_t)r * K + e];
    }
    s[warp][lane] = v;
    __syncthreads();
    if (warp == 0 && e < K) {
        for (int k = 1; k < 16; ++k) v += s[k][lane];
        g[e] += (float)v;
    }
}

// mean squared error over count values and its gradient dy = 2 (y - t) / count
// (a double per block: per warp, the atomics on the one sum took most of the time)
__global__ void __launch_bounds__(256) mse_kernel(const float *y, const float *t, float *dy, size_t count, double *loss) {
    __shared__ double sw[8];
    const float scale = (float)count;
    double s = 0;
    auto one = [&](float a, float b) -> float {
        const float d = a - b;
        s += (double)d * d;
        return 2.f * d / scale;
    };
    const size_t i0 = blockIdx.x * (size_t)blockDim.x + threadIdx.x, stride = (size_t)gridDim.x * blockDim.x;
    const bool vec = (((uintptr_t)y | (uintptr_t)t | (uintptr_t)dy) & 15) == 0;
    const size_t n4 = vec ? count / 4 : 0;
    for (size_t i = i0; i < n4; i += stride) {
        const float4 a = ((const float4 *)y)[i], b = ((const float4 *)t)[i];
        ((float4 *)dy)[i] = make_float4(one(a.x, b.x), one(a.y, b.y), one(a.z, b.z), one(a.w, b.w));
    }
    for (size_t i = n4 * 4 + i0; i < count; i += stride) dy[i] = one(y[i], t[i]);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) sw[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < 8; ++k) s += sw[k];
        if (s != 0) atomicAdd(loss, s / (double)count);
    }
}

// Adam on FP32 master weights; refreshes the BF16 copy used by the products
__global__ void adam_kernel(float *p, const float *g, float *m, float *v, __nv_bfloat16 *pb, size_t n, float lr,
                            float b1, float b2, float eps, float bc1, float bc2) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float upd = lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
        p[i] -= upd;
        pb[i] = __float2bfloat16(p[i]);
    }
}

__global__ void to_bf16_kernel(const float *p, __nv_bfloat16 *pb, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        pb[i] = __float2bfloat16(p[i]);
}

// ---- inference on the tensor cores -----------------------------------------------
// Implicit GEMM per 16x16 output tile: for each of the nine taps,
// D[pixel][co] += A[pixel][ci] * B[ci][co], A being the input tile shifted by
// the tap.  The input tile (halo 1) is staged once in shared memory as BF16
// rows [pixel][channel] padded to KIN + 8 elements (80 or 48 bytes: the eight
// rows one ldmatrix reads fall in distinct banks); the layer's weights as
// [tap][co][ci] rows of the same padding.  mma.sync m16n8k16 takes BF16
// operands with FP32 accumulation; a warp computes two output rows (M = 16
// pixels each) and shares every B fragment between them.  Activations between
// layers are BF16 NHWC with 32 channels; the first layer reads the FP32 NCHW
// network input, the last writes FP32 NCHW.
constexpr int kIT = 16;       // output tile edge
constexpr int kIH = kIT + 2;  // staged tile edge

__device__ __forceinline__ void ldsm_x4(const void *p, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(a));
}

__device__ __forceinline__ void ldsm_x2(const void *p, uint32_t &r0, uint32_t &r1) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];\n" : "=r"(r0), "=r"(r1) : "r"(a));
}

__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

template <int KIN, int NOUT>
constexpr size_t conv_mma_smem() {
    return (size_t)(9 * NOUT + kIH * kIH) * (KIN + 8) * 2 + NOUT * 4;
}

template <int KIN, int NOUT, bool IN_F32, bool OUT_F32, bool RELU>
__global__ void __launch_bounds__(256) conv3x3_mma_kernel(const void *__restrict__ in, int cin,
                                                          const __nv_bfloat16 *__restrict__ w,
                                                          const float *__restrict__ bias, void *__restrict__ out,
                                                          int cout, int N, int H, int W) {
    constexpr int AS = KIN + 8;  // BF16 elements per staged row
    constexpr int NT = NOUT / 8; // n-tiles of 8 output channels
    constexpr int KS = KIN / 16; // k-steps per tap
    extern __shared__ __align__(16) unsigned char smraw[];
    __nv_bfloat16 *s_w = (__nv_bfloat16 *)smraw;          // [9][NOUT][AS]
    __nv_bfloat16 *s_a = s_w + 9 * NOUT * AS;              // [kIH * kIH][AS]
    float *s_bias = (float *)(s_a + kIH * kIH * AS);       // [NOUT]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int i = tid; i < 9 * NOUT * KIN; i += blockDim.x) {
        const int tap = i / (NOUT * KIN), co = (i / KIN) % NOUT, ci = i % KIN;
        s_w[(tap * NOUT + co) * AS + ci] =
            (co < cout && ci < cin) ? w[((size_t)co * cin + ci) * 9 + tap] : __float2bfloat16(0.f);
    }
    for (int i = tid; i < NOUT; i += blockDim.x) s_bias[i] = i < cout ? bias[i] : 0.f;
    const int tiles_x = (W + kIT - 1) / kIT, tiles_y = (H + kIT - 1) / kIT;
    const long long per_img = (long long)tiles_x * tiles_y, tiles = per_img * N;
    for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int n = (int)(t / per_img), rem = (int)(t % per_img);
        const int oy = (rem / tiles_x) * kIT, ox = (rem % tiles_x) * kIT;
        __syncthreads();  // the previous tile's reads of s_a are done
        if constexpr (IN_F32) {
            const float *x = (const float *)in + (size_t)n * cin * H * W;
            for (int i = tid; i < KIN * kIH * kIH; i += blockDim.x) {
                const int c = i / (kIH * kIH), p = i % (kIH * kIH);
                const int gy = oy + p / kIH - 1, gx = ox + p % kIH - 1;
                float v = 0.f;
                if (c < cin && gy >= 0 && gy < H && gx >= 0 && gx < W) v = x[((size_t)c * H + gy) * W + gx];
                s_a[p * AS + c] = __float2bfloat16(v);
            }
        } else {
            const __nv_bfloat16 *x = (const __nv_bfloat16 *)in + (size_t)n * H * W * KIN;
            constexpr int CH = KIN / 8;  // 16-byte chunks per pixel
            for (int i = tid; i < kIH * kIH * CH; i += blockDim.x) {
                const int p = i / CH, q = i % CH;
                const int gy = oy + p / kIH - 1, gx = ox + p % kIH - 1;
                uint4 v = make_uint4(0u, 0u, 0u, 0u);
                if (gy >= 0 && gy < H && gx >= 0 && gx < W)
                    v = *(const uint4 *)(x + ((size_t)gy * W + gx) * KIN + q * 8);
                *(uint4 *)(s_a + p * AS + q * 8) = v;
            }
        }
        __syncthreads();
        // warp w computes output rows w and w + 8 of the tile
        const int rows[2] = {warp, warp + 8};
        float acc[2][NT][4];
#pragma unroll
        for (int rr = 0; rr < 2; ++rr)
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[rr][j][e] = s_bias[j * 8 + 2 * (lane & 3) + (e & 1)];
        const int am = (lane & 7) + 8 * ((lane >> 3) & 1);  // A row (pixel) this lane addresses
        const int ak = 8 * (lane >> 4);                    // A column offset
#pragma unroll
        for (int tap = 0; tap < 9; ++tap) {
            const int ky = tap / 3, kx = tap % 3;
#pragma unroll
            for (int ks = 0; ks < KS; ++ks) {
                uint32_t a[2][4];
#pragma unroll
                for (int rr = 0; rr < 2; ++rr)
                    ldsm_x4(s_a + ((rows[rr] + ky) * kIH + am + kx) * AS + ks * 16 + ak, a[rr][0], a[rr][1],
                            a[rr][2], a[rr][3]);
                if constexpr (NT == 1) {
                    uint32_t b0, b1;
                    ldsm_x2(s_w + (tap * NOUT + (lane & 7)) * AS + ks * 16 + 8 * ((lane >> 3) & 1), b0, b1);
#pragma unroll
                    for (int rr = 0; rr < 2; ++rr) mma_bf16_16816(acc[rr][0], a[rr], b0, b1);
                } else {
#pragma unroll
                    for (int j2 = 0; j2 < NT / 2; ++j2) {
                        const int mat = lane >> 3;
                        const int nt = 2 * j2 + (mat >> 1), kh = mat & 1;
                        uint32_t b0, b1, b2, b3;
                        ldsm_x4(s_w + (tap * NOUT + nt * 8 + (lane & 7)) * AS + ks * 16 + kh * 8, b0, b1, b2, b3);
#pragma unroll
                        for (int rr = 0; rr < 2; ++rr) {
                            mma_bf16_16816(acc[rr][2 * j2], a[rr], b0, b1);
                            mma_bf16_16816(acc[rr][2 * j2 + 1], a[rr], b2, b3);
                        }
                    }
                }
            }
        }
        // accumulator (e = 0,1: pixel g; e = 2,3: pixel g + 8), channels j*8 + 2c, +1
        const int g8 = lane >> 2, cq = lane & 3;
#pragma unroll
        for (int rr = 0; rr < 2; ++rr) {
            const int py = oy + rows[rr];
            if (py >= H) continue;
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    const int px = ox + g8 + 8 * hf;
                    if (px >= W) continue;
                    float v0 = acc[rr][j][2 * hf], v1 = acc[rr][j][2 * hf + 1];
                    if (RELU) {
                        v0 = fmaxf(v0, 0.f);
                        v1 = fmaxf(v1, 0.f);
                    }
                    const int co = j * 8 + 2 * cq;
                    if constexpr (OUT_F32) {
                        float *y = (float *)out + (size_t)n * cout * H * W;
                        if (co < cout) y[((size_t)co * H + py) * W + px] = v0;
                        if (co + 1 < cout) y[((size_t)(co + 1) * H + py) * W + px] = v1;
                    } else {
                        __nv_bfloat16 *y = (__nv_bfloat16 *)out + ((size_t)n * H * W + (size_t)py * W + px) * NOUT;
                        *(__nv_bfloat162 *)(y + co) = __floats2bfloat162_rn(v0, v1);
                    }
                }
        }
    }
}

// ---- host side ---------------------------------------------------------------
template <int CIN, int COUT, bool RELU, bool TRANS, bool MASK>
static cudaError_t conv(const float *x, const __nv_bfloat16 *w, const float *b, const float *act, float *y, int N, int H,
                        int W, cudaStream_t s) {
    using C = ConvCfg<CIN, COUT>;
    auto k = conv3x3_kernel<CIN, COUT, RELU, TRANS, MASK>;
    const cudaError_t e = ensure_smem_attr((const void *)k, (int)C::smem);
    if (e != cudaSuccess) return e;
    dim3 grid((W + 31) / 32, (H + C::TH - 1) / C::TH, N);
    k<<<grid, C::NWARP * 32, C::smem, s>>>(x, w, b, act, y, H, W);
    return cudaGetLastError();
}

template <int KIN, int NOUT, bool IN_F32, bool OUT_F32, bool RELU>
static cudaError_t conv_mma(const void *x, int cin, const __nv_bfloat16 *w, const float *b, void *y, int cout, int N,
                            int H, int W, cudaStream_t s) {
    constexpr size_t smem = conv_mma_smem<KIN, NOUT>();
    auto kern = conv3x3_mma_kernel<KIN, NOUT, IN_F32, OUT_F32, RELU>;
    static int blocks_per_sm = 0, sms = 0;
    if (!blocks_per_sm) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        int dev = 0;
        if (e == cudaSuccess) e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks_per_sm, kern, 256, smem);
        if (e != cudaSuccess) return e;
        if (blocks_per_sm < 1) return cudaErrorInvalidConfiguration;
    }
    const long long tiles = (long long)((W + kIT - 1) / kIT) * ((H + kIT - 1) / kIT) * N;
    const int grid = (int)std::min<long long>(tiles, (long long)blocks_per_sm * sms);
    kern<<<grid, 256, smem, s>>>(x, cin, w, b, y, cout, N, H, W);
    return cudaGetLastError();
}

// partial sums of a layer's weight gradients: blocks * RGW rows of K floats
static int wgrad_blocks() { return device_sms() * 2; }
template <int CIN, int COUT> constexpr size_t kWgradPart = (size_t)WgradCfg<CIN, COUT>::RGW *WgradCfg<CIN, COUT>::K;
// a block's share of the workspace: the most any layer writes (9248 floats, the
// 32 -> 32 layers; the narrow last layers write 6936 and 5780 in several row groups)
constexpr size_t kWgradPartMax = std::max({kWgradPart<6, 32>, kWgradPart<10, 32>, kWgradPart<32, 32>, kWgradPart<32, 6>,
                                           kWgradPart<32, 10>});

template <int CIN, int COUT>
static cudaError_t conv_wgrad(const float *x, const float *dy, float *part, float *g, int N, int H, int W,
                              cudaStream_t s) {
    using C = WgradCfg<CIN, COUT>;
    static_assert(kWgradPart<CIN, COUT> <= kWgradPartMax, "partial sums");
    auto k = conv3x3_wgrad_kernel<CIN, COUT>;
    const cudaError_t e = ensure_smem_attr((const void *)k, (int)C::smem);
    if (e != cudaSuccess) return e;
    const long long tiles = (long long)((W + 15) / 16) * ((H + 15) / 16) * N;
    const int grid = (int)std::min<long long>(tiles, wgrad_blocks());
    k<<<grid, C::NT, C::smem, s>>>(x, dy, part, N, H, W);
    wgrad_reduce_kernel<<<(C::K + 31) / 32, 512, 0, s>>>(part, grid * C::RGW, C::K, g);
    return cudaGetLastError();
}

// (cin, cout, relu) dispatch over the layer shapes the network uses
static cudaError_t conv_fwd_any(int cin, int cout, bool relu, const float *x, const __nv_bfloat16 *w, const float *b,
                                float *y, int N, int H, int W, cudaStream_t s) {
    if (cin == 6 && cout == 32 && relu) return conv<6, 32, true, false, false>(x, w, b, nullptr, y, N, H, W, s);
    if (cin == 10 && cout == 32 && relu) return conv<10, 32, true, false, false>(x, w, b, nullptr, y, N, H, W, s);
    if (cin == 32 && cout == 32 && relu) return conv<32, 32, true, false, false>(x, w, b, nullptr, y, N, H, W, s);
    if (cin == 32 && cout == 6 && !relu) return conv<32, 6, false, false, false>(x, w, b, nullptr, y, N, H, W, s);
    if (cin == 32 && cout == 10 && !relu) return conv<32, 10, false, false, false>(x, w, b, nullptr, y, N, H, W, s);
    return cudaErrorInvalidValue;
}

// input gradient of a layer cin -> cout, with the ReLU mask of the layer below
// (act: its output): dx has cin = 32 channels
static cudaError_t conv_dgrad_any(int cin, int cout, const float *dy, const __nv_bfloat16 *w, const float *act, float *dx,
                                  int N, int H, int W, cudaStream_t s) {
    if (cin == 32 && cout == 32) return conv<32, 32, false, true, true>(dy, w, nullptr, act, dx, N, H, W, s);
    if (cin == 32 && cout == 6) return conv<6, 32, false, true, true>(dy, w, nullptr, act, dx, N, H, W, s);
    if (cin == 32 && cout == 10) return conv<10, 32, false, true, true>(dy, w, nullptr, act, dx, N, H, W, s);
    return cudaErrorInvalidValue;
}

static cudaError_t conv_wgrad_any(int cin, int cout, const float *x, const float *dy, float *part, float *g, int N,
                                  int H, int W, cudaStream_t s) {
    if (cin == 6 && cout == 32) return conv_wgrad<6, 32>(x, dy, part, g, N, H, W, s);
    if (cin == 10 && cout == 32) return conv_wgrad<10, 32>(x, dy, part, g, N, H, W, s);
    if (cin == 32 && cout == 32) return conv_wgrad<32, 32>(x, dy, part, g, N, H, W, s);
    if (cin == 32 && cout == 6) return conv_wgrad<32, 6>(x, dy, part, g, N, H, W, s);
    if (cin == 32 && cout == 10) return conv_wgrad<32, 10>(x, dy, part, g, N, H, W, s);
    return cudaErrorInvalidValue;
}

}  // namespace mf

using namespace mf;

struct mf_cnn {
    int ch[5];                 // channels: in, 32, 32, 32, out
    size_t woff[5], boff[5];   // offsets of layer weights / biases in the parameter vector
    size_t nparam = 0;
    float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;  // master params, grads, Adam moments
    __nv_bfloat16 *pb = nullptr;                                   // BF16 copy used by the products
    float *part = nullptr;                                         // partial weight gradients of a backward pass (11 MB)
    float *act[5] = {nullptr, nullptr, nullptr, nullptr, nullptr}; // layer outputs of the last kept forward
    float *dbuf[2] = {nullptr, nullptr};                           // gradient ping-pong buffers
    double *dloss = nullptr;
    __nv_bfloat16 *ibuf[2] = {nullptr, nullptr};                   // inference activations, BF16 NHWC x 32
    size_t icap_pix = 0;
    size_t cap_pix = 0;        // N*H*W the activation buffers hold
    int N = 0, H = 0, W = 0;
    long long steps = 0;
    cudaStream_t stream = nullptr;
    std::string err;
};

static mf_status cnn_fail(mf_cnn *c, mf_status s, const std::string &m) {
    if (c) c->err = m;
    else set_static_error(m);
    return s;
}

#define CKC(call)                                                                                  \
    do {                                                                                           \
        cudaError_t e_ = (call);                                                                   \
        if (e_ != cudaSuccess) {                                                                   \
            cudaGetLastError(); /* reported here: the next launch check must not see it again */   \
            return cnn_fail(c, e_ == cudaErrorMemoryAllocation ? MF_ENOMEM : MF_ECUDA,             \
                            std::string(#call) + ": " + cudaGetErrorString(e_));                   \
        }                                                                                          \
    } while (0)

static void cnn_free_acts(mf_cnn *c) {
    for (auto &a : c->act)
        if (a) { cudaFree(a); a = nullptr; }
    for (auto &d : c->dbuf)
        if (d) { cudaFree(d); d = nullptr; }
    c->cap_pix = 0;
    c->N = 0;  // the last forward's activations are gone: no backward on them
}

static mf_status cnn_ensure_infer(mf_cnn *c, int N, int H, int W) {
    const size_t pix = (size_t)N * H * W;
    if (pix <= c->icap_pix) return MF_OK;
    for (auto &b : c->ibuf)
        if (b) { cudaFree(b); b = nullptr; }
    c->icap_pix = 0;
    for (auto &b : c->ibuf) CKC(cudaMalloc(&b, pix * 32 * 2));
    c->icap_pix = pix;
    return MF_OK;
}

// all that a forward and the backward after it write: a backward allocates
// nothing (it may run while a stream is captured)
static mf_status cnn_ensure(mf_cnn *c, int N, int H, int W) {
    const size_t pix = (size_t)N * H * W;
    if (!c->part) CKC(cudaMalloc(&c->part, wgrad_blocks() * kWgradPartMax * 4));
    if (pix <= c->cap_pix) return MF_OK;
    cnn_free_acts(c);
    for (int l = 1; l <= 3; ++l) CKC(cudaMalloc(&c->act[l], pix * c->ch[l] * 4));
    for (auto &d : c->dbuf) CKC(cudaMalloc(&d, pix * 32 * 4));
    c->cap_pix = pix;
    return MF_OK;
}

extern "C" {

mf_status mf_cnn_create(mf_cnn **out, int in_ch, int out_ch, uint64_t seed, void *cuda_stream) {
    if (!out) return cnn_fail(nullptr, MF_EINVAL, "out is NULL");
    *out = nullptr;
    if (!((in_ch == 6 && out_ch == 6) || (in_ch == 10 && out_ch == 10)))
        return cnn_fail(nullptr, MF_EINVAL, "channels must be 6/6 (4-connected) or 10/10 (8-connected)");
    mf_cnn *c = new mf_cnn();
    const int ch[5] = {in_ch, 32, 32, 32, out_ch};
    for (int i = 0; i < 5; ++i) c->ch[i] = ch[i];
    size_t off = 0;
    for (int l = 1; l <= 4; ++l) {
        c->woff[l] = off;
        off += (size_t)ch[l] * ch[l - 1] * 9;
        c->boff[l] = off;
        off += ch[l];
    }
    c->nparam = off;
    c->stream = (cudaStream_t)cuda_stream;
    // He-uniform initial weights from a SplitMix64 stream, zero biases
    std::vector<float> h(off, 0.f);
    uint64_t st = seed;
    auto next = [&]() {
        uint64_t z = (st += 0x9E3779B97F4A7C15ull);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z ^= z >> 31;
        return (double)(z >> 11) * (1.0 / 9007199254740992.0);
    };
    for (int l = 1; l <= 4; ++l) {
        const double fan_in = 9.0 * ch[l - 1];
        const double a = (l == 4 ? 0.5 : 1.0) * std::sqrt(6.0 / fan_in);
        for (size_t i = 0; i < (size_t)ch[l] * ch[l - 1] * 9; ++i) h[c->woff[l] + i] = (float)((2 * next() - 1) * a);
    }
    cudaError_t e = cudaMalloc(&c->p, off * 4);
    if (e == cudaSuccess) e = cudaMalloc(&c->g, off * 4);
    if (e == cudaSuccess) e = cudaMalloc(&c->m, off * 4);
    if (e == cudaSuccess) e = cudaMalloc(&c->v, off * 4);
    if (e == cudaSuccess) e = cudaMalloc(&c->pb, off * 2);
    if (e == cudaSuccess) e = cudaMalloc(&c->dloss, 8);
    if (e == cudaSuccess) e = cudaMemcpy(c->p, h.data(), off * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(c->g, 0, off * 4);
    if (e == cudaSuccess) e = cudaMemset(c->m, 0, off * 4);
    if (e == cudaSuccess) e = cudaMemset(c->v, 0, off * 4);
    if (e == cudaSuccess) {
        to_bf16_kernel<<<64, 256, 0, c->stream>>>(c->p, c->pb, off);
        e = cudaStreamSynchronize(c->stream);
    }
    if (e != cudaSuccess) {
        std::string m = cudaGetErrorString(e);
        mf_cnn_destroy(c);
        return cnn_fail(nullptr, MF_ECUDA, "mf_cnn_create: " + m);
    }
    *out = c;
    return MF_OK;
}

mf_status mf_cnn_destroy(mf_cnn *c) {
    if (!c) return MF_OK;
    cnn_free_acts(c);
    void *ps[] = {c->p, c->g, c->m, c->v, c->pb, c->part, c->dloss, c->ibuf[0], c->ibuf[1]};
    for (void *q : ps)
        if (q) cudaFree(q);
    delete c;
    return MF_OK;
}

const char *mf_cnn_last_error(const mf_cnn *c) { return c ? c->err.c_str() : mf_last_error(nullptr); }

int64_t mf_cnn_num_params(const mf_cnn *c) { return c ? (int64_t)c->nparam : 0; }

mf_status mf_cnn_get_params(mf_cnn *c, float *out, int on_device) {
    if (!c || !out) return cnn_fail(c, MF_EINVAL, "null argument");
    CKC(cudaMemcpyAsync(out, c->p, c->nparam * 4, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                        c->stream));
    CKC(cudaStreamSynchronize(c->stream));
    return MF_OK;
}

mf_status mf_cnn_set_params(mf_cnn *c, const float *in, int on_device) {
    if (!c || !in) return cnn_fail(c, MF_EINVAL, "null argument");
    CKC(cudaMemcpyAsync(c->p, in, c->nparam * 4, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                        c->stream));
    to_bf16_kernel<<<64, 256, 0, c->stream>>>(c->p, c->pb, c->nparam);
    CKC(cudaGetLastError());
    CKC(cudaMemsetAsync(c->m, 0, c->nparam * 4, c->stream));
    CKC(cudaMemsetAsync(c->v, 0, c->nparam * 4, c->stream));
    c->steps = 0;
    CKC(cudaStreamSynchronize(c->stream));
    return MF_OK;
}

// Parameters from a NumPy .npy file holding a little-endian float32 vector
// of exactly num_params entries (format versions 1-3).
mf_status mf_load_model(mf_cnn *c, const char *path) {
    if (!c || !path) return cnn_fail(c, MF_EINVAL, "null argument");
    FILE *f = fopen(path, "rb");
    if (!f) return cnn_fail(c, MF_EINVAL, std::string("cannot open ") + path);
    auto bad = [&](const std::string &m) {
        fclose(f);
        return cnn_fail(c, MF_EINVAL, std::string(path) + ": " + m);
    };
    unsigned char pre[8];
    if (fread(pre, 1, 8, f) != 8 || memcmp(pre, "\x93NUMPY", 6) != 0) return bad("not a .npy file");
    size_t hlen = 0;
    if (pre[6] == 1) {
        unsigned char b[2];
        if (fread(b, 1, 2, f) != 2) return bad("truncated header");
        hlen = (size_t)b[0] | ((size_t)b[1] << 8);
    } else if (pre[6] == 2 || pre[6] == 3) {
        unsigned char b[4];
        if (fread(b, 1, 4, f) != 4) return bad("truncated header");
        hlen = (size_t)b[0] | ((size_t)b[1] << 8) | ((size_t)b[2] << 16) | ((size_t)b[3] << 24);
    } else {
        return bad("unsupported .npy version");
    }
    if (hlen > (1u << 20)) return bad("header too long");
    std::string h(hlen, '\0');
    if (fread(&h[0], 1, hlen, f) != hlen) return bad("truncated header");
    if (h.find("'descr': '<f4'") == std::string::npos) return bad("dtype is not little-endian float32");
    if (h.find("'fortran_order': False") == std::string::npos) return bad("Fortran order");
    const size_t sp = h.find("'shape': (");
    if (sp == std::string::npos) return bad("no shape");
    const long long cnt = strtoll(h.c_str() + sp + 10, nullptr, 10);
    if (cnt != (long long)c->nparam || h.find(",)", sp) == std::string::npos)
        return bad("shape does not match the network's " + std::to_string(c->nparam) + " parameters");
    std::vector<float> buf(c->nparam);
    if (fread(buf.data(), 4, c->nparam, f) != c->nparam) return bad("truncated data");
    fclose(f);
    return mf_cnn_set_params(c, buf.data(), 0);
}

mf_status mf_cnn_get_grads(mf_cnn *c, float *out, int on_device) {
    if (!c || !out) return cnn_fail(c, MF_EINVAL, "null argument");
    CKC(cudaMemcpyAsync(out, c->g, c->nparam * 4, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                        c->stream));
    CKC(cudaStreamSynchronize(c->stream));
    return MF_OK;
}

mf_status mf_cnn_forward(mf_cnn *c, const float *x, int N, int H, int W, float *y) {
    if (!c || !x || !y || N < 1 || H < 1 || W < 1) return cnn_fail(c, MF_EINVAL, "bad forward arguments");
    mf_status s = cnn_ensure(c, N, H, W);
    if (s != MF_OK) return s;
    c->N = N;
    c->H = H;
    c->W = W;
    const float *in = x;
    for (int l = 1; l <= 4; ++l) {
        float *o = l == 4 ? y : c->act[l];
        CKC(conv_fwd_any(c->ch[l - 1], c->ch[l], l < 4, in, c->pb + c->woff[l], c->p + c->boff[l], o, N, H, W,
                         c->stream));
        in = o;
    }
    return MF_OK;
}

mf_status mf_cnn_infer(mf_cnn *c, const float *x, int N, int H, int W, float *y) {
    if (!c || !x || !y || N < 1 || H < 1 || W < 1) return cnn_fail(c, MF_EINVAL, "bad infer arguments");
    mf_status s = cnn_ensure_infer(c, N, H, W);
    if (s != MF_OK) return s;
    const int cin = c->ch[0], cout = c->ch[4];
    __nv_bfloat16 *b0 = c->ibuf[0], *b1 = c->ibuf[1];
    CKC((conv_mma<16, 32, true, false, true>(x, cin, c->pb + c->woff[1], c->p + c->boff[1], b0, 32, N, H, W,
                                             c->stream)));
    CKC((conv_mma<32, 32, false, false, true>(b0, 32, c->pb + c->woff[2], c->p + c->boff[2], b1, 32, N, H, W,
                                              c->stream)));
    CKC((conv_mma<32, 32, false, false, true>(b1, 32, c->pb + c->woff[3], c->p + c->boff[3], b0, 32, N, H, W,
                                              c->stream)));
    if (cout <= 8)
        CKC((conv_mma<32, 8, false, true, false>(b0, 32, c->pb + c->woff[4], c->p + c->boff[4], y, cout, N, H, W,
                                                 c->stream)));
    else
        CKC((conv_mma<32, 16, false, true, false>(b0, 32, c->pb + c->woff[4], c->p + c->boff[4], y, cout, N, H, W,
                                                  c->stream)));
    return MF_OK;
}

mf_status mf_cnn_zero_grad(mf_cnn *c) {
    if (!c) return cnn_fail(c, MF_EINVAL, "null network");
    CKC(cudaMemsetAsync(c->g, 0, c->nparam * 4, c->stream));
    return MF_OK;
}

mf_status mf_cnn_backward(mf_cnn *c, const float *x, const float *dy) {
    if (!c || !x || !dy || !c->N) return cnn_fail(c, MF_EINVAL, "backward needs the last forward's input and dy");
    const int N = c->N, H = c->H, W = c->W;
    // gradient of layer l's output lives in cur, with the layer's ReLU applied
    // (layer 4 has none)
    const float *cur = dy;
    int slot = 0;
    for (int l = 4; l >= 1; --l) {
        const float *lin = l == 1 ? x : c->act[l - 1];
        float *dx = c->dbuf[slot];
        CKC(conv_wgrad_any(c->ch[l - 1], c->ch[l], lin, cur, c->part, c->g + c->woff[l], N, H, W, c->stream));
        if (l > 1) {
            CKC(conv_dgrad_any(c->ch[l - 1], c->ch[l], cur, c->pb + c->woff[l], c->act[l - 1], dx, N, H, W, c->stream));
            cur = dx;
            slot ^= 1;
        }
    }
    return MF_OK;
}

mf_status mf_cnn_mse(mf_cnn *c, const float *y, const float *target, float *dy, int64_t count, double *loss) {
    if (!c || !y || !target || !dy || count < 1) return cnn_fail(c, MF_EINVAL, "bad loss arguments");
    CKC(cudaMemsetAsync(c->dloss, 0, 8, c->stream));
    mse_kernel<<<device_sms() * 8, 256, 0, c->stream>>>(y, target, dy, (size_t)count, c->dloss);
    CKC(cudaGetLastError());
    double h = 0;
    CKC(cudaMemcpyAsync(&h, c->dloss, 8, cudaMemcpyDeviceToHost, c->stream));
    CKC(cudaStreamSynchronize(c->stream));
    if (loss) *loss = h;
    return MF_OK;
}

mf_status mf_cnn_adam_step(mf_cnn *c, float lr, float beta1, float beta2, float eps) {
    if (!c) return cnn_fail(c, MF_EINVAL, "null network");
    c->steps += 1;
    const float bc1 = 1.f - (float)std::pow((double)beta1, (double)c->steps);
    const float bc2 = 1.f - (float)std::pow((double)beta2, (double)c->steps);
    adam_kernel<<<64, 256, 0, c->stream>>>(c->p, c->g, c->m, c->v, c->pb, c->nparam, lr, beta1, beta2, eps, bc1, bc2);
    CKC(cudaGetLastError());
    return MF_OK;
}

}  // extern "C"
