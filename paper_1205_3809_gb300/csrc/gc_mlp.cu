// Learned vertex priority: per-vertex features, a 6-32-32-1 ReLU MLP with
// bf16 operands and fp32 accumulation (forward, loss gradient, Adam), and
// the monotone map from a score to a uint32 key for gc_color's priority.
// The paper colors in index order (Sec. 3.2) and cites ordering heuristics
// for Greedy (smallest-last, largest-first: Sec. 1, Sec. 3.1); the network
// is trained to place a vertex where such an ordering would put it.
//
// Parameter vector (fp32 master copy, kMlpParams floats):
//   W1[32][6] | b1[32] | W2[32][32] | b2[32] | W3[32] | b3
// Forward, per sample x (6 features):
//   a0 = bf16(x); z1 = bf16(W1) a0 + b1; a1 = bf16(relu(z1));
//   z2 = bf16(W2) a1 + b2; a2 = bf16(relu(z2)); y = bf16(W3) . a2 + b3
// with every dot product accumulated in fp32 in index order (bf16 = round
// to nearest even).  The loss of a batch of B samples is mean (y - t)^2; its
// gradient uses the same bf16 weights and activations.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "gc.h"

namespace {

constexpr int kIn = 6, kH = 32;
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kH * kIn, kOffW2 = kOffB1 + kH, kOffB2 = kOffW2 + kH * kH,
              kOffW3 = kOffB2 + kH, kOffB3 = kOffW3 + kH, kMlpParams = kOffB3 + 1;
static_assert(kMlpParams == 1313, "parameter layout");
constexpr int kTile = 128;  // samples per tile of the gradient kernel, one per thread

__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// Two fp32 values side by side, each lane of the arithmetic rounded as the
// scalar instruction rounds it.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 x, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(x));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// The parameters as the forward kernel reads them: weights rounded to bf16 and
// stored input by input, so that the weights of neighbouring units sit side by
// side (a row of 36 floats spreads the stores over the banks).
constexpr int kRow = kH + 4;
struct __align__(16) ForwardParams {
    float w1[kIn][kRow];
    float w2[kH][kRow];
    float w3[kH], b1[kH], b2[kH];  // (b1, b2: read two at a time)
    float b3;
};
__device__ __forceinline__ void load_forward_params(const float* __restrict__ params, ForwardParams& s) {
    for (int i = threadIdx.x; i < kMlpParams; i += blockDim.x) {
        const float p = params[i];
        if (i < kOffB1) {
            s.w1[i % kIn][i / kIn] = bf16r(p);
        } else if (i < kOffW2) {
            s.b1[i - kOffB1] = p;
        } else if (i < kOffB2) {
            s.w2[(i - kOffW2) % kH][(i - kOffW2) / kH] = bf16r(p);
        } else if (i < kOffW3) {
            s.b2[i - kOffB2] = p;
        } else if (i < kOffB3) {
            s.w3[i - kOffW3] = bf16r(p);
        } else {
            s.b3 = p;
        }
    }
}

// One layer of one sample: every unit's sum runs over the inputs in index order,
// two units to an instruction.
template <int IN, int OUT>
__device__ __forceinline__ void layer_units(const float (*w)[kRow], const float* bias, const float (&in)[IN],
                                            float (&out)[OUT]) {
    f32x2 acc[OUT / 2];
#pragma unroll
    for (int q = 0; q < OUT / 2; ++q) acc[q] = 0ull;
#pragma unroll
    for (int i = 0; i < IN; ++i) {
        const f32x2 a = pack2(in[i], in[i]);
#pragma unroll
        for (int q = 0; q < OUT / 2; q += 2) {
            const ulonglong2 wq = *reinterpret_cast<const ulonglong2*>(&w[i][2 * q]);
            acc[q] = fma2(wq.x, a, acc[q]);
            acc[q + 1] = fma2(wq.y, a, acc[q + 1]);
        }
    }
#pragma unroll
    for (int q = 0; q < OUT / 2; ++q) {
        float x, y;
        unpack2(acc[q], x, y);
        out[2 * q] = bf16r(fmaxf(x + bias[2 * q], 0.f));
        out[2 * q + 1] = bf16r(fmaxf(y + bias[2 * q + 1], 0.f));
    }
}

// Two bf16 values in a word, the first in its low half: rounding to nearest
// even (NaN stays NaN), max(., 0) of both (NaN gives 0, as fmaxf does; rounding
// keeps the sign, so it commutes with the maximum), and a value back.
__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi) {
    uint32_t w;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w) : "f"(hi), "f"(lo));
    return w;
}
__device__ __forceinline__ uint32_t relu_pair(uint32_t w) {
    uint32_t m;
    asm("max.bf16x2 %0, %1, %2;" : "=r"(m) : "r"(w), "r"(0u));
    return m;
}
__device__ __forceinline__ float bf16_of(uint32_t w, int half) {
    return __uint_as_float(half ? w & 0xffff0000u : w << 16);
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// The same for R samples and units j0 .. j0 + J - 1, a weight read from shared
// memory serving all samples, with the activations kept as pairs of bf16 (half the
// registers, and bias, rounding and maximum take one instruction each for two
// units).
template <int IN, int J, int R>
__device__ __forceinline__ void layer_pairs(const float (*w)[kRow], const float* bias, int j0,
                                            const uint32_t (&in)[R][IN / 2], uint32_t (&out)[R][J / 2]) {
    f32x2 acc[R][J / 2];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int q = 0; q < J / 2; ++q) acc[r][q] = 0ull;
#pragma unroll
    for (int i = 0; i < IN; ++i) {
        f32x2 a[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float v = bf16_of(in[r][i / 2], i & 1);
            a[r] = pack2(v, v);
        }
#pragma unroll
        for (int q = 0; q < J / 2; q += 2) {
            const ulonglong2 wq = *reinterpret_cast<const ulonglong2*>(&w[i][j0 + 2 * q]);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                acc[r][q] = fma2(wq.x, a[r], acc[r][q]);
                acc[r][q + 1] = fma2(wq.y, a[r], acc[r][q + 1]);
            }
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int q = 0; q < J / 2; ++q) {
            float x, y;
            unpack2(add2(acc[r][q], *reinterpret_cast<const f32x2*>(&bias[j0 + 2 * q])), x, y);
            out[r][q] = relu_pair(bf16_pair(x, y));
        }
}

// R samples per thread, kForwardUnits units at a time.
// Bound: the fp32 multiply-adds (1,248 a sample; 70 % of the fp32 rate) and the
// 16-byte weight reads beside them, one for R * 4 multiply-adds.  4,194,301
// samples take 195 us, 16,000,001 take 719 with R = 4 (one sample a thread,
// scalar arithmetic: 319 for the first; two samples with activations as floats,
// 128 registers: 223 and 818; two as pairs: 206 and 745; three 201 and 736;
// four, 8 or 32 units at a time: 199 and 217).
//
// A thread takes its R samples whether they are there or not, so R is the
// smallest of 1, 2 and 4 that covers n in one turn of the grid (one block per
// SM).  On the device, 1,000 to 38,912 samples take 5.4 to 5.6 us
// with R = 1 and 9.9 with 4 (5.2 to 5.5 before any of this, a sample a thread),
// 39,000 to 77,824 take 6.9 with R = 2 and 9.9 with 4 (6.4 to 8.2 before).
constexpr int kForwardUnits = 16, kForwardThreads = 256;
template <int R>
__global__ void __launch_bounds__(kForwardThreads, 1) mlp_forward_kernel(const float* __restrict__ params,
                                                          const float* __restrict__ x, int64_t n,
                                                          float* __restrict__ y) {
    constexpr int J = kForwardUnits;
    __shared__ ForwardParams s;
    load_forward_params(params, s);
    __syncthreads();
    const int64_t T = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r0 < n; r0 += T * R) {
        uint32_t a0[R][kIn / 2], a1[R][kH / 2];
        float out[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int64_t row = r0 + r * T < n ? r0 + r * T : r0;
#pragma unroll
            for (int i = 0; i < kIn; i += 2)
                a0[r][i / 2] = bf16_pair(__ldg(x + row * kIn + i), __ldg(x + row * kIn + i + 1));
            out[r] = 0.f;
        }
#pragma unroll
        for (int j0 = 0; j0 < kH; j0 += J) {
            uint32_t h[R][J / 2];
            layer_pairs<kIn, J, R>(s.w1, s.b1, j0, a0, h);
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int q = 0; q < J / 2; ++q) a1[r][j0 / 2 + q] = h[r][q];
        }
        // output = bf16(W3) . a2 + b3, accumulated in unit order
#pragma unroll 1
        for (int j0 = 0; j0 < kH; j0 += J) {
            uint32_t a2[R][J / 2];
            layer_pairs<kH, J, R>(s.w2, s.b2, j0, a1, a2);
#pragma unroll
            for (int j = 0; j < J; ++j)
#pragma unroll
                for (int r = 0; r < R; ++r) out[r] = fmaf(s.w3[j0 + j], bf16_of(a2[r][j / 2], j & 1), out[r]);
        }
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (r0 + r * T < n) y[r0 + r * T] = out[r] + s.b3;
    }
}

// Gradient of scale * sum_b (y_b - t_b)^2 over n samples, added into grad;
// the sum of squared errors is added into *sse.  Rounding to bf16 passes
// gradients straight through, and the backward pass uses the same bf16
// weights and activations as the forward.
//
// A block takes kTile samples at a time.  First a thread runs one sample
// forward and backward (weights from shared memory, two units to an
// instruction) and leaves its activations and deltas in shared memory; then
// every warp takes 32 of the samples and adds their outer products to sums
// that it keeps in registers over all tiles: lane l holds units 4 (l / 4) ..
// + 3 by inputs 8 (l % 4) .. + 7 of W2's gradient (three reads of 16 bytes for
// 32 multiply-adds), and unit l of the other gradients.  The warps' sums meet
// once, at the end.
//
// Bound: reads of weights and activations from shared memory and the fp32
// multiply-adds (3,552 a sample), about level.  With a thread per parameter
// walking the tile (two reads a multiply-add) and 64 threads a block, 65,536
// samples took 51 us, now 26 (262,144: 149 us, now 63).
//
// Error: a warp's sums run over all of its samples, n / 1,216 terms in a row, and
// then over the blocks by atomics, which set the error: from 4,096 to 16.8 million
// samples each part of the gradient is off by at most 5e-7 of itself (against 64
// bits over the same activations; 9e-7 with a sum a parameter and tile).
constexpr int kTileWarps = kTile / 32;
struct __align__(16) GradShared {
    ForwardParams p;
    float w2r[kH][kRow];        // W2 by unit, for the way back
    float a1[kTile][kRow], a2[kTile][kRow], d1[kTile][kRow], d2[kTile][kRow];
    float a0[kTile][8];         // the inputs, then 1 and dy
    float sum[kMlpParams];
    float sse[kTileWarps];
};

__global__ void __launch_bounds__(kTile) mlp_grad_kernel(const float* __restrict__ params,
                                                         const float* __restrict__ x,
                                                         const float* __restrict__ t, int64_t n,
                                                         float scale, float* grad, float* sse) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    GradShared& s = *reinterpret_cast<GradShared*>(s_raw);
    load_forward_params(params, s.p);
    for (int i = threadIdx.x; i < kH * kH; i += blockDim.x) s.w2r[i / kH][i % kH] = bf16r(params[kOffW2 + i]);
    for (int i = threadIdx.x; i < kMlpParams; i += blockDim.x) s.sum[i] = 0.f;
    __syncthreads();
    const int q = threadIdx.x, lane = q & 31, warp = q >> 5;
    const int j0 = 4 * (lane >> 2), i0 = 8 * (lane & 3);
    f32x2 gw2[4][4];             // W2: units j0 .. + 3, inputs i0 + 2 u, + 1
    f32x2 gw1[4];                // W1 and b1 of unit `lane`: inputs 0 .. 5, then the bias and a term unused
    float gb2 = 0.f, gw3 = 0.f, gb3 = 0.f, sse_local = 0.f;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        gw1[u] = 0ull;
#pragma unroll
        for (int v = 0; v < 4; ++v) gw2[u][v] = 0ull;
    }
    for (int64_t base = (int64_t)blockIdx.x * kTile; base < n; base += (int64_t)gridDim.x * kTile) {
        {
            const int64_t r = base + q;
            const bool valid = r < n;
            float a0[kIn], a1[kH], a2[kH], d2[kH];
#pragma unroll
            for (int i = 0; i < kIn; ++i) a0[i] = valid ? bf16r(x[r * kIn + i]) : 0.f;
            layer_units(s.p.w1, s.p.b1, a0, a1);
            layer_units(s.p.w2, s.p.b2, a1, a2);
            float out = 0.f;
#pragma unroll
            for (int j = 0; j < kH; ++j) out = fmaf(s.p.w3[j], a2[j], out);
            out += s.p.b3;
            const float err = valid ? out - t[r] : 0.f;
            sse_local += err * err;
            const float dy = 2.f * scale * err;
            // relu masks: a > 0 exactly when z > 0 (rounding to bf16 keeps a positive value positive)
#pragma unroll
            for (int j = 0; j < kH; ++j) d2[j] = a2[j] > 0.f ? dy * s.p.w3[j] : 0.f;
#pragma unroll
            for (int j = 0; j < kH; j += 4) {
                *reinterpret_cast<float4*>(&s.a1[q][j]) = make_float4(a1[j], a1[j + 1], a1[j + 2], a1[j + 3]);
                *reinterpret_cast<float4*>(&s.a2[q][j]) = make_float4(a2[j], a2[j + 1], a2[j + 2], a2[j + 3]);
                *reinterpret_cast<float4*>(&s.d2[q][j]) = make_float4(d2[j], d2[j + 1], d2[j + 2], d2[j + 3]);
            }
            *reinterpret_cast<float4*>(&s.a0[q][0]) = make_float4(a0[0], a0[1], a0[2], a0[3]);
            *reinterpret_cast<float4*>(&s.a0[q][4]) = make_float4(a0[4], a0[5], 1.f, dy);
            f32x2 acc[kH / 2];
#pragma unroll
            for (int u = 0; u < kH / 2; ++u) acc[u] = 0ull;
#pragma unroll
            for (int j = 0; j < kH; ++j) {
                const f32x2 dj = pack2(d2[j], d2[j]);
#pragma unroll
                for (int u = 0; u < kH / 2; u += 2) {
                    const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(&s.w2r[j][2 * u]);
                    acc[u] = fma2(w.x, dj, acc[u]);
                    acc[u + 1] = fma2(w.y, dj, acc[u + 1]);
                }
            }
#pragma unroll
            for (int u = 0; u < kH / 2; u += 2) {
                float4 d;
                unpack2(acc[u], d.x, d.y);
                unpack2(acc[u + 1], d.z, d.w);
                d.x = a1[2 * u] > 0.f ? d.x : 0.f;
                d.y = a1[2 * u + 1] > 0.f ? d.y : 0.f;
                d.z = a1[2 * u + 2] > 0.f ? d.z : 0.f;
                d.w = a1[2 * u + 3] > 0.f ? d.w : 0.f;
                *reinterpret_cast<float4*>(&s.d1[q][2 * u]) = d;
            }
        }
        __syncwarp();  // a warp adds up its own 32 samples: no other warp's are read
#pragma unroll 2
        for (int b = warp * 32; b < warp * 32 + 32; ++b) {
            const float4 d = *reinterpret_cast<const float4*>(&s.d2[b][j0]);
            const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(&s.a1[b][i0]);
            const ulonglong2 c = *reinterpret_cast<const ulonglong2*>(&s.a1[b][i0 + 4]);
            const float dd[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const f32x2 e = pack2(dd[u], dd[u]);
                gw2[u][0] = fma2(e, a.x, gw2[u][0]);
                gw2[u][1] = fma2(e, a.y, gw2[u][1]);
                gw2[u][2] = fma2(e, c.x, gw2[u][2]);
                gw2[u][3] = fma2(e, c.y, gw2[u][3]);
            }
            const ulonglong2 f = *reinterpret_cast<const ulonglong2*>(&s.a0[b][0]);
            const ulonglong2 g = *reinterpret_cast<const ulonglong2*>(&s.a0[b][4]);
            const f32x2 e = pack2(s.d1[b][lane], s.d1[b][lane]);
            gw1[0] = fma2(e, f.x, gw1[0]);
            gw1[1] = fma2(e, f.y, gw1[1]);
            gw1[2] = fma2(e, g.x, gw1[2]);
            gw1[3] = fma2(e, g.y, gw1[3]);
            float one, dy;
            unpack2(g.y, one, dy);
            gb2 += s.d2[b][lane];
            gw3 = fmaf(dy, s.a2[b][lane], gw3);
            gb3 += dy;
        }
        __syncwarp();
    }
    for (int o = 16; o > 0; o >>= 1) sse_local += __shfl_xor_sync(0xffffffffu, sse_local, o);
    if (lane == 0) s.sse[warp] = sse_local;
    // the warps' sums, one warp after another
    for (int w = 0; w < kTileWarps; ++w) {
        if (w == warp) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    float lo, hi;
                    unpack2(gw2[u][v], lo, hi);
                    s.sum[kOffW2 + (j0 + u) * kH + i0 + 2 * v] += lo;
                    s.sum[kOffW2 + (j0 + u) * kH + i0 + 2 * v + 1] += hi;
                }
                float lo, hi;
                unpack2(gw1[u], lo, hi);
                if (u < 3) {
                    s.sum[kOffW1 + lane * kIn + 2 * u] += lo;
                    s.sum[kOffW1 + lane * kIn + 2 * u + 1] += hi;
                } else {
                    s.sum[kOffB1 + lane] += lo;
                }
            }
            s.sum[kOffB2 + lane] += gb2;
            s.sum[kOffW3 + lane] += gw3;
            if (lane == 0) s.sum[kOffB3] += gb3;
        }
        __syncthreads();
    }
    for (int p = threadIdx.x; p < kMlpParams; p += blockDim.x) atomicAdd(&grad[p], s.sum[p]);
    if (threadIdx.x == 0) {
        float total = s.sse[0];
        for (int w = 1; w < kTileWarps; ++w) total += s.sse[w];
        atomicAdd(sse, total);
    }
}

// Adam (Kingma & Ba): m <- b1 m + (1-b1) g; v <- b2 v + (1-b2) g^2;
// p <- p - lr * (m / (1-b1^step)) / (sqrt(v / (1-b2^step)) + eps).
__global__ void mlp_adam_kernel(float* params, float* m, float* v, const float* grad, float lr,
                                float b1, float b2, float eps, float c1, float c2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kMlpParams) return;
    const float gi = grad[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    params[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// Per-vertex features (deg = degree; nbr = the neighbours' degrees), every
// degree-like count on a log2 scale, since R-MAT degrees span five decades:
//   f0 = L(deg)                   f1 = floor(log2(1 + deg))
//   f2 = L(floor(sum nbr / deg))  f3 = L(max nbr)
//   f4 = L(sum nbr)               f5 = L(min nbr)
// (f2..f5 = 0 for an isolated vertex; sum nbr counts the walks of length 2).
// L(x) is Mitchell's piecewise-linear log2(1 + x) (J. N. Mitchell, 1962):
// with m = 1 + x = 2^e (1 + f), 0 <= f < 1, L = e + f, f truncated to 16
// bits.  It is exact in integer arithmetic, so every feature is an exact
// float, equal on any machine; it matches log2 at powers of two and is off by
// less than 0.087 elsewhere.
__device__ __forceinline__ float mitchell_log2_1p(unsigned long long x) {
    const unsigned long long m = x + 1ull;
    const int e = 63 - __clzll((long long)m);
    const unsigned long long r = m - (1ull << e);
    const unsigned long long frac = e >= 16 ? (r >> (e - 16)) : (r << (16 - e));
    return (float)((unsigned long long)e * 65536ull + frac) * (1.f / 65536.f);
}

__device__ __forceinline__ void write_features(float* f, int32_t d, unsigned long long sum, int32_t mx,
                                               int32_t mn) {
    float2 x, y, z;
    x.x = mitchell_log2_1p((unsigned long long)d);
    x.y = (float)(31 - __clz(d + 1));
    y = z = make_float2(0.f, 0.f);
    if (d > 0) {
        y.x = mitchell_log2_1p(sum / (unsigned long long)d);
        y.y = mitchell_log2_1p((unsigned long long)mx);
        z.x = mitchell_log2_1p(sum);
        z.y = mitchell_log2_1p((unsigned long long)mn);
    }
    if (((uintptr_t)f & 7u) == 0) {
        float2* o = reinterpret_cast<float2*>(f);
        o[0] = x;
        o[1] = y;
        o[2] = z;
    } else {
        f[0] = x.x; f[1] = x.y; f[2] = y.x; f[3] = y.y; f[4] = z.x; f[5] = z.y;
    }
}

// What the features need of a row's neighbours.
struct RowDegrees {
    unsigned long long sum = 0;
    int32_t mx = 0, mn = 0x7fffffff;
    __device__ __forceinline__ void add(int32_t d) {
        sum += (unsigned long long)d;
        mx = max(mx, d);
        mn = min(mn, d);
    }
    // over the lanes of a group of L
    template <int L>
    __device__ __forceinline__ void combine() {
#pragma unroll
        for (int o = 1; o < L; o <<= 1) {
            sum += __shfl_xor_sync(0xffffffffu, sum, o);
            mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        }
    }
};

// A graph as the features read it.
struct FeatureGraph {
    const int32_t* __restrict__ rowptr;
    const int32_t* __restrict__ colidx;
    int32_t nnz;
    uint32_t col_mis;  // entries from a 32-byte boundary to colidx

    // (one line, most often one sector)
    __device__ __forceinline__ int32_t degree(int32_t w) const { return __ldg(rowptr + w + 1) - __ldg(rowptr + w); }

    // Lane j of a group of L: every L-th 32-byte chunk of the row [b, b + d).
    template <int L>
    __device__ __forceinline__ RowDegrees row(int32_t b, int32_t d, unsigned j) const {
        RowDegrees r;
        for (int64_t off = 8 * (int64_t)j - (int64_t)(((uint32_t)b + col_mis) & 7u); off < d; off += 8 * L) {
            int32_t w[8];
            const int64_t a = b + off;
            if (a >= 0 && a + 8 <= nnz) {
                asm volatile("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                             : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]),
                               "=r"(w[7])
                             : "l"(colidx + a));
            } else {
#pragma unroll
                for (int u = 0; u < 8; ++u) w[u] = a + u >= 0 && a + u < nnz ? __ldg(colidx + a + u) : 0;
            }
            int32_t dw[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) dw[u] = off + u >= 0 && off + u < d ? degree(w[u]) : -1;
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (dw[u] >= 0) r.add(dw[u]);
        }
        return r;
    }
};

// Its own row by each lane, four entries at a time.
__device__ __forceinline__ RowDegrees lane_row(const FeatureGraph& g, int32_t b, int32_t d) {
    RowDegrees r;
    for (int32_t i = 0; i < d; i += 4) {
        int32_t w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) w[u] = i + u < d ? __ldg(g.colidx + b + i + u) : 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) w[u] = i + u < d ? g.degree(w[u]) : -1;
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (w[u] >= 0) r.add(w[u]);
    }
    return r;
}

// The rows of a warp's vertices by four lanes each, eight side by side, in
// `steps` steps: lane s of each group of four holds the row of step s.
__device__ __forceinline__ RowDegrees small_rows(const FeatureGraph& g, unsigned lane, int32_t b, int32_t d, unsigned steps) {
    RowDegrees mine;
#pragma unroll 1
    for (unsigned s = 0; s < steps; ++s) {
        const int src = (int)((lane & ~3u) | s);
        RowDegrees r = g.row<4>(__shfl_sync(0xffffffffu, b, src), __shfl_sync(0xffffffffu, d, src), lane & 3u);
        r.combine<4>();
        if ((lane & 3u) == s) mine = r;
    }
    return mine;
}

// A warp takes 32 vertices.  When none of their rows is longer than 16, each lane
// reads its own; otherwise rows of up to 57 entries are read by 4 lanes, 8 rows
// side by side, rows of up to 121 by 16 lanes and longer ones by the whole warp,
// a 32-byte chunk a lane at a time.  A small graph (rows of 6 entries and more on
// average) is dealt out 8 or 16 vertices a warp (STEPS = 1, 2: in as many steps of
// 8 rows), so that all SMs have some.
//
// Bound: one random L2 sector per entry (the neighbour's row starts; a probe
// that only gathers reaches 208 G/s).  With a thread per short row and the
// longest rows read 32 entries at a time with two waits each, R-MAT-B of 2^22
// vertices took 441 us, now 391; R-MAT-ER 386 us, now 313 (214 G entries/s).
// Six blocks an SM: with four (62 registers) 436 us for the first.
//
// In the natural order of a mesh or band neighbouring lanes gather neighbouring
// words when each has a row of its own: grid of 2,000 x 2,000 67.8 us (thread per
// row, 8 entries at a time), 89.7 (two lanes in chunks), 55.2 now; 12 entries a
// row 43.4, 79.1, 40.1; 26 entries 42.2, 168 (16 lanes), 47.7 (4 lanes, two chunks
// each).  With own rows up to 12 only, a geometric graph of 1M vertices in random
// order (8 a row) takes 46.2 us, not 52.4 (thread per row 53.4), but 200 graphs of
// 4,096 vertices in a batch, 8 a row and near each other, 71, not 66 (65).
// Few vertices: G(3000, 12000) 3.0 us, 5.3 in warps of 32, 3.2 now; K(1500) 111, 132
// and 33.7.
constexpr int kFeatureBlocks = 6;
template <unsigned STEPS>
__global__ void __launch_bounds__(256, kFeatureBlocks) features_kernel(const int32_t* __restrict__ rowptr,
                                                       const int32_t* __restrict__ colidx, int32_t n,
                                                       float* __restrict__ out) {
    constexpr int32_t kOwn = 16, kSmall = 57, kMid = 8 * 16 - 7;
    FeatureGraph g;
    g.rowptr = rowptr;
    g.colidx = colidx;
    g.nnz = __ldg(rowptr + n);
    g.col_mis = (uint32_t)((uintptr_t)colidx >> 2) & 7u;
    const unsigned lane = threadIdx.x & 31u;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t W = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const unsigned steps = STEPS == 4u || g.nnz / 6 >= n ? STEPS : 4u;
    const unsigned rows = 8u * steps, own = (lane >> 2) * steps + (lane & 3u);
    for (int64_t base = gw * rows; base < n; base += W * rows) {
        const int64_t v = base + own;
        const bool valid = (lane & 3u) < steps && v < n;
        const int32_t b = valid ? __ldg(rowptr + v) : 0, d = valid ? __ldg(rowptr + v + 1) - b : 0;
        RowDegrees mine;
        if (steps == 4u && __all_sync(0xffffffffu, d <= kOwn)) {
            mine = lane_row(g, b, d);
        } else {
            mine = small_rows(g, lane, b, d <= kSmall ? d : 0, steps);
        }
        unsigned mid = __ballot_sync(0xffffffffu, d > kSmall && d <= kMid);
        while (mid) {
            // the lower half of the warp takes the first of them, the upper half the second
            const unsigned rest = mid & (mid - 1);
            const unsigned from = lane < 16u ? mid : rest;
            const int o = __ffs(from) - 1;
            const int32_t ob = __shfl_sync(0xffffffffu, b, o & 31), od = __shfl_sync(0xffffffffu, d, o & 31);
            RowDegrees r = g.row<16>(ob, from ? od : 0, lane & 15u);
            r.combine<16>();
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                RowDegrees x;
                x.sum = __shfl_sync(0xffffffffu, r.sum, 16 * h);
                x.mx = __shfl_sync(0xffffffffu, r.mx, 16 * h);
                x.mn = __shfl_sync(0xffffffffu, r.mn, 16 * h);
                const unsigned set = h == 0 ? mid : rest;
                if (set && (int)lane == __ffs(set) - 1) mine = x;
            }
            mid = rest & (rest - 1);
        }
        unsigned big = __ballot_sync(0xffffffffu, d > kMid);
        while (big) {
            const int o = __ffs(big) - 1;
            big &= big - 1;
            RowDegrees r = g.row<32>(__shfl_sync(0xffffffffu, b, o), __shfl_sync(0xffffffffu, d, o), lane);
            r.combine<32>();
            if ((int)lane == o) mine = r;
        }
        if (valid) write_features(out + v * 6, d, mine.sum, mine.mx, mine.mn);
    }
}

// Score -> key with the same order: smaller score = smaller key (higher
// precedence).  IEEE order of floats is the order of their bit patterns
// with the sign bit flipped (positives) or all bits flipped (negatives).
__global__ void keys_kernel(const float* __restrict__ y, int64_t n, uint32_t* __restrict__ keys) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        float f = y[i];
        if (f != f) f = __int_as_float(0x7f800000);  // NaN sorts last
        if (f == 0.f) f = 0.f;                        // -0 and +0 alike
        const uint32_t u = (uint32_t)__float_as_int(f);
        keys[i] = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    }
}

int grid_for(int64_t items, int per_block, int cap) {
    int64_t g = (items + per_block - 1) / per_block;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (int)g;
}

int sm_count() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 148;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 148;
    return sms;
}

int check_launch() {
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? GC_OK : GC_ERR_CUDA;
}

}  // namespace

extern "C" {

int gc_features(const int32_t* rowptr, const int32_t* colidx, int32_t n, float* features, void* stream) {
    if (n < 0 || (n > 0 && (!rowptr || !features))) return GC_ERR_INVALID;
    if (n == 0) return GC_OK;
    const int sms = sm_count();
    const int64_t warps = (int64_t)sms * kFeatureBlocks * 8;
    const cudaStream_t s = (cudaStream_t)stream;
    if (n <= 8 * warps) {
        features_kernel<1><<<grid_for((int64_t)n, 64, sms * 16), 256, 0, s>>>(rowptr, colidx, n, features);
    } else if (n <= 16 * warps) {
        features_kernel<2><<<grid_for((int64_t)n, 128, sms * 16), 256, 0, s>>>(rowptr, colidx, n, features);
    } else {
        features_kernel<4><<<grid_for((int64_t)n, 256, sms * 16), 256, 0, s>>>(rowptr, colidx, n, features);
    }
    return check_launch();
}

int gc_mlp_forward(const float* params, const float* x, int64_t n, float* y, void* stream) {
    if (n < 0 || !params || (n > 0 && (!x || !y))) return GC_ERR_INVALID;
    if (n == 0) return GC_OK;
    const cudaStream_t s = (cudaStream_t)stream;
    const int most = sm_count();
    const int64_t turn = (int64_t)most * kForwardThreads;
    if (n <= turn) {
        mlp_forward_kernel<1><<<grid_for(n, kForwardThreads, most), kForwardThreads, 0, s>>>(params, x, n, y);
    } else if (n <= 2 * turn) {
        mlp_forward_kernel<2><<<most, kForwardThreads, 0, s>>>(params, x, n, y);
    } else {
        mlp_forward_kernel<4><<<most, kForwardThreads, 0, s>>>(params, x, n, y);
    }
    return check_launch();
}

int gc_mlp_grad(const float* params, const float* x, const float* t, int64_t n, float scale, float* grad,
                float* sse, void* stream) {
    if (n < 0 || !params || !grad || !sse || (n > 0 && (!x || !t))) return GC_ERR_INVALID;
    if (n == 0) return GC_OK;
    // (two blocks an SM: their shared memory)
    if (cudaFuncSetAttribute(mlp_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GradShared)) !=
        cudaSuccess) {
        (void)cudaGetLastError();
        return GC_ERR_CUDA;
    }
    mlp_grad_kernel<<<grid_for(n, kTile, sm_count() * 2), kTile, sizeof(GradShared), (cudaStream_t)stream>>>(
        params, x, t, n, scale, grad, sse);
    return check_launch();
}

int gc_mlp_adam(float* params, float* m, float* v, const float* grad, int32_t step, float lr, float beta1,
                float beta2, float eps, void* stream) {
    if (!params || !m || !v || !grad || step < 1) return GC_ERR_INVALID;
    const float c1 = 1.f - (float)std::pow((double)beta1, (double)step);
    const float c2 = 1.f - (float)std::pow((double)beta2, (double)step);
    mlp_adam_kernel<<<(kMlpParams + 255) / 256, 256, 0, (cudaStream_t)stream>>>(params, m, v, grad, lr, beta1,
                                                                                 beta2, eps, c1, c2);
    return check_launch();
}

int gc_priority_keys(const float* scores, int64_t n, uint32_t* keys, void* stream) {
    if (n < 0 || (n > 0 && (!scores || !keys))) return GC_ERR_INVALID;
    if (n == 0) return GC_OK;
    keys_kernel<<<grid_for(n, 256, sm_count() * 8), 256, 0, (cudaStream_t)stream>>>(scores, n, keys);
    return check_launch();
}

int gc_mlp_train_step(float* params, float* m, float* v, float* grad, float* sse, const float* x,
                      const float* t, int64_t n, int32_t step, float lr, float beta1, float beta2, float eps,
                      void* stream) {
    if (n < 1 || !params || !m || !v || !grad || !sse || !x || !t || step < 1) return GC_ERR_INVALID;
    const cudaStream_t st = (cudaStream_t)stream;
    if (cudaMemsetAsync(grad, 0, sizeof(float) * kMlpParams, st) != cudaSuccess) return GC_ERR_CUDA;
    if (cudaMemsetAsync(sse, 0, sizeof(float), st) != cudaSuccess) return GC_ERR_CUDA;
    const int rc = gc_mlp_grad(params, x, t, n, 1.f / (float)n, grad, sse, stream);
    if (rc != GC_OK) return rc;
    return gc_mlp_adam(params, m, v, grad, step, lr, beta1, beta2, eps, stream);
}

int gc_mlp_param_count(void) { return kMlpParams; }

}  // extern "C"
