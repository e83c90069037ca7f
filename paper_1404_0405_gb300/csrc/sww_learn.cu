// Learned refinement proposal: per-patch features of the wavelet coefficients, a
// two-layer perceptron (BF16 weights, FP32 accumulation) that proposes patches for
// the next mask, and its training kernels (loss gradient and Adam).  The exact
// threshold rules still build the mask; a proposed patch only adds its nodes to
// the set T before the graded closure, so the plain criterion keeps the last word.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <type_traits>

#include "sww_core.cuh"
#include "sww_kernels.h"
#include "sww_internal.h"
#include "sww_learn.h"

namespace sww {

namespace {

__device__ __forceinline__ int64_t lgid() { return int64_t(blockIdx.x) * blockDim.x + threadIdx.x; }

__device__ __forceinline__ float bf16_round(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// ------------------------------------------------------------------ training

// The perceptron's weights in FP32 (W1 and w2 rounded to BF16 and widened: the values
// the products use), in shared memory: W1[f][h], b1, w2, b2.
struct __align__(16) WeightsF {
    float w1[NF][NH], b1[NH], w2[NH], b2;
};

// by the whole block, one parameter a thread (a single thread's 321 dependent loads
// and conversions took most of k_mlp_predict's 9.7 us on 54 565 samples)
__device__ __forceinline__ void stage_weights(const float* __restrict__ params, WeightsF& w) {
    float* dst = reinterpret_cast<float*>(&w);   // the members in the order of params
    for (int k = threadIdx.x; k < MLP_PARAMS; k += blockDim.x) {
        const bool bias = (k >= NF * NH && k < NF * NH + NH) || k == MLP_PARAMS - 1;
        dst[k] = bias ? params[k] : bf16_round(params[k]);
    }
    __syncthreads();
}

// Two FP32 numbers in one 64-bit register: fma.rn.f32x2 does two multiply-adds, each
// rounded as fmaf rounds it, in one issue slot.
using F2 = unsigned long long;
__device__ __forceinline__ F2 pack2(float a, float b) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 unpack2(F2 x) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(x));
    return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// Logits of K samples of one thread (xx[k][f]: feature f of sample k, twice), with the
// operations of mlp_logit in its order: hidden units in pairs by f32x2, and each
// 16-byte load of four weights serves K samples.
template <int K>
__device__ __forceinline__ void logits(const WeightsF& w, const F2 (&xx)[K][NF], float (&out)[K]) {
#pragma unroll
    for (int k = 0; k < K; ++k) out[k] = w.b2;
#pragma unroll 2
    for (int h = 0; h < NH; h += 4) {
        const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(&w.b1[h]);
        F2 z[K][2];
#pragma unroll
        for (int k = 0; k < K; ++k) z[k][0] = b.x, z[k][1] = b.y;
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(&w.w1[f][h]);
#pragma unroll
            for (int k = 0; k < K; ++k) z[k][0] = fma2(xx[k][f], v.x, z[k][0]), z[k][1] = fma2(xx[k][f], v.y, z[k][1]);
        }
        const float4 v2 = *reinterpret_cast<const float4*>(&w.w2[h]);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const float2 p = unpack2(z[k][0]), q = unpack2(z[k][1]);
            out[k] = fmaf(fmaxf(p.x, 0.f), v2.x, out[k]);
            out[k] = fmaf(fmaxf(p.y, 0.f), v2.y, out[k]);
            out[k] = fmaf(fmaxf(q.x, 0.f), v2.z, out[k]);
            out[k] = fmaf(fmaxf(q.y, 0.f), v2.w, out[k]);
        }
    }
}

// the features of sample i, each as an (x, x) pair; zero past the end.  X rows are
// NF floats; `vec`: X is 16-byte aligned (two 16-byte loads a row)
__device__ __forceinline__ void load_row(const float* __restrict__ X, int64_t i, int64_t n, bool vec, float (&x)[NF]) {
    static_assert(NF == 8, "row loads");
    if (i >= n) {
#pragma unroll
        for (int f = 0; f < NF; ++f) x[f] = 0.f;
    } else if (vec) {
        const float4 a = *reinterpret_cast<const float4*>(X + i * NF), b = *reinterpret_cast<const float4*>(X + i * NF + 4);
        x[0] = a.x, x[1] = a.y, x[2] = a.z, x[3] = a.w, x[4] = b.x, x[5] = b.y, x[6] = b.z, x[7] = b.w;
    } else {
#pragma unroll
        for (int f = 0; f < NF; ++f) x[f] = X[i * NF + f];
    }
}

// Partial sums of the weighted binary cross-entropy and its gradient with respect to
// the FP32 master parameters (the BF16 rounding is passed straight through), one row
// of MLP_PARAMS + 1 sums per block.
//
// About 600 multiply-adds a sample against 36 bytes read: bound by the FP32 pipe's
// issue slots (15 us for a million samples if nothing else were issued).  A warp
// takes tiles of 64 samples by itself, no block barrier between them:
//   forward   lane = two samples, the logit as in mlp_logit; features and d loss /
//             d logit left in shared memory, transposed;
//   backward  lane = one hidden unit: z again (eight multiply-adds are cheaper than
//             passing 32 activations through shared memory), then the unit's ten sums in
//             registers, even and odd samples in the halves of an f32x2.
// A tile's sums (chains of 32) join the lane's totals, so no chain of additions is long;
// warps and blocks are added in FP64.  A million samples: 388 us with one thread per
// parameter reading activations from shared memory, 51 us now.
constexpr int GRAD_WARPS = 20, GRAD_TPB = 32 * GRAD_WARPS, TILE_S = 64;

__global__ void __launch_bounds__(GRAD_TPB, 1)
    k_mlp_grad(const float* __restrict__ X, const float* __restrict__ y, int64_t n, const float* __restrict__ params,
               float pos_w, float* __restrict__ part, int vec) {
    constexpr int NP = MLP_PARAMS + 1;
    __shared__ WeightsF w;
    __shared__ __align__(16) float tile[GRAD_WARPS][NF + 1][TILE_S];   // features by sample, then d loss / d logit
    static_assert(NP <= (NF + 1) * TILE_S, "a warp's sums reuse its tile");
    stage_weights(params, w);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float(*xs)[TILE_S] = tile[warp];
    // this lane's hidden unit, each value twice
    F2 wv[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) wv[f] = pack2(w.w1[f][lane], w.w1[f][lane]);
    const F2 bv = pack2(w.b1[lane], w.b1[lane]);
    const float w2 = w.w2[lane];
    float tot[NF + 2], tg = 0.f, tl = 0.f;   // W1 column, b1, w2; sums of d loss / d logit and of the loss
#pragma unroll
    for (int r = 0; r < NF + 2; ++r) tot[r] = 0.f;
    const int64_t tiles = (n + TILE_S - 1) / TILE_S;
    for (int64_t t = int64_t(warp) * gridDim.x + blockIdx.x; t < tiles; t += int64_t(GRAD_WARPS) * gridDim.x) {
        {
            F2 xx[2][NF];
            float lg[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                float x[NF];
                load_row(X, t * TILE_S + 32 * k + lane, n, vec != 0, x);
#pragma unroll
                for (int f = 0; f < NF; ++f) xs[f][32 * k + lane] = x[f], xx[k][f] = pack2(x[f], x[f]);
            }
            logits<2>(w, xx, lg);
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int64_t i = t * TILE_S + 32 * k + lane;
                float g = 0.f;
                if (i < n) {
                    const float logit = lg[k], tt = y[i];
                    const float p = 1.f / (1.f + expf(-logit));
                    g = pos_w * tt * (p - 1.f) + (1.f - tt) * p;   // d loss / d logit
                    const float sp = logit > 0 ? logit + log1pf(expf(-logit)) : log1pf(expf(logit));   // softplus
                    tl += pos_w * tt * (sp - logit) + (1.f - tt) * sp;
                    tg += g;
                }
                xs[NF][32 * k + lane] = g;
            }
        }
        __syncwarp();
        F2 acc[NF + 2];
#pragma unroll
        for (int r = 0; r < NF + 2; ++r) acc[r] = 0ull;
        // the last tile's samples past the end take no part whatever the weights hold
        const int m = int(n - t * TILE_S < TILE_S ? n - t * TILE_S : TILE_S);
        auto backward = [&](auto whole, int s) {
            auto in = [&](int q) { return decltype(whole)::value || s + q < m; };
            ulonglong2 x[NF];   // samples s, s + 1 and s + 2, s + 3
#pragma unroll
            for (int f = 0; f < NF; ++f) x[f] = *reinterpret_cast<const ulonglong2*>(&xs[f][s]);
            const ulonglong2 gg = *reinterpret_cast<const ulonglong2*>(&xs[NF][s]);
            F2 z0 = bv, z1 = bv;
#pragma unroll
            for (int f = 0; f < NF; ++f) z0 = fma2(x[f].x, wv[f], z0), z1 = fma2(x[f].y, wv[f], z1);
            const float2 ga = unpack2(gg.x), gb = unpack2(gg.y);
            float2 za = unpack2(z0), zb = unpack2(z1);
            if (!in(0)) za.x = 0.f;
            if (!in(1)) za.y = 0.f;
            if (!in(2)) zb.x = 0.f;
            if (!in(3)) zb.y = 0.f;
            const F2 d0 = pack2(za.x > 0.f ? ga.x * w2 : 0.f, za.y > 0.f ? ga.y * w2 : 0.f);
            const F2 d1 = pack2(zb.x > 0.f ? gb.x * w2 : 0.f, zb.y > 0.f ? gb.y * w2 : 0.f);
#pragma unroll
            for (int f = 0; f < NF; ++f) acc[f] = fma2(d1, x[f].y, fma2(d0, x[f].x, acc[f]));
            acc[NF] = add2(add2(acc[NF], d0), d1);
            acc[NF + 1] = fma2(gg.x, pack2(fmaxf(za.x, 0.f), fmaxf(za.y, 0.f)), acc[NF + 1]);
            acc[NF + 1] = fma2(gg.y, pack2(fmaxf(zb.x, 0.f), fmaxf(zb.y, 0.f)), acc[NF + 1]);
        };
        if (m == TILE_S) {
#pragma unroll 2
            for (int s = 0; s < TILE_S; s += 4) backward(std::true_type(), s);
        } else {
#pragma unroll 1
            for (int s = 0; s < m; s += 4) backward(std::false_type(), s);
        }
#pragma unroll
        for (int r = 0; r < NF + 2; ++r) {
            const float2 v = unpack2(acc[r]);
            tot[r] += v.x + v.y;
        }
        __syncwarp();   // the next tile's features overwrite this one's
    }
    for (int o = 16; o > 0; o >>= 1) tg += __shfl_xor_sync(0xffffffffu, tg, o), tl += __shfl_xor_sync(0xffffffffu, tl, o);
    __syncwarp();
    float* row = &xs[0][0];   // the warp's NP sums, in the order of params
#pragma unroll
    for (int f = 0; f < NF; ++f) row[f * NH + lane] = tot[f];
    row[NF * NH + lane] = tot[NF];
    row[NF * NH + NH + lane] = tot[NF + 1];
    if (lane == 0) row[MLP_PARAMS - 1] = tg, row[MLP_PARAMS] = tl;
    __syncthreads();
    for (int k = threadIdx.x; k < NP; k += GRAD_TPB) {
        double s = 0;
        for (int q = 0; q < GRAD_WARPS; ++q) s += double((&tile[q][0][0])[k]);
        part[int64_t(blockIdx.x) * NP + k] = float(s);
    }
}

// out[k] = sum of the blocks' rows / n: 32 outputs a block, eight threads an output
// (one thread an output waited for 256 loads in turn: 24 us; 5.5 us now)
__global__ void __launch_bounds__(256) k_mlp_grad_final(const float* __restrict__ part, int nblk, int64_t n,
                                                        float* __restrict__ out) {
    constexpr int NP = MLP_PARAMS + 1;
    __shared__ double sh[8][32];
    const int c = threadIdx.x & 31, r = threadIdx.x >> 5, k = int(blockIdx.x) * 32 + c;
    double s = 0;
    if (k < NP) {
#pragma unroll 8
        for (int b = r; b < nblk; b += 8) s += double(part[int64_t(b) * NP + k]);
    }
    sh[r][c] = s;
    __syncthreads();
    if (r == 0 && k < NP) {
        for (int q = 1; q < 8; ++q) s += sh[q][c];
        out[k] = float(s / double(n > 0 ? n : 1));
    }
}

__global__ void k_adam(float* __restrict__ params, const float* __restrict__ grad, float* __restrict__ m,
                       float* __restrict__ v, int t, float lr, float b1, float b2, float eps) {
    const int k = int(lgid());
    if (k >= MLP_PARAMS) return;
    const float g = grad[k];
    m[k] = b1 * m[k] + (1.f - b1) * g;
    v[k] = b2 * v[k] + (1.f - b2) * g * g;
    const float mh = m[k] / (1.f - powf(b1, float(t)));
    const float vh = v[k] / (1.f - powf(b2, float(t)));
    params[k] -= lr * mh / (sqrtf(vh) + eps);
}

// One thread a sample: 32 bytes read for 290 multiply-adds, but a usual call (the
// patches of one adaptation) is a single wave, bound by the latency of staging the
// weights and of the logit's chain of 32.  54 565 samples: 9.7 us with the weights
// staged by one thread, 3.3 us now.
__global__ void __launch_bounds__(256) k_mlp_predict(const float* __restrict__ X, int64_t n,
                                                     const float* __restrict__ params, float* __restrict__ out, int vec) {
    __shared__ WeightsF w;
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    int64_t i = lgid();
    float x[NF];
    load_row(X, i, n, vec != 0, x);   // in flight while the weights are staged
    stage_weights(params, w);
    while (i < n) {
        F2 xx[1][NF];
#pragma unroll
        for (int f = 0; f < NF; ++f) xx[0][f] = pack2(x[f], x[f]);
        load_row(X, i + stride, n, vec != 0, x);
        float lg[1];
        logits<1>(w, xx, lg);
        out[i] = 1.f / (1.f + expf(-lg[0]));
        i += stride;
    }
}

}  // namespace

MlpWeights mlp_weights(const float* params) {
    MlpWeights w{};
    for (int k = 0; k < NF * NH; ++k) w.w1[k] = __float2bfloat16_rn(params[k]);
    for (int h = 0; h < NH; ++h) w.b1[h] = params[NF * NH + h];
    for (int h = 0; h < NH; ++h) w.w2[h] = __float2bfloat16_rn(params[NF * NH + NH + h]);
    w.b2 = params[NF * NH + 2 * NH];
    return w;
}

// 16-byte row loads need an aligned X (rows are 32 bytes)
static int row_vec(const float* X) { return (reinterpret_cast<uintptr_t>(X) & 15) == 0; }

void launch_mlp_grad(const float* X, const float* y, int64_t n, const float* params, float pos_w, float* work,
                     float* out, cudaStream_t s) {
    // a block an SM, fewer when there are fewer tiles (the tiles of a small set go to
    // different SMs first); work holds MLP_GRAD_BLOCKS rows
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        nsm = 1;
    const int64_t tiles = (n + TILE_S - 1) / TILE_S;
    const int blocks = int(std::max<int64_t>(1, std::min<int64_t>(tiles, std::min(nsm, MLP_GRAD_BLOCKS))));
    count_launch(2);
    k_mlp_grad<<<blocks, GRAD_TPB, 0, s>>>(X, y, n, params, pos_w, work, row_vec(X));
    k_mlp_grad_final<<<blocks_for(MLP_PARAMS + 1, 32), 256, 0, s>>>(work, blocks, n, out);
}

void launch_adam(float* params, const float* grad, float* m, float* v, int t, float lr, cudaStream_t s) {
    count_launch(1);
    k_adam<<<blocks_for(MLP_PARAMS, 128), 128, 0, s>>>(params, grad, m, v, t, lr, 0.9f, 0.999f, 1e-8f);
}

void launch_mlp_predict(const float* X, int64_t n, const float* params, float* out, cudaStream_t s) {
    if (n <= 0) return;
    count_launch(1);
    k_mlp_predict<<<unsigned(std::min<int64_t>(blocks_for(n, 256), 4096)), 256, 0, s>>>(X, n, params, out, row_vec(X));
}

}  // namespace sww

// ------------------------------------------------------------------ C ABI (training)

namespace {
int learn_fail(int code, const char* msg) { return sww::set_error(code, msg); }
}  // namespace

extern "C" int sww_mlp_loss_grad(const float* X, const float* y, int64_t n, const float* params, float pos_weight,
                                 float* work, float* out, void* stream) {
    if (!X || !y || !params || !work || !out || n < 0) return learn_fail(SWW_E_ARG, "sww_mlp_loss_grad: bad argument");
    sww::launch_mlp_grad(X, y, n, params, pos_weight, work, out, static_cast<cudaStream_t>(stream));
    if (cudaGetLastError() != cudaSuccess) return learn_fail(SWW_E_CUDA, "sww_mlp_loss_grad: launch failed");
    return SWW_OK;
}

extern "C" int sww_mlp_adam(float* params, const float* grad, float* m, float* v, int t, float lr, void* stream) {
    if (!params || !grad || !m || !v || t < 1) return learn_fail(SWW_E_ARG, "sww_mlp_adam: bad argument");
    sww::launch_adam(params, grad, m, v, t, lr, static_cast<cudaStream_t>(stream));
    if (cudaGetLastError() != cudaSuccess) return learn_fail(SWW_E_CUDA, "sww_mlp_adam: launch failed");
    return SWW_OK;
}

extern "C" int sww_mlp_predict(const float* X, int64_t n, const float* params, float* out, void* stream) {
    if (!X || !params || !out || n < 0) return learn_fail(SWW_E_ARG, "sww_mlp_predict: bad argument");
    sww::launch_mlp_predict(X, n, params, out, static_cast<cudaStream_t>(stream));
    if (cudaGetLastError() != cudaSuccess) return learn_fail(SWW_E_CUDA, "sww_mlp_predict: launch failed");
    return SWW_OK;
}
