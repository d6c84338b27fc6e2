// FP32 tile MLP on CUDA cores (reference-precision path of every network in the renderer).
#pragma once

#include "nedf_device.cuh"

namespace nedf {

constexpr int kTileRows = 64;        // rows per SIMT MLP tile
constexpr int kXStride = kTileRows + 4;
constexpr int kThreads = 256;

// ---------------------------------------------------------------------------------------------
// FP32 tile MLP on CUDA cores.  X is a feature-major tile [K][kXStride] in shared memory;
// a layer overwrites it with its N outputs.  256 threads: 8 row groups x 32 column groups, each thread
// 8 rows x N/32 columns, every output one FMA chain over k in ascending order from its bias.
//
// Weights come through shared memory in double-buffered blocks of kWBlock inputs by 16-byte cp.async: Wt is
// 16-byte aligned (a layer's K N + N floats are a multiple of 4 at every width, and types are strided so).  A warp holds 4 row x 8
// column groups, so that one k step at N = 256 is 64 FMAs for four 16-byte loads of one wavefront each: the
// FMA pipe is the bound.  (Four rows a thread with the weights read by 4-byte global loads took 17 loads
// for the same 64 FMAs: 48-instance FP32 frame at 256 x 256 2.58 -> 1.81 ms, 49 k queries of an 8 x 128
// network 687 -> 346 us.)
// ---------------------------------------------------------------------------------------------
constexpr int kWBlock = 8;

template <int N>
__device__ __forceinline__ void load_weights_f32(float *dst, const float *__restrict__ src, int rows)
{
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    for (int e = threadIdx.x; e < rows * (N / 4); e += kThreads)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d + 16u * e), "l"(src + 4 * e) : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
}

template <int N>
__device__ __forceinline__ void dense_f32(float *X, int K, const float *__restrict__ Wt,
                                          const float *__restrict__ b, bool relu)
{
    constexpr int NC = N / 32;                       // columns per thread: quads 128 apart (or one pair)
    constexpr int NV = NC < 4 ? NC : 4;              // ... read NV at a time
    __shared__ __align__(16) float ws[2][kWBlock * N];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cg = (warp & 3) * 8 + (lane & 7), rg = (warp >> 2) * 4 + (lane >> 3);
    float acc[8][NC];
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        const float bj = __ldg(b + (j / NV) * 128 + cg * NV + j % NV);
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i][j] = bj;
    }
    const int nb = (K + kWBlock - 1) / kWBlock;
    load_weights_f32<N>(ws[0], Wt, min(kWBlock, K));
    for (int blk = 0; blk < nb; ++blk) {
        const int k0 = blk * kWBlock, kc = min(kWBlock, K - k0);
        if (blk + 1 < nb) {
            load_weights_f32<N>(ws[(blk + 1) & 1], Wt + (size_t)(k0 + kWBlock) * N, min(kWBlock, K - k0 - kWBlock));
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const float *xp = X + (size_t)k0 * kXStride + rg * 8, *wp = ws[blk & 1] + cg * NV;
        auto step = [&](int k) {
            const float4 x0 = *reinterpret_cast<const float4 *>(xp + k * kXStride);
            const float4 x1 = *reinterpret_cast<const float4 *>(xp + k * kXStride + 4);
            const float x[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
            float w[NC];
#pragma unroll
            for (int q = 0; q < NC / NV; ++q) {
                if (NV == 4) {
                    const float4 v = *reinterpret_cast<const float4 *>(wp + k * N + q * 128);
                    w[q * NV] = v.x; w[q * NV + 1] = v.y; w[q * NV + 2 < NC ? q * NV + 2 : 0] = v.z; w[q * NV + 3 < NC ? q * NV + 3 : 0] = v.w;
                } else {
                    const float2 v = *reinterpret_cast<const float2 *>(wp + k * N);
                    w[0] = v.x; w[NC > 1 ? 1 : 0] = v.y;
                }
            }
#pragma unroll
            for (int j = 0; j < NC; ++j)
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[i][j] = fmaf(x[i], w[j], acc[i][j]);
        };
        if (kc == kWBlock) {
#pragma unroll
            for (int k = 0; k < kWBlock; ++k) step(k);
        } else {
            for (int k = 0; k < kc; ++k) step(k);
        }
        __syncthreads();                             // the buffer is refilled, and X overwritten, after every read
    }
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        float4 *dst = reinterpret_cast<float4 *>(X + (size_t)((j / NV) * 128 + cg * NV + j % NV) * kXStride + rg * 8);
        if (relu)
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[i][j] = fmaxf(acc[i][j], 0.0f);
        dst[0] = make_float4(acc[0][j], acc[1][j], acc[2][j], acc[3][j]);
        dst[1] = make_float4(acc[4][j], acc[5][j], acc[6][j], acc[7][j]);
    }
    __syncthreads();
}

template <int N>
__device__ __forceinline__ void mlp_hidden_f32(float *X, int K0, int hidden, const float *w)
{
    // layer 0: K0 -> N, then hidden-1 layers N -> N; w advanced past each (Wt, b)
    dense_f32<N>(X, K0, w, w + (size_t)K0 * N, true);
    w += (size_t)K0 * N + N;
    for (int l = 1; l < hidden; ++l) {
        dense_f32<N>(X, N, w, w + (size_t)N * N, true);
        w += (size_t)N * N + N;
    }
}

// Output layer with n_out <= 4 outputs: y[r][o] for the tile's rows.
__device__ __forceinline__ void out_layer_f32(const float *X, int K, const float *__restrict__ Wt,
                                              const float *__restrict__ b, int n_out, float (*y)[4])
{
    for (int e = threadIdx.x; e < kTileRows * n_out; e += blockDim.x) {
        int r = e / n_out, o = e - r * n_out;
        float acc = __ldg(b + o);
        for (int k = 0; k < K; ++k) acc = fmaf(X[k * kXStride + r], __ldg(Wt + k * n_out + o), acc);
        y[r][o] = acc;
    }
    __syncthreads();
}

// gamma(x) of an n-wide input with L frequencies written as features [f0, f0 + n (1 + 2L)).
__device__ __forceinline__ float posenc_feature(const float *x, int n, int L, int f)
{
    if (f < n) return x[f];
    f -= n;
    int blk = f / n, c = f - blk * n;
    if (blk < L) return sinf(ldexpf(x[c], blk));
    return cosf(ldexpf(x[c], blk - L));
}

}  // namespace nedf
