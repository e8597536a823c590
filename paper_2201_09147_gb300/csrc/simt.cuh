// Building blocks of the FP32 SIMT kernels (inference and training): a
// 128-row activation tile held transposed in shared memory and a
// register-tiled GEMM against a weight matrix streamed from global memory.
#pragma once

#include <cstdint>

#include "common.cuh"

namespace sdfnn {
namespace simt {

constexpr int kSimtThreads = 256;
constexpr int kChunkK = 16;  // rows of W^T staged per step

// Activation tile X^T[k][r] (k = feature, r = row) with 4-float groups of r
// permuted by (k / 4) % 8 to keep the epilogue's column stores conflict free.
__device__ __forceinline__ int xt_index(int k, int r) { return k * 128 + ((((r >> 2) ^ ((k >> 2) & 7))) << 2) + (r & 3); }


// One k of acc[i][j] += X[r0 + i][k] * W[n_j][k], wk = row k of W^T from the
// thread's first feature on (its groups of four features are 64 apart).
// Packed FMAs (two lanes an instruction, each rounded as a scalar FMA in the
// same order): the FMA pipe then takes half the issue slots, and the loads and
// address work fit beside it.  One group pairs rows (four weights to
// duplicate), more pair features (eight activations).
template <int G>
__device__ __forceinline__ void simt_step(const float* __restrict__ xt, const float* __restrict__ wk,
                                          float (&acc)[8][4 * G], int k, int r0) {
    const int sw = (k >> 2) & 7;
    const float4 xa = *reinterpret_cast<const float4*>(xt + k * 128 + ((((r0 >> 2)) ^ sw) << 2));
    const float4 xb = *reinterpret_cast<const float4*>(xt + k * 128 + ((((r0 >> 2) + 1) ^ sw) << 2));
    if (G == 1) {
        const float2 x2[4] = {make_float2(xa.x, xa.y), make_float2(xa.z, xa.w), make_float2(xb.x, xb.y),
                              make_float2(xb.z, xb.w)};
        const float4 wv = *reinterpret_cast<const float4*>(wk);
        const float w4[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 r = __ffma2_rn(x2[i], make_float2(w4[e], w4[e]), make_float2(acc[2 * i][e], acc[2 * i + 1][e]));
                acc[2 * i][e] = r.x;
                acc[2 * i + 1][e] = r.y;
            }
    } else {
        const float x[8] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y, xb.z, xb.w};
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const float4 wv = *reinterpret_cast<const float4*>(wk + g * 64);
            const float2 w2[2] = {make_float2(wv.x, wv.y), make_float2(wv.z, wv.w)};
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int j = g * 4 + 2 * e;
                    const float2 r = __ffma2_rn(make_float2(x[i], x[i]), w2[e], make_float2(acc[i][j], acc[i][j + 1]));
                    acc[i][j] = r.x;
                    acc[i][j + 1] = r.y;
                }
        }
    }
}

// acc[i][j] = sum_k X[r0 + i][k] * W[n_j][k] for the thread's 8 rows and its
// features n_j = feat_of(4 g0 + j, fg).  W^T is streamed from global memory (L2
// resident) through a double-buffered shared-memory stage by all T threads;
// T / 256 threads share a row and group of lanes, each with its own feature
// groups from g0 on.  A warp with on = false (warp-uniform) only helps staging.
// Starts and ends with the block synchronised.
template <int W, int T = kSimtThreads>
__device__ __forceinline__ void simt_gemm(const float* __restrict__ xt, const float* __restrict__ wt_g,
                                          float* __restrict__ ws, float (&acc)[8][W / 16 * kSimtThreads / T], int r0,
                                          int fg, int g0 = 0, bool on = true) {
    constexpr int G = W / 64 * kSimtThreads / T;  // feature groups per thread
    constexpr int NCH = W / kChunkK;
    constexpr int F4_PER_CHUNK = kChunkK * W / 4;
    constexpr int PER_T = F4_PER_CHUNK / T;
    static_assert(PER_T >= 1, "chunk too small");
    const int tid = threadIdx.x;
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4 * G; ++j) acc[i][j] = 0.0f;

    const float4* src = reinterpret_cast<const float4*>(wt_g);
    float4 pre[PER_T];
#pragma unroll
    for (int u = 0; u < PER_T; ++u) pre[u] = __ldg(src + tid + u * T);
#pragma unroll
    for (int u = 0; u < PER_T; ++u) reinterpret_cast<float4*>(ws)[tid + u * T] = pre[u];
    __syncthreads();

    for (int c = 0; c < NCH; ++c) {
        const float* wsc = ws + (c & 1) * kChunkK * W + g0 * 64 + fg * 4;
        if (c + 1 < NCH) {
#pragma unroll
            for (int u = 0; u < PER_T; ++u) pre[u] = __ldg(src + (c + 1) * F4_PER_CHUNK + tid + u * T);
        }
        constexpr int kUnroll = W == 64 ? 4 : 2;  // (registers)
#pragma unroll kUnroll
        for (int kk = 0; on && kk < kChunkK; ++kk) simt_step<G>(xt, wsc + kk * W, acc, c * kChunkK + kk, r0);
        if (c + 1 < NCH) {
            float4* dst = reinterpret_cast<float4*>(ws + ((c + 1) & 1) * kChunkK * W);
#pragma unroll
            for (int u = 0; u < PER_T; ++u) dst[tid + u * T] = pre[u];
        }
        __syncthreads();
    }
}

// The same with W^T resident in shared memory (width 64): no staging, one
// barrier at the end.
__device__ __forceinline__ void simt_gemm_resident64(const float* __restrict__ xt, const float* __restrict__ wt_s,
                                                     float (&acc)[8][4], int r0, int fg, bool on) {
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;
#pragma unroll 4
    for (int k = 0; on && k < 64; ++k) simt_step<1>(xt, wt_s + k * 64 + fg * 4, acc, k, r0);
    __syncthreads();
}

__device__ __forceinline__ int feat_of(int j, int fg) { return (j >> 2) * 64 + fg * 4 + (j & 3); }

// Sum over the 16 lanes that share a row group (lanes l and l ^ 1, 2, 4, 8).
__device__ __forceinline__ float reduce16(float v) {
    v += __shfl_xor_sync(0xffffffffu, v, 8);
    v += __shfl_xor_sync(0xffffffffu, v, 4);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v;
}

}  // namespace simt
}  // namespace sdfnn
