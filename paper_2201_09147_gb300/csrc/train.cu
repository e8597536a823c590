// Training path: the parameter vector's layout, the FP32 forward of a fitting
// step, the fitting objective with its adjoints, and Adam.  The other forward
// and backward kernels are in train32_tc.cu (FP32) and train_tc.cu (16-bit
// operands).
#include <cstdint>

#include "common.cuh"
#include "internal.h"
#include "launch_cache.h"
#include "simt.cuh"

namespace sdfnn {

TrainShape train_shape(int in_dim, int width, int n_hidden) {
    TrainShape s{};
    s.in_dim = in_dim;
    s.width = width;
    s.n_hidden = n_hidden;
    int64_t o = 0;
    s.off_w0 = o;
    o += static_cast<int64_t>(width) * in_dim;
    s.off_b0 = o;
    o += width;
    for (int l = 0; l < n_hidden; ++l) {
        s.off_w[l] = o;
        o += static_cast<int64_t>(width) * width;
        s.off_b[l] = o;
        o += width;
    }
    s.off_wout = o;
    o += width;
    s.off_bout = o;
    o += 1;
    s.count = o;
    return s;
}

namespace {

using namespace simt;

// ---------------------------------------------------------------------------
// forward of a fitting step
// ---------------------------------------------------------------------------
// f and grad f as chains of FP32 FMAs in a fixed order.  A fitting step reports
// its objective in double, summed over f and grad f: the last bits of their
// contractions show there, so it keeps this forward, whose values do not
// depend on the tensor core's accumulation (train32_tc.cu has the other one,
// for gradients through autograd).
constexpr int kTilePts = 32;  // 32 points x 4 streams = the 128 rows of a tile

// W^T of every hidden layer (the forward GEMM streams W^T).
__global__ void transpose_hidden_kernel(const float* __restrict__ theta, TrainShape sh, float* __restrict__ wt) {
    __shared__ float t[32][33];
    const int W = sh.width, l = blockIdx.z;
    const float* src = theta + sh.off_w[l];
    float* dst = wt + static_cast<size_t>(l) * W * W;
    const int bx = blockIdx.x * 32, by = blockIdx.y * 32;
    for (int y = threadIdx.y; y < 32; y += blockDim.y) t[y][threadIdx.x] = src[(by + y) * W + bx + threadIdx.x];
    __syncthreads();
    for (int y = threadIdx.y; y < 32; y += blockDim.y) dst[(bx + y) * W + by + threadIdx.x] = t[threadIdx.x][y];
}

// ---------------------------------------------------------------------------
// forward with saved pre-activations
// ---------------------------------------------------------------------------
template <int W>
struct FwdSmem {
    float xt[W * 128];
    float ws[2 * kChunkK * W];
    float px[kTilePts], py[kTilePts], pz[kTilePts], pt[kTilePts];
    long long tile;
};

template <int W>
__global__ void __launch_bounds__(kSimtThreads, W == 64 ? 3 : W == 128 ? 2 : 1) train_fwd_kernel(const TrainArgs a) {
    extern __shared__ float4 smem_f4[];
    FwdSmem<W>& S = *reinterpret_cast<FwdSmem<W>*>(smem_f4);
    constexpr int FPT = W / 16;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rg = warp * 2 + (lane >> 4), fg = lane & 15, r0 = rg * 8, p0 = r0 >> 2;
    const TrainShape& sh = a.sh;
    const int IN = sh.in_dim, KH = sh.n_hidden;
    const float* W0 = a.theta + sh.off_w0;
    const float* B0 = a.theta + sh.off_b0;
    const float* WO = a.theta + sh.off_wout;
    const float bout = a.theta[sh.off_bout];
    const int64_t n = a.n;

    while (true) {
        if (tid == 0) S.tile = static_cast<long long>(atomicAdd(&a.w.counters[0], 1ull));
        __syncthreads();
        const int64_t base = S.tile * kTilePts;
        if (base >= n) break;
        if (tid < kTilePts) {
            const int64_t i = base + tid;
            const bool v = i < n;
            S.px[tid] = v ? a.pts[i] : 0.0f;
            S.py[tid] = v ? a.pts[n + i] : 0.0f;
            S.pz[tid] = v ? a.pts[2 * n + i] : 0.0f;
            S.pt[tid] = (v && a.pt_time) ? a.pt_time[i] : 0.0f;
        }
        __syncthreads();

        // layer 0: A_0 = W_0 (p, t) + b_0;  P_0 = sin A_0;  G_0^c = W_0[:, c] cos A_0
#pragma unroll
        for (int jg = 0; jg < FPT / 4; ++jg) {
            float za[2][4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int nn = feat_of(jg * 4 + e, fg);
                const float wx = W0[nn * IN], wy = W0[nn * IN + 1], wz = W0[nn * IN + 2];
                const float wt = IN == 4 ? W0[nn * IN + 3] : 0.0f;
                const float bb = B0[nn];
#pragma unroll
                for (int pp = 0; pp < 2; ++pp) {
                    const int p = p0 + pp;
                    const float z = fmaf(wx, S.px[p], fmaf(wy, S.py[p], fmaf(wz, S.pz[p], fmaf(wt, S.pt[p], bb))));
                    za[pp][e] = z;
                    float sn, cs;
                    sincos_r(z, &sn, &cs);
                    *reinterpret_cast<float4*>(S.xt + xt_index(nn, r0 + pp * 4)) =
                        make_float4(sn, wx * cs, wy * cs, wz * cs);
                }
            }
#pragma unroll
            for (int pp = 0; pp < 2; ++pp) {
                const int64_t i = base + p0 + pp;
                if (i < n)
                    *reinterpret_cast<float4*>(a.w.z0 + i * W + feat_of(jg * 4, fg)) =
                        make_float4(za[pp][0], za[pp][1], za[pp][2], za[pp][3]);
            }
        }
        __syncthreads();

        float acc[8][FPT];
        for (int l = 0; l < KH; ++l) {
            simt_gemm<W>(S.xt, a.w.wt + static_cast<size_t>(l) * W * W, S.ws, acc, r0, fg);
            const float* bl = a.theta + sh.off_b[l];
            float4* zl = reinterpret_cast<float4*>(a.w.z) + static_cast<size_t>(l) * n * W;
            const bool last = l + 1 == KH;
            float dot[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) dot[i] = 0.0f;
#pragma unroll
            for (int jg = 0; jg < FPT / 4; ++jg) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int j = jg * 4 + e, nn = feat_of(j, fg);
                    const float bb = bl[nn];
                    const float wo = last ? WO[nn] : 0.0f;
#pragma unroll
                    for (int pp = 0; pp < 2; ++pp) {
                        const float A = acc[pp * 4][j] + bb;
                        const float h0 = acc[pp * 4 + 1][j], h1 = acc[pp * 4 + 2][j], h2 = acc[pp * 4 + 3][j];
                        const int64_t i = base + p0 + pp;
                        if (i < n) zl[i * W + nn] = make_float4(A, h0, h1, h2);
                        float sn, cs;
                        sincos_r(A, &sn, &cs);
                        if (!last) {
                            *reinterpret_cast<float4*>(S.xt + xt_index(nn, r0 + pp * 4)) =
                                make_float4(sn, cs * h0, cs * h1, cs * h2);
                        } else {
                            dot[pp * 4 + 0] = fmaf(wo, sn, dot[pp * 4 + 0]);
                            dot[pp * 4 + 1] = fmaf(wo, cs * h0, dot[pp * 4 + 1]);
                            dot[pp * 4 + 2] = fmaf(wo, cs * h1, dot[pp * 4 + 2]);
                            dot[pp * 4 + 3] = fmaf(wo, cs * h2, dot[pp * 4 + 3]);
                        }
                    }
                }
            }
            if (!last) {
                __syncthreads();
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i) dot[i] = reduce16(dot[i]);
                if (fg == 0) {
#pragma unroll
                    for (int pp = 0; pp < 2; ++pp) {
                        const int64_t i = base + p0 + pp;
                        if (i < n) {
                            a.out_f[i] = dot[pp * 4] + bout;
                            a.out_grad[i] = dot[pp * 4 + 1];
                            a.out_grad[n + i] = dot[pp * 4 + 2];
                            a.out_grad[2 * n + i] = dot[pp * 4 + 3];
                        }
                    }
                }
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// fitting objective and its adjoints
// ---------------------------------------------------------------------------
__global__ void count_near_kernel(const uint8_t* __restrict__ near, int64_t n, unsigned long long* cnt) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    unsigned c = 0;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride) c += near[i] != 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(cnt, static_cast<unsigned long long>(c));
}

__device__ __forceinline__ float sign_of(float x) { return x > 0.0f ? 1.0f : (x < 0.0f ? -1.0f : 0.0f); }

// Per point: the three terms of the objective and dL/df, dL/d(grad f):
//   value:      |f - g|                       -> sign(f - g) / n
//   direction:  1 - <a, b> / (|a| |b|)  (near) -> -(b / (|a| |b|) - cos a / |a|^2) * lam_n / n_near
//   Eikonal:    | |a| - 1 |                    -> sign(|a| - 1) a / |a| * lam_e / n
// (a = grad f, b = the target gradient).  Sums of the terms go to sums[0..2];
// the last block to finish (*ticket, zero at launch) writes out = (mean |f - g|,
// mean over near points of (1 - cos), mean | |grad f| - 1 |, total).
__global__ void fit_loss_kernel(const float* __restrict__ f, const float* __restrict__ grad,
                                const float* __restrict__ tf, const float* __restrict__ tgrad,
                                const uint8_t* __restrict__ near, int64_t n, float lam_n, float lam_e,
                                const unsigned long long* n_near, float* __restrict__ df, float* __restrict__ dgrad,
                                double* sums, unsigned int* ticket, double* out) {
    __shared__ double red[3][8];
    __shared__ bool last;
    const unsigned long long nn = *n_near;
    const float inv_n = 1.0f / static_cast<float>(n);
    const float dir_w = nn ? lam_n / static_cast<float>(nn) : 0.0f;
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += stride) {
        const float e = f[i] - tf[i];
        df[i] = sign_of(e) * inv_n;
        s0 += fabs(static_cast<double>(e));
        const float ax = grad[i], ay = grad[n + i], az = grad[2 * n + i];
        const float bx = tgrad[i], by = tgrad[n + i], bz = tgrad[2 * n + i];
        const float na = sqrtf(ax * ax + ay * ay + az * az), nb = sqrtf(bx * bx + by * by + bz * bz);
        float gx = 0.0f, gy = 0.0f, gz = 0.0f;
        if (na > 0.0f) {
            const float ek = sign_of(na - 1.0f) * lam_e * inv_n / na;
            gx = ek * ax;
            gy = ek * ay;
            gz = ek * az;
        }
        s2 += fabs(static_cast<double>(na) - 1.0);
        if (near[i] && na > 0.0f && nb > 0.0f) {
            const float inv_ab = 1.0f / (na * nb);
            const float cs = (ax * bx + ay * by + az * bz) * inv_ab;
            s1 += 1.0 - static_cast<double>(cs);
            const float ca = cs / (na * na);
            gx -= dir_w * (bx * inv_ab - ca * ax);
            gy -= dir_w * (by * inv_ab - ca * ay);
            gz -= dir_w * (bz * inv_ab - ca * az);
        }
        dgrad[i] = gx;
        dgrad[n + i] = gy;
        dgrad[2 * n + i] = gz;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s0 += __shfl_xor_sync(0xffffffffu, s0, o);
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    }
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        red[0][w] = s0;
        red[1][w] = s1;
        red[2][w] = s2;
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        double t = 0.0;
        for (int k = 0; k < (blockDim.x >> 5); ++k) t += red[threadIdx.x][k];
        atomicAdd(&sums[threadIdx.x], t);
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) + 1u == gridDim.x;
    __syncthreads();
    if (last && threadIdx.x == 0) {
        __threadfence();
        const double lv = __ldcg(sums) / static_cast<double>(n);
        const double ld = nn ? __ldcg(sums + 1) / static_cast<double>(nn) : 0.0;
        const double le = __ldcg(sums + 2) / static_cast<double>(n);
        out[0] = lv;
        out[1] = ld;
        out[2] = le;
        out[3] = lv + static_cast<double>(lam_n) * ld + static_cast<double>(lam_e) * le;
    }
}

// Adam (Kingma and Ba): m <- b1 m + (1 - b1) g;  v <- b2 v + (1 - b2) g^2;
// theta <- theta - lr (m / (1 - b1^t)) / (sqrt(v / (1 - b2^t)) + eps)
__global__ void adam_kernel(float* __restrict__ theta, const float* __restrict__ grad, float* __restrict__ m,
                            float* __restrict__ v, int64_t count, float lr, float beta1, float beta2, float eps,
                            float c1, float c2) {
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < count; i += stride) {
        const float g = grad[i];
        const float mi = fmaf(beta1, m[i], (1.0f - beta1) * g);
        const float vi = fmaf(beta2, v[i], (1.0f - beta2) * g * g);
        m[i] = mi;
        v[i] = vi;
        theta[i] -= lr * (mi * c1) / (sqrtf(vi * c2) + eps);
    }
}

template <class Kernel>
cudaError_t launch_simt_persistent(Kernel k, size_t smem, int num_sms, cudaStream_t s, const void* arg) {
    // the attributes are set and the occupancy counted once per kernel and device; the
    // largest shared-memory carveout lets the occupancy query (and the launch) place as
    // many CTAs per SM as shared memory allows
    cudaError_t e = ensure_smem_attributes(k);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = launch_cached(reinterpret_cast<const void*>(k), smem, kSimtThreads, &per_sm, [&](int* v) {
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(v, k, kSimtThreads, smem);
    });
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    void* args[] = {const_cast<void*>(arg)};
    return cudaLaunchKernel(reinterpret_cast<const void*>(k), dim3(num_sms * per_sm), dim3(kSimtThreads), args, smem,
                            s);
}

template <int W>
cudaError_t forward_w(const TrainArgs& a, int num_sms, cudaStream_t s) {
    if (a.sh.n_hidden > 0) {
        dim3 grid(W / 32, W / 32, a.sh.n_hidden);
        transpose_hidden_kernel<<<grid, dim3(32, 8), 0, s>>>(a.theta, a.sh, a.w.wt);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    cudaError_t e = cudaMemsetAsync(a.w.counters, 0, 4 * sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    return launch_simt_persistent(train_fwd_kernel<W>, sizeof(FwdSmem<W>), num_sms, s, &a);
}

}  // namespace

cudaError_t launch_fit_forward(const TrainArgs& a, int num_sms, cudaStream_t s) {
    cudaError_t e = launch_pack32_backward(a, num_sms, s);
    if (e != cudaSuccess) return e;
    switch (a.sh.width) {
    case 64:
        return forward_w<64>(a, num_sms, s);
    case 128:
        return forward_w<128>(a, num_sms, s);
    case 256:
        return forward_w<256>(a, num_sms, s);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_fit_loss(const float* f, const float* grad, const float* tf, const float* tgrad,
                            const uint8_t* near, int64_t n, float lam_n, float lam_e, float* d_f, float* d_grad,
                            FitScratch* sc, double* out, int num_sms, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(sc, 0, sizeof(FitScratch), s);
    if (e != cudaSuccess) return e;
    int blocks = static_cast<int>((n + 255) / 256);
    if (blocks > 4 * num_sms) blocks = 4 * num_sms;
    if (blocks < 1) blocks = 1;
    count_near_kernel<<<blocks, 256, 0, s>>>(near, n, &sc->n_near);
    fit_loss_kernel<<<blocks, 256, 0, s>>>(f, grad, tf, tgrad, near, n, lam_n, lam_e, &sc->n_near, d_f, d_grad, sc->sums,
                                           &sc->ticket, out);
    return cudaGetLastError();
}

cudaError_t launch_adam(float* theta, const float* grad, float* m, float* v, int64_t count, float lr, float beta1,
                        float beta2, float eps, int step, int num_sms, cudaStream_t s) {
    const double c1 = 1.0 / (1.0 - std::pow(static_cast<double>(beta1), step));
    const double c2 = 1.0 / (1.0 - std::pow(static_cast<double>(beta2), step));
    int blocks = static_cast<int>((count + 255) / 256);
    if (blocks > 4 * num_sms) blocks = 4 * num_sms;
    if (blocks < 1) blocks = 1;
    adam_kernel<<<blocks, 256, 0, s>>>(theta, grad, m, v, count, lr, beta1, beta2, eps, static_cast<float>(c1),
                                       static_cast<float>(c2));
    return cudaGetLastError();
}

}  // namespace sdfnn
