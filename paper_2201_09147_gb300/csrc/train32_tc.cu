// FP32 training path on the tensor cores (SDF_FP32): the three kernels of
// train_tc.cu with operands split so that the products keep FP32 accuracy.
//
//   forward:  grad32_tc_kernel<W, true>; saves A_0 and (A_l, H_l) in FP32;
//   backward: train32_bwd_kernel, D_l = (dA_l, dH_l) from Y_l and the saved
//             (A_l, H_l), then Y_{l-1} = W_l^T D_l;
//   weights:  train32_wgrad_kernel, dW_l = sum over point-streams of D_l X_{l-1}^T.
//
// The parameters change from step to step and the adjoints span many binades
// (1 / n of the loss, growing and shrinking from layer to layer and point to
// point), beyond a half's exponents.  So all three split every FP32 operand into
// three bfloat16 values x0 + x1 + x2 (24 significand bits, a float's exponent
// range) and keep the six products x_i y_j with i + j <= 2; what is left out is
// below 2^-24 of the product.  x0 y0 has an accumulator of its own
// (grad32_tc.cuh says why).
//
// A fitting step takes its forward from train.cu (launch_fit_forward): its
// objective is reported in double and shows the last bits of f.
//
// The kernels before these ran the same contractions on the FP32 FMA units:
// forward and backward of the (128,2) at 50,001 points through autograd 1,502
// -> 354 us; a fitting step 984 -> 395 us ((128,2), 30,000 points), 448 -> 224
// ((256,1), 9,001), 549 -> 268 ((256,3), 2,000).  Errors of dL/dtheta against FP64
// on five networks at 20,011 points 4 to 22 % lower.
#include <algorithm>
#include <cstdint>

#include "grad32_tc.cuh"
#include "internal.h"
#include "tc_common.cuh"

namespace sdfnn {

namespace {

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }
size_t rows_pad_of(size_t W) { return W < 128 ? 128 : W; }

}  // namespace

// Counters, then the W_l and W_l^T images (three bfloat16 planes each), their rows'
// gains, W_l^T in FP32, A_0, (A_l, H_l) and (dA_l, dH_l).
size_t train_workspace_bytes(const TrainShape& sh, int64_t n) {
    const size_t W = sh.width, k = sh.n_hidden, N = static_cast<size_t>(n), img = rows_pad_of(W) * W * 2;
    return 2 * align256(3 * k * img) + align256(2 * k * W * 4) + align256(k * W * W * 4) + align256(N * W * 4) + 2 * align256(k * N * 4 * W * 4) + 256;
}

TrainWork train_work(const TrainShape& sh, int64_t n, void* ws) {
    const size_t W = sh.width, k = sh.n_hidden, N = static_cast<size_t>(n), img = rows_pad_of(W) * W * 2;
    uint8_t* p = static_cast<uint8_t*>(ws);
    TrainWork w{};
    w.counters = reinterpret_cast<unsigned long long*>(p);
    p += 256;
    w.wbf = p;
    p += align256(3 * k * img);
    w.wbft = p;
    p += align256(3 * k * img);
    w.gain = reinterpret_cast<float*>(p);
    p += align256(2 * k * W * 4);
    w.wt = reinterpret_cast<float*>(p);
    p += align256(k * W * W * 4);
    w.z0 = reinterpret_cast<float*>(p);
    p += align256(N * W * 4);
    w.z = reinterpret_cast<float*>(p);
    p += align256(k * N * 4 * W * 4);
    w.d = reinterpret_cast<float*>(p);
    return w;
}

namespace {

// Two points (four streams each) of one feature as 16-byte chunks of the three planes.
__device__ __forceinline__ void store_split3(uint32_t x_s, uint32_t plane, uint32_t off, const float4& a,
                                             const float4& b) {
    uint32_t q[4][3];
    split3x2(a.x, a.y, q[0]);
    split3x2(a.z, a.w, q[1]);
    split3x2(b.x, b.y, q[2]);
    split3x2(b.z, b.w, q[3]);
#pragma unroll
    for (int i = 0; i < 3; ++i) st_shared_v4(x_s + i * plane + off, q[0][i], q[1][i], q[2][i], q[3][i]);
}

// ---------------------------------------------------------------------------
// weight images
// ---------------------------------------------------------------------------
// W_l (rows = output units) and W_l^T (rows = inputs) in three bfloat16 planes per K block, and the correction of
// each row's sums (grad32_tc.cuh).  wimg NULL: without the W_l images.  256 threads: a block's elements are whole
// rows.
__global__ void __launch_bounds__(256) train32_pack_kernel(const float* __restrict__ theta, TrainShape sh, int rows_pad,
                                                           uint8_t* wimg, uint8_t* wtimg, float* gain) {
    __shared__ float sq[2][16];  // sums of squares over 16 elements: W_l, W_l^T
    const int W = sh.width, tid = threadIdx.x;
    const int per = rows_pad * W, total = per * sh.n_hidden;
    const size_t block = static_cast<size_t>(rows_pad) * 128u;  // one plane of a K block
    for (int i0 = blockIdx.x * 256; i0 < total; i0 += gridDim.x * 256) {
        const int i = i0 + tid, l = i / per, r = (i % per) / W, k = i % W;
        const float* Wl = theta + sh.off_w[l];
        uint32_t w[3] = {0u, 0u, 0u}, t[3] = {0u, 0u, 0u};
        float x = 0.0f, y = 0.0f;
        if (r < W) {
            x = Wl[r * W + k];
            y = Wl[k * W + r];
            split3x2(x, 0.0f, w);
            split3x2(y, 0.0f, t);
        }
        const size_t at = (static_cast<size_t>(l) * (W / 64) + k / 64) * 3 * block + sw128_offset(r, k & 63, rows_pad);
#pragma unroll
        for (int p = 0; p < 3; ++p) {
            if (wimg != nullptr) *reinterpret_cast<uint16_t*>(wimg + at + p * block) = static_cast<uint16_t>(w[p]);
            *reinterpret_cast<uint16_t*>(wtimg + at + p * block) = static_cast<uint16_t>(t[p]);
        }
        // scaled by the row's largest, so that no square leaves a float's range
        float mx = fabsf(x), my = fabsf(y);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            my = fmaxf(my, __shfl_xor_sync(0xffffffffu, my, o));
        }
        if ((tid & 15) == 0) {
            sq[0][tid >> 4] = mx;
            sq[1][tid >> 4] = my;
        }
        __syncthreads();
        const int s0 = tid / W * (W / 16);  // the row's first step in sq
        for (int s = s0; s < s0 + W / 16; ++s) {
            mx = fmaxf(mx, sq[0][s]);
            my = fmaxf(my, sq[1][s]);
        }
        __syncthreads();
        float vx = mx > 0.0f ? (x / mx) * (x / mx) : 0.0f, vy = my > 0.0f ? (y / my) * (y / my) : 0.0f;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
            vx += __shfl_xor_sync(0xffffffffu, vx, o);
            vy += __shfl_xor_sync(0xffffffffu, vy, o);
        }
        if ((tid & 15) == 0) {
            sq[0][tid >> 4] = vx;
            sq[1][tid >> 4] = vy;
        }
        __syncthreads();
        if (k < 2 && r < W) {
            float sum = 0.0f, shares = 0.0f;
            for (int s = s0; s < s0 + W / 16; ++s) {
                sum += sq[k][s];
                if (sq[k][s] > 0.0f) shares += sum;
            }
            gain[(static_cast<size_t>(k) * sh.n_hidden + l) * W + r] =
                sum > 0.0f ? 1.0f + static_cast<float>(kStepLoss) * (shares / sum) : 1.0f;
        }
        __syncthreads();
    }
}

struct Train32Args {
    TrainShape sh;
    const float* theta;
    const float* pts;      // SoA (3, n)
    const float* pt_time;  // (n) or NULL
    int64_t n;
    const float* d_f;      // (n)
    const float* d_grad;   // SoA (3, n)
    const uint8_t* wt;     // W_l^T images
    const float* a0;       // [n][W] A_0
    const float4* z;       // [k][n][W] (A_l, H_l^x, H_l^y, H_l^z)
    float4* d;             // [k][n][W] (dA_l, dH_l^x, dH_l^y, dH_l^z)
    const float* gain;     // [k][W] the correction of a row's sums, W_l^T
    float* d_theta;
    int* status;
};

// ---------------------------------------------------------------------------
// backward through the hidden layers and the input layer
// ---------------------------------------------------------------------------
template <int W>
struct B32 : G32<W, 3> {
    using G = G32<W, 3>;
    static constexpr uint32_t RING = G::NH * 3u * G::PLANE, ADJ = RING + G::NS * G::UNIT;
    static constexpr uint32_t BARS = ADJ + G::NH * G::HPTS * 16u, MISC = BARS + (2 * G::NS + 2 * G::NH) * 8u;
    static constexpr uint32_t TOTAL = MISC + 32u;
    static_assert(TOTAL + 1024u <= 227u * 1024u, "shared memory");
};

// The warp roles and tiles of grad32_tc_kernel, run from the top layer down.  Bound by the MMAs (six
// instructions per K step and TMEM tile, 384 clocks at least) and the reads of the saved (A, H), which are loaded a
// chunk of four points ahead.  Sums over the batch (biases, W_0, w_out) stay in registers of the thread that
// owns the feature until the end.
template <int W>
__global__ void __launch_bounds__(B32<W>::THREADS, 1) train32_bwd_kernel(const Train32Args a) {
    using C = B32<W>;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t raw_s = smem_u32(smem_raw);
    const uint32_t base_s = (raw_s + 1023u) & ~1023u;
    uint8_t* base = smem_raw + (base_s - raw_s);
    const TrainShape& sh = a.sh;
    const int KH = sh.n_hidden, IN = sh.in_dim;
    float4* adj = reinterpret_cast<float4*>(base + C::ADJ);  // (df, dg_x, dg_y, dg_z) per point
    const uint32_t bar_full = base_s + C::BARS, bar_empty = bar_full + 8u * C::NS;
    const uint32_t bar_xready = bar_empty + 8u * C::NS, bar_dfull = bar_xready + 8u * C::NH;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(base + C::MISC);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(base + C::MISC + 4);
    const uint32_t ring_s = base_s + C::RING;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (tid == 0) {
        for (int s = 0; s < C::NS; ++s) {
            mbar_init(bar_full + 8u * s, 1);
            mbar_init(bar_empty + 8u * s, 1);
        }
        for (int h = 0; h < C::NH; ++h) {
            mbar_init(bar_xready + 8u * h, C::GROUP_THREADS);
            mbar_init(bar_dfull + 8u * h, 1);
        }
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(smem_u32(tmem_slot), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    const long long n_sets = (a.n + C::NH * C::HPTS - 1) / (C::NH * C::HPTS);
    const long long G = gridDim.x;
    const int my_sets = static_cast<int>(n_sets > blockIdx.x ? (n_sets - blockIdx.x + G - 1) / G : 0);
    const int n_groups = my_sets * KH;
    bool ok = true;

    if (warp == C::PRODUCER_WARP) {
        if (lane == 0) {
            uint32_t g = 0;
            int l = KH - 1;
            for (int k = 0; k < n_groups && ok; ++k) {
                const uint8_t* src = a.wt + static_cast<size_t>(l) * C::UNITS * C::UNIT;
                for (int h = 0; h < C::NH && ok; ++h)
                    for (int u = 0; u < C::UNITS && ok; ++u, ++g) {
                        const uint32_t stage = g % C::NS, use = g / C::NS;
                        if (use > 0) ok = mbar_wait_bounded(bar_empty + 8u * stage, (use - 1) & 1u, a.status, abort_flag);
                        if (!ok) break;
                        mbar_arrive_expect_tx(bar_full + 8u * stage, C::UNIT);
                        bulk_g2s(ring_s + stage * C::UNIT, src + u * C::UNIT, C::UNIT, bar_full + 8u * stage);
                    }
                l = l == 0 ? KH - 1 : l - 1;
            }
            for (uint32_t gg = g > C::NS ? g - C::NS : 0; gg < g; ++gg)
                mbar_drain(bar_full + 8u * (gg % C::NS), (gg / C::NS) & 1u);
        }
    } else if (warp == C::MMA_WARP) {
        if (lane == 0) {
            uint32_t g = 0;
            for (int k = 0; k < n_groups && ok; ++k)
                for (int h = 0; h < C::NH && ok; ++h) {
                    ok = mbar_wait_bounded(bar_xready + 8u * h, k & 1, a.status, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t xd0 = desc_mnmajor_sw128(base_s + h * 3u * C::PLANE, W * 128u);
                    ok = mma_layer32<C>(tmem, h, xd0, ring_s, bar_full, bar_empty, g, a.status, abort_flag);
                    if (ok) mma_commit(bar_dfull + 8u * h);
                }
        }
    } else {
        const int h = warp / C::GROUP_WARPS, ge = warp % C::GROUP_WARPS;
        const int mt = (ge >> 2) % C::MT, cs = (ge >> 2) / C::MT, quad = ge & 3;
        const int m = mt * 128 + quad * 32 + lane;
        const bool live = mt * 128 + quad * 32 < W;  // warp-uniform
        const int gt = ge * 32 + lane;
        const uint32_t d_s = tmem + (static_cast<uint32_t>(quad * 32) << 16) + (mt + h) * 256u + cs * (C::CPTS * 4u);
        const uint32_t xh = base_s + h * 3u * C::PLANE;
        const int p0 = h * C::HPTS, q0 = p0 + cs * C::CPTS;
        const bool timed = a.pt_time != nullptr && IN == 4;
        float wo = 0.0f, w0x = 0.0f, w0y = 0.0f, w0z = 0.0f;
        if (live) {
            const float* w0 = a.theta + sh.off_w0 + m * IN;
            wo = __ldg(a.theta + sh.off_wout + m);
            w0x = __ldg(w0);
            w0y = __ldg(w0 + 1);
            w0z = __ldg(w0 + 2);
        }
        float s_b[kMaxHidden + 1] = {}, s_o = 0.0f, s_w[4] = {}, s_bout = 0.0f;
        uint32_t df_phase = 0;
        for (int i = 0; i < my_sets; ++i) {
            const int64_t base_p = ((static_cast<int64_t>(i) * G + blockIdx.x) * C::NH + h) * C::HPTS;
            if (gt < C::HPTS) {
                const int64_t k = base_p + gt;
                const bool v = k < a.n;
                const float4 ad = v ? make_float4(a.d_f[k], a.d_grad[k], a.d_grad[a.n + k], a.d_grad[2 * a.n + k])
                                    : make_float4(0.f, 0.f, 0.f, 0.f);
                adj[p0 + gt] = ad;
                s_bout += ad.x;
            }
            bar_named(1 + h, C::GROUP_THREADS);
            const int64_t pb = base_p + cs * C::CPTS;  // this thread's first point; nv of its points are in the batch
            const int nv = static_cast<int>(min(max(a.n - pb, static_cast<int64_t>(0)), static_cast<int64_t>(C::CPTS)));
            for (int l = KH - 1; l >= 0 && ok; --l) {
                const bool top = l == KH - 1;
                const size_t at = (static_cast<size_t>(l) * a.n + pb) * W + m;
                const float4* zp = a.z + at;
                float4* dp = a.d + at;
                float4 zn[4];
                if (live)
#pragma unroll
                    for (int e = 0; e < 4; ++e) zn[e] = e < nv ? __ldg(zp + e * W) : make_float4(0.f, 0.f, 0.f, 0.f);
                if (!top) {
                    ok = __all_sync(0xffffffffu, mbar_wait_bounded(bar_dfull + 8u * h, df_phase, a.status, abort_flag));
                    df_phase ^= 1u;
                    if (!ok) break;
                    tc_fence_after();
                }
                float sb = 0.0f, so = 0.0f;
                const float gain = !top && live ? __ldg(a.gain + (l + 1) * W + m) : 1.0f;
#pragma unroll 1
                for (int q = 0; live && q < C::CPTS / 4; ++q) {
                    // Y of four points (16 columns); at the top w_out times the adjoints
                    float v[16];
                    if (top) {
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float4 ad = adj[q0 + 4 * q + e];
                            v[4 * e] = ad.x * wo;
                            v[4 * e + 1] = ad.y * wo;
                            v[4 * e + 2] = ad.z * wo;
                            v[4 * e + 3] = ad.w * wo;
                        }
                    } else {
                        float c[16];
                        tmem_ld16(d_s + q * 16u, v);
                        tmem_ld16(d_s + 128u + q * 16u, c);
                        tmem_wait_ld();
#pragma unroll
                        for (int j = 0; j < 16; ++j) v[j] = (v[j] + c[j]) * gain;
                    }
                    float4 Z[4];
                    zp += 4 * W;
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        Z[e] = zn[e];
                        if (q + 1 < C::CPTS / 4)
                            zn[e] = 4 * (q + 1) + e < nv ? __ldg(zp + e * W) : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float y0 = v[4 * e], y1 = v[4 * e + 1], y2 = v[4 * e + 2], y3 = v[4 * e + 3];
                        float sn, cn;
                        sincos_r(Z[e].x, &sn, &cn);
                        if (top) {
                            const float4 ad = adj[q0 + 4 * q + e];
                            so += ad.x * sn + cn * (ad.y * Z[e].y + ad.z * Z[e].z + ad.w * Z[e].w);
                        }
                        const float dA = y0 * cn - sn * (y1 * Z[e].y + y2 * Z[e].z + y3 * Z[e].w);
                        sb += dA;
                        Z[e] = make_float4(dA, y1 * cn, y2 * cn, y3 * cn);
                        if (4 * q + e < nv) dp[e * W] = Z[e];
                    }
                    dp += 4 * W;
                    store_split3(xh, C::PLANE, xoff32<W>(m, cs * (C::CPTS / 2) + 2 * q), Z[0], Z[1]);
                    store_split3(xh, C::PLANE, xoff32<W>(m, cs * (C::CPTS / 2) + 2 * q + 1), Z[2], Z[3]);
                }
#pragma unroll
                for (int j = 0; j < kMaxHidden; ++j) s_b[j] += j == l ? sb : 0.0f;
                s_o += so;
                fence_proxy_async_smem();
                tc_fence_before();
                mbar_arrive(bar_xready + 8u * h);
            }
            // input layer: dA_0 = dP_0 cos A_0 - sin A_0 sum_c dG_0^c W_0[:, c];
            // dW_0[:, c] += dA_0 x_c + dG_0^c cos A_0 (c < 3), dA_0 t (c = 3); db_0 += dA_0
            if (ok) {
                ok = __all_sync(0xffffffffu, mbar_wait_bounded(bar_dfull + 8u * h, df_phase, a.status, abort_flag));
                df_phase ^= 1u;
                tc_fence_after();
            }
            if (ok && live) {
                const float* ap = a.a0 + pb * W + m;
                const float* xp = a.pts + pb;  // the points: the same address for the whole warp
                float sb = 0.0f, sw[4] = {};   // sums over the tile first: shorter chains of roundings
                const float gain = __ldg(a.gain + m);
#pragma unroll 1
                for (int q = 0; q < C::CPTS / 4; ++q) {
                    float A0[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) A0[e] = 4 * q + e < nv ? __ldg(ap + e * W) : 0.0f;
                    ap += 4 * W;
                    float v[16], c[16];
                    tmem_ld16(d_s + q * 16u, v);
                    tmem_ld16(d_s + 128u + q * 16u, c);
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 16; ++j) v[j] = (v[j] + c[j]) * gain;
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        if (4 * q + e >= nv) continue;  // Y is zero past the batch
                        const float y1 = v[4 * e + 1], y2 = v[4 * e + 2], y3 = v[4 * e + 3];
                        float sn, cn;
                        sincos_r(A0[e], &sn, &cn);
                        const float dA = v[4 * e] * cn - sn * (y1 * w0x + y2 * w0y + y3 * w0z);
                        sb += dA;
                        sw[0] += dA * __ldg(xp + e) + y1 * cn;
                        sw[1] += dA * __ldg(xp + a.n + e) + y2 * cn;
                        sw[2] += dA * __ldg(xp + 2 * a.n + e) + y3 * cn;
                        if (timed) sw[3] += dA * __ldg(a.pt_time + pb + 4 * q + e);
                    }
                    xp += 4;
                }
                s_b[kMaxHidden] += sb;
#pragma unroll
                for (int c = 0; c < 4; ++c) s_w[c] += sw[c];
            }
            tc_fence_before();
            // the next tile's point data overwrites this half's; one stop decision for the group
            if (bar_or(1 + h, C::GROUP_THREADS, !ok || *abort_flag != 0)) break;
        }
        if (live && my_sets > 0) {
#pragma unroll
            for (int l = 0; l < kMaxHidden; ++l)
                if (l < KH) atomicAdd(a.d_theta + sh.off_b[l] + m, s_b[l]);
            atomicAdd(a.d_theta + sh.off_b0 + m, s_b[kMaxHidden]);
            atomicAdd(a.d_theta + sh.off_wout + m, s_o);
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (c < IN) atomicAdd(a.d_theta + sh.off_w0 + m * IN + c, s_w[c]);
        }
        if (gt < C::HPTS) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s_bout += __shfl_xor_sync(0xffffffffu, s_bout, o);
            if (lane == 0 && my_sets > 0) atomicAdd(a.d_theta + sh.off_bout, s_bout);
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// ---------------------------------------------------------------------------
// weight gradients dW_l = sum over point-streams of D_l X_{l-1}^T
// ---------------------------------------------------------------------------
// A job is a block of NB x NB weights of one layer; the K blocks (16 points = 64
// point-streams) of all jobs are dealt out evenly, so a CTA runs one or two
// jobs.  Builder threads load a K block's D_l (A operand, rows = output units)
// or saved (A, H) (B operand, rows = inputs), split into three planes and store
// them K-major; one thread multiplies.  The accumulator is added to FP32
// registers every kFlush K blocks: 16 truncations of the tensor core at most
// meet a sum (root mean square error below that of the 600-term FMA chains
// this replaces), and one K block late, so that the next block is being
// multiplied meanwhile.
template <int W>
struct Wg32 {
    static constexpr int NB = W < 128 ? W : 128;          // inputs (and output units) of a job
    static constexpr int JB = W / NB;                     // job rows, job columns per layer
    static constexpr uint32_t A_PLANE = 16384u, X_PLANE = NB * 128u;
    static constexpr uint32_t STAGE = 3u * (A_PLANE + X_PLANE);
    static constexpr int NS = 2;
    static constexpr int BUILDERS = 512;                  // first half: D, second half: X
    static constexpr int SPAN = 256 / NB;                 // threads per row
    static constexpr int PPT = 16 / SPAN;                 // points per thread
    static constexpr int THREADS = BUILDERS + 32;
    static constexpr int TMEM_COLS = 2 * NB;
    static constexpr uint32_t BARS = NS * STAGE, MISC = BARS + (2 * NS + 2) * 8u, TOTAL = MISC + 32u;
};
constexpr int kFlush = 4;
// The correction of a flush's sums over `steps` K steps of points (grad32_tc.cuh: terms of one size).
__device__ __forceinline__ float flush_gain(int steps) {
    return 1.0f + static_cast<float>(0.5 * kStepLoss) * static_cast<float>(steps + 1);
}

template <int W>
__global__ void __launch_bounds__(Wg32<W>::THREADS, 1) train32_wgrad_kernel(const Train32Args a) {
    using C = Wg32<W>;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t raw_s = smem_u32(smem_raw);
    const uint32_t base_s = (raw_s + 1023u) & ~1023u;
    uint8_t* base = smem_raw + (base_s - raw_s);
    const TrainShape& sh = a.sh;
    const int KH = sh.n_hidden;
    const uint32_t bar_full = base_s + C::BARS, bar_empty = bar_full + 8u * C::NS;
    const uint32_t bar_done = bar_empty + 8u * C::NS, bar_flushed = bar_done + 8u;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(base + C::MISC);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(base + C::MISC + 4);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (tid == 0) {
        for (int s = 0; s < C::NS; ++s) {
            mbar_init(bar_full + 8u * s, C::BUILDERS);
            mbar_init(bar_empty + 8u * s, 1);
        }
        mbar_init(bar_done, 1);
        mbar_init(bar_flushed, C::BUILDERS);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(smem_u32(tmem_slot), C::TMEM_COLS);
        tmem_relinquish();
    }
    // width 64: the A operand's rows 64 .. 127 stay zero
    if (W < 128)
        for (int s = 0; s < C::NS; ++s)
            for (int p = 0; p < 3; ++p)
                for (uint32_t i = W * 128u + tid * 16u; i < C::A_PLANE; i += C::THREADS * 16u)
                    st_shared_v4(base_s + s * C::STAGE + p * C::A_PLANE + i, 0u, 0u, 0u, 0u);
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    const int64_t nkb = (a.n + 15) / 16;                     // K blocks per job
    const int64_t total = nkb * KH * C::JB * C::JB;
    const int64_t lo = total * blockIdx.x / gridDim.x, hi = total * (blockIdx.x + 1) / gridDim.x;
    bool ok = true;
    // Both roles walk the same list: block t belongs to job t / nkb; a flush follows every kFlush blocks of a
    // job and its last one.
    if (hi > lo && warp == C::BUILDERS / 32) {
        if (lane == 0) {
            constexpr uint32_t idesc = idesc_f32acc(128, C::NB, false);
            uint32_t g = 0, flushes = 0;
            int in_acc = 0;
            for (int64_t t = lo; t < hi && ok; ++t, ++g) {
                const uint32_t stage = g % C::NS;
                ok = mbar_wait_bounded(bar_full + 8u * stage, (g / C::NS) & 1u, a.status, abort_flag);
                if (ok && in_acc == 0 && flushes > 0)
                    ok = mbar_wait_bounded(bar_flushed, (flushes - 1) & 1u, a.status, abort_flag);
                if (!ok) break;
                tc_fence_after();
                const uint32_t sa = base_s + stage * C::STAGE, sx = sa + 3u * C::A_PLANE;
                const uint64_t ad0 = desc_kmajor_sw128(sa), xd0 = desc_kmajor_sw128(sx);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const uint64_t a0 = desc_add(ad0, kk * 32u), x0 = desc_add(xd0, kk * 32u);
                    const uint64_t a1 = desc_add(a0, C::A_PLANE), a2 = desc_add(a0, 2 * C::A_PLANE);
                    const uint64_t x1 = desc_add(x0, C::X_PLANE), x2 = desc_add(x0, 2 * C::X_PLANE);
                    mma_f16kind(tmem, a0, x0, idesc, (in_acc | kk) != 0);
                    mma_f16kind(tmem + C::NB, a0, x1, idesc, (in_acc | kk) != 0);
                    mma_f16kind(tmem + C::NB, a0, x2, idesc, 1u);
                    mma_f16kind(tmem + C::NB, a1, x0, idesc, 1u);
                    mma_f16kind(tmem + C::NB, a1, x1, idesc, 1u);
                    mma_f16kind(tmem + C::NB, a2, x0, idesc, 1u);
                }
                mma_commit(bar_empty + 8u * stage);
                if (++in_acc == kFlush || t + 1 == hi || (t + 1) % nkb == 0) {
                    mma_commit(bar_done);
                    ++flushes;
                    in_acc = 0;
                }
            }
        }
    } else if (hi > lo) {
        const bool is_x = tid >= 256;
        const int row = (tid & 255) % C::NB, p_off = ((tid & 255) / C::NB) * C::PPT;
        const int quad = warp & 3, cg = warp >> 2;              // TMEM lanes and quarter of the columns to flush
        constexpr int FC = C::NB / 4;                           // columns per thread
        const uint32_t d_s = tmem + (static_cast<uint32_t>(quad * 32) << 16) + cg * FC;
        float acc[FC];
#pragma unroll
        for (int j = 0; j < FC; ++j) acc[j] = 0.0f;
        // the flush of the blocks multiplied so far; `job` >= 0 also adds the registers to dL/dtheta
        uint32_t flushes = 0;
        auto flush = [&](int job, float gain) {
            ok = __all_sync(0xffffffffu, mbar_wait_bounded(bar_done, flushes & 1u, a.status, abort_flag)) && ok;
            ++flushes;
            if (!ok) return;
            tc_fence_after();
#pragma unroll
            for (int j = 0; j < FC; j += 16) {
                float v[16], c[16];
                tmem_ld16(d_s + j, v);
                tmem_ld16(d_s + C::NB + j, c);
                tmem_wait_ld();
#pragma unroll
                for (int e = 0; e < 16; ++e) acc[j + e] = fmaf(v[e] + c[e], gain, acc[j + e]);
            }
            tc_fence_before();
            mbar_arrive(bar_flushed);
            if (job >= 0) {
                const int l = job / (C::JB * C::JB), b = job % (C::JB * C::JB);
                const int unit = (b / C::JB) * C::NB + quad * 32 + lane;
                if (quad * 32 < C::NB) {
                    float4* out = reinterpret_cast<float4*>(a.d_theta + sh.off_w[l] + static_cast<size_t>(unit) * W +
                                                            (b % C::JB) * C::NB + cg * FC);
#pragma unroll
                    for (int j = 0; j < FC / 4; ++j)
                        atomicAdd(out + j, make_float4(acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]));
                }
#pragma unroll
                for (int j = 0; j < FC; ++j) acc[j] = 0.0f;
            }
        };
        uint32_t g = 0;
        int in_acc = 0;
        float gain = 1.0f;     // of the pending flush
        int pending = -2;      // the flush to run after the next build: -2 none, -1 to registers, >= 0 to that job
        for (int64_t t = lo; t < hi && ok; ++t, ++g) {
            const int job = static_cast<int>(t / nkb);
            const int64_t pbase = (t % nkb) * 16 + p_off;
            const int l = job / (C::JB * C::JB), b = job % (C::JB * C::JB);
            const int feat = (is_x ? b % C::JB : b / C::JB) * C::NB + row;
            // this thread's points of the K block: D_l, or the layer below's (A, H) (A_0 and W_0 for layer 0)
            float4 q[C::PPT];
            if (!is_x || l > 0) {
                const float4* src = (is_x ? a.z + static_cast<size_t>(l - 1) * a.n * W
                                          : a.d + static_cast<size_t>(l) * a.n * W) + feat;
#pragma unroll
                for (int e = 0; e < C::PPT; ++e)
                    q[e] = pbase + e < a.n ? __ldg(src + (pbase + e) * W) : make_float4(0.f, 0.f, 0.f, 0.f);
            } else {
                const float* w0 = a.theta + sh.off_w0 + feat * sh.in_dim;
                const float wx = __ldg(w0), wy = __ldg(w0 + 1), wz = __ldg(w0 + 2);
#pragma unroll
                for (int e = 0; e < C::PPT; ++e)
                    q[e] = make_float4(pbase + e < a.n ? __ldg(a.a0 + (pbase + e) * W + feat) : 0.0f, wx, wy, wz);
            }
            const uint32_t stage = g % C::NS, use = g / C::NS;
            if (use > 0)
                ok = __all_sync(0xffffffffu, mbar_wait_bounded(bar_empty + 8u * stage, (use - 1) & 1u, a.status, abort_flag));
            if (!ok) break;
            const uint32_t st = base_s + stage * C::STAGE + (is_x ? 3u * C::A_PLANE : 0u) + (row >> 3) * 1024u + (row & 7) * 128u;
            const uint32_t plane = is_x ? C::X_PLANE : C::A_PLANE;
#pragma unroll
            for (int e = 0; e < C::PPT; ++e)
                if (is_x) {
                    // points past the batch: D is zero there, X only has to be finite
                    float sn, cn;
                    sincos_r(q[e].x, &sn, &cn);
                    q[e] = make_float4(sn, cn * q[e].y, cn * q[e].z, cn * q[e].w);
                }
#pragma unroll
            for (int e = 0; e < C::PPT; e += 2) {
                const uint32_t c = static_cast<uint32_t>((p_off + e) >> 1);
                store_split3(st, plane, (c ^ (row & 7u)) << 4, q[e], q[e + 1]);
            }
            fence_proxy_async_smem();
            mbar_arrive(bar_full + 8u * stage);
            if (pending != -2) {
                flush(pending, gain);
                pending = -2;
            }
            const bool job_end = t + 1 == hi || (t + 1) % nkb == 0;
            if (++in_acc == kFlush || job_end) {
                pending = job_end ? job : -1;
                // four K steps a block; the batch's last block has one per four points
                gain = flush_gain(4 * in_acc - (pbase - p_off + 16 > a.n ? static_cast<int>(pbase - p_off + 16 - a.n) / 4 : 0));
                in_acc = 0;
            }
        }
        if (ok && pending != -2) flush(pending, gain);
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, C::TMEM_COLS);
    }
}

cudaError_t pack32(const TrainArgs& a, uint8_t* wimg, int num_sms, cudaStream_t s) {
    const int W = a.sh.width, rows_pad = static_cast<int>(rows_pad_of(W));
    const int blocks = std::min((rows_pad * W * a.sh.n_hidden + 255) / 256, 8 * num_sms);
    train32_pack_kernel<<<blocks, 256, 0, s>>>(a.theta, a.sh, rows_pad, wimg, a.w.wbft, a.w.gain);
    return cudaGetLastError();
}

template <int W>
cudaError_t forward32_w(const TrainArgs& a, int num_sms, cudaStream_t s) {
    const TrainShape& sh = a.sh;
    const int rows_pad = static_cast<int>(rows_pad_of(W));
    cudaError_t e = pack32(a, a.w.wbf, num_sms, s);
    if (e != cudaSuccess) return e;
    GradArgs ga{};
    ga.net.in_dim = sh.in_dim;
    ga.net.width = W;
    ga.net.n_hidden = sh.n_hidden;
    ga.net.w0 = a.theta + sh.off_w0;
    ga.net.b0 = a.theta + sh.off_b0;
    for (int l = 0; l < sh.n_hidden; ++l) ga.net.bh[l] = a.theta + sh.off_b[l];
    ga.net.wout = a.theta + sh.off_wout;
    ga.net.wbf = a.w.wbf;
    ga.net.wbf_layer_bytes = static_cast<uint32_t>(rows_pad) * W * 6u;
    ga.net.rows_pad = rows_pad;
    ga.net.s32 = a.w.gain;
    ga.pt_time = a.pt_time;
    ga.pts = a.pts;
    ga.n = a.n;
    ga.out = a.out_grad;
    ga.status = a.status;
    ga.save_a0 = a.w.z0;
    ga.save_a = a.w.z;
    ga.out_f = a.out_f;
    ga.out_bias = a.theta + sh.off_bout;
    using C = G32<W, 3>;
    return launch_tc(grad32_tc_kernel<W, true>, C::THREADS, g32_layout<C>().total + 1024, C::TMEM_COLS, num_sms, s, &ga);
}

template <int W>
cudaError_t backward32_w(const TrainArgs& a, int num_sms, cudaStream_t s) {
    Train32Args t{};
    t.sh = a.sh;
    t.theta = a.theta;
    t.pts = a.pts;
    t.pt_time = a.pt_time;
    t.n = a.n;
    t.d_f = a.d_f;
    t.d_grad = a.d_grad;
    t.wt = a.w.wbft;
    t.a0 = a.w.z0;
    t.z = reinterpret_cast<const float4*>(a.w.z);
    t.d = reinterpret_cast<float4*>(a.w.d);
    t.gain = a.w.gain + static_cast<size_t>(a.sh.n_hidden) * W;
    t.d_theta = a.d_theta;
    t.status = a.status;
    cudaError_t e = launch_tc(train32_bwd_kernel<W>, B32<W>::THREADS, B32<W>::TOTAL + 1024, 512, num_sms, s, &t);
    if (e != cudaSuccess) return e;
    return launch_tc(train32_wgrad_kernel<W>, Wg32<W>::THREADS, Wg32<W>::TOTAL + 1024, 512, num_sms, s, &t);
}

}  // namespace

cudaError_t launch_pack32_backward(const TrainArgs& a, int num_sms, cudaStream_t s) {
    return pack32(a, nullptr, num_sms, s);
}

cudaError_t launch_train_forward(const TrainArgs& a, int num_sms, cudaStream_t s) {
    switch (a.sh.width) {
    case 64:
        return forward32_w<64>(a, num_sms, s);
    case 128:
        return forward32_w<128>(a, num_sms, s);
    case 256:
        return forward32_w<256>(a, num_sms, s);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_train_backward(const TrainArgs& a, int num_sms, cudaStream_t s) {
    switch (a.sh.width) {
    case 64:
        return backward32_w<64>(a, num_sms, s);
    case 128:
        return backward32_w<128>(a, num_sms, s);
    case 256:
        return backward32_w<256>(a, num_sms, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace sdfnn
