// Analytic-gradient kernel (Alg. 2) of the FP32 path on the tensor cores,
// shared by normal mapping and the FP32 training forward.
//
// Normal mapping holds every FP32 operand as two half-precision values, the
// rounding h and the rounding l of 2^11 (x - h): 2 x 11 significand bits and the
// remainder's sign, so the pair misses x by at most 2^-24 of its binade, the half
// unit of a float, down to |x| = 2^-12 (below, by 2^-36).  A product is h h' +
// 2^-11 (l h' + h l') (l l' is below 2^-24), three tcgen05.mma per K step.  The
// operands are scaled by powers of two for it, unit by unit (split_image32 in
// api.cu, which also says how far a unit's tangents may stay below their bound).
//
// The training forward, whose parameters only the device knows, holds them as
// three bfloat16 values x0 + x1 + x2 instead (24 significand bits, a float's
// exponents, no scales) and keeps the six products x_i y_j with i + j <= 2;
// what is left out is below 2^-24 of the product.
//
// What decides the accuracy is the accumulation: the tensor core truncates
// the running sum to 24 bits once per K step of 16 (measured with random
// operands: the mean error has the sign opposite to the sum).  So h h' (x0 y0)
// has its own accumulator (the small products would otherwise truncate the
// large sum two to five more times per step), and the mean of the truncation is
// multiplied back in: a step takes about kStepLoss of the sum that it leaves, and
// after step s of a row w that sum is, in the mean, sum_{k <= s} w_k^2 / sum w_k^2
// of the whole.  So a row's gain is 1 + kStepLoss times the sum of these shares
// over the steps in which it has weights: 8.5 kStepLoss = 2.7e-7 for a dense row
// of 256, next to nothing for a row of a few weights, whose sums lose little.  (One
// gain for all rows would be an error of its own there.)  Contractions of 128 x K
// sines with K x 64 uniform weights on GB300, halves, root mean square error
// against FP64 in units of 1e-7, for K = 64 / 128 / 256: a chain of FP32 FMAs 1.8 /
// 3.7 / 7.2, one accumulator for all three products 3.9 / 9.7 / 24.9, two
// accumulators 1.6 / 3.5 / 8.7, with the gain 1.4 / 2.4 / 5.2.  (h h' of the upper
// half of K added to the complete small products instead, without a gain: 8
// truncations per accumulator, gradients of the (256,3) up to 18 % further off and 6 %
// slower.)
#pragma once

#include "tc_common.cuh"

namespace sdfnn {
namespace {

// P operand planes: 2 halves (head, remainder) or 3 bfloat16 values.
template <int W, int P>
struct G32 {
    static constexpr int PLANES = P;
    static constexpr bool F16 = P == 2;
    static constexpr int MT = (W + 127) / 128;      // TMEM tiles of 128 feature rows
    static constexpr int KB = W / 64;               // 64-wide K blocks of the contraction
    static constexpr int ROWS_PAD = MT * 128;
    static constexpr int NH = 2 / MT;               // independent tiles of 32 points ("halves") per CTA
    static constexpr int CS = 2;                    // threads per feature and half: each takes 32 / CS points
    static constexpr int HPTS = 32;
    static constexpr int CPTS = HPTS / CS;
    static constexpr int HROWS = 4 * HPTS;          // point-streams of a half = MMA N
    static constexpr uint32_t PLANE = W * 256u;     // bytes of one operand plane of a half
    // A ring unit is one plane of a K block for one TMEM tile (16 KB, consecutive in the weight image).
    static constexpr uint32_t UNIT = 16384u;
    static constexpr int UNITS = KB * P * MT;       // units per layer
    static constexpr int NS = P == 2 || W == 64 ? 6 : 2;  // (three planes of 64 KB leave room for two units)
    static constexpr int GROUP_WARPS = 4 * MT * CS;
    static constexpr int GROUP_THREADS = GROUP_WARPS * 32;
    static constexpr int EPI_WARPS = NH * GROUP_WARPS;
    static constexpr int PRODUCER_WARP = EPI_WARPS;
    static constexpr int MMA_WARP = EPI_WARPS + 1;
    static constexpr int THREADS = (EPI_WARPS + 2) * 32;
    static constexpr int TMEM_COLS = 512;           // (half or TMEM tile) * 256 + {0: h h' or x0 y0, 128: the small products}
};

struct G32Layout {
    uint32_t x, ring, pts, bars, misc, total;
};

template <class C>
__host__ __device__ inline G32Layout g32_layout() {
    G32Layout L;
    uint32_t o = 0;
    L.x = o;
    o += C::NH * C::PLANES * C::PLANE;
    L.ring = o;
    o += C::NS * C::UNIT;
    L.pts = o;
    o += C::NH * C::HPTS * 16u;
    L.bars = o;
    o += (2 * C::NS + 2 * C::NH) * 8u;
    o = (o + 15u) & ~15u;
    L.misc = o;
    o += 32u;
    L.total = o;
    return L;
}

// A remainder is held times 2^11: as large as its head, it is no smaller a half than the head is.
constexpr float kRemScale = 2048.0f;

// Two half planes of a pair of floats: the rounding of x and of 2^11 times what is left (exact).
__device__ __forceinline__ void split2x2(float a, float b, uint32_t (&p)[2]) {
    p[0] = pack16x2<true>(a, b);
    const float2 h = make_float2(from16<true>(static_cast<uint16_t>(p[0] & 0xFFFFu)),
                                 from16<true>(static_cast<uint16_t>(p[0] >> 16)));
    const float2 r = __fmul2_rn(__ffma2_rn(h, make_float2(-1.0f, -1.0f), make_float2(a, b)), make_float2(kRemScale, kRemScale));
    p[1] = pack16x2<true>(r.x, r.y);
}

// Three bfloat16 planes of a pair of floats: the rounding of x, of x minus
// that, and of what is left (the subtractions are exact).
__device__ __forceinline__ void split3x2(float a, float b, uint32_t (&p)[3]) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        p[i] = pack_bf16x2(a, b);
        if (i < 2) {
            const float2 r = __ffma2_rn(make_float2(__uint_as_float(p[i] << 16), __uint_as_float(p[i] & 0xFFFF0000u)),
                                        make_float2(-1.0f, -1.0f), make_float2(a, b));
            a = r.x;
            b = r.y;
        }
    }
}

// Two points (four streams each) of one feature as 16-byte chunks of the P planes.
template <int P>
__device__ __forceinline__ void store_split(uint32_t x_s, uint32_t plane, uint32_t off, const float (&v)[8]) {
    uint32_t q[4][P];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        if constexpr (P == 2)
            split2x2(v[2 * e], v[2 * e + 1], q[e]);
        else
            split3x2(v[2 * e], v[2 * e + 1], q[e]);
    }
#pragma unroll
    for (int i = 0; i < P; ++i) st_shared_v4(x_s + i * plane + off, q[0][i], q[1][i], q[2][i], q[3][i]);
}

// Byte offset in a half's MN-major plane of the chunk holding points 2c, 2c + 1 for feature m.
template <int W>
__device__ __forceinline__ uint32_t xoff32(int m, int c) {
    return static_cast<uint32_t>(c >> 3) * (W * 128u) + static_cast<uint32_t>(m >> 3) * 1024u +
           static_cast<uint32_t>(m & 7) * 128u + (static_cast<uint32_t>((c & 7) ^ (m & 7)) << 4);
}

// Sum over the 32 lanes of a warp of each of v[0..15]: afterwards lane L holds,
// in v[0], the sum of entry L / 2 (recursive halving, 16 shuffles).
__device__ __forceinline__ void warp_sum16(float (&v)[16], int lane) {
#pragma unroll
    for (int s = 8; s >= 1; s >>= 1) {
        const bool upper = (lane & (2 * s)) != 0;
#pragma unroll
        for (int i = 0; i < s; ++i) {
            const float send = upper ? v[i] : v[i + s];
            const float keep = upper ? v[i + s] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * s);
        }
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// Index of point j (j < 0: none) of half h of this CTA's set i (-1 past the work).
template <int NH, int HPTS>
__device__ __forceinline__ int g32_index(const GradArgs& a, long long n_work, int h, int j, int i) {
    const long long k = ((static_cast<long long>(i) * gridDim.x + blockIdx.x) * NH + h) * HPTS + j;
    if (j < 0 || k >= n_work) return -1;
    return a.list ? __ldg(a.list + k) : static_cast<int>(k);
}

// Copies (x, y, z, t) of point idx into the float4 at shared address dst
// (zeros for idx < 0); complete after cp_async_wait_all in the same thread.
__device__ __forceinline__ void g32_point_async(uint32_t dst, const GradArgs& a, bool timed, int idx) {
    if (idx < 0) {
        st_shared_v4(dst, 0u, 0u, 0u, 0u);
        return;
    }
    cp_async4(dst, a.pts + idx);
    cp_async4(dst + 4u, a.pts + a.n + idx);
    cp_async4(dst + 8u, a.pts + 2 * a.n + idx);
    if (timed)
        cp_async4(dst + 12u, a.pt_time + idx);
    else
        st_shared_u32(dst + 12u, 0u);
}

// The MMAs of one layer for one half: Y = W X in the ring's order of units (per K block the planes of W, per plane
// the TMEM tiles).  d holds x0 y0, d + 128 the small products.  One accumulator and one shape per chain of MMAs:
// only such instructions are ordered among themselves.  (The first plane times two planes of X as one instruction of
// N = 256 over both accumulators would overlap the other products' N = 128 with nothing between them.)
template <class C>
__device__ __forceinline__ bool mma_layer32(uint32_t tmem, int h, uint64_t xd0, uint32_t ring_s, uint32_t bar_full,
                                            uint32_t bar_empty, uint32_t& g, int* status, volatile int* abort_flag) {
    constexpr uint32_t idesc = idesc_f32acc(128, C::HROWS, C::F16) | kIdescMajorMnB;
    for (int kb = 0; kb < C::KB; ++kb)
        for (int p = 0; p < C::PLANES; ++p)
            for (int mt = 0; mt < C::MT; ++mt, ++g) {
                const uint32_t stage = g % C::NS, use = g / C::NS;
                if (!mbar_wait_bounded(bar_full + 8u * stage, use & 1u, status, abort_flag)) return false;
                tc_fence_after();
                const uint64_t wd0 = desc_kmajor_sw128(ring_s + stage * C::UNIT);
                const uint32_t d = tmem + (mt + h) * 256u;
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const uint64_t wd = desc_add(wd0, kk * 32u);
                    const uint64_t xd = desc_add(xd0, static_cast<uint32_t>(kb * 8 + kk * 2) * 1024u);
                    if (p == 0) {
                        mma_f16kind(d, wd, xd, idesc, (kb | kk) != 0);
                        mma_f16kind(d + 128u, wd, desc_add(xd, C::PLANE), idesc, (kb | kk) != 0);
                        if (C::PLANES == 3) mma_f16kind(d + 128u, wd, desc_add(xd, 2 * C::PLANE), idesc, 1u);
                    } else {
                        mma_f16kind(d + 128u, wd, xd, idesc, 1u);
                        if (C::PLANES == 3 && p == 1) mma_f16kind(d + 128u, wd, desc_add(xd, C::PLANE), idesc, 1u);
                    }
                }
                mma_commit(bar_empty + 8u * stage);
            }
    return true;
}

// Same skeleton as grad_tc_kernel (features as MMA rows, N = 32 points x 4
// streams, a producer warp streaming the weights, an MMA warp, epilogue groups
// that own a feature per thread), with these differences: operands in
// planes and two accumulators; at width 256 the planes of one half fill
// the activation memory, so the CTA runs one half of 32 points (its MMAs, 96 of
// about 77 clocks a layer, and epilogue, about as long, take turns; an MMA of N =
// 64 costs its issuer the same 77, so two halves of 16 points lose: the training
// forward of the (128,2) 93 -> 113 us); two threads share a
// feature, so 16 epilogue warps hide the sines' latency; the output layer
// runs in FP32 on the CUDA cores (w_out times the last tangents, summed over
// the features by a warp butterfly and, in a fixed order, over the warps).
// The FP32 FMA units did the same products before (grad_simt_kernel, now for
// networks beyond the scales only): a call of 20,011 points of a (256,3) 0.73
// -> 0.124 ms, of a (128,2) 0.168 -> 0.040, of a (64,2) 0.074 -> 0.049 (the
// last two bound by the host), the error against FP64 4 to 14 % lower on each
// of six networks.  What bounds the (256,3) now is the alternation of MMAs and
// epilogue (14.7 k clocks a layer and tile).
//
// TRAIN: the training forward.  It saves A_0 ([n][W]) and (A_l, H_l^x, H_l^y,
// H_l^z) ([k][n][W] float4: a warp's store is 512 consecutive bytes) and also
// writes f (no list, no normalisation).  Bound by its MMAs, six per K step: 93 us
// for 50,001 points of the (128,2), where halves under a scale per layer, which
// some networks exceed, took 68.
template <int W, bool TRAIN = false>
__global__ void __launch_bounds__(G32<W, TRAIN ? 3 : 2>::THREADS, 1) grad32_tc_kernel(const GradArgs a) {
    using C = G32<W, TRAIN ? 3 : 2>;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t raw_s = smem_u32(smem_raw);
    const uint32_t base_s = (raw_s + 1023u) & ~1023u;
    uint8_t* base = smem_raw + (base_s - raw_s);
    const NetView& net = a.net;
    const int KH = net.n_hidden;
    const G32Layout L = g32_layout<C>();
    const float4* pts = reinterpret_cast<const float4*>(base + L.pts);
    const uint32_t bar_full = base_s + L.bars;
    const uint32_t bar_empty = bar_full + 8u * C::NS;
    const uint32_t bar_xready = bar_empty + 8u * C::NS;
    const uint32_t bar_dfull = bar_xready + 8u * C::NH;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(base + L.misc);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(base + L.misc + 4);
    const uint32_t x_s = base_s + L.x, ring_s = base_s + L.ring;
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
        tmem_alloc(smem_u32(tmem_slot), C::TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    // Static schedule: half h of CTA b takes the tiles of 32 points b * NH + h, + G * NH, ...; all halves
    // of a CTA run the same number of tiles (one beyond the work has no valid point).
    const long long n_work = a.list ? static_cast<long long>(*a.count) : a.n;
    const long long n_sets = (n_work + C::NH * C::HPTS - 1) / (C::NH * C::HPTS);
    const long long G = gridDim.x;
    const int my_sets = static_cast<int>(n_sets > blockIdx.x ? (n_sets - blockIdx.x + G - 1) / G : 0);
    const int n_groups = my_sets * KH;  // (tile, hidden layer) pairs of each half, in order
    bool ok = true;

    if (warp == C::PRODUCER_WARP) {
        if (lane == 0) {
            uint32_t g = 0;
            int l = 0;
            for (int k = 0; k < n_groups && ok; ++k) {
                const uint8_t* src = net.wbf + static_cast<size_t>(l) * net.wbf_layer_bytes;
                for (int h = 0; h < C::NH && ok; ++h)
                    for (int u = 0; u < C::UNITS && ok; ++u, ++g) {
                        const uint32_t stage = g % C::NS, use = g / C::NS;
                        if (use > 0) ok = mbar_wait_bounded(bar_empty + 8u * stage, (use - 1) & 1u, a.status, abort_flag);
                        if (!ok) break;
                        mbar_arrive_expect_tx(bar_full + 8u * stage, C::UNIT);
                        bulk_g2s(ring_s + stage * C::UNIT, src + u * C::UNIT, C::UNIT, bar_full + 8u * stage);
                    }
                l = l + 1 == KH ? 0 : l + 1;
            }
            // every copy issued must land before the block exits
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
                    const uint64_t xd0 = desc_mnmajor_sw128(x_s + h * C::PLANES * C::PLANE, W * 128u);
                    ok = mma_layer32<C>(tmem, h, xd0, ring_s, bar_full, bar_empty, g, a.status, abort_flag);
                    if (ok) mma_commit(bar_dfull + 8u * h);
                }
        }
    } else {
        // epilogue group h: thread <-> feature m, points cs * CPTS .. of half h
        const int h = warp / C::GROUP_WARPS, ge = warp % C::GROUP_WARPS;
        const int mt = (ge >> 2) % C::MT, cs = (ge >> 2) / C::MT, quad = ge & 3;
        const int m = mt * 128 + quad * 32 + lane;
        const bool live = mt * 128 + quad * 32 < W;  // warp-uniform
        const int gt = ge * 32 + lane;
        const uint32_t d_s = tmem + (static_cast<uint32_t>(quad * 32) << 16) + (mt + h) * 256u + cs * (C::CPTS * 4u);
        const uint32_t xh = x_s + h * C::PLANES * C::PLANE;
        const int p0 = h * C::HPTS, q0 = p0 + cs * C::CPTS;
        // output sums of the half: one row of HROWS floats per 32 features, in the half's activation
        // memory (free between the last MMA of a tile and the next tile's input layer)
        float* red = reinterpret_cast<float*>(base + L.x + h * C::PLANES * C::PLANE);
        const bool timed = a.pt_time != nullptr && net.in_dim == 4;
        float4 u0 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        float ut = 0.0f, wo = 0.0f;
        if (live) {
            const float* w0 = net.w0 + m * net.in_dim;
            u0 = make_float4(__ldg(w0), __ldg(w0 + 1), __ldg(w0 + 2), __ldg(net.b0 + m));
            const float wt = net.in_dim == 4 ? __ldg(w0 + 3) : 0.0f;
            if (timed)
                ut = wt;
            else
                u0.w = fmaf(wt, a.time, u0.w);
            wo = __ldg(net.wout + m);
        }
        // normal mapping: this feature's scales (split_image32 in api.cu), entry 0 for the input layer
        const float4* scales = reinterpret_cast<const float4*>(net.s32) + m;
        float4 sc = make_float4(1.0f, 1.0f, 1.0f, 0.0f);
        if (!TRAIN && live) sc = __ldg(scales);
        const float p_in = sc.x, g_in = sc.y;
        // Thread gt < HPTS holds the index of point gt; the next tile's index is loaded a tile ahead and its
        // coordinates are copied during this tile's layers, so no global load sits between two tiles.
        int idx = -1, nidx = -1;
        if (gt < C::HPTS) {
            nidx = g32_index<C::NH, C::HPTS>(a, n_work, h, my_sets > 0 ? gt : -1, 0);
            g32_point_async(base_s + L.pts + static_cast<uint32_t>(p0 + gt) * 16u, a, timed, nidx);
        }
        uint32_t df_phase = 0;
        for (int i = 0; i < my_sets; ++i) {
            if (gt < C::HPTS) {
                cp_async_wait_all();
                idx = nidx;
                nidx = g32_index<C::NH, C::HPTS>(a, n_work, h, i + 1 < my_sets ? gt : -1, i + 1);
            }
            bar_named(1 + h, C::GROUP_THREADS);
            // TRAIN: this thread's first point, and how many of its points are in the batch
            const long long pb = ((static_cast<long long>(i) * G + blockIdx.x) * C::NH + h) * C::HPTS + cs * C::CPTS;
            const int nv = TRAIN ? static_cast<int>(min(max(a.n - pb, 0ll), static_cast<long long>(C::CPTS))) : 0;
            // input layer: P_0 = sin(A_0), G_0^c = W_0[:, c] (.) cos(A_0), at the feature's scales
            if (live) {
#pragma unroll 2
                for (int c = 0; c < C::CPTS / 2; ++c) {
                    float v[8];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const float4 q = pts[q0 + 2 * c + e];
                        const float z = fmaf(u0.x, q.x, fmaf(u0.y, q.y, fmaf(u0.z, q.z, fmaf(ut, q.w, u0.w))));
                        if (TRAIN && 2 * c + e < nv) a.save_a0[(pb + 2 * c + e) * W + m] = z;
                        float sn, cn;
                        sincos_r(z, &sn, &cn);
                        cn *= g_in;
                        v[4 * e] = TRAIN ? sn : sn * p_in;
                        v[4 * e + 1] = u0.x * cn;
                        v[4 * e + 2] = u0.y * cn;
                        v[4 * e + 3] = u0.z * cn;
                    }
                    store_split<C::PLANES>(xh, C::PLANE, xoff32<W>(m, cs * (C::CPTS / 2) + c), v);
                }
            }
            fence_proxy_async_smem();
            tc_fence_before();
            mbar_arrive(bar_xready + 8u * h);

            for (int l = 0; l < KH && ok; ++l) {
                ok = __all_sync(0xffffffffu, mbar_wait_bounded(bar_dfull + 8u * h, df_phase, a.status, abort_flag));
                df_phase ^= 1u;
                if (!ok) break;
                if (l == 0 && gt < C::HPTS)
                    g32_point_async(base_s + L.pts + static_cast<uint32_t>(p0 + gt) * 16u, a, timed, nidx);
                tc_fence_after();
                if (!live) {
                    fence_proxy_async_smem();
                    tc_fence_before();
                    if (l + 1 < KH) mbar_arrive(bar_xready + 8u * h);
                    continue;
                }
                const bool last = l + 1 == KH;
                const float gain = TRAIN ? __ldg(net.s32 + l * W + m) : 1.0f;
                // from the accumulators to A, from the tangents' to the next operand (the last layer: to values
                // times w_out), and the next operand's scale of the sines
                sc = TRAIN ? make_float4(gain, gain, 1.0f, 0.0f) : __ldg(scales + (l + 1) * W);
                const float bb = __ldg(net.bh[l] + m), mg = last ? wo * sc.y : sc.y;
                constexpr float lo = TRAIN ? 1.0f : 1.0f / kRemScale;
                float4* save = TRAIN ? reinterpret_cast<float4*>(a.save_a) + (static_cast<size_t>(l) * a.n + pb) * W + m : nullptr;
#pragma unroll 1
                for (int q = 0; q < C::CPTS / 4; ++q) {
                    // four points: 16 columns of each accumulator
                    float v[16], c[16];
                    tmem_ld16(d_s + q * 16u, v);
                    tmem_ld16(d_s + 128u + q * 16u, c);
                    tmem_wait_ld();
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int j = 4 * e;
#pragma unroll
                        for (int s = 0; s < 4; s += 2) {
                            const float2 r = __ffma2_rn(make_float2(c[j + s], c[j + s + 1]), make_float2(lo, lo),
                                                        make_float2(v[j + s], v[j + s + 1]));
                            v[j + s] = r.x;
                            v[j + s + 1] = r.y;
                        }
                        const float A = fmaf(v[j], sc.x, bb);
                        if (TRAIN && 4 * q + e < nv)
                            save[(4 * q + e) * W] = make_float4(A, v[j + 1] * sc.y, v[j + 2] * sc.y, v[j + 3] * sc.y);
                        float sn, cn;
                        sincos_r(A, &sn, &cn);
                        cn *= mg;
                        const float ps = TRAIN ? (last ? wo : 1.0f) : sc.z;
                        const float2 r01 = __fmul2_rn(make_float2(sn, v[j + 1]), make_float2(ps, cn));
                        const float2 r23 = __fmul2_rn(make_float2(v[j + 2], v[j + 3]), make_float2(cn, cn));
                        v[j] = r01.x;
                        v[j + 1] = r01.y;
                        v[j + 2] = r23.x;
                        v[j + 3] = r23.y;
                    }
                    if (last) {
                        warp_sum16(v, lane);
                        if ((lane & 1) == 0) red[(mt * 4 + quad) * C::HROWS + cs * (C::CPTS * 4) + q * 16 + (lane >> 1)] = v[0];
                    } else {
                        const float(&lo8)[8] = *reinterpret_cast<const float(*)[8]>(&v[0]);
                        const float(&hi8)[8] = *reinterpret_cast<const float(*)[8]>(&v[8]);
                        store_split<C::PLANES>(xh, C::PLANE, xoff32<W>(m, cs * (C::CPTS / 2) + 2 * q), lo8);
                        store_split<C::PLANES>(xh, C::PLANE, xoff32<W>(m, cs * (C::CPTS / 2) + 2 * q + 1), hi8);
                    }
                }
                fence_proxy_async_smem();
                tc_fence_before();
                if (!last) mbar_arrive(bar_xready + 8u * h);
            }
            // one decision for the group; the output rows of red are complete
            if (bar_or(1 + h, C::GROUP_THREADS, !ok || *abort_flag != 0)) break;
            if (gt < C::HPTS) {
                if (idx >= 0) {
                    float f = 0.0f, gx = 0.0f, gy = 0.0f, gz = 0.0f;
#pragma unroll
                    for (int r = 0; r < W / 32; ++r) {
                        const float4 t = *reinterpret_cast<const float4*>(red + r * C::HROWS + gt * 4);
                        f += t.x;
                        gx += t.y;
                        gy += t.z;
                        gz += t.w;
                    }
                    if (TRAIN) a.out_f[idx] = f + __ldg(a.out_bias);
                    if (a.normalize) {
                        const float len = sqrtf(gx * gx + gy * gy + gz * gz);
                        const float inv = len >= 1e-12f ? 1.0f / len : 0.0f;
                        gx *= inv;
                        gy *= inv;
                        gz *= inv;
                    }
                    a.out[idx] = gx;
                    a.out[a.n + idx] = gy;
                    a.out[2 * a.n + idx] = gz;
                }
            }
            // the barrier at the top of the next tile orders these reads of red before its input layer
        }
        if (gt < C::HPTS) cp_async_wait_all();
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, C::TMEM_COLS);
    }
}

}  // namespace
}  // namespace sdfnn
