// Trace kernel with several threads per ray (tcgen05; 16-bit and E4M3 operands).
#pragma once

#include "rays.cuh"
#include "tc_common.cuh"

namespace sdfnn {
namespace {

// The state machine and arithmetic of trace_level_tc_kernel, arranged for short
// steps instead of many tiles: CS threads share a ray, each computing W / CS
// units of layer 0 and of every epilogue.  A step is a serial chain (layer 0,
// MMAs, epilogues, output, step) that a ray repeats tens of times; with one
// thread per ray the W sines of a layer are one warp's instruction stream, and a
// frame of few rays, or the long rays of any frame, waits on its latency while
// the SM idles.
//
//   width 64 (weights resident, one tile, CS = 4): calls of few rays.
//   width 128, head + remainder operands (resident, one tile, CS = 4): the
//     weights of two layers leave room for one tile of activations per SM, which
//     had 128 threads; with one layer, small calls only.
//   width 256 (weights streamed through a ring; large calls of a single layer
//     run trace_single_tc_kernel): two tiles that share every weight unit, CS =
//     2; for calls of at most 128 rays per SM one tile, CS = 4 and a third ring
//     stage (a lone tile's MMAs consume a unit faster than two outstanding copies
//     bring them).
//
// What it measured (one call, us, before -> after): a 128 x 128 trace of the
// Lipschitz-stepped (64,1) 159 .. 191 -> 80; the plain (256,3) trace of 100^2 rays
// 822 -> 461 (one tile, third stage), of 1280 x 720 2,704 -> 2,492; a nested (64,2) > (128,2) > (256,2) frame of 150^2 rays 700 -> 554, of
// 512^2 1,046 -> 999.  At width 256 the two tiles' MMAs and epilogues still take turns, and
// a lone tile waits for its weights (9 k clocks a layer with two stages).
// Handing the rays left at the end of a level to a second, one-tile launch was
// tried: 3 % faster on the plain 1280 x 720 trace, 6 to 20 % slower on the
// nested frames, whose levels are short.
//
// Every value is computed as trace_level_tc_kernel computes it, whatever the
// kernel, tile or thread: the same MMAs in the same order, and the output
// layer's two FMA chains run over the units in order (the first part's thread
// continues them over the other parts' sines, left in shared memory).
template <int W, int OP, bool SPLIT, int TILES = W == 256 ? 2 : 1>
struct WideCfg {
    static constexpr bool FP8 = OP == kOpE4M3, F16 = OP == kOpF16;
    static constexpr int EB = FP8 ? 1 : 2;          // operand bytes per element
    static constexpr bool RES = W < 256;
    static constexpr int ST = TILES;                // tiles of 128 rays
    static constexpr int CS = 4 / ST;
    static constexpr int TT = 128 * CS;             // threads of a tile
    static constexpr int NRT = TT * ST;             // ray threads
    static constexpr int THREADS = NRT + 32;        // and the producer warp
    static constexpr int PL = SPLIT ? 2 : 1;        // operand planes (head, remainder)
    static constexpr int KB = W * EB / 128;         // K blocks of 128 bytes
    static constexpr uint32_t PLANE = 128u * W * EB;
    static constexpr uint32_t UNIT = W * 128u;      // one plane of a K block of the weights
    static constexpr int NS = ST == 1 ? 3 : 2;      // ring stages (streamed weights)
    static constexpr int UPT = W / CS;              // units per thread
    static constexpr uint32_t SINES = (W - UPT) * ST * 128u * 4u;  // last-layer sines of parts 1 .. CS-1
    static constexpr uint32_t X = ST * PL * PLANE > SINES ? ST * PL * PLANE : SINES;
    static constexpr int TMEM_COLS = W * ST;
};

struct WideLayout {
    uint32_t w, w0, wt, bh, wout, pos, act, bars, misc, total;
};

constexpr int kWideRegroup = 4;  // steps between two regroupings of the remaining rays

template <class C, int W>
__host__ __device__ inline WideLayout wide_layout(int KH) {
    WideLayout L;
    uint32_t o = C::X;
    L.w = o;
    o += (C::RES ? KH * C::PL * C::KB : C::NS) * C::UNIT;
    L.w0 = o;
    o += W * 16u;
    L.wt = o;
    o += W * 4u;
    L.bh = o;
    o += static_cast<uint32_t>(KH) * W * 4u;
    L.wout = o;
    o += W * 4u;
    L.pos = o;
    o += C::ST * 128u * 16u;
    L.act = o;
    o += 32u;
    L.bars = o;
    o += 8u * (2 * C::NS + 1);
    o = (o + 15u) & ~15u;
    L.misc = o;
    o += 32u;
    L.total = o;
    return L;
}

// 16 sines of one ray row (units u0 .. u0+15) into X.
template <class C>
__device__ __forceinline__ void wide_store16(uint32_t x_s, int row, int u0, const float (&v)[16]) {
    if constexpr (C::FP8) {
        uint32_t w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e)
            w[e] = pack_e4m3x4(kFp8ActScale * v[4 * e], kFp8ActScale * v[4 * e + 1], kFp8ActScale * v[4 * e + 2],
                               kFp8ActScale * v[4 * e + 3]);
        st_shared_v4(x_s + sw128_chunk_offset(row, u0 >> 4, 128), w[0], w[1], w[2], w[3]);
    } else {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            uint32_t h[4], l[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (C::PL == 2)
                    pack_split<C::F16>(v[8 * q + 2 * e], v[8 * q + 2 * e + 1], h[e], l[e]);
                else
                    h[e] = pack16x2<C::F16>(v[8 * q + 2 * e], v[8 * q + 2 * e + 1]);
            }
            const uint32_t off = sw128_chunk_offset(row, (u0 >> 3) + q, 128);
            st_shared_v4(x_s + off, h[0], h[1], h[2], h[3]);
            if (C::PL == 2) st_shared_v4(x_s + C::PLANE + off, l[0], l[1], l[2], l[3]);
        }
    }
}

// Polls without suspending the thread: the waits of a step are short and all
// on its critical path.
__device__ __forceinline__ bool mbar_wait_spin(uint32_t bar, uint32_t parity, int* status, volatile int* abort_flag) {
    if (mbar_test_wait(bar, parity)) return true;
    const uint64_t t0 = globaltimer_ns();
    while (true) {
#pragma unroll 1
        for (int i = 0; i < 64; ++i)
            if (mbar_test_wait(bar, parity)) return true;
        if (*abort_flag) return false;
        if (globaltimer_ns() - t0 > kWaitBudgetNs) {
            raise_status(status, kStatusTimeout);
            *abort_flag = 1;
            return false;
        }
    }
}

// refill_ray, without the work counter once this CTA has seen it run out
// (*dry): an atomic's round trip would delay every step in which a ray ends.
// Other warps set *dry meanwhile and refill_ray is a collective of the warp, so
// the warp decides as one: by what any of its lanes has read.
__device__ __forceinline__ void wide_refill(const LevelArgs& a, Ray& r, long long n_work, volatile int* dry) {
    if (__any_sync(0xffffffffu, *dry != 0)) {
        if (r.state == kSlotEmpty) r.state = kSlotDone;
        return;
    }
    refill_ray(a, r, n_work);
    if (r.state == kSlotDone) *dry = 1;
}

template <int W, int OP, bool SPLIT, int TILES>
__global__ void __launch_bounds__(WideCfg<W, OP, SPLIT, TILES>::THREADS, 1) trace_wide_kernel(const LevelArgs a) {
    using C = WideCfg<W, OP, SPLIT, TILES>;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t raw_s = smem_u32(smem_raw);
    const uint32_t base_s = (raw_s + 1023u) & ~1023u;
    uint8_t* base = smem_raw + (base_s - raw_s);
    const NetView& net = a.net;
    const int KH = net.n_hidden;
    const WideLayout L = wide_layout<C, W>(KH);
    float* w0s = reinterpret_cast<float*>(base + L.w0);
    float* wts = reinterpret_cast<float*>(base + L.wt);
    float* bhs = reinterpret_cast<float*>(base + L.bh);
    float* wos = reinterpret_cast<float*>(base + L.wout);
    float4* pos = reinterpret_cast<float4*>(base + L.pos);
    volatile int* act = reinterpret_cast<volatile int*>(base + L.act);  // [4 ST]: any active ray in an owner warp
    float4* sines = reinterpret_cast<float4*>(base);  // [(W - UPT) / 4][ST * 128], while X is free
    const uint32_t bar_full = base_s + L.bars, bar_empty = bar_full + 8u * C::NS, bar_mma = bar_empty + 8u * C::NS;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(base + L.misc);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(base + L.misc + 4);
    volatile int* done_flag = reinterpret_cast<volatile int*>(base + L.misc + 8);
    volatile uint32_t* consumed = reinterpret_cast<volatile uint32_t*>(base + L.misc + 12);
    volatile int* dry = reinterpret_cast<volatile int*>(base + L.misc + 16);  // the level's work has run out
    int* left = reinterpret_cast<int*>(base + L.misc + 20);                   // rays counted by a regrouping
    const uint32_t w_s = base_s + L.w;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (tid == 0) {
        for (int s = 0; s < C::NS; ++s) {
            mbar_init(bar_full + 8u * s, 1);
            mbar_init(bar_empty + 8u * s, 1);
        }
        mbar_init(bar_mma, 1);
        *abort_flag = 0;
        *done_flag = 0;
        *consumed = 0;
        *dry = 0;
        *left = 0;
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(smem_u32(tmem_slot), C::TMEM_COLS);
        tmem_relinquish();
    }
    const bool timed = a.ray_time != nullptr && net.in_dim == 4;
    for (int i = tid; i < W; i += C::THREADS) {
        stage_layer0_pairs(net, a.time, timed, i, w0s, wts);
        wos[i] = net.wout[i];
        for (int l = 0; l < KH; ++l) bhs[l * W + i] = net.bh[l][i];
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == C::NRT / 32) {
        if (lane == 0 && C::RES) {
            // resident weights: per layer and K block the head, then the remainder
            mbar_arrive_expect_tx(bar_full, static_cast<uint32_t>(KH * C::PL * C::KB) * C::UNIT);
            uint32_t dst = w_s;
            for (int l = 0; l < KH; ++l)
                for (int kb = 0; kb < C::KB; ++kb) {
                    const size_t src = static_cast<size_t>(l) * net.wbf_layer_bytes + static_cast<size_t>(kb) * net.rows_pad * 128u;
                    bulk_g2s(dst, net.wbf + src, C::UNIT, bar_full);
                    dst += C::UNIT;
                    if (C::PL == 2) {
                        bulk_g2s(dst, net.wbf_lo + src, C::UNIT, bar_full);
                        dst += C::UNIT;
                    }
                }
            mbar_drain(bar_full, 0u);
        } else if (lane == 0) {
            // streamed weights: the K blocks of layer 0 .. KH-1 in consumption order, cyclically, until the rays
            // are done
            uint32_t g = 0;
            int l = 0, kb = 0;
            while (true) {
                const uint32_t stage = g % C::NS, use = g / C::NS;
                if (use > 0) {
                    const uint32_t bar = bar_empty + 8u * stage, par = (use - 1) & 1u;
                    const uint64_t t0 = globaltimer_ns();
                    bool got = false;
                    while (!(got = mbar_try_wait(bar, par))) {
                        if (*done_flag || *abort_flag) break;
                        if (globaltimer_ns() - t0 > kWaitBudgetNs) {
                            raise_status(a.status, kStatusTimeout);
                            *abort_flag = 1;
                            break;
                        }
                    }
                    if (!got) break;
                }
                mbar_arrive_expect_tx(bar_full + 8u * stage, C::UNIT);
                bulk_g2s(w_s + stage * C::UNIT,
                         net.wbf + static_cast<size_t>(l) * net.wbf_layer_bytes + static_cast<size_t>(kb) * net.rows_pad * 128u,
                         C::UNIT, bar_full + 8u * stage);
                if (++kb == C::KB) {
                    kb = 0;
                    l = l + 1 == KH ? 0 : l + 1;
                }
                ++g;
            }
            // every copy issued must land before the block exits
            for (uint32_t gg = *consumed; gg < g; ++gg) mbar_drain(bar_full + 8u * (gg % C::NS), (gg / C::NS) & 1u);
        }
    } else {
        const long long n_work = a.in_list ? static_cast<long long>(*a.in_count) : a.n;
        const int row = tid & 127, tile = tid / C::TT, part = (tid / 128) % C::CS, u0 = part * C::UPT;
        const int slot = tile * 128 + row;
        const bool owner = part == 0;
        const bool issuer = tid == C::NRT - 128;  // lane 0 of the last part's first warp
        const uint32_t x_s = base_s + static_cast<uint32_t>(tile) * (C::PL * C::PLANE);
        const uint32_t d_s = tmem + static_cast<uint32_t>(tile * W + u0) + (static_cast<uint32_t>((row >> 5) * 32) << 16);
        // E4M3: the format fields 0 of this descriptor select E4M3 under kind::f8f6f4
        constexpr uint32_t idesc = idesc_f32acc(128, W, C::F16 || C::FP8);
        const uint64_t xd0 = desc_kmajor_sw128(base_s), wd0 = desc_kmajor_sw128(w_s);
        uint32_t mma_phase = 0, g = 0;
        bool issue_ok = true;  // the issuer: every weight unit so far arrived in time
        int regroup = 0;  // 0: the work lasts; else the steps to the next regrouping, + 1
        Ray ray;
        // Few rays: in the first turn one warp of owners per CTA takes them, or two, ..., as far as the work needs: a
        // CTA's step is shorter with fewer.  If work is left then (not every CTA has an SM yet), the others take part.
        // With layer 0 below, the (64,1) coarse trace of 49 x 38 rays takes 79 us (first come, first served: 97;
        // trace_level_tc_kernel: 93), of 64 x 64 78.5 (97; 109), the Lipschitz-stepped one of 32 x 32 64 (79; 95).
        bool holds = static_cast<long long>(slot >> 5) * 32 * gridDim.x >= n_work;
        // Layer 0 of a row is computed by warps of all four schedulers.  (TMEM lanes go by the warp's number, so the
        // warps that read a row's accumulators share one, and late in a level few rows have a ray.)
        const int row0 = (row + 32 * part) & 127, slot0 = tile * 128 + row0;
        // Stop decisions go through the ray threads' barrier: a timed-out wait drops the rays (the status
        // word reports it) instead of leaving the loop.
        while (true) {
            if (C::ST == 2 && regroup == 1) {
                // two tiles, and no more work: every kWideRegroup steps the rays that remain are dealt out again to
                // the first slots, so that the second tile (its MMAs, then its epilogues) drops out early
                bar_named(1, C::NRT);  // the sines have been read: X is free for the records
                float4* rec = reinterpret_cast<float4*>(base);
                if (owner && ray.state == kSlotActive) {
                    float4* q = rec + 3 * atomicAdd(left, 1);
                    q[0] = make_float4(__int_as_float(ray.idx), __int_as_float(ray.nlev), __int_as_float(ray.ntot), ray.tau);
                    q[1] = make_float4(ray.px, ray.py, ray.pz, ray.vx);
                    q[2] = make_float4(ray.vy, ray.vz, 0.0f, 0.0f);
                }
                bar_named(1, C::NRT);
                if (owner) {
                    ray.state = kSlotDone;
                    if (slot < *left) {
                        const float4 u = rec[3 * slot], v = rec[3 * slot + 1], w = rec[3 * slot + 2];
                        ray.idx = __float_as_int(u.x);
                        ray.nlev = __float_as_int(u.y);
                        ray.ntot = __float_as_int(u.z);
                        ray.tau = u.w;
                        ray.px = v.x;
                        ray.py = v.y;
                        ray.pz = v.z;
                        ray.vx = v.w;
                        ray.vy = w.x;
                        ray.vz = w.y;
                        ray.state = kSlotActive;
                    }
                }
            }
            if (owner) {
                if (!holds) wide_refill(a, ray, n_work, dry);
                holds = false;
                const bool on = ray.state == kSlotActive;
                pos[slot] = make_float4(ray.px, ray.py, ray.pz, timed && on ? __ldg(a.ray_time + ray.idx) : 0.0f);
                const bool any = __any_sync(0xffffffffu, on);
                if (lane == 0) act[slot >> 5] = any ? 1 : 0;
            }
            if (!bar_or(1, C::NRT, owner && ray.state == kSlotActive)) break;
            if (C::ST == 2 && a.cap > 0) {
                // *dry and *left change before that barrier only (another one follows this read): the same decision
                // in every thread.  A level without steps has one barrier per turn and nothing to regroup.
                if (regroup == 1 && tid == 0) *left = 0;
                regroup = *dry == 0 ? 0 : regroup <= 1 ? kWideRegroup + (regroup == 0 ? 0 : 1) : regroup - 1;
            }
            if (a.cap <= 0) {
                if (owner) pass_ray(a, ray);
                continue;
            }
            const bool wact = act[slot >> 5] != 0;  // rows of 32 slots without a ray are skipped (warp-uniform)
            if (act[slot0 >> 5] != 0) {
                const float4 p = pos[slot0];
                const float2 px = make_float2(p.x, p.x), py = make_float2(p.y, p.y), pz = make_float2(p.z, p.z),
                             pt = make_float2(p.w, p.w);
#pragma unroll 1
                for (int j = 0; j < C::UPT / 16; ++j) {
                    float v[16];
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const int pr = (u0 >> 1) + j * 8 + q;
                        const float4 A = reinterpret_cast<const float4*>(w0s)[2 * pr];
                        const float4 B = reinterpret_cast<const float4*>(w0s)[2 * pr + 1];
                        float2 c = make_float2(B.z, B.w);
                        if (timed) c = __ffma2_rn(reinterpret_cast<const float2*>(wts)[pr], pt, c);
                        const float2 z = __ffma2_rn(
                            make_float2(A.x, A.y), px,
                            __ffma2_rn(make_float2(A.z, A.w), py, __ffma2_rn(make_float2(B.x, B.y), pz, c)));
                        v[2 * q] = sin_fast(z.x);
                        v[2 * q + 1] = sin_fast(z.y);
                    }
                    wide_store16<C>(x_s, row0, u0 + j * 16, v);
                }
            }
            fence_proxy_async_smem();
            tc_fence_before();
            bar_named(1, C::NRT);

            bool good = true;
            float2 acc01 = make_float2(0.0f, 0.0f), acc23 = make_float2(0.0f, 0.0f);
            for (int l = 0; l < KH; ++l) {
                if (issuer) {
                    tc_fence_after();
                    if (C::RES) {
                        if (g == 0) issue_ok = mbar_wait_spin(bar_full, 0u, a.status, abort_flag);
                        g = 1;
                        if (issue_ok) {
                            const uint64_t wl = desc_add(wd0, static_cast<uint32_t>(l * C::PL * C::KB) * C::UNIT);
#pragma unroll
                            for (int k = 0; k < 4 * C::KB; ++k) {
                                const uint64_t xd = desc_add(xd0, (k >> 2) * 128u * 128u + (k & 3) * 32u);
                                const uint64_t wd = desc_add(wl, (k >> 2) * C::PL * C::UNIT + (k & 3) * 32u);
                                mma_f16kind(tmem, xd, wd, idesc, k != 0);
                                if (C::PL == 2) {
                                    mma_f16kind(tmem, xd, desc_add(wd, C::UNIT), idesc, 1u);
                                    mma_f16kind(tmem, desc_add(xd, C::PLANE), wd, idesc, 1u);
                                }
                            }
                        }
                    }
                    for (int kb = 0; !C::RES && kb < C::KB && issue_ok; ++kb, ++g) {
                        const uint32_t stage = g % C::NS;
                        issue_ok = mbar_wait_spin(bar_full + 8u * stage, (g / C::NS) & 1u, a.status, abort_flag);
                        if (!issue_ok) break;
                        tc_fence_after();
#pragma unroll
                        for (int t = 0; t < C::ST; ++t) {
                            // a tile without a ray: nothing reads its accumulator
                            if ((act[4 * t] | act[4 * t + 1] | act[4 * t + 2] | act[4 * t + 3]) == 0) continue;
#pragma unroll
                            for (int kk = 0; kk < 4; ++kk) {
                                const uint64_t xd = desc_add(xd0, t * C::PLANE + kb * 128u * 128u + kk * 32u);
                                const uint64_t wd = desc_add(wd0, stage * C::UNIT + kk * 32u);
                                if (C::FP8)
                                    mma_f8kind(tmem + t * W, xd, wd, idesc, (kb | kk) != 0);
                                else
                                    mma_f16kind(tmem + t * W, xd, wd, idesc, (kb | kk) != 0);
                            }
                        }
                        mma_commit(bar_empty + 8u * stage);
                    }
                    if (issue_ok) mma_commit(bar_mma);
                }
                // a warp either reads the accumulator whole or not at all
                good = __all_sync(0xffffffffu, mbar_wait_spin(bar_mma, mma_phase, a.status, abort_flag) && good);
                mma_phase ^= 1u;
                tc_fence_after();
                const bool last = l + 1 == KH;
                // E4M3: accumulator -> value (the operand scales q_w and 256 divided out)
                const float mf = C::FP8 ? 1.0f / (net.q_w[l] * kFp8ActScale) : 1.0f;
                const float2 mf2 = make_float2(mf, mf);
                if (good && wact) {
#pragma unroll 1
                    for (int j = 0; j < C::UPT / 16; ++j) {
                        float v[16];
                        tmem_ld16(d_s + j * 16u, v);
                        tmem_wait_ld();
                        const float4* b4 = reinterpret_cast<const float4*>(bhs + l * W + u0 + j * 16);
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const float4 b = b4[q];
                            const float2 v01 = make_float2(v[4 * q], v[4 * q + 1]), v23 = make_float2(v[4 * q + 2], v[4 * q + 3]);
                            const float2 x01 = C::FP8 ? __ffma2_rn(v01, mf2, make_float2(b.x, b.y))
                                                      : __fadd2_rn(v01, make_float2(b.x, b.y));
                            const float2 x23 = C::FP8 ? __ffma2_rn(v23, mf2, make_float2(b.z, b.w))
                                                      : __fadd2_rn(v23, make_float2(b.z, b.w));
                            v[4 * q] = sin_fast(x01.x);
                            v[4 * q + 1] = sin_fast(x01.y);
                            v[4 * q + 2] = sin_fast(x23.x);
                            v[4 * q + 3] = sin_fast(x23.y);
                        }
                        if (!last) {
                            wide_store16<C>(x_s, row, u0 + j * 16, v);
                        } else if (owner) {
                            const float4* w4 = reinterpret_cast<const float4*>(wos + j * 16);
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                const float4 w = w4[q];
                                acc01 = __ffma2_rn(make_float2(w.x, w.y), make_float2(v[4 * q], v[4 * q + 1]), acc01);
                                acc23 = __ffma2_rn(make_float2(w.z, w.w), make_float2(v[4 * q + 2], v[4 * q + 3]), acc23);
                            }
                        } else {
                            float4* dst = sines + ((u0 - C::UPT) / 4 + j * 4) * (C::ST * 128) + slot;
#pragma unroll
                            for (int q = 0; q < 4; ++q)
                                dst[q * (C::ST * 128)] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
                        }
                    }
                }
                if (!last) fence_proxy_async_smem();
                tc_fence_before();
                bar_named(1, C::NRT);
            }
            if (owner) {
                if (good && wact) {
                    const float4* w4 = reinterpret_cast<const float4*>(wos + C::UPT);
#pragma unroll 8
                    for (int q = 0; q < (W - C::UPT) / 4; ++q) {
                        const float4 w = w4[q], s = sines[q * (C::ST * 128) + slot];
                        acc01 = __ffma2_rn(make_float2(w.x, w.y), make_float2(s.x, s.y), acc01);
                        acc23 = __ffma2_rn(make_float2(w.z, w.w), make_float2(s.z, s.w), acc23);
                    }
                }
                const float f = ((acc01.x + acc01.y) + (acc23.x + acc23.y)) + net.bout;
                // step_ray is a collective of the warp, and another warp may set the flag between two lanes' reads
                if (!__any_sync(0xffffffffu, !good || *abort_flag != 0))
                    step_ray(a, ray, f);
                else
                    ray.state = kSlotDone;
            }
        }
        if (issuer) *consumed = g;
        bar_named(1, C::NRT);
        if (issuer) {
            __threadfence_block();
            *done_flag = 1;
        }
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
