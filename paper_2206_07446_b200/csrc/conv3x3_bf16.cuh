// 3x3 / stride 1 / pad 1 convolution with BF16 math straight from the fp32 activation.  Included by gemm_tc.cu (inside namespace
// nnv, after the PTX helpers).
//
// Bound: the issue of 18 MMAs (M = 128, N <= 128, K = 16), ~82 cycles each, per patch and 32 input channels by one thread; the chain
// of box load, rounding and MMAs comes right behind (256 -> 256 @56: without the rounding after two boxes, or without the weights'
// loads after the first ring, the same time within 1 %; with half the MMAs 9.3 us instead of 11.0).  A CTA owns an
// output patch of 16 rows x 8 columns and BN output channels.  Per block of 32 input channels it fetches ONE fp32 halo box of
// 18 x 10 pixels, eight warps round it to bf16 into the un-swizzled core-matrix layout [8-channel chunk][pixel][16 bytes],
// and all nine taps read that one copy: a tap (r, s) is a shift of the descriptor's start address by 10 r + s pixels, and the
// eight-row groups of the A operand (the image rows of the patch) lie 160 bytes apart.  The implicit GEMM converts and fetches
// every tap's tile by itself (9 x 16 KB against 23 KB), the earlier form of this kernel three boxes.
// The weights of a filter row's three taps arrive as bf16, 64-byte swizzled, through one three-dimensional box.  K splits over
// the channel blocks use a cluster whose CTAs push their partial rows to the rows' owners, as in gemm_tc_kernel.
// Measured (chained launches, with bias, us; the better of the converting implicit GEMM and the earlier form -> this one):
// 256 -> 256 @56 21.0 -> 11.0, 64 -> 64 @224 20.3 -> 17.5, 128 -> 128 @112 20.5 -> 9.1, 512 -> 512 @28 19.7 -> 11.9, 64 -> 64 @56
// 6.9 -> 4.7, 128 -> 128 @28 6.7 -> 4.7, 256 -> 256 @14 7.4 -> 5.2.
#pragma once

struct ConvBDev {
    unsigned long long* stamp;
    float* D;
    const float* bias;
    const float* addend;
    int C, H, W, K, BN, act, tmem_cols, splits, nb, cblk, tiles_w;
    int tma_out;                      // 0: plain stores; else the column width of the sub-tiles stored by TMA
    uint32_t b_off, bar_off, recv_off;
};

constexpr int CB_THREADS = 384;
constexpr int CB_PIX = 180;                                   // pixels of a halo box: 18 rows x 10
constexpr uint32_t CB_A32 = 23 * 1024;                        // fp32 box slot (180 x 128 bytes, padded)
constexpr uint32_t CB_ABF = 92 * 128;                         // bf16 box slot (4 x 180 x 16 bytes, padded)
constexpr uint32_t CB_RINGS_A = 2 * (CB_A32 + CB_ABF);
constexpr int CB_MAX_NB = 8;
constexpr int CB_BAR_BYTES = 8 * (6 + 2 * CB_MAX_NB + 4) + 512;

__global__ void __launch_bounds__(CB_THREADS, 1)
conv3x3_bf16_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                    const __grid_constant__ CUtensorMap tmD, const ConvBDev g) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* const sm = smem_raw + (sbase - smem_u32(smem_raw));
    const int BN = g.BN, NB = g.nb, splits = g.splits;
    const uint32_t b_slot = (uint32_t)BN * 192u;              // three taps x BN rows x 64 bytes
    const uint32_t bars = sbase + g.bar_off;
    auto a_full = [&](int s) { return bars + 8u * s; };
    auto a_conv = [&](int s) { return bars + 8u * (2 + s); };
    auto a_empty = [&](int s) { return bars + 8u * (4 + s); };
    auto b_full = [&](int s) { return bars + 8u * (6 + s); };
    auto b_empty = [&](int s) { return bars + 8u * (6 + CB_MAX_NB + s); };
    const uint32_t tmem_full_bar = bars + 8u * (6 + 2 * CB_MAX_NB), recv_bar = tmem_full_bar + 8u, holder = recv_bar + 8u;
    float* const s_bias = reinterpret_cast<float*>(sm + g.bar_off + 8 * (6 + 2 * CB_MAX_NB + 4));
    const volatile uint32_t* holder_ptr = reinterpret_cast<const volatile uint32_t*>(sm + (holder - sbase));

    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int sp = (int)blockIdx.z;
    const int tile_h = (int)blockIdx.x / g.tiles_w, tile_w = (int)blockIdx.x - tile_h * g.tiles_w;
    const int oh0 = tile_h * 16, ow0 = tile_w * 8, n0 = blockIdx.y * BN;
    const int cb0 = g.cblk * sp / splits, ncb = g.cblk * (sp + 1) / splits - cb0;

    if (warp == 0 && lane == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmA)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB)) : "memory");
        if (g.tma_out) asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmD)) : "memory");
        for (int s = 0; s < 2; ++s) { mbar_init(a_full(s), 1); mbar_init(a_conv(s), 8); mbar_init(a_empty(s), 1); }
        for (int s = 0; s < NB; ++s) { mbar_init(b_full(s), 1); mbar_init(b_empty(s), 1); }
        mbar_init(tmem_full_bar, 1);
        mbar_init(recv_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(holder), "r"((uint32_t)g.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const int rows_per = 128 / splits, r0 = sp * rows_per, nch = BN / 4;
    if (splits > 1) {
        if (threadIdx.x == 64) mbar_expect_tx(recv_bar, (uint32_t)(splits * rows_per * BN) * 4u);
        __syncwarp();
        cluster_arrive_relaxed();
    }
    const uint32_t tmem_base = *holder_ptr;
    pdl_wait();
    pdl_trigger();
    if (threadIdx.x == 32) stamp_start(g.stamp);

    // Warps 2-5 and 8-11: round box after box, 32 pixels x 8 channels at a time.
    auto convert_boxes = [&](int cw) -> bool {
        for (int it = 0; it < ncb; ++it) {
            const int s = it & 1;
            const uint32_t ph = (uint32_t)(it >> 1) & 1u;
            if (!mbar_wait(a_full(s), ph)) return false;
            if (it >= 2 && !mbar_wait(a_empty(s), ph ^ 1u)) return false;      // the slot's former bf16 box has been multiplied
            const uint8_t* const src = sm + (uint32_t)s * CB_A32;
            uint8_t* const dst = sm + 2 * CB_A32 + (uint32_t)s * CB_ABF;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int item = cw + 8 * i;                                   // 6 groups of 32 pixels x 4 chunks
                const int r = (item >> 2) * 32 + lane;
                if (r < CB_PIX) convert_chunk<false>(src, dst, dst, r, item & 3, CB_PIX);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");       // generic writes -> visible to the MMA's reads
            __syncwarp();
            if (lane == 0) mbar_arrive(a_conv(s));
        }
        return true;
    };

    bool cluster_arrived = false;
    if (warp == 0) {
        if (elect_one()) {
            bool ok = true;
            for (int it = 0; it < ncb; ++it) {
                const int s = it & 1;
                if (it >= 2) ok = mbar_wait(a_conv(s), ((uint32_t)(it >> 1) & 1u) ^ 1u);   // the slot's former fp32 box has been rounded
                if (!ok) break;
                mbar_expect_tx(a_full(s), CB_PIX * 128u);
                tma_load_3d(sbase + (uint32_t)s * CB_A32, &tmA, (cb0 + it) * 32, ow0 - 1, oh0 - 1, a_full(s));
            }
            if (!ok) {
                atomicExch(&g_device_status, (int)NNV_ERR_TIMEOUT);
                for (int i = 0; i < 1000; ++i) __nanosleep(1000);              // let loads already in flight land
            }
        }
        __syncwarp();
        if (splits > 1) cluster_wait();
    } else if (warp == 7) {
        if (elect_one()) {
            bool ok = true;
            int s = 0;
            uint32_t ph = 0;
            for (int it = 0; it < 3 * ncb; ++it) {
                if (it >= NB) ok = mbar_wait(b_empty(s), ph ^ 1u);
                if (!ok) break;
                const int cb = it / 3, r = it - 3 * cb;
                mbar_expect_tx(b_full(s), b_slot);
                tma_load_3d(sbase + g.b_off + (uint32_t)s * b_slot, &tmB, (cb0 + cb) * 32, n0, 3 * r, b_full(s));
                if (++s == NB) { s = 0; ph ^= 1u; }
            }
            if (!ok) {
                atomicExch(&g_device_status, (int)NNV_ERR_TIMEOUT);
                for (int i = 0; i < 1000; ++i) __nanosleep(1000);
            }
        }
        __syncwarp();
        if (splits > 1) cluster_wait();
    } else if (warp == 1) {
        if (elect_one()) {
            // instruction descriptor: fp32 accumulate, bf16 operands, both K-major, N = BN, M = 128
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | (8u << 24);
            constexpr uint32_t lbo_a = CB_PIX * 16u;
            bool ok = true;
            int sb = 0, refill_b = 3 * ncb - NB;              // releases that the producer waits for
            uint32_t pb = 0;
            for (int it = 0; it < ncb && ok; ++it) {
                const int sa = it & 1;
                ok = mbar_wait(a_conv(sa), (uint32_t)(it >> 1) & 1u);
                if (!ok) break;
                const uint32_t a = sbase + 2 * CB_A32 + (uint32_t)sa * CB_ABF;
                for (int r = 0; r < 3; ++r) {
                    ok = mbar_wait(b_full(sb), pb);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t b = sbase + g.b_off + (uint32_t)sb * b_slot;
#pragma unroll
                    for (int s = 0; s < 3; ++s)
#pragma unroll
                        for (int kk = 0; kk < 2; ++kk)
                            umma<true>(tmem_base, make_smem_desc_plain(a + (uint32_t)(r * 10 + s) * 16u + kk * 2u * lbo_a, lbo_a, 160),
                                       make_smem_desc64(b + (uint32_t)s * BN * 64u) + (uint64_t)(kk * 2), idesc,
                                       (it | r | s | kk) ? 1u : 0u);
                    if (refill_b-- > 0) umma_commit(b_empty(sb));
                    if (++sb == NB) { sb = 0; pb ^= 1u; }
                }
                if (ok && it + 2 < ncb) umma_commit(a_empty(sa));
            }
            if (ok) umma_commit(tmem_full_bar);
            else atomicExch(&g_device_status, (int)NNV_ERR_TIMEOUT);
        }
        __syncwarp();
        if (splits > 1) cluster_wait();
    } else if (warp == 6) {
        if (splits > 1) cluster_wait();
    } else if (warp >= 8) {
        if (!convert_boxes(warp - 4) && lane == 0) atomicExch(&g_device_status, (int)NNV_ERR_TIMEOUT);
        __syncwarp();
        if (splits > 1) cluster_wait();
    } else {
        // Warps 2-5: conversion, then the write-out (the indices and the bias before the wait for the accumulator).
        const int quarter = warp & 3, q0 = quarter * 32, t = (int)threadIdx.x - 64;
        const float bias = (g.bias && t < BN && n0 + t < g.K) ? __ldg(g.bias + n0 + t) : 0.f;
        const float hi = g.act == 2 ? 6.f : INFINITY;
        auto act4 = [&](float4& v) {
            if (g.act) {
                v.x = fminf(fmaxf(v.x, 0.f), hi); v.y = fminf(fmaxf(v.y, 0.f), hi);
                v.z = fminf(fmaxf(v.z, 0.f), hi); v.w = fminf(fmaxf(v.w, 0.f), hi);
            }
        };
        auto acc16 = [&](int c0, float (&v)[16]) {
            uint32_t r[16];
            tmem_ld16_nowait(tmem_base + ((uint32_t)q0 << 16) + (uint32_t)c0, r);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
        };
        bool ok = convert_boxes(warp - 2);
        if (t < BN) s_bias[t] = bias;
        asm volatile("barrier.sync 1, 128;" ::: "memory");
        const bool vec = (g.K & 3) == 0 && (reinterpret_cast<uintptr_t>(g.D) & 15) == 0 && (!g.addend || (reinterpret_cast<uintptr_t>(g.addend) & 15) == 0);
        auto wait_acc = [&]() {
            ok = ok && mbar_wait(tmem_full_bar, 0);
            tc_fence_after();
            if (!ok && lane == 0) atomicExch(&g_device_status, (int)NNV_ERR_TIMEOUT);
            ok = __all_sync(0xffffffffu, ok);
        };
        if (splits == 1) {
            // MMA row = 8 * (patch row) + (patch column): a warp holds 4 image rows x 8 pixels
            const int oh = oh0 + quarter * 4 + (lane >> 3), ow = ow0 + (lane & 7);
            const bool inside = oh < g.H && ow < g.W;
            const long long off = ((long long)oh * g.W + ow) * g.K + n0;
            const int CW = g.tma_out ? g.tma_out : 16;
            const uint32_t swz = CW == 32 ? (uint32_t)(lane & 7) : (uint32_t)((lane >> 1) & 3);
            const uint32_t sub = 32u * (uint32_t)CW * 4u;
            uint8_t* row0 = sm + (uint32_t)quarter * sub + (uint32_t)lane * (uint32_t)CW * 4u;    // both A rings are idle by then
            wait_acc();
            if (ok) {
#pragma unroll 1
                for (int c0 = 0; c0 < BN; c0 += 16) {
                    float v[16];
                    float4 aa[4];
                    if (g.addend && vec) {
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            aa[c] = inside && n0 + c0 + 4 * c < g.K ? __ldg(reinterpret_cast<const float4*>(g.addend + off + c0 + 4 * c)) : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                    acc16(c0, v);
                    const uint32_t h = CW == 32 ? (uint32_t)(c0 >> 2) & 4u : 0u;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const float4 bb = *reinterpret_cast<const float4*>(s_bias + c0 + c * 4);
                        float4 o = make_float4(v[c * 4] + bb.x, v[c * 4 + 1] + bb.y, v[c * 4 + 2] + bb.z, v[c * 4 + 3] + bb.w);
                        if (g.addend && vec) { o.x += aa[c].x; o.y += aa[c].y; o.z += aa[c].z; o.w += aa[c].w; }
                        if (vec) act4(o);
                        if (g.tma_out) {
                            *reinterpret_cast<float4*>(row0 + (((h + (uint32_t)c) ^ swz) << 4)) = o;
                        } else if (inside) {
                            const float vv[4] = {o.x, o.y, o.z, o.w};
                            for (int j = 0; j < 4 && n0 + c0 + 4 * c + j < g.K; ++j) {
                                const long long at = off + c0 + 4 * c + j;
                                g.D[at] = vec ? vv[j] : act_fn(g.addend ? vv[j] + __ldg(g.addend + at) : vv[j], g.act);
                            }
                        }
                    }
                    if (g.tma_out && (CW == 16 || h)) {       // the sub-tile is complete
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        __syncwarp();
                        if (lane == 0 && oh0 + quarter * 4 < g.H && n0 + c0 + 16 - CW < g.K) {
                            tma_store_3d(&tmD, smem_u32(row0), n0 + c0 + 16 - CW, ow0, oh0 + quarter * 4);
                            tma_store_commit();
                        }
                        row0 += 4u * sub;
                    }
                }
                if (g.tma_out && lane == 0) tma_store_wait_read();
            }
        } else {
            uint8_t* const prow = sm + (uint32_t)(q0 + lane) * (uint32_t)BN * 4u;
            int pos = (q0 + lane) % nch;
            const int a0 = max(q0, lane * rows_per), a1 = min(q0 + 32, (lane + 1) * rows_per);
            const bool sends = lane < splits && a1 > a0;
            uint32_t push_dst = 0, push_bar = 0;
            if (sends) {
                push_dst = cluster_addr(sbase + g.recv_off + (uint32_t)((r0 + a0 - lane * rows_per) * BN) * 4u, lane);
                push_bar = cluster_addr(recv_bar, lane);
            }
            const int qstep = 128 / nch, rstep = 128 - qstep * nch;
            int rr = t / nch, cc = t - rr * nch, rot = (r0 + rr) % nch;
            const int rot_step = qstep % nch;
            const uint8_t* const recv = sm + g.recv_off;
            const uint32_t part_stride = (uint32_t)(rows_per * BN) * 4u;
            cluster_wait();                                   // every CTA's barriers are initialised
            wait_acc();
            if (ok) {
#pragma unroll 1
                for (int c0 = 0; c0 < BN; c0 += 16) {
                    float v[16];
                    acc16(c0, v);
#pragma unroll
                    for (int j = 0; j < 16; j += 4) {
                        *reinterpret_cast<float4*>(prow + pos * 16) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
                        pos = pos + 1 == nch ? 0 : pos + 1;
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes -> visible to the bulk copies
                __syncwarp();
                if (sends) bulk_push(push_dst, sbase + (uint32_t)(a0 * BN) * 4u, (uint32_t)((a1 - a0) * BN) * 4u, push_bar);
            }
            int total = rows_per * nch;
            if (!mbar_wait(recv_bar, 0)) {
                if (lane == 0) atomicExch(&g_device_status, (int)NNV_ERR_TIMEOUT);
                total = 0;
            }
            __syncwarp();
            cluster_arrive_relaxed();                         // this CTA's rows have arrived: their senders may leave
            cluster_arrived = true;
            auto reduce = [&](auto nsplits) {
                constexpr int NS = decltype(nsplits)::value;
#pragma unroll 1
                for (int idx = t; idx < total; idx += 128) {
                    const int p = cc + rot >= nch ? cc + rot - nch : cc + rot;
                    const uint8_t* src = recv + (uint32_t)(rr * BN) * 4u + (uint32_t)p * 16u;
                    float4 v[NS];
#pragma unroll
                    for (int rk = 0; rk < NS; ++rk) v[rk] = *reinterpret_cast<const float4*>(src + rk * part_stride);
                    float4 o = *reinterpret_cast<const float4*>(s_bias + cc * 4);
                    float4 a = v[0];
#pragma unroll
                    for (int rk = 1; rk < NS; ++rk) { a.x += v[rk].x; a.y += v[rk].y; a.z += v[rk].z; a.w += v[rk].w; }
                    o.x += a.x; o.y += a.y; o.z += a.z; o.w += a.w;
                    const int m = r0 + rr, oh = oh0 + (m >> 3), ow = ow0 + (m & 7), n = n0 + cc * 4;
                    if (oh < g.H && ow < g.W && n < g.K) {
                        const long long at = ((long long)oh * g.W + ow) * g.K + n;
                        if (vec) {
                            if (g.addend) {
                                const float4 aa = __ldg(reinterpret_cast<const float4*>(g.addend + at));
                                o.x += aa.x; o.y += aa.y; o.z += aa.z; o.w += aa.w;
                            }
                            act4(o);
                            *reinterpret_cast<float4*>(g.D + at) = o;
                        } else {
                            const float vv[4] = {o.x, o.y, o.z, o.w};
                            for (int j = 0; j < 4 && n + j < g.K; ++j)
                                g.D[at + j] = act_fn(g.addend ? vv[j] + __ldg(g.addend + at + j) : vv[j], g.act);
                        }
                    }
                    rr += qstep; cc += rstep; rot += rot_step;
                    if (cc >= nch) { cc -= nch; ++rr; ++rot; }
                    if (rot >= nch) rot -= nch;
                }
            };
            if (splits == 8) reduce(std::integral_constant<int, 8>());
            else if (splits == 4) reduce(std::integral_constant<int, 4>());
            else reduce(std::integral_constant<int, 2>());
        }
    }
    __syncwarp();
    if (splits > 1) {
        if (!cluster_arrived) cluster_arrive_relaxed();
        cluster_wait();                                       // nobody leaves while its rows may still be on their way
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0) stamp_end(g.stamp);
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)g.tmem_cols) : "memory");
    }
}
