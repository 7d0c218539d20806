// 3x3 / stride 1 / pad 1 convolution with BF16 math straight from the fp32 activation.  Included by gemm_tc.cu (inside namespace
// nnv, after the PTX helpers).
//
// Bound: shared memory.  Per patch and block of 32 input channels the copies write 60 KB (64 output channels), the rounding reads 23 and
// writes 12, and 18 MMAs (M = 128, N = 64, K = 16) read 6 KB each: 200 KB, 1590 cycles at 128 bytes a cycle, where a block takes 1500
// (device-clock probes, 256 -> 256 @56).  One thread issues an MMA per 82 cycles; two, with an accumulator each and the filter rows in
// turn, reach that bound, and four boxes in flight keep it fed.  (A copy of the box for each filter column, so that the rows of the A
// operand start on 128 bytes, costs more traffic than it saves: 11.5 us against 10.8.)  A CTA owns an
// output patch of 16 rows x 8 columns and BN output channels.  Per block of 32 input channels it fetches ONE fp32 halo box of
// 18 x 10 pixels, eight warps round it to bf16 into the un-swizzled core-matrix layout [8-channel chunk][pixel][16 bytes],
// and all nine taps read that one copy: a tap (r, s) is a shift of the descriptor's start address by 10 r + s pixels, and the
// eight-row groups of the A operand (the image rows of the patch) lie 160 bytes apart.  The implicit GEMM converts and fetches
// every tap's tile by itself (9 x 16 KB against 23 KB).
// The weights of a filter row's three taps arrive as bf16, 64-byte swizzled, through one three-dimensional box.  K splits over
// the channel blocks use a cluster whose CTAs push their partial rows to the rows' owners, as in gemm_tc_kernel.
// The write-out is that of gemm_tc_kernel: eight warps, rows from shared memory as coalesced stores.  It took 1.7 us of the 10.8.
// Measured (chained launches, with bias, us; one issuer, two boxes, TMA stores by four warps -> this one): 256 -> 256 @56 10.9 -> 9.9,
// 64 -> 64 @224 16.8 -> 15.0, 128 -> 128 @112 9.1 -> 8.2, 64 -> 64 @56 4.55 -> 4.16, 320 -> 640 @24 9.7 -> 8.7, 128 -> 128 @28 4.53 -> 4.37,
// 512 -> 512 @14 7.3 -> 7.0.
#pragma once

struct ConvBDev {
    unsigned long long* stamp;
    float* D;
    const float* bias;
    const float* addend;
    int C, H, W, K, BN, act, tmem_cols, splits, na, nb, cblk, tiles_w, issuers;
    uint32_t b_off, bar_off, recv_off;
};

constexpr int CB_THREADS = 384;
constexpr int CB_PIX = 180;                                   // pixels of a halo box: 18 rows x 10
constexpr uint32_t CB_A32 = 23 * 1024;                        // fp32 box slot (180 x 128 bytes, padded)
constexpr uint32_t CB_ABF = 92 * 128;                         // bf16 box slot (4 x 180 x 16 bytes, padded)
constexpr int CB_MAX_NA = 4;
constexpr int CB_MAX_NB = 8;
constexpr int CB_BAR_BYTES = 8 * (2 * CB_MAX_NA + 4 + 2 * CB_MAX_NB + 4) + 512;

template <bool SPLIT>
__global__ void __launch_bounds__(CB_THREADS, 1)
conv3x3_bf16_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                    const ConvBDev g) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* const sm = smem_raw + (sbase - smem_u32(smem_raw));
    const int BN = g.BN, NA = g.na, NB = g.nb, splits = SPLIT ? g.splits : 1;
    const uint32_t abf0 = (uint32_t)NA * CB_A32;              // the bf16 boxes lie behind the fp32 ones
    const uint32_t b_slot = (uint32_t)BN * 192u;              // three taps x BN rows x 64 bytes
    const uint32_t bars = sbase + g.bar_off;
    auto a_full = [&](int s) { return bars + 8u * s; };                        // an fp32 box has landed
    auto a_free = [&](int s) { return bars + 8u * (CB_MAX_NA + s); };          // it has been rounded
    auto a_conv = [&](int s) { return bars + 8u * (2 * CB_MAX_NA + s); };      // a bf16 box is complete
    auto a_empty = [&](int s) { return bars + 8u * (2 * CB_MAX_NA + 2 + s); }; // it has been multiplied
    auto b_full = [&](int s) { return bars + 8u * (2 * CB_MAX_NA + 4 + s); };
    auto b_empty = [&](int s) { return bars + 8u * (2 * CB_MAX_NA + 4 + CB_MAX_NB + s); };
    const uint32_t tmem_full_bar = bars + 8u * (2 * CB_MAX_NA + 4 + 2 * CB_MAX_NB), recv_bar = tmem_full_bar + 8u, holder = recv_bar + 8u;
    const uint32_t sbias = bars + (uint32_t)CB_BAR_BYTES - 512u;
    const volatile uint32_t* holder_ptr = reinterpret_cast<const volatile uint32_t*>(sm + (holder - sbase));

    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int sp = (int)blockIdx.z;
    const int tile_h = (int)blockIdx.x / g.tiles_w, tile_w = (int)blockIdx.x - tile_h * g.tiles_w;
    const int oh0 = tile_h * 16, ow0 = tile_w * 8, n0 = blockIdx.y * BN;
    const int cb0 = g.cblk * sp / splits, ncb = g.cblk * (sp + 1) / splits - cb0;

    if (warp == 0 && lane == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmA)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB)) : "memory");
        for (int s = 0; s < NA; ++s) { mbar_init(a_full(s), 1); mbar_init(a_free(s), 8); }
        for (int s = 0; s < 2; ++s) { mbar_init(a_conv(s), 8); mbar_init(a_empty(s), (uint32_t)g.issuers); }
        for (int s = 0; s < NB; ++s) { mbar_init(b_full(s), 1); mbar_init(b_empty(s), 1); }
        mbar_init(tmem_full_bar, (uint32_t)g.issuers);
        mbar_init(recv_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(holder), "r"((uint32_t)g.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // What the write-out needs besides the accumulator is worked out here, under the previous kernel's tail.
    const int cw = warp >= 8 ? warp - 4 : warp - 2;           // of the eight converting warps
    const int quarter = warp & 3, q0 = quarter * 32, half = warp >> 3, t = half * 128 + (cw & 3) * 32 + lane;
    const bool vec = (g.K & 3) == 0 && (reinterpret_cast<uintptr_t>(g.D) & 15) == 0 && (!g.addend || (reinterpret_cast<uintptr_t>(g.addend) & 15) == 0);
    uint32_t sub = sbase + (uint32_t)(cw & 7) * 2048u;        // a warp's sub-tile: 32 pixels x 16 columns
    long long row_pitch = (long long)g.W * g.K;
    int rows_live = ow0 + (lane >> 2) < g.W ? g.H - oh0 - quarter * 4 : 0;        // image rows of the quarter that exist where this lane stores
    float* out = g.D + ((long long)(oh0 + quarter * 4) * g.W + ow0 + (lane >> 2)) * g.K + n0 + half * 16 + (lane & 3) * 4;
    const int rows_per = 128 / splits, r0 = sp * rows_per;
    int nch = BN / 4, rot0 = 0, qstep = 0, rstep = 0, rot_step = 0, rr = 0, cc = 0, rot = 0;
    uint32_t push_dst = 0, push_bar = 0, push_src = 0, push_bytes = 0;
    if constexpr (!SPLIT) {
        asm volatile("" : "+r"(sub), "+l"(row_pitch), "+r"(rows_live), "+l"(out));
    } else {
        rot0 = (q0 + lane) % nch;
        const int a0 = max(q0, lane * rows_per), a1 = min(q0 + 32, (lane + 1) * rows_per);
        if (half == 0 && lane < splits && a1 > a0) {
            push_dst = cluster_addr(sbase + g.recv_off + (uint32_t)((r0 + a0 - lane * rows_per) * BN) * 4u, lane);
            push_bar = cluster_addr(recv_bar, lane);
            push_src = sbase + (uint32_t)(a0 * BN) * 4u;
            push_bytes = (uint32_t)((a1 - a0) * BN) * 4u;
        }
        qstep = 256 / nch; rstep = 256 - qstep * nch;
        rr = t / nch; cc = t - rr * nch; rot = (r0 + rr) % nch;
        rot_step = qstep % nch;
        asm volatile("" : "+r"(nch), "+r"(rot0), "+r"(push_dst), "+r"(push_bar), "+r"(push_src), "+r"(push_bytes));
        asm volatile("" : "+r"(qstep), "+r"(rstep), "+r"(rr), "+r"(cc), "+r"(rot), "+r"(rot_step));
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if constexpr (SPLIT) {
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
        int sa = 0;
        uint32_t pa = 0;
        for (int it = 0; it < ncb; ++it) {
            const int s = it & 1;
            if (!mbar_wait(a_full(sa), pa)) return false;
            if (it >= 2 && !mbar_wait(a_empty(s), ((uint32_t)(it >> 1) & 1u) ^ 1u)) return false;      // the slot's former bf16 box has been multiplied
            const uint8_t* const src = sm + (uint32_t)sa * CB_A32;
            uint8_t* const dst = sm + abf0 + (uint32_t)s * CB_ABF;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int item = cw + 8 * i;                                   // 6 groups of 32 pixels x 4 chunks
                const int r = (item >> 2) * 32 + lane;
                if (r < CB_PIX) convert_chunk<false>(src, dst, dst, r, item & 3, CB_PIX);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");       // generic writes -> visible to the MMA's reads
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(a_conv(s));
                if (it + NA < ncb) mbar_arrive(a_free(sa));                    // only where the producer waits for it
            }
            if (++sa == NA) { sa = 0; pa ^= 1u; }
        }
        return true;
    };

    bool cluster_arrived = false;
    if (warp == 0) {
        if (elect_one()) {
            bool ok = true;
            int s = 0;
            uint32_t ph = 0;
            for (int it = 0; it < ncb; ++it) {
                if (it >= NA) ok = mbar_wait(a_free(s), ph ^ 1u);
                if (!ok) break;
                mbar_expect_tx(a_full(s), CB_PIX * 128u);
                tma_load_3d(sbase + (uint32_t)s * CB_A32, &tmA, (cb0 + it) * 32, ow0 - 1, oh0 - 1, a_full(s));
                if (++s == NA) { s = 0; ph ^= 1u; }
            }
            if (!ok) {
                atomicExch(&g_device_status, (int)NNV_ERR_TIMEOUT);
                for (int i = 0; i < 1000; ++i) __nanosleep(1000);              // let loads already in flight land
            }
        }
        __syncwarp();
        if constexpr (SPLIT) cluster_wait();
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
        if constexpr (SPLIT) cluster_wait();
    } else if (warp == 1 || warp == 6) {
        const int iss = warp == 1 ? 0 : 1;
        if (iss < g.issuers && elect_one()) {
            // instruction descriptor: fp32 accumulate, bf16 operands, both K-major, N = BN, M = 128
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | (8u << 24);
            constexpr uint32_t lbo_a = CB_PIX * 16u;
            bool ok = true;
            const uint32_t acc = tmem_base + (uint32_t)(iss * BN);
            int sb = 0, stage = 0;                            // filter rows are stages; with two issuers, this one's are the even or the odd ones
            uint32_t pb = 0, more = 0;                        // 0: the accumulator's first MMA overwrites it
            for (int it = 0; it < ncb && ok; ++it) {
                const int sa = it & 1;
                ok = mbar_wait(a_conv(sa), (uint32_t)(it >> 1) & 1u);
                if (!ok) break;
                const uint32_t a = sbase + abf0 + (uint32_t)sa * CB_ABF;
                for (int r = 0; r < 3; ++r, ++stage, sb = sb + 1 == NB ? 0 : sb + 1, pb ^= sb == 0 ? 1u : 0u) {
                    if (g.issuers == 2 && (stage & 1) != iss) continue;
                    ok = mbar_wait(b_full(sb), pb);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t b = sbase + g.b_off + (uint32_t)sb * b_slot;
#pragma unroll
                    for (int s = 0; s < 3; ++s)
#pragma unroll
                        for (int kk = 0; kk < 2; ++kk)
                            umma<true>(acc, make_smem_desc_plain(a + (uint32_t)(r * 10 + s) * 16u + kk * 2u * lbo_a, lbo_a, 160),
                                       make_smem_desc64(b + (uint32_t)s * BN * 64u) + (uint64_t)(kk * 2), idesc,
                                       (s | kk) ? 1u : more);
                    more = 1u;
                    if (stage + NB < 3 * ncb) umma_commit(b_empty(sb));   // only where the producer waits for it
                }
                if (ok && it + 2 < ncb) umma_commit(a_empty(sa));
            }
            if (ok) umma_commit(tmem_full_bar);
            else atomicExch(&g_device_status, (int)NNV_ERR_TIMEOUT);
        }
        __syncwarp();
        if constexpr (SPLIT) cluster_wait();
    } else {
        // Warps 2-5 and 8-11: conversion, then the write-out.  The TMEM lanes a warp may read are those of its number modulo four, so
        // each quarter of the tile's rows (4 image rows x 8 pixels) has two warps, which take the 16-column chunks in turn.
        const float bias = (g.bias && t < BN && n0 + t < g.K) ? __ldg(g.bias + n0 + t) : 0.f;
        auto act4 = [&](float4& v) {
            if (g.act) {
                const float hi = g.act == 2 ? 6.f : INFINITY;
                v.x = fminf(fmaxf(v.x, 0.f), hi); v.y = fminf(fmaxf(v.y, 0.f), hi);
                v.z = fminf(fmaxf(v.z, 0.f), hi); v.w = fminf(fmaxf(v.w, 0.f), hi);
            }
        };
        const uint32_t tacc = tmem_base + ((uint32_t)q0 << 16);
        const bool two = g.issuers == 2;
        // 16 columns of this lane's row, the issuers' accumulators added in order
        auto acc16 = [&](int c0, float (&v)[16]) {
            uint32_t r[16], q[16];
            tmem_ld16_nowait(tacc + (uint32_t)c0, r);
            tmem_ld16_nowait(tacc + (uint32_t)(two ? BN + c0 : c0), q);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = two ? __uint_as_float(r[i]) + __uint_as_float(q[i]) : __uint_as_float(r[i]);
        };
        bool ok = convert_boxes(cw);
        if (t < BN) asm volatile("st.shared.f32 [%0], %1;" ::"r"(sbias + 4u * (uint32_t)t), "f"(bias) : "memory");
        asm volatile("barrier.sync 1, 256;" ::: "memory");
        auto wait_acc = [&]() {
            ok = ok && mbar_wait(tmem_full_bar, 0);
            tc_fence_after();
            if (!ok && lane == 0) atomicExch(&g_device_status, (int)NNV_ERR_TIMEOUT);
            ok = __all_sync(0xffffffffu, ok);
        };
        if (!SPLIT && vec) {
            // Per 16 columns: TMEM -> registers (lane = one pixel), + bias -> a sub-tile in shared memory (both A rings are idle by then)
            // -> (+ residual, activation) -> memory, an image row of 8 pixels x 64 bytes at a time.
            auto fetch_addend = [&](int c0, float4 (&a)[4]) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    a[i] = g.addend && c0 < BN && i < rows_live && n0 + c0 + 4 * (lane & 3) < g.K
                               ? __ldg(reinterpret_cast<const float4*>(g.addend + (out - g.D) + (c0 - half * 16) + (long long)i * row_pitch))
                               : make_float4(0.f, 0.f, 0.f, 0.f);
            };
            float4 aa[4];
            fetch_addend(half * 16, aa);
            wait_acc();
            if (ok && half * 16 < BN) {
#pragma unroll 1
                for (int c0 = half * 16; c0 < BN; c0 += 32) {
                    float v[16];
                    acc16(c0, v);
                    const uint32_t swz = (uint32_t)((lane >> 1) & 3) << 4;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const float4 bb = lds128(sbias + (uint32_t)(c0 + 4 * c) * 4u);
                        sts128(sub + (uint32_t)lane * 64u + (((uint32_t)c << 4) ^ swz),
                               make_float4(v[c * 4] + bb.x, v[c * 4 + 1] + bb.y, v[c * 4 + 2] + bb.z, v[c * 4 + 3] + bb.w));
                    }
                    __syncwarp();
                    const int r1 = lane >> 2;
                    const uint32_t src = sub + (uint32_t)r1 * 64u + (uint32_t)(((lane & 3) ^ ((r1 >> 1) & 3)) << 4);
                    float4 q[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        q[i] = lds128(src + (uint32_t)i * 512u);
                        if (g.addend) { q[i].x += aa[i].x; q[i].y += aa[i].y; q[i].z += aa[i].z; q[i].w += aa[i].w; }
                        act4(q[i]);
                    }
                    float* const at = out + (c0 - half * 16);
                    if (n0 + c0 + 4 * (lane & 3) < g.K) {
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            if (i < rows_live) *reinterpret_cast<float4*>(at + (long long)i * row_pitch) = q[i];
                    }
                    if (g.addend) fetch_addend(c0 + 32, aa);
                    __syncwarp();                             // the sub-tile is free again
                }
            }
        } else if (!SPLIT) {
            const int oh = oh0 + quarter * 4 + (lane >> 3), ow = ow0 + (lane & 7);
            const long long off = ((long long)oh * g.W + ow) * g.K + n0;
            wait_acc();
            if (ok) {
#pragma unroll 1
                for (int c0 = half * 16; c0 < BN; c0 += 32) {
                    float v[16];
                    acc16(c0, v);
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        if (oh < g.H && ow < g.W && n0 + c0 + j < g.K) {
                            float bb;
                            asm volatile("ld.shared.f32 %0, [%1];" : "=f"(bb) : "r"(sbias + (uint32_t)(c0 + j) * 4u) : "memory");
                            const float o = v[j] + bb;
                            g.D[off + c0 + j] = act_fn(g.addend ? o + __ldg(g.addend + off + c0 + j) : o, g.act);
                        }
                }
            }
        } else {
            const uint32_t prow = sbase + (uint32_t)(q0 + lane) * (uint32_t)BN * 4u, recv = sbase + g.recv_off, part_stride = (uint32_t)(rows_per * BN) * 4u;
            cluster_wait();                                   // every CTA's barriers are initialised
            wait_acc();
            if (ok) {
#pragma unroll 1
                for (int c0 = half * 16; c0 < BN; c0 += 32) {
                    float v[16];
                    acc16(c0, v);
                    int pos = rot0 + c0 / 4;
                    if (pos >= nch) pos -= nch;
#pragma unroll
                    for (int j = 0; j < 16; j += 4) {
                        sts128(prow + (uint32_t)pos * 16u, make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]));
                        pos = pos + 1 == nch ? 0 : pos + 1;
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes -> visible to the bulk copies
            }
            __syncwarp();
            asm volatile("barrier.sync %0, 64;" ::"r"(2 + quarter) : "memory");   // both warps' columns of these rows are parked
            if (ok && push_bytes) bulk_push(push_dst, push_src, push_bytes, push_bar);
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
                for (int idx = t; idx < total; idx += 256) {
                    const int p = cc + rot >= nch ? cc + rot - nch : cc + rot;
                    const uint32_t src = recv + (uint32_t)(rr * BN) * 4u + (uint32_t)p * 16u;
                    float4 v[NS];
#pragma unroll
                    for (int rk = 0; rk < NS; ++rk) v[rk] = lds128(src + (uint32_t)rk * part_stride);
                    float4 o = lds128(sbias + (uint32_t)cc * 16u);
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
    if constexpr (SPLIT) {
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
