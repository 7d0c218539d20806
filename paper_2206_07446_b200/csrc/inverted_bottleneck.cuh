// An inverted-residual block (1x1 expansion -> 3x3 depthwise -> 1x1 projection) as one launch.  Included by gemm_tc.cu.
//
// A CTA owns a patch of ph x pw output pixels and some of the expanded channels, in blocks of 32.  It multiplies the pixels the patch
// needs (its halo, at most 128 of them: the rows of one MMA tile) with its rows of the expansion's weights, writes bias + activation into
// shared memory as one [pixel][32 channels] tile a block, runs the depthwise filter from there, and multiplies the result, already in
// the layout of an A operand, with its columns of the projection's weights.  The CTAs that share a patch form a cluster and push their
// partial rows to the CTA that owns them, as the split launches of gemm_tc_kernel do.  Both intermediate tensors are written to memory as
// well (every pixel by the patch that owns it, 128-byte lines, nobody waits for them), so that a layer's output is there to be read.
//
// Same bits as the three launches: a GEMM launch adds its K blocks in an order of its own (K splits, and in each split an accumulator
// for the even blocks and one for the odd ones, added in order at the end), and this kernel keeps to the order that the projection's
// tiling has: a CTA holds a split (`both`) or one of its accumulators, and the owner of a row adds them in the same order.
//
// What bounds it: a chain of dependent phases, each long because a warp pays ~5 cycles an instruction with few others on its scheduler
// (cycles, 64 -> 384 -> 64 @10, 60 CTAs of 48 pixels x 32 channels): pixels from L2 and first MMAs 1580, accumulators to tiles 650, depthwise
// 920, second MMAs 680, partial rows parked 610 and pushed 840, added up 690.  Sixteen warps, for the passes are bound by issue slots (eight with
// twice the columns and pixels each: as long), in 64 registers, so that the next kernel's CTAs fit beside.  A strip of pixels a thread with a
// sliding window, four channels a thread and paired multiply-adds issued less and took as long or longer.
// us a block in a row of them, three launches / this one (TF32): 16 -> 96 -> 24 /2 @112 12.1 / 8.2, 24 -> 144 -> 24 @56 10.1 / 8.4,
// 32 -> 192 -> 32 @28 7.6 / 6.0, 64 -> 384 -> 64 @14 7.7 / 5.0, 96 -> 576 -> 96 @14 8.4 / 6.2, 160 -> 960 -> 160 @7 7.9 / 5.8, 160 -> 960 -> 320
// @7 8.2 / 7.3; of 145 blocks of 96 - 224 pixel images (BF16 too) every one was faster.  Warm MobileNetV2-shaped inference @160 168.6 -> 131.0.
constexpr int IB_MAX_KB = 8;             // 32-channel blocks of the block's input
constexpr int IB_MAX_NB = 8;             // 32-channel blocks of the expansion in one CTA
constexpr int IB_THREADS = 512;
constexpr int IB_PITCH = 144;            // bytes from a pixel to the next in the expansion's tiles
constexpr int IB_BAR_BYTES = 8 * (2 * IB_MAX_KB + 8);

struct IbDev {
    float* e; float* d; float* y;                             // outputs: expansion, depthwise, projection
    const float* b1; const float* b2; const float* b3;        // biases or null
    const float* addend; const float* wd;                     // residual of the projection or null; raw depthwise weights [E][9]
    int E, K, H, W, OH, OW, stride, act3, early;
    float most1, most2;                                       // upper bounds of the first two activations
    int ph, pw, hw, rows, px, tiles_w;                        // patch, width and pixels of its halo, pixels of the patch
    int nkb1, nb_most, step, both, ranks, splits, BN2, w2_boxes, issuers, tmem_cols;
    uint32_t magic_hw, magic_pw, magic_px, magic_nch, magic_n;
    uint32_t w1_off, conv_off, d_off, w2_off, bar_off, par_off;    // byte offsets from the aligned base; E and the received rows at 0
    uint16_t first[IB_MAX_RANKS];                             // a rank's first channel block, and how many it has (every step-th)
    uint8_t count[IB_MAX_RANKS];
    uint32_t pairs;                                           // bit k: split k's accumulators are with two ranks
};

// Bulk copy of `bytes` (a multiple of 16) from memory into this CTA's shared memory.
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
// (By one warp, before the next kernel is let in: CTAs let in earlier could take columns that this grid's still need.)
__device__ __forceinline__ void tmem_take(uint32_t holder, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(holder), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ float lds32(uint32_t addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}
template <int OFF> __device__ __forceinline__ float2 lds64_at(uint32_t addr) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2+%3];" : "=f"(v.x), "=f"(v.y) : "r"(addr), "n"(OFF) : "memory");
    return v;
}
// Eight accumulator columns of this lane's row; of two accumulators (`other` columns apart) the sum.  (Selects instead of branches, here and
// below: a branch that depends on the launch costs a lone warp 30 cycles.)
__device__ __forceinline__ void ib_acc8(uint32_t taddr, bool two, uint32_t other, float (&v)[8]) {
    uint32_t r[8], q[8];
    tmem_ld8_nowait(taddr, r);
    tmem_ld8_nowait(two ? taddr + other : taddr, q);
    tmem_wait_ld();
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = two ? __uint_as_float(r[i]) + __uint_as_float(q[i]) : __uint_as_float(r[i]);
}

template <bool BF16, bool SPLIT>
__global__ void __launch_bounds__(IB_THREADS, 2)
inverted_bottleneck_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW1,
                           const __grid_constant__ CUtensorMap tmW2, const IbDev g) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* const sm = smem_raw + (sbase - smem_u32(smem_raw));
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int rank = SPLIT ? (int)blockIdx.z : 0;
    const int first = g.first[rank], nb = g.count[rank], N1 = nb * 32;
    const int th = (int)blockIdx.x / g.tiles_w, oh0 = th * g.ph, ow0 = ((int)blockIdx.x - th * g.tiles_w) * g.pw;
    const int ih0 = oh0 * g.stride - 1, iw0 = ow0 * g.stride - 1;
    constexpr uint32_t W1_BOX = BF16 ? 2048u : 4096u, W_ROW = BF16 ? 64u : 128u;      // 32 rows of 32 channels; a row
    const uint32_t x_stage = a_stage_of(g.rows), d_stage = BF16 ? (uint32_t)pad8(g.px) * 64u : a_stage_of(g.px);
    const uint32_t w2_stage = (uint32_t)g.BN2 * W_ROW;
    const int rp = pad8(g.rows);

    const uint32_t bars = sbase + g.bar_off;
    auto full_bar = [&](int kb) { return bars + 8u * kb; };
    auto conv_bar = [&](int kb) { return bars + 8u * (IB_MAX_KB + kb); };
    const uint32_t w2_bar = bars + 8u * (2 * IB_MAX_KB), acc1_bar = w2_bar + 8, acc2_bar = w2_bar + 16, recv_bar = w2_bar + 24,
                   par_bar = w2_bar + 32, holder = w2_bar + 40;
    float* const par = reinterpret_cast<float*>(sm + g.par_off);      // biases 1, 2 [nb_most * 32], 3 [BN2], taps [nb_most][32][9]
    float* const sb1 = par;
    float* const sb2 = par + g.nb_most * 32;
    float* const sb3 = par + g.nb_most * 64;
    float* const swd = sb3 + g.BN2;

    const int rows_per = (g.px + g.ranks - 1) / g.ranks;      // output pixels this CTA adds up
    const int my_rows = max(0, min(rows_per, g.px - rank * rows_per));
    if (warp == 0 && lane == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmX)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmW1)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmW2)) : "memory");
        for (int kb = 0; kb < g.nkb1; ++kb) {
            mbar_init(full_bar(kb), (uint32_t)(1 + nb));      // the pixels' box and one of weights a channel block
            mbar_init(conv_bar(kb), 4);
        }
        mbar_init(w2_bar, 1);
        mbar_init(acc1_bar, (uint32_t)g.issuers);
        mbar_init(acc2_bar, 2);
        mbar_init(recv_bar, 1);
        mbar_init(par_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_take(holder, (uint32_t)g.tmem_cols);
    const int quarter = warp & 3, grp = warp >> 2;            // the rows of the accumulators that this warp may read, its share of the columns
    const int row = quarter * 32 + lane;                      // this lane's accumulator row: a pixel of the halo, later one of the patch
    const int hr = div_magic(row, g.hw, g.magic_hw), ih = ih0 + hr, iw = iw0 + (row - hr * g.hw);
    const bool inside = ih >= 0 && ih < g.H && iw >= 0 && iw < g.W;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if constexpr (SPLIT) {
        if (threadIdx.x == 64 && my_rows) mbar_expect_tx(recv_bar, (uint32_t)(g.ranks * my_rows * g.BN2) * 4u);
        __syncwarp();
    }
    const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(sm + (holder - sbase));
    const uint32_t tacc = tmem_base + ((uint32_t)(quarter * 32) << 16);
    // Loads, dealt to the warps (each costs its thread ~165 cycles): the pixels by warps 0 and 7, what later phases need by them as well, the
    // expansion's weights by warps 2 - 5 and 8 - 15.  Weights that nothing before this launch in its stream still writes are fetched before the wait for
    // the previous kernel.
    auto load_weights = [&]() {
        if (warp == 0) {
            // a block's biases and raw depthwise taps [channel][9], as far as its channels exist
            uint32_t bytes = g.b3 ? (uint32_t)g.K * 4u : 0u;
            for (int j = 0; j < nb; ++j)
                bytes += (uint32_t)min(32, g.E - (first + j * g.step) * 32) * (36u + (g.b1 ? 4u : 0u) + (g.b2 ? 4u : 0u));
            mbar_expect_tx(par_bar, bytes);
            for (int j = 0; j < nb; ++j) {
                const int c = (first + j * g.step) * 32;
                const uint32_t n = (uint32_t)min(32, g.E - c);
                if (g.b1) bulk_load(smem_u32(sb1 + j * 32), g.b1 + c, n * 4u, par_bar);
                bulk_load(smem_u32(swd + j * 288), g.wd + (long long)c * 9, n * 36u, par_bar);
                if (g.b2) bulk_load(smem_u32(sb2 + j * 32), g.b2 + c, n * 4u, par_bar);
            }
            if (g.b3) bulk_load(smem_u32(sb3), g.b3, (uint32_t)g.K * 4u, par_bar);
        } else if (warp == 7) {
            mbar_expect_tx(w2_bar, (uint32_t)nb * w2_stage);
            const int box = g.BN2 / g.w2_boxes;
            for (int j = 0; j < nb; ++j)
                for (int h = 0; h < g.w2_boxes; ++h)
                    tma_load_3d(sbase + g.w2_off + j * w2_stage + (uint32_t)(h * box) * W_ROW, &tmW2, (first + j * g.step) * 32, h * box, 0, w2_bar);
        } else if (warp != 1 && warp != 6) {
            for (int i = warp < 8 ? warp - 2 : warp - 4; i < g.nkb1 * nb; i += 12) {
                const int kb = i / nb, j = i - kb * nb;
                mbar_expect_tx(full_bar(kb), W1_BOX);
                tma_load_3d(sbase + g.w1_off + (uint32_t)i * W1_BOX, &tmW1, kb * 32, (first + j * g.step) * 32, 0, full_bar(kb));
            }
        }
    };
    if (g.early) {
        if (elect_one()) load_weights();
        __syncwarp();
    }
    pdl_wait();
    pdl_trigger();
    bool ok = true;
    if ((warp == 0 || warp == 7) && elect_one()) {
        for (int kb = warp == 0 ? 0 : 1; kb < g.nkb1; kb += 2) {
            mbar_expect_tx(full_bar(kb), (uint32_t)g.rows * 128u);
            tma_load_3d(sbase + kb * x_stage, &tmX, kb * 32, iw0, ih0, full_bar(kb));
        }
    }
    __syncwarp();
    if (!g.early && elect_one()) load_weights();
    __syncwarp();
    if (warp == 0 || warp == 7) {
        // (through with their loads)
    } else if (warp != 1 && warp != 6) {
        if constexpr (BF16) {
            // the pixels, rounded to bf16 (a row a thread; warps 8 - 11 and 12 - 15 take the blocks in turn): what the MMAs read
            if (warp >= 8)
                for (int kb = (warp - 8) >> 2; kb < g.nkb1; kb += 2) {
                    ok = ok && mbar_wait(full_bar(kb), 0);
                    if (ok && row < g.rows) {
#pragma unroll
                        for (int c = 0; c < 4; ++c) convert_chunk<false>(sm + kb * x_stage, sm + g.conv_off + kb * rp * 64, nullptr, row, c, rp);
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(conv_bar(kb));
                }
        }
        __syncwarp();
    } else {
        const int iss = warp == 1 ? 0 : 1;
        if (iss < g.issuers && elect_one()) {
            const uint32_t fmt = BF16 ? 1u : 2u;
            const uint32_t idesc = (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(N1 >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
            const uint32_t acc = tmem_base + (uint32_t)(iss * N1);
            for (int kb = iss; kb < g.nkb1; kb += g.issuers) {
                ok = mbar_wait(BF16 ? conv_bar(kb) : full_bar(kb), 0);
                if (!ok) break;
                tc_fence_after();
                const uint32_t first_mma = kb != iss ? 1u : 0u;
                const uint32_t b_src = sbase + g.w1_off + (uint32_t)(kb * nb) * W1_BOX;
                if constexpr (BF16) {
                    const uint32_t a_src = sbase + g.conv_off + (uint32_t)(kb * rp) * 64u, lbo = (uint32_t)rp * 16u;
                    const uint64_t bdesc = make_smem_desc64(b_src);
#pragma unroll
                    for (int kk = 0; kk < 2; ++kk)
                        umma<true>(acc, make_smem_desc_plain(a_src + kk * 2 * lbo, lbo, 128), bdesc + (uint64_t)(kk * 2), idesc, kk ? 1u : first_mma);
                } else {
                    const uint64_t adesc = make_smem_desc(sbase + kb * x_stage), bdesc = make_smem_desc(b_src);
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        umma<false>(acc, adesc + (uint64_t)(kk * 2), bdesc + (uint64_t)(kk * 2), idesc, kk ? 1u : first_mma);
                }
            }
            if (ok) umma_commit(acc1_bar);
        }
        __syncwarp();
    }

    // Expansion out of the accumulators: + bias, activation, zero outside the image, into the tiles that the depthwise pass reads (in the
    // place of the operands, which the MMAs are through with).  Their rows are IB_PITCH bytes apart: sixteen more than a block's, so that
    // neither the lanes' rows here nor the pixels' words there meet in a bank.
    auto gave_up = [&]() {
        if (!ok && lane == 0) atomicExch(&g_device_status, (int)NNV_ERR_TIMEOUT);
        ok = __all_sync(0xffffffffu, ok);
    };
    const uint32_t e_stage = (uint32_t)g.rows * IB_PITCH;
    ok = ok && mbar_wait(par_bar, 0) && mbar_wait(acc1_bar, 0);
    tc_fence_after();
    gave_up();
    if (ok && quarter * 32 < g.rows) {
        const bool two = min(g.issuers, g.nkb1) > 1;
        uint32_t dst = sbase + (uint32_t)row * IB_PITCH + (uint32_t)grp * 32u;
#pragma unroll 1
        for (int c0 = grp * 8; c0 < N1; c0 += 32, dst += e_stage) {
            float v[8];
            ib_acc8(tacc + (uint32_t)c0, two, (uint32_t)N1, v);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const float4 bb = g.b1 ? *reinterpret_cast<const float4*>(sb1 + c0 + 4 * c) : make_float4(0.f, 0.f, 0.f, 0.f);
                v[4 * c] += bb.x; v[4 * c + 1] += bb.y; v[4 * c + 2] += bb.z; v[4 * c + 3] += bb.w;
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = fminf(fmaxf(v[i], 0.f), g.most1);
            if (row < g.rows) {
                const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
                sts128(dst, inside ? make_float4(v[0], v[1], v[2], v[3]) : none);
                sts128(dst + 16u, inside ? make_float4(v[4], v[5], v[6], v[7]) : none);
            }
        }
    }
    tc_fence_before();                                        // (the projection's accumulators take the same columns)
    __syncthreads();

    // Depthwise: sixteen lanes to a pixel and channel block, two channels each.
    {
        const int q = lane & 15;
        const uint32_t down = (uint32_t)g.hw * IB_PITCH;
#pragma unroll 1
        for (int u = warp * 2 + (lane >> 4); u < nb * g.px; u += IB_THREADS / 16) {
            const int j = div_magic(u, g.px, g.magic_px), p = u - j * g.px, pr = div_magic(p, g.pw, g.magic_pw), pc = p - pr * g.pw;
            const int c = (first + j * g.step) * 32 + 2 * q, oh = oh0 + pr, ow = ow0 + pc;
            const uint32_t top = sbase + (uint32_t)j * e_stage + (uint32_t)((pr * g.hw + pc) * g.stride) * IB_PITCH + (uint32_t)q * 8u;
            const uint32_t taps = smem_u32(swd) + (uint32_t)(j * 288 + q * 18) * 4u;       // [channel 0, 1][tap 0..8]
            float2 v[9], t[9];
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                v[3 * r] = lds64_at<0>(top + r * down);
                v[3 * r + 1] = lds64_at<IB_PITCH>(top + r * down);
                v[3 * r + 2] = lds64_at<2 * IB_PITCH>(top + r * down);
            }
            t[0] = lds64_at<0>(taps); t[1] = lds64_at<8>(taps); t[2] = lds64_at<16>(taps); t[3] = lds64_at<24>(taps); t[4] = lds64_at<32>(taps);
            t[5] = lds64_at<40>(taps); t[6] = lds64_at<48>(taps); t[7] = lds64_at<56>(taps); t[8] = lds64_at<64>(taps);
            const float w[18] = {t[0].x, t[0].y, t[1].x, t[1].y, t[2].x, t[2].y, t[3].x, t[3].y, t[4].x,
                                 t[4].y, t[5].x, t[5].y, t[6].x, t[6].y, t[7].x, t[7].y, t[8].x, t[8].y};
            float2 o = g.b2 ? *reinterpret_cast<const float2*>(sb2 + j * 32 + 2 * q) : make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                o.x = fmaf(v[k].x, w[k], o.x);
                o.y = fmaf(v[k].y, w[9 + k], o.y);
            }
            const bool real = c < g.E;                        // (padding of the last block has no taps)
            o.x = real ? fminf(fmaxf(o.x, 0.f), g.most2) : 0.f;
            o.y = real ? fminf(fmaxf(o.y, 0.f), g.most2) : 0.f;
            if constexpr (BF16) {
                *reinterpret_cast<__nv_bfloat162*>(sm + g.d_off + j * d_stage + (uint32_t)((q >> 2) * pad8(g.px) + p) * 16u + (uint32_t)(q & 3) * 4u) =
                    __floats2bfloat162_rn(o.x, o.y);
            } else {
                *reinterpret_cast<float2*>(sm + g.d_off + j * d_stage + (uint32_t)p * 128u + (uint32_t)(((q >> 1) ^ (p & 7)) << 4) + (uint32_t)(q & 1) * 8u) = o;
            }
            if (real && oh < g.OH && ow < g.OW) {
                *reinterpret_cast<float2*>(g.d + ((oh * g.OW + ow) * g.E + c)) = o;
                // the expansion's pixels that this one owns: itself, or with stride 2 the 2 x 2 from itself on
                const int eh = oh * g.stride, ew = ow * g.stride;
                float* const e = g.e + ((eh * g.W + ew) * g.E + c);
                *reinterpret_cast<float2*>(e) = v[4];
                if (g.stride == 2) {
                    if (ew + 1 < g.W) *reinterpret_cast<float2*>(e + g.E) = v[5];
                    if (eh + 1 < g.H) {
                        *reinterpret_cast<float2*>(e + g.W * g.E) = v[7];
                        if (ew + 1 < g.W) *reinterpret_cast<float2*>(e + (g.W + 1) * g.E) = v[8];
                    }
                }
            }
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the tiles -> the MMAs' reads; the expansion's place -> the peers' pushes
    __syncthreads();
    tc_fence_after();
    __syncwarp();
    // (Relaxed: a release would wait for the stores above to reach memory, 0.6 us.  What the peers write next nobody here reads any more.)
    if constexpr (SPLIT) cluster_arrive_relaxed();            // this CTA's barriers and the place of its received rows may be used from here on

    // Projection.  With both accumulators of a split here the issuers take its blocks in turn, else each half of the columns.
    if ((warp == 1 || warp == 6) && ok) {
        const int iss = warp == 1 ? 0 : 1;
        if (elect_one()) {
            ok = mbar_wait(w2_bar, 0);
            if (ok) {
                tc_fence_after();
                const int half = ((g.BN2 >> 5) << 4) + ((g.BN2 & 16) ? 16 : 0);      // columns of the first half, a multiple of 16
                const int n = g.both ? g.BN2 : iss == 0 ? half : g.BN2 - half;
                const uint32_t fmt = BF16 ? 1u : 2u;
                const uint32_t idesc = (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
                const uint32_t col = g.both ? (uint32_t)(iss * g.BN2) : (uint32_t)(iss * half);
                const int j0 = g.both ? iss : 0, dj = g.both ? 2 : 1;
                if (n > 0)
                    for (int j = j0; j < nb; j += dj) {
                        const uint32_t a_src = sbase + g.d_off + j * d_stage;
                        const uint32_t b_src = sbase + g.w2_off + j * w2_stage + (g.both ? 0u : col * W_ROW);
                        if constexpr (BF16) {
                            const uint32_t lbo = (uint32_t)pad8(g.px) * 16u;
                            const uint64_t bdesc = make_smem_desc64(b_src);
#pragma unroll
                            for (int kk = 0; kk < 2; ++kk)
                                umma<true>(tmem_base + col, make_smem_desc_plain(a_src + kk * 2 * lbo, lbo, 128), bdesc + (uint64_t)(kk * 2), idesc,
                                           kk || j != j0 ? 1u : 0u);
                        } else {
                            const uint64_t adesc = make_smem_desc(a_src), bdesc = make_smem_desc(b_src);
#pragma unroll
                            for (int kk = 0; kk < 4; ++kk)
                                umma<false>(tmem_base + col, adesc + (uint64_t)(kk * 2), bdesc + (uint64_t)(kk * 2), idesc, kk || j != j0 ? 1u : 0u);
                        }
                    }
                umma_commit(acc2_bar);
            }
        }
        __syncwarp();
    }

    // Partial rows: parked as rows of BN2 words (16-byte words rotated by the row's index) over the operands, pushed to their owners.
    const int nch = g.BN2 / 4;
    auto rotation = [&](int r) { return r - div_magic(r, nch, g.magic_nch) * nch; };
    const uint32_t park = sbase + g.d_off;
    ok = ok && mbar_wait(acc2_bar, 0);
    tc_fence_after();
    gave_up();
    if (ok && quarter * 32 < g.px) {
        const bool two = g.both && nb > 1;
        const uint32_t prow = park + (uint32_t)row * (uint32_t)g.BN2 * 4u;
        int pos = rotation(row) + 2 * grp;
        if (pos >= nch) pos -= nch;
#pragma unroll 1
        for (int c0 = grp * 8; c0 < g.BN2; c0 += 32) {
            float v[8];
            ib_acc8(tacc + (uint32_t)c0, two, (uint32_t)g.BN2, v);
            if (row < g.px) {
                sts128(prow + (uint32_t)pos * 16u, make_float4(v[0], v[1], v[2], v[3]));
                sts128(prow + (uint32_t)(pos + 1 == nch ? 0 : pos + 1) * 16u, make_float4(v[4], v[5], v[6], v[7]));
            }
            pos += 8;
            if (pos >= nch) pos -= nch;                       // (rows of sixteen columns have four words, and end here)
        }
    }
    uint32_t recv = park, part_stride = 0;
    int total = my_rows * g.BN2;
    if constexpr (SPLIT) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        cluster_wait();                                       // every CTA is through with the place where its rows go
        __syncthreads();
        for (int to = warp; ok && to < g.ranks; to += IB_THREADS / 32) {      // (a push costs its thread as much as a load)
            const int a0 = to * rows_per, n = min(rows_per, g.px - a0);
            if (n > 0 && elect_one())
                bulk_push(cluster_addr(sbase + (uint32_t)(rank * n * g.BN2) * 4u, to), park + (uint32_t)(a0 * g.BN2) * 4u, (uint32_t)(n * g.BN2) * 4u,
                          cluster_addr(recv_bar, to));
            __syncwarp();
        }
        recv = sbase;
        part_stride = (uint32_t)(my_rows * g.BN2) * 4u;
    } else {
        __syncthreads();
    }
    // Owner: partial rows in rank order, + bias, + residual, activation.  A thread adds up single words: there are few of them.
    const int row0 = rank * rows_per;
    int rr = 0, cc = 0, off = 0;                              // of the word in hand: row, column, place in the output (-1: nowhere)
    auto place = [&](int idx) {
        rr = div_magic(idx, g.BN2, g.magic_n); cc = idx - rr * g.BN2;
        const int p = row0 + rr, pr = div_magic(p, g.pw, g.magic_pw), oh = oh0 + pr, ow = ow0 + (p - pr * g.pw);
        off = idx < total && oh < g.OH && ow < g.OW && cc < g.K ? (oh * g.OW + ow) * g.K + cc : -1;
    };
    place((int)threadIdx.x);
    float aa = g.addend && off >= 0 ? __ldg(g.addend + off) : 0.f;
    if constexpr (SPLIT) {
        ok = !my_rows || mbar_wait(recv_bar, 0);
        gave_up();
        if (!ok) total = 0;
        __syncwarp();
        cluster_arrive_relaxed();                             // this CTA's rows have arrived: their senders may leave
    } else if (!ok) {
        total = 0;
    }
#pragma unroll 1
    for (int idx = threadIdx.x; idx < total; idx += IB_THREADS) {
        int pos = (cc >> 2) + rotation(row0 + rr);
        if (pos >= nch) pos -= nch;
        uint32_t src = recv + (uint32_t)(rr * g.BN2 + pos * 4 + (cc & 3)) * 4u;
        float a;
        if constexpr (SPLIT) {
            // a split's accumulators first, then the splits; -0 in place of an accumulator that is none leaves every sum as it is
            uint32_t pairs = g.pairs;
            a = -0.f;
#pragma unroll 1
            for (int k = 0; k < g.splits; k += 4) {
                float v[8];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const bool here = k + u < g.splits, two = here && (pairs & 1u);
                    v[2 * u] = here ? lds32(src) : -0.f;
                    v[2 * u + 1] = two ? lds32(src + part_stride) : -0.f;
                    src += two ? 2u * part_stride : here ? part_stride : 0u;
                    pairs >>= 1;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) a += v[2 * u] + v[2 * u + 1];
            }
        } else {
            a = lds32(src);
        }
        a += g.b3 ? sb3[cc] : 0.f;
        if (g.addend) a += aa;
        if (g.act3) a = fminf(fmaxf(a, 0.f), g.act3 == 2 ? 6.f : INFINITY);
        const int to = off;
        place(idx + IB_THREADS);                              // (the next residual word leaves before this one's store)
        aa = g.addend && off >= 0 ? __ldg(g.addend + off) : 0.f;
        if (to >= 0) g.y[to] = a;
    }
    __syncwarp();
    if constexpr (SPLIT) cluster_wait();                      // nobody leaves while its rows may still be on their way
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)g.tmem_cols) : "memory");
    }
}
