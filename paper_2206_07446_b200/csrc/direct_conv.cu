// fp32 direct convolution: an implicit GEMM on the FP32 pipes straight from the raw OIHW weights (no weight transform).
//
// Bound: the L1 / shared-memory data path (4 x 4 outputs a thread: ~6.5 cycles of shared-memory reads for 4 cycles of
// FMAs), and on the small layers a cold run picks this kernel for, latency.  A block owns 32 pixels x 32 channels and
// walks the reduction in chunks of JC (channel, tap) pairs in raw weight order; the next chunk's global loads are in
// flight while this one is multiplied out of shared memory.
//   - Eight lanes read 128 contiguous bytes (32 channels of one pixel and tap; 32 weights of one row), so a warp's
//     gather touches four lines; with 32-byte pieces of 16 lines the gathers alone cost as much L1 time as the
//     multiplication.  The pairs are stored transposed, [pair][pixel] and [pair][channel], with the 16-byte words of a
//     row permuted by the pair's index / 4, which makes the stores and the reads free of bank conflicts.
//   - The block's threads form four groups of 8 x 8 that take a quarter of every chunk each and are summed at the end.
//   - `splits` blocks of a cluster share the chunks of one tile and add their partial tiles through distributed shared
//     memory in rank order (the result does not depend on timing).
// Measured (back to back calls, us): 3 -> 32 3x3 / 2 @224 7.1; the kernel further below, on larger tiles, takes most layers on channels in fours:
// this kernel / that one 64 -> 128 3x3 / 2 @56 10.9 / 9.6, 256 -> 256 3x3 @14 17.6 / 16.5, 512 -> 512 3x3 @7 23.2 / 16.4, 64 -> 64 3x3 @112 45.2 / 37.7,
// 1024 -> 256 1x1 @14 9.5 / 7.5, 2048 -> 512 1x1 @7 11.9 / 7.5, 320 -> 1280 1x1 @7 7.4 / 5.6.
#include <algorithm>
#include <type_traits>

#include "nnv_internal.h"

namespace nnv {
namespace {

constexpr int DC_T = 32;                                      // pixels and channels of a tile
constexpr int DC_THREADS = 256;
constexpr int DC_GROUPS = 4;

struct DirectDev {
    const float* x; const float* w; const float* bias; const float* add; float* y;
    int act, C, H, W, K, R, S, stride, pad, OH, OW, splits;
    int* status;                                               // the device status word (blocks that wait for one another)
};

__device__ __forceinline__ float direct_act(float v, int act) {
    if (act == 1) return fmaxf(v, 0.f);
    if (act == 2) return fminf(fmaxf(v, 0.f), 6.f);
    return v;
}

// Reduction pairs per chunk: 32 channels x 9 taps, 64 channels x 1 tap, or 64 flat (c, r, s) positions (TAPS = 0: any filter).
template <int TAPS> struct DcChunk {
    static constexpr int CB = TAPS == 9 ? 32 : 64;
    static constexpr int JC = TAPS == 9 ? 288 : 64;
};

// Shared memory of a block: both staged operands, at least the four groups' partial tiles.
__host__ __device__ constexpr int dc_smem_floats(int jc) {
    return 2 * jc * DC_T > DC_GROUPS * DC_T * (DC_T + 4) ? 2 * jc * DC_T : DC_GROUPS * DC_T * (DC_T + 4);
}

// Word of (pair j, element e) in a staged operand.
__device__ __forceinline__ int dc_word(int j, int e) { return j * DC_T + (e ^ (((j >> 2) & 7) << 2)); }

template <int TAPS>
__global__ void __launch_bounds__(DC_THREADS, 2)
direct_conv_kernel(const DirectDev g) {
    pdl_wait();
    constexpr int JC = DcChunk<TAPS>::JC, CB = DcChunk<TAPS>::CB, T = DC_T, G = DC_GROUPS, GT = DC_THREADS / G;
    extern __shared__ __align__(16) float sm[];
    float* const As = sm;
    float* const Bs = sm + JC * T;

    const int tid = threadIdx.x;
    const int RS = g.R * g.S, Q = g.C * RS, P = g.OH * g.OW;
    const int p0 = blockIdx.x * T, k0 = blockIdx.y * T;
    const int sp = blockIdx.z;
    const int chunks_all = (Q + JC - 1) / JC;
    const int ch0 = chunks_all * sp / g.splits, ch1 = chunks_all * (sp + 1) / g.splits;

    // Loader role: element e (pixel of A, channel of B) and word l8 of its eight.  Word loads move four channels / weights;
    // the flat form moves single positions.
    constexpr int VW = TAPS ? 4 : 1;
    constexpr int N = JC / (8 * VW);                           // words a thread fetches per operand and chunk
    using Word = typename std::conditional<TAPS != 0, float4, float>::type;
    const int e = tid >> 3, l8 = tid & 7;
    const int pa = p0 + e, kb = k0 + e;
    const int oh = pa / g.OW, ow = pa - oh * g.OW;
    const int ih0 = pa < P ? oh * g.stride - g.pad : -(1 << 20), iw0 = ow * g.stride - g.pad;   // a pixel beyond the grid is outside the image
    const float* const wrow = g.w + (long long)kb * Q;
    Word ra[N], rb[N];
    // Positions outside the image, the filter bank or the reduction are fetched from a valid address and zeroed on
    // their way into shared memory, so that all loads of a chunk leave back to back.
    uint32_t live_a = 0, live_b = 0;
    auto fetch = [&](int ch) {
        live_a = live_b = 0;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            int c, r, s;
            if constexpr (TAPS != 0) {
                r = TAPS == 9 ? i / 3 : 0;
                s = TAPS == 9 ? i % 3 : 0;
                c = ch * CB + (TAPS == 9 ? 0 : 32 * i) + 4 * l8;
            } else {
                const int q = ch * JC + 8 * i + l8;
                if (ch * JC + 8 * i >= Q) break;
                c = q / RS;
                const int rs = q - c * RS;
                r = rs / g.S;
                s = rs - r * g.S;
            }
            const int ih = ih0 + r, iw = iw0 + s;
            const bool ok = c < g.C && ih >= 0 && ih < g.H && iw >= 0 && iw < g.W;
            ra[i] = __ldg(reinterpret_cast<const Word*>(ok ? g.x + ((long long)ih * g.W + iw) * g.C + c : g.x));
            live_a |= ok ? 1u << i : 0u;
        }
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const int q = ch * JC + (8 * i + l8) * VW;
            const bool ok = kb < g.K && q < Q;
            rb[i] = __ldg(reinterpret_cast<const Word*>(ok ? wrow + q : g.w));
            live_b |= ok ? 1u << i : 0u;
        }
    };
    auto stash = [&](int ch) {
        const int left = (Q - ch * JC + 3) & ~3;               // pairs from here on are never read
#pragma unroll
        for (int i = 0; i < N; ++i) {
            if ((TAPS == 9 ? 36 * l8 : (8 * i + l8) * VW) >= left) break;
            const float* v = reinterpret_cast<const float*>(&ra[i]);
#pragma unroll
            for (int u = 0; u < VW; ++u) {
                const int j = TAPS == 9 ? (4 * l8 + u) * 9 + i : (8 * i + l8) * VW + u;      // raw weight order: channel-major
                As[dc_word(j, e)] = (live_a >> i) & 1u ? v[u] : 0.f;
            }
        }
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const float* v = reinterpret_cast<const float*>(&rb[i]);
            if ((8 * i + l8) * VW >= left) break;
#pragma unroll
            for (int u = 0; u < VW; ++u) Bs[dc_word((8 * i + l8) * VW + u, e)] = (live_b >> i) & 1u ? v[u] : 0.f;
        }
    };

    const int grp = tid / GT, gt = tid - grp * GT;
    const int tx = gt & 7, ty = gt >> 3;                       // tx -> channels, ty -> pixels
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;

    fetch(ch0);
    for (int ch = ch0; ch < ch1; ++ch) {
        if (ch > ch0) __syncthreads();                         // the previous chunk has been multiplied
        stash(ch);
        __syncthreads();
        if (ch + 1 < ch1) fetch(ch + 1);
        const int words = (min(JC, Q - ch * JC) + 3) >> 2;     // groups of four pairs that exist
        const int w1 = words * (grp + 1) / G;
#pragma unroll 1
        for (int wd = words * grp / G; wd < w1; ++wd) {
            const float* a = As + wd * 4 * T + ((ty ^ (wd & 7)) << 2);
            const float* b = Bs + wd * 4 * T + ((tx ^ (wd & 7)) << 2);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float4 av = *reinterpret_cast<const float4*>(a + j * T);
                const float4 bv = *reinterpret_cast<const float4*>(b + j * T);
                const float aa[4] = {av.x, av.y, av.z, av.w}, bb[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int jj = 0; jj < 4; ++jj) acc[i][jj] = fmaf(aa[i], bb[jj], acc[i][jj]);
            }
        }
    }
    // The next kernel's blocks are let in only now: released at the start they would pile up on the SMs this grid leaves
    // idle and run there several to an SM (22.5 us a call back to back where one call takes 14, 64 -> 128 3x3 / 2 @56).
    pdl_trigger();
    __syncthreads();

    // Partial tiles of the groups, then of the cluster, each summed in index order.
    constexpr int RP = T + 4;
    float* red = sm;
    static_assert(G * T * RP <= dc_smem_floats(JC), "the partial tiles reuse the staging buffers");
#pragma unroll
    for (int i = 0; i < 4; ++i)
        *reinterpret_cast<float4*>(red + (grp * T + ty * 4 + i) * RP + tx * 4) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    __syncthreads();
    auto group_sum = [&](int row, int c4) {
        float4 s = *reinterpret_cast<const float4*>(red + row * RP + c4);
#pragma unroll
        for (int q = 1; q < G; ++q) {
            const float4 v = *reinterpret_cast<const float4*>(red + (q * T + row) * RP + c4);
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
        return s;
    };
    if (g.splits > 1) {
        for (int idx = tid; idx < T * (T / 4); idx += DC_THREADS) {      // into group 0's place: every thread its own words
            const int row = idx / (T / 4), c4 = (idx % (T / 4)) * 4;
            *reinterpret_cast<float4*>(red + row * RP + c4) = group_sum(row, c4);
        }
        __syncwarp();                                          // the cluster barrier is one instruction of the whole warp
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
    const bool vec = (g.K & 3) == 0;
    const int rows = T / g.splits;                             // splits is a power of two up to 8
    for (int idx = tid; idx < rows * (T / 4); idx += DC_THREADS) {
        const int row = sp * rows + idx / (T / 4), c4 = (idx % (T / 4)) * 4;
        float4 s;
        if (g.splits == 1) {
            s = group_sum(row, c4);
        } else {
            const uint32_t local = (uint32_t)__cvta_generic_to_shared(red + row * RP + c4);
            float4 part[8];                                    // all remote loads leave before the first is used
#pragma unroll
            for (int rk = 0; rk < 8; ++rk)
                if (rk < g.splits) {
                    uint32_t remote;
                    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(rk));
                    asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];"
                                 : "=f"(part[rk].x), "=f"(part[rk].y), "=f"(part[rk].z), "=f"(part[rk].w) : "r"(remote));
                }
            s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int rk = 0; rk < 8; ++rk)
                if (rk < g.splits) { s.x += part[rk].x; s.y += part[rk].y; s.z += part[rk].z; s.w += part[rk].w; }
        }
        const int p = p0 + row, k = k0 + c4;
        if (p >= P || k >= g.K) continue;
        const long long o = (long long)p * g.K + k;
        float v[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (k + j >= g.K) break;
            if (g.bias) v[j] += __ldg(g.bias + k + j);
            if (g.add) v[j] += __ldg(g.add + o + j);
            v[j] = direct_act(v[j], g.act);
            if (!vec) g.y[o + j] = v[j];
        }
        if (vec) *reinterpret_cast<float4*>(g.y + o) = make_float4(v[0], v[1], v[2], v[3]);
    }
    if (g.splits > 1) {                                        // nobody leaves while its partial tile may still be read
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}

// 3x3 and 1x1 filters on channels in fours.  A block owns T pixels x T channels (T = 32 or 64) and walks the reduction in 16-byte pieces, four
// channels of one tap each.  Both operands arrive by asynchronous copies: pixels as rows of pieces, weights as rows in their raw order (in
// which a piece's four words lie nine apart, so they are read word by word); the next chunk's fly while one is multiplied.  A thread owns 8 x 8
// outputs (8 x 4 where T is 32), so the threads form groups that take the pieces in turn and are summed at the end.
// Bound: the FP32 pipes, with the shared-memory reads beside them: a warp's piece takes 256 multiply-adds and 40 reads (3x3), which two blocks on
// an SM overlap (one block with the next piece's words read between the multiply-adds of the one before: no faster; paired multiply-adds change
// nothing; 4 x 4 outputs a thread need as many reads for a quarter of the work).  Rows are an odd number of pieces apart: eight neighbouring
// rows never meet in a bank.
template <int TAPS, int T> struct DtShape {
    static constexpr int QUADS = TAPS == 9 ? 128 / T : 1024 / T;       // channels of a chunk, in fours
    static constexpr int PIECES = QUADS * TAPS;
    static constexpr uint32_t PITCH = (PIECES | 1) * 16, STAGE = 2 * T * PITCH;
    static constexpr int NJ = T / 8;                           // channels of a thread
    static constexpr int GT = T, G = 256 / GT;                 // threads of a group, groups
    static constexpr int RED = T + 8;                          // words of a partial tile's row
    static constexpr uint32_t RECV = (uint32_t)G * T * RED * 4;        // place of received rows
    static constexpr size_t SMEM = 2 * STAGE > RECV + (T + 8) * RED * 4 ? 2 * STAGE : RECV + (T + 8) * RED * 4;
};
constexpr int DT_THREADS = 256;

__device__ __forceinline__ void copy16(uint32_t dst, const void* src, bool live) {       // (not live: zeros, nothing is read)
    const int n = live ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ float4 lds4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ float lds1(uint32_t addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void sts4(uint32_t addr, float x, float y, float z, float w) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}
__device__ __forceinline__ void add4(float4& a, const float4& b) { a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w; }

template <int TAPS, int T>
__global__ void __launch_bounds__(DT_THREADS, 2)
direct_tile_kernel(const DirectDev g) {
    using D = DtShape<TAPS, T>;
    constexpr int QUADS = D::QUADS, RED = D::RED;
    extern __shared__ __align__(16) float sm[];
    __shared__ __align__(8) unsigned long long recv_bar;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(sm), bar = (uint32_t)__cvta_generic_to_shared(&recv_bar);
    const int tid = threadIdx.x, P = g.OH * g.OW, CQ = g.C >> 2, Q = g.C * TAPS;
    const int p0 = blockIdx.x * T, k0 = blockIdx.y * T, sp = blockIdx.z;
    const int q_first = CQ * sp / g.splits, q_last = CQ * (sp + 1) / g.splits;       // this block's channels, in fours
    const int rows = (T + g.splits - 1) / g.splits, my_rows = max(0, min(rows, T - sp * rows));    // the tile's rows that this block adds up

    // Loader role.  3x3: the lower half of the threads copies a channel quad of a pixel each, nine taps, the upper half as much of a weight row.  1x1:
    // every thread a channel quad of four pixels and four weight rows.
    constexpr int LR = TAPS == 9 ? T : DT_THREADS / QUADS, ROWS = T / LR;
    const int unit = TAPS == 9 ? tid & 127 : tid, lq = unit % QUADS, lr = unit / QUADS;
    const float* px[ROWS];                                     // the pixel's window: its first channel at tap (0, 0), and the taps inside the image
    uint32_t inside[ROWS];
#pragma unroll
    for (int i = 0; i < ROWS; ++i) {
        const int p = p0 + lr + i * LR, oh = p / g.OW, ow = p - oh * g.OW, ih = oh * g.stride - g.pad, iw = ow * g.stride - g.pad;
        px[i] = g.x + ((long long)ih * g.W + iw) * g.C;
        inside[i] = 0;
#pragma unroll
        for (int t = 0; t < TAPS; ++t)
            if (p < P && ih + t / 3 >= 0 && ih + t / 3 < g.H && iw + t % 3 >= 0 && iw + t % 3 < g.W) inside[i] |= 1u << t;
    }
    const long long wrow = (long long)g.W * g.C;
    auto issue = [&](int q0, uint32_t stage) {                 // the chunk's copies
        const int q = q0 + lq;
        if constexpr (TAPS == 9) {
            if (tid < 128) {
                const uint32_t taps = q < q_last ? inside[0] : 0u, dst = stage + (uint32_t)lr * D::PITCH + (uint32_t)lq * 144u;
                const float* src = px[0] + 4 * q;
#pragma unroll
                for (int t = 0; t < 9; ++t) copy16(dst + 16u * t, taps >> t & 1u ? src + (t / 3) * wrow + (t % 3) * g.C : g.x, taps >> t & 1u);
            } else {
                const int left = k0 + lr < g.K ? (q_last - q0) * 9 : 0;      // pieces of the weight row that exist
                const uint32_t dst = stage + (uint32_t)(T + lr) * D::PITCH + 16u * lq;
                const float* src = g.w + (long long)(k0 + lr) * Q + 36 * q0 + 4 * lq;
#pragma unroll
                for (int u = 0; u < 9; ++u) {
                    const bool in = lq + u * QUADS < left;
                    copy16(dst + 16u * u * QUADS, in ? src + 4 * u * QUADS : g.w, in);
                }
            }
        } else {
            const bool here = q < q_last;
            uint32_t dst = stage + (uint32_t)lr * D::PITCH + 16u * lq;
#pragma unroll
            for (int i = 0; i < ROWS; ++i, dst += LR * D::PITCH) {
                const bool in_x = here && inside[i], in_w = here && k0 + lr + i * LR < g.K;
                copy16(dst, in_x ? px[i] + 4 * q : g.x, in_x);
                copy16(dst + T * D::PITCH, in_w ? g.w + (long long)(k0 + lr + i * LR) * Q + 4 * q : g.w, in_w);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (g.splits > 1 && tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }

    constexpr int GX = 8, GY = T / 8, NJ = D::NJ;              // threads of a group along channels and pixels
    const int grp = tid / D::GT, gx = tid % GX, gy = tid % D::GT / GX;         // outputs: pixels gy + GY i, channels gx + GX j
    float acc[8][NJ];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < NJ; ++j) acc[i][j] = 0.f;

    pdl_wait();
    issue(q_first, base);
    if (g.splits > 1 && tid == 0 && my_rows)
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"((uint32_t)(g.splits * my_rows * RED) * 4u) : "memory");
    uint32_t stage = base;
    for (int q0 = q_first; q0 < q_last; q0 += QUADS) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();                                       // the chunk is there, and nobody multiplies the one before any more
        const uint32_t next = base + (stage == base ? D::STAGE : 0u);
        const bool more = q0 + QUADS < q_last;
        if (more) issue(q0 + QUADS, next);
        const int n = min(QUADS, q_last - q0) * TAPS;
        const uint32_t a = stage + (uint32_t)gy * D::PITCH, b = stage + (uint32_t)(T + gx) * D::PITCH;
        int tap = grp % TAPS;
        uint32_t at = TAPS == 1 ? 16u * grp : (uint32_t)(grp / TAPS * 144 + tap * 4);          // the piece's first word in a weight row
#pragma unroll 1
        for (int t = grp; t < n; t += D::G) {
            float4 bv[NJ];
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                const uint32_t row = b + (uint32_t)(GX * j) * D::PITCH + at;
                if constexpr (TAPS == 1) bv[j] = lds4(row);
                else bv[j] = make_float4(lds1(row), lds1(row + 36u), lds1(row + 72u), lds1(row + 108u));
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float4 av = lds4(a + (uint32_t)(GY * i) * D::PITCH + 16u * t);
#pragma unroll
                for (int j = 0; j < NJ; ++j) acc[i][j] = fmaf(av.x, bv[j].x, acc[i][j]);
#pragma unroll
                for (int j = 0; j < NJ; ++j) acc[i][j] = fmaf(av.y, bv[j].y, acc[i][j]);
#pragma unroll
                for (int j = 0; j < NJ; ++j) acc[i][j] = fmaf(av.z, bv[j].z, acc[i][j]);
#pragma unroll
                for (int j = 0; j < NJ; ++j) acc[i][j] = fmaf(av.w, bv[j].w, acc[i][j]);
            }
            if constexpr (TAPS == 1) at += 16u * D::G;
            else {
                tap += D::G;
                at += 4u * D::G;
                if (tap >= TAPS) { tap -= TAPS; at += 144u - 4u * TAPS; }
            }
        }
        stage = next;
    }
    // The next kernel's blocks are let in only now: released at the start they would pile up on the SMs this grid leaves idle and run there
    // several to an SM.
    pdl_trigger();
    __syncthreads();
    if (g.splits > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");     // the place of received rows is free, the barrier there

    // The groups' partial tiles, summed in order.
    {
        float* red = sm + (grp * T + gy) * RED + gx;
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < NJ; ++j) red[i * GY * RED + j * GX] = acc[i][j];
    }
    __syncthreads();
    const bool vec = (g.K & 3) == 0 && (reinterpret_cast<uintptr_t>(g.add) & 15) == 0;
    auto finish = [&](int r, int c4, float4 s) {
        const int p = p0 + r, k = k0 + c4;
        if (p >= P || k >= g.K) return;
        const long long o = (long long)p * g.K + k;
        if (vec) {
            if (g.bias) add4(s, make_float4(__ldg(g.bias + k), __ldg(g.bias + k + 1), __ldg(g.bias + k + 2), __ldg(g.bias + k + 3)));
            if (g.add) add4(s, __ldg(reinterpret_cast<const float4*>(g.add + o)));
            *reinterpret_cast<float4*>(g.y + o) = make_float4(direct_act(s.x, g.act), direct_act(s.y, g.act), direct_act(s.z, g.act), direct_act(s.w, g.act));
        } else {
            const float v[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (k + j >= g.K) break;
                float f = v[j];
                if (g.bias) f += __ldg(g.bias + k + j);
                if (g.add) f += __ldg(g.add + o + j);
                g.y[o + j] = direct_act(f, g.act);
            }
        }
    };
#pragma unroll 1
    for (int idx = tid; idx < T * T / 4; idx += DT_THREADS) {
        const int r = idx / (T / 4), c4 = (idx % (T / 4)) * 4;
        const uint32_t at = base + (uint32_t)(r * RED + c4) * 4u;
        float4 s = lds4(at);
#pragma unroll
        for (int q = 1; q < D::G; ++q) add4(s, lds4(at + (uint32_t)(q * T * RED) * 4u));
        if (g.splits == 1) finish(r, c4, s);
        else sts4(at, s.x, s.y, s.z, s.w);
    }
    if (g.splits == 1) return;

    // The cluster's: every block pushes the others their rows of its tile, which they add up in rank order.
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (tid < g.splits) {
        const int n = min(rows, T - tid * rows);
        if (n > 0) {
            uint32_t dst, there;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"(base + D::RECV + (uint32_t)(sp * n * RED) * 4u), "r"(tid));
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(there) : "r"(bar), "r"(tid));
            asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(dst), "r"(base + (uint32_t)(tid * rows * RED) * 4u), "r"((uint32_t)(n * RED) * 4u), "r"(there) : "memory");
        }
    }
    __syncwarp();
    bool arrived = my_rows == 0;
    for (uint32_t i = 0; !arrived && i < (1u << 20); ++i) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(done) : "r"(bar) : "memory");
        arrived = done != 0;
    }
    if (!arrived && tid == 0) atomicExch(g.status, (int)NNV_ERR_TIMEOUT);
    __syncwarp();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");      // this block's rows have arrived: their senders may leave
    for (int idx = tid; arrived && idx < my_rows * (T / 4); idx += DT_THREADS) {
        const int r = idx / (T / 4), c4 = (idx % (T / 4)) * 4;
        float4 part[8];
#pragma unroll
        for (int rk = 0; rk < 8; ++rk)
            if (rk < g.splits) part[rk] = lds4(base + D::RECV + (uint32_t)((rk * my_rows + r) * RED + c4) * 4u);
        float4 s = part[0];
#pragma unroll
        for (int rk = 1; rk < 8; ++rk)
            if (rk < g.splits) add4(s, part[rk]);
        finish(sp * rows + r, c4, s);
    }
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <int TAPS, int T>
nnv_status_t launch_dt(const DirectDev& g, cudaStream_t st) {
    constexpr size_t smem = DtShape<TAPS, T>::SMEM;
    static const cudaError_t attr = cudaFuncSetAttribute(direct_tile_kernel<TAPS, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    NNV_CUDA(attr);
    const dim3 grid(ceil_div(g.OH * g.OW, T), ceil_div(g.K, T), g.splits);
    NNV_REQUIRE(grid.y <= 65535, NNV_ERR_UNSUPPORTED, "too many output channels for the direct kernel");
    const dim3 outputs(ceil_div(g.OH * g.OW, DC_T), ceil_div(g.K, DC_T));     // (as for direct_conv_kernel; 260 layers take the same either way)
    NNV_CUDA(launch_pdl_attrs(stream_carveout(STREAM_LONE, outputs, dim3(DT_THREADS)), g.splits, direct_tile_kernel<TAPS, T>, grid, dim3(DT_THREADS), smem, st, g));
    return NNV_OK;
}

// The device status word's address, asked for once per thread and device.
nnv_status_t status_word(int** out) {
    static thread_local int of = -1;
    static thread_local const int* word = nullptr;
    int dev = 0;
    NNV_CUDA(cudaGetDevice(&dev));
    if (dev != of) {
        NNV_TRY(device_status_address(&word));
        of = dev;
    }
    *out = const_cast<int*>(word);
    return NNV_OK;
}

// direct_tile_kernel's tile and split for a layer, if it is to run it: by estimated time, us, of calls one behind the other.  Fitted to 260 layers of 16 -
// 2048 channels on 7 - 160 pixels a side (11 % off on average, either kernel): they take 0.825 of direct_conv_kernel's time (geometric mean; 0.80
// with the best of all tiles, splits and kernels), three of them 2 % longer or more (of 260 others five, 24 -> 32 3x3 @106x84 by 8 %).  direct_conv_kernel keeps what it is estimated to run within 3 %
// as fast, and within 20 % on up to 32 input or output channels, where the estimates are worst (32 -> 32 3x3 @80 8.5 us against 9.9).
struct DirectSplit { int splits; double us; };
DirectSplit pick_split(int P, int C, int K, int jc, int chunks, int taps) {
    // The split with the least estimated time, in cycles: an SM's blocks share its L1, so a chunk costs blocks per SM x ~16 cycles a pair; a split
    // adds two cluster barriers and the remote reads.
    const long long tiles = (long long)ceil_div(P, DC_T) * ceil_div(K, DC_T);
    DirectSplit d{1, 0.0};
    double best = 1e30;
    for (int s = 1; s <= 8 && s <= chunks; s *= 2) {
        const double t = (double)((tiles * s + 147) / 148) * ceil_div(chunks, s) * jc * 16.0 + (s > 1 ? 3000.0 : 0.0);
        if (t < best - 1e-9) { best = t; d.splits = s; }
    }
    const double blocks = (double)tiles * d.splits, eff = std::max(1.0, blocks / 148), n = ceil_div(chunks, d.splits), last = std::min(1.0, (double)C * taps / jc);
    d.us = 1.05 + (d.splits > 1 ? 1.31 : 0.0) + 0.268 * blocks / 148 + (taps == 9 ? 0.836 * n + eff * (3.2 * n + 0.624 * last) : 0.469 * n + eff * (0.549 * n + 0.533 * last));
    return d;
}
bool pick_tile(int P, int C, int K, int taps, int* tile, int* splits) {
    double best = 1e30;
    for (int t = 32; t <= 64; t *= 2)
        for (int s = 1; s <= 8 && s <= C / 4; s *= 2) {
            const double blocks = (double)ceil_div(P, t) * ceil_div(K, t) * s, slots = s == 8 ? 264 : s == 4 ? 284 : 296;
            const int per = taps == 9 ? 128 / t : 1024 / t, g = 256 / t, quads = ceil_div(C / 4, s);      // quads a chunk, groups
            const int rounds = quads / per * ceil_div(per * taps, g) + ceil_div(quads % per * taps, g);
            const double waves = std::ceil(blocks / slots), w = waves < 3 ? waves : blocks / slots + 0.5;
            const double pair = waves > 1 ? 1.0 : std::min(1.0, std::max(0.0, (blocks - 100) / 60));       // blocks that share an SM
            const double us = 1.89 + (s > 1 ? 0.4 + 0.167 * w : 0.0) + 0.913 * (w - 1) + 0.058 * w * (1 - pair) * ceil_div(quads, per) +
                              w * (t == 64 ? rounds * (0.687 * (1 - pair) + 0.932 * pair) + 1.76 * pair : rounds * (0.384 * (1 - pair) + 0.646 * pair) + 0.34 * pair);
            if (us < best - 1e-9) { best = us; *tile = t; *splits = s; }
        }
    const int jc = taps == 9 ? 288 : 64;
    return best < (C <= 32 || K <= 32 ? 0.8 : 0.97) * pick_split(P, C, K, jc, ceil_div(C * taps, jc), taps).us;
}

template <int TAPS>
nnv_status_t launch_dc(const DirectDev& g, cudaStream_t st) {
    constexpr size_t smem = sizeof(float) * dc_smem_floats(DcChunk<TAPS>::JC);
    static const cudaError_t attr = cudaFuncSetAttribute(direct_conv_kernel<TAPS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    NNV_CUDA(attr);
    const dim3 grid(ceil_div(g.OH * g.OW, DC_T), ceil_div(g.K, DC_T), g.splits);
    NNV_REQUIRE(grid.y <= 65535, NNV_ERR_UNSUPPORTED, "too many output channels for the direct kernel");
    NNV_CUDA(launch_pdl_attrs(stream_carveout(STREAM_LONE, grid, dim3(DC_THREADS)), g.splits, direct_conv_kernel<TAPS>, grid, dim3(DC_THREADS), smem, st, g));
    return NNV_OK;
}

}  // namespace

nnv_status_t launch_direct(const float* x, const float* w, const float* bias, const float* add, float* y, int act,
                           int C, int H, int W, int K, int R, int S, int stride, int pad, int OH, int OW,
                           cudaStream_t st) {
    DirectDev g{x, w, bias, add, y, act, C, H, W, K, R, S, stride, pad, OH, OW, 1, nullptr};
    const bool al16 = ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(w) | reinterpret_cast<uintptr_t>(y)) & 15) == 0;
    const int taps = (C % 4) == 0 && al16 ? ((R == 3 && S == 3) ? 9 : (R == 1 && S == 1) ? 1 : 0) : 0;
    const int jc = taps == 9 ? 288 : 64, chunks = ceil_div(C * R * S, jc);
    int tile = 0;
    if (taps != 0 && pick_tile(OH * OW, C, K, taps, &tile, &g.splits)) {
        if (g.splits > 1) NNV_TRY(status_word(&g.status));
        if (taps == 9) return tile == 32 ? launch_dt<9, 32>(g, st) : launch_dt<9, 64>(g, st);
        return tile == 32 ? launch_dt<1, 32>(g, st) : launch_dt<1, 64>(g, st);
    }
    g.splits = pick_split(OH * OW, C, K, jc, chunks, taps).splits;
    return taps == 9 ? launch_dc<9>(g, st) : taps == 1 ? launch_dc<1>(g, st) : launch_dc<0>(g, st);
}

}  // namespace nnv

// Which kernel runs a direct layer of P pixels on channels in fours (9 or 1 taps), for the tests: the tile of direct_tile_kernel (0: the other one), the split.
extern "C" void nnv_internal_direct_rule(int P, int C, int K, int taps, int32_t* out) {
    using namespace nnv;
    const int jc = taps == 9 ? 288 : 64;
    int tile = 0, splits = 0;
    if (!pick_tile(P, C, K, taps, &tile, &splits)) {
        tile = 0;
        splits = pick_split(P, C, K, jc, ceil_div(C * taps, jc), taps).splits;
    }
    out[0] = tile;
    out[1] = splits;
}
