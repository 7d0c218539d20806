// A whole Winograd layer F(4x4,3x3) or F(6x6,3x3) on a small image from its raw weights, as one launch: both data transforms, the filter
// transform and the tile GEMM, in fp32.  For passes that transform their weights anew: neither U (36 or 64 words for nine of a filter) nor V
// nor M exists in memory.
//
// Bound: on few tiles the bytes of U, 38 MB for 512 -> 512 F(4,3), which the transform kernel writes and the tile GEMM reads back; here 9.4 MB of raw
// weights are read once, under the previous kernel's tail, and instruction issue sets the pace: ~90 instructions a filter and T (M + 2)^2
// products with a shared-memory read for every four.
//   - A block owns 32 output channels, T tiles and a slice of the input channels, an eighth or two of the quads of every 32; a cluster's blocks the
//     slices of the same outputs.
//   - A lane owns an output channel.  It transforms a filter in registers, a column of U at a time, and multiplies it with V's words of that
//     input channel, which are the same for the whole warp: a broadcast read feeds four products a lane, and nothing is
//     reduced across lanes.  The eight warps are two halves of U's columns x four shares of the slice's channels.
//   - The shares' sums are added through shared memory, the slices' by bulk pushes: each block gets an equal part of the (tile, channel) pairs,
//     whole, adds the slices and applies the output transform and the epilogue.
//   - Every transform and sum is in the order of the kernels for transformed weights (wino_tables.cuh, wino_small.cu): the bits are theirs.
// 512 -> 512 F(4,3) @7 between layers alike: 13.3 us against 23.4.  A block of 512 -> 512 @4 takes 5.6 us alone on an SM: input transform 1.1, products 2.4, the
// shares' sums 0.6, the exchange 0.8, output transform 0.7; two on an SM 8.4.
#include <algorithm>
#include <type_traits>

#include "nnv_internal.h"
#include "wino_tables.cuh"

namespace nnv {
namespace {

constexpr int WL_THREADS = 256, WL_K = 32, WL_SHARES = 4;

struct WlDev {
    const float* x; const float* w; const float* bias; const float* add; float* y;
    int C, H, W, K, pad, OH, OW, TW, tiles, act, slices, quads;       // quads: a block's groups of four input channels
    int early;                                                        // the weights do not depend on the kernel before
    int* status;
};

// Words of a row of raw weights: an odd multiple of four, so that 16-byte reads of 32 rows have no conflicts.
__host__ __device__ constexpr int wl_raw_pitch(int quads) { return 36 * quads + (quads & 1 ? 8 : 4); }

template <int M, int T>
struct WlShape {
    static constexpr int A = M + 2, A2 = A * A, N = A / 2;     // N: columns of U of a half
    static constexpr int VP = A2 * T + 4;                      // words of a channel of V: an odd multiple of four, so that the transform's stores spread over the banks
    static constexpr int SP = 2 * A2 + 1;                      // words of a (tile, channel) pair's sums, of each half of the input channels
    static constexpr uint32_t SUMS = (uint32_t)(WL_K * T * SP) * 4u;
    static constexpr uint32_t PARK = (uint32_t)(WL_SHARES * A2 * T * WL_K) * 4u;   // parked sums, later those received; behind them the added ones: all
    static size_t bytes(int quads) {                                               // where the weights and V were
        return std::max(((size_t)WL_K * wl_raw_pitch(quads) + (size_t)(4 * quads) * VP) * 4, (size_t)PARK + SUMS);
    }
};
// Columns of U: a half has both of each pair of points +-p, which share their even part.
template <int M> __host__ __device__ constexpr int wl_column(int half, int n) { return M == 4 ? half * 3 + n : half ? 3 + n : n < 3 ? n : 7; }

// One input channel: the filter w[0..8] of this lane's output channel, its half of U times V's words at `v`.
template <int M, int T, int HALF>
__device__ __forceinline__ void wl_channel(const float* w, const float* v, float (&acc)[M / 2 + 1][(M + 2) * T]) {
    constexpr int A = M + 2, N = A / 2;
#pragma unroll
    for (int n = 0; n < N; ++n) {
        constexpr int Q = A * T / 4;
        const int nu = wl_column<M>(HALF, n);
        float t[3], u[A];
#pragma unroll
        for (int r = 0; r < 3; ++r) t[r] = wino_filter<M>(nu, w[3 * r], w[3 * r + 1], w[3 * r + 2]);
#pragma unroll
        for (int xi = 0; xi < A; ++xi) u[xi] = wino_filter<M>(xi, t[0], t[1], t[2]);
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const float4 y = *reinterpret_cast<const float4*>(v + nu * A * T + 4 * q);
            acc[n][4 * q] = fmaf(u[(4 * q) / T], y.x, acc[n][4 * q]);
            acc[n][4 * q + 1] = fmaf(u[(4 * q + 1) / T], y.y, acc[n][4 * q + 1]);
            acc[n][4 * q + 2] = fmaf(u[(4 * q + 2) / T], y.z, acc[n][4 * q + 2]);
            acc[n][4 * q + 3] = fmaf(u[(4 * q + 3) / T], y.w, acc[n][4 * q + 3]);
        }
    }
}

template <int M, int T>
__global__ void __launch_bounds__(WL_THREADS, 2)
wino_layer_kernel(const WlDev g) {
    using S = WlShape<M, T>;
    using B = WinoBA<M>;
    constexpr int A = S::A, A2 = S::A2, N = S::N;
    extern __shared__ __align__(16) float sm[];
    __shared__ __align__(8) unsigned long long bar;            // received sums
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(sm), recv_bar = (uint32_t)__cvta_generic_to_shared(&bar);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int k0 = blockIdx.x * WL_K, t0 = blockIdx.y * T, sp = blockIdx.z;
    // Quad q of the slice: channels 4 (8 (q / per) + sp + 4 (q % per)) ...
    const int rp = wl_raw_pitch(g.quads), per = 8 / g.slices, groups = g.slices / 2, blocks = g.quads / per;
    auto channel = [&](int q) { return g.slices == 8 ? 4 * (8 * q + sp) : 4 * (8 * (q >> 1) + sp + 4 * (q & 1)); };
    float* const V = sm + WL_K * rp;
    const int pairs = WL_K * T / g.slices, p0 = sp * pairs;    // this block's (tile, channel) pairs of the write-out
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(recv_bar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(recv_bar), "r"((uint32_t)(g.slices * pairs * S::SP) * 4u) : "memory");
    }
    auto load_weights = [&]() {                                // four rows a warp
        for (int r = warp * 4; r < warp * 4 + 4; ++r) {
            if (k0 + r >= g.K) break;
            const float* const row = g.w + (long long)(k0 + r) * g.C * 9;
            for (int i = lane; i < g.quads * 9; i += 32) {
                const int q = i / 9, c = channel(q);
                if (c < g.C)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(base + (uint32_t)(r * rp + 4 * i) * 4u), "l"(row + c * 9 + 4 * (i - 9 * q)) : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (g.early) load_weights();
    pdl_wait();
    pdl_trigger();
    if (!g.early) load_weights();

    // V of the slice's channels: two threads per tile and channel, half of the rows each.
    {
        constexpr int CL = 32 / T;
        const int nc = 4 * g.quads, items = (nc + CL - 1) / CL * 2;
        for (int i = warp; i < items; i += WL_THREADS / 32) {
            const int t = lane % T, c = (i >> 1) * CL + lane / T, ch = channel(c >> 2) + (c & 3);
            if (c >= nc || ch >= g.C) continue;
            const int tile = t0 + t, th = tile / g.TW, h0 = th * M - g.pad, w0 = (tile - th * g.TW) * M - g.pad;
            const uint32_t pixel = (uint32_t)g.C * 4u, at = (uint32_t)((h0 * g.W + w0) * g.C + ch) * 4u;
            float d[A][A];
#pragma unroll
            for (int r = 0; r < A; ++r)
#pragma unroll
                for (int s = 0; s < A; ++s) {
                    const bool in = tile < g.tiles && (uint32_t)(h0 + r) < (uint32_t)g.H && (uint32_t)(w0 + s) < (uint32_t)g.W;
                    const uint32_t off = at + (uint32_t)(r * g.W + s) * pixel;
                    d[r][s] = in ? __ldg(reinterpret_cast<const float*>(reinterpret_cast<const char*>(g.x) + off)) : 0.f;
                }
            auto rows = [&](auto first) {
                constexpr int R0 = decltype(first)::value;
                float e[A / 2][A];                             // of B^T d
#pragma unroll
                for (int s = 0; s < A; ++s) {
                    float col[A], v[A];
#pragma unroll
                    for (int r = 0; r < A; ++r) col[r] = d[r][s];
                    wino_input(col, v);
#pragma unroll
                    for (int r = 0; r < A / 2; ++r) e[r][s] = v[R0 + r];
                }
#pragma unroll
                for (int r = 0; r < A / 2; ++r) {
                    float v[A];
                    wino_input(e[r], v);                       // (B^T d) B
#pragma unroll
                    for (int j = 0; j < A; ++j) V[c * S::VP + (j * A + R0 + r) * T + t] = v[j];
                }
            };
            if (i & 1) rows(std::integral_constant<int, A / 2>());
            else rows(std::integral_constant<int, 0>());
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();

    // Products.
    const int half = warp & 1, share = warp >> 1, group = g.slices == 8 ? share : share >> 1;     // a share: a quarter of the blocks of 32, or one of the two quads of half of them
    float acc[N][A * T];
#pragma unroll
    for (int n = 0; n < N; ++n)
#pragma unroll
        for (int i = 0; i < A * T; ++i) acc[n][i] = 0.f;
    auto multiply = [&](auto h) {
#pragma unroll 1
        for (int i = blocks * group / groups; i < blocks * (group + 1) / groups; ++i) {
            const int q = g.slices == 8 ? i : 2 * i + (share & 1);
            if (channel(q) >= g.C) break;
            float w[36];
            const float *const src = sm + lane * rp + q * 36, *const v = V + 4 * q * S::VP;
#pragma unroll
            for (int e = 0; e < 9; ++e) {
                const float4 f = *reinterpret_cast<const float4*>(src + 4 * e);
                w[4 * e] = f.x; w[4 * e + 1] = f.y; w[4 * e + 2] = f.z; w[4 * e + 3] = f.w;
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) wl_channel<M, T, decltype(h)::value>(w + 9 * c, v + c * S::VP, acc);
        }
    };
    if (half) multiply(std::integral_constant<int, 1>());
    else multiply(std::integral_constant<int, 0>());
    __syncthreads();                                           // weights and V are read no more

    // The shares' sums: parked, added in order, laid out by (tile, channel).
    auto park = [&](auto h) {
        float* const dst = sm + share * (A2 * T * WL_K) + lane;
#pragma unroll
        for (int n = 0; n < N; ++n)
#pragma unroll
            for (int i = 0; i < A * T; ++i) dst[(wl_column<M>(decltype(h)::value, n) * A * T + i) * WL_K] = acc[n][i];
    };
    if (half) park(std::integral_constant<int, 1>());
    else park(std::integral_constant<int, 0>());
    __syncthreads();
    float* const sums = sm + S::PARK / 4;
#pragma unroll 4
    for (int i = warp; i < A2 * T; i += WL_THREADS / 32) {
        const float* const p = sm + i * WL_K + lane;
        float* const to = sums + ((i % T) * WL_K + lane) * S::SP + i / T;
        to[0] = p[0] + p[A2 * T * WL_K];
        to[A2] = p[2 * (A2 * T * WL_K)] + p[3 * (A2 * T * WL_K)];
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");               // generic writes -> visible to the bulk copies
    __syncthreads();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");      // the parked sums' place is free for received ones

    // What the write-out reads from memory, under the exchange: a thread has a row of an output tile.
    auto place = [&](int idx, int* oh, int* ow, int* k) {
        const int pr = p0 + idx % pairs, tile = t0 + pr / WL_K, th = tile / g.TW;
        *k = k0 + pr % WL_K;
        *oh = th * M + idx / pairs; *ow = (tile - th * g.TW) * M;
        return tile < g.tiles && *k < g.K && *oh < g.OH;
    };
    auto epilogue_reads = [&](int idx, float (&a)[M], float& b) {
        int oh, ow, k;
        const bool live = idx < pairs * M && place(idx, &oh, &ow, &k);
        b = live && g.bias ? __ldg(g.bias + k) : 0.f;
#pragma unroll
        for (int j = 0; j < M; ++j) a[j] = live && g.add && ow + j < g.OW ? __ldg(g.add + ((long long)oh * g.OW + ow + j) * g.K + k) : 0.f;
    };
    float av[M], bv;
    epilogue_reads(tid, av, bv);
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (tid < g.slices) {
        const uint32_t bytes = (uint32_t)(pairs * S::SP) * 4u;
        uint32_t dst, there;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"(base + (uint32_t)sp * bytes), "r"(tid));
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(there) : "r"(recv_bar), "r"(tid));
        asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(dst), "r"(base + S::PARK + (uint32_t)tid * bytes), "r"(bytes), "r"(there) : "memory");
    }
    __syncwarp();
    bool ok = false;
    for (uint32_t i = 0; !ok && i < (1u << 20); ++i) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(done) : "r"(recv_bar) : "memory");
        ok = done != 0;
    }
    if (!ok && tid == 0) atomicExch(g.status, (int)NNV_ERR_TIMEOUT);
    __syncwarp();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");      // this block's sums have arrived: their senders may leave
    const float* const recv = sm;
    // Output transform, columns, then rows with the epilogue.
    float* const tmp = sm + S::SUMS / 4;                       // [M][A][pairs], behind the received sums
    for (int idx = tid; ok && idx < pairs * A; idx += WL_THREADS) {
        const int pr = idx % pairs, nu = idx / pairs;
        float m[A];
#pragma unroll
        for (int l = 0; l < A; ++l) {
            float y[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float* const r = recv + pr * S::SP + h * A2 + nu * A + l;
                const int step = pairs * S::SP;
                y[h] = g.slices == 8 ? ((r[0] + r[4 * step]) + (r[2 * step] + r[6 * step])) + ((r[step] + r[5 * step]) + (r[3 * step] + r[7 * step]))
                                     : (r[0] + r[2 * step]) + (r[step] + r[3 * step]);
            }
            m[l] = y[0] + y[1];
        }
#pragma unroll
        for (int i = 0; i < M; ++i) {
            float s = 0.f;
#pragma unroll
            for (int l = 0; l < A; ++l)
                if (B::at(i, l) != 0.f) s += B::at(i, l) * m[l];
            tmp[(i * A + nu) * pairs + pr] = s;
        }
    }
    __syncthreads();
    for (int idx = tid; ok && idx < pairs * M; idx += WL_THREADS) {
        int oh, ow, k;
        if (idx != tid) epilogue_reads(idx, av, bv);
        if (!place(idx, &oh, &ow, &k)) continue;
        const int pr = idx % pairs, i = idx / pairs;
        float m[A];
#pragma unroll
        for (int l = 0; l < A; ++l) m[l] = tmp[(i * A + l) * pairs + pr];
        float* const out = g.y + ((long long)oh * g.OW + ow) * g.K + k;
#pragma unroll
        for (int j = 0; j < M; ++j) {
            float s = 0.f;
#pragma unroll
            for (int l = 0; l < A; ++l)
                if (B::at(j, l) != 0.f) s += m[l] * B::at(j, l);
            if (ow + j >= g.OW) continue;
            s += bv;
            if (g.add) s += av[j];
            if (g.act) s = fmaxf(s, 0.f);
            if (g.act == 2) s = fminf(s, 6.f);
            out[(long long)j * g.K] = s;
        }
    }
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Estimated us of a layer inside a pass: here, and as the filter transform on its own stream with the three kernels for transformed weights.  Here: a base,
// the slice's quads one after the other, dearer as blocks begin to share an SM (clusters of four and eight: from about 56 blocks on, all of
// them from 80) and fill the wave; F(6,3) pays for a second tile a block.  There: the bytes of U beyond the ~6 MB that the transform's own
// launches hide, channels and outputs.  Fitted to 1483 layers of 16 - 1024 channels on 1 - 12 tiles in rows of eight (5 - 8 % off).
double wl_us(int m, int T, int slices, int quads, long long blocks) {
    const double q = std::max(quads, 4), shared = std::min(1.0, std::max(0.0, (blocks - 56) / 24.0)), full = std::max(0.0, (blocks - 80) / 184.0);
    return (m == 6 ? 3.5 : 2.7) + (slices == 8 ? 0.45 : 0.0) + 0.194 * q * (1 + shared) + full * (1.7 + 0.08 * q) + (m == 6 && T == 2 ? 3.3 : 0.0);
}
double wl_separate_us(int m, int C, int K, int tiles) {
    const double mb = 4e-6 * (m + 2) * (m + 2) * C * K, hidden = m == 6 ? 6.0 : 5.0;
    return (m == 6 ? 3.86 : 3.35) + 0.005 * C + (m == 6 ? 0.0058 : 0.0035) * K + 0.6 * std::min(10.0, std::max(0.0, mb - hidden)) +
           0.37 * std::max(0.0, mb - 16) + 0.11 * std::max(0, tiles - 8) + (m == 6 ? 0.0005 : 0.0008) * tiles * C;
}

// Tiles a block, slices and whether the layer is to run here: where it fits one wave at two blocks an SM (more pays the filter transform too often:
// F(4,3) 512 -> 512 @14 23.7 us without, 38 with, 384 -> 384 @14 15.3 / 25), wino_small.cu runs the tile GEMM for transformed weights, whose sums it
// follows, and the estimate is lower.  Two tiles a block (four: as fast alone, but then only eight SMs of a wave have a second block, which sets the time:
// 512 -> 512 @7 13.4 us against 12.5), F(6,3) one where that fits the wave.
// us a layer in a row of such layers, separate / here: F(4,3) 64 -> 64 @8 4.2 / 3.6, 128 -> 128 4.8 / 4.3, 256 -> 256 8.6 / 6.1, 512 -> 512 23.0 / 12.9, @4
// 20.8 / 8.8, F(6,3) 64 -> 64 @12 4.8 / 4.4, 384 -> 384 23.7 / 16.1, 192 -> 192 @6 7.8 / 6.0, 256 -> 256 12.9 / 6.8.  What the estimate leaves to the separate
// kernels: F(6,3) 16 -> 192 @12x24 4.9 / 6.4, 64 -> 128 @18 5.5 / 6.4, 192 -> 32 @12 5.1 / 6.0, F(4,3) 192 -> 192 @8x16 6.5 / 7.5, 256 -> 160 @8x16 7.1 / 8.6.
// Of the 1483 layers 203 would be more than 3 % slower here without it, 12 - 17 are with it.  Cold passes, where the link hides the filter transform, gain less:
// a ResNet-18-shaped model @224 with F(4,3) 902 / 892 us, staged three deep 991 / 979.
struct WlPlan { bool fits, use; int T, slices, quads; };
WlPlan wl_plan(int m, int C, int K, int tiles) {
    constexpr long long WAVE = 264;                            // clusters of eight, two blocks an SM
    WlPlan p{false, false, m == 4 ? 2 : 1, 4, 0};
    if (C % 4 != 0 || C > 512 || (m == 6 && (tiles == 1 ? C < 128 : tiles > 4 && C > 64)) || !wino_small_applies(m, tiles, align_up(C, 8), K)) return p;
    if (C > 256) {
        if (tiles > 4) return p;                               // (the GEMM for transformed weights would need more registers to follow)
        p.slices = 8;
    }
    auto blocks = [&]() { return (long long)ceil_div(K, WL_K) * ceil_div(tiles, p.T) * p.slices; };
    if (m == 6 && tiles <= 4 && blocks() > WAVE) p.T = 2;
    p.fits = blocks() <= WAVE;
    p.quads = ceil_div(C, 32) * 8 / p.slices;
    p.use = p.fits && wl_us(m, p.T, p.slices, p.quads, blocks()) < 0.98 * wl_separate_us(m, C, K, tiles);
    return p;
}

template <int M, int T>
nnv_status_t launch_wl(WlDev g, cudaStream_t st) {
    using S = WlShape<M, T>;
    const size_t smem = S::bytes(g.quads);
    static const cudaError_t attr = cudaFuncSetAttribute(wino_layer_kernel<M, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::bytes(16));
    NNV_CUDA(attr);
    NNV_CUDA(launch_pdl_cluster(wino_layer_kernel<M, T>, dim3(ceil_div(g.K, WL_K), ceil_div(g.tiles, T), g.slices), dim3(WL_THREADS), smem, st, g.slices, g));
    return NNV_OK;
}

}  // namespace

bool wino_layer_applies(int m, int C, int K, int tiles) { return wl_plan(m, C, K, tiles).use; }
int wino_layer_parts(int m, int C, int K, int tiles) {
    const WlPlan p = wl_plan(m, C, K, tiles);
    return !p.fits ? 0 : p.slices == 8 ? 4 : 2;
}

nnv_status_t launch_wino_layer(int m, const float* x, const float* w, const float* bias, const float* add, float* y, int act, int C, int H, int W,
                               int K, int pad, int OH, int OW, bool early, cudaStream_t st) {
    const int TW = ceil_div(OW, m), tiles = ceil_div(OH, m) * TW;
    const WlPlan p = wl_plan(m, C, K, tiles);
    NNV_REQUIRE(p.fits, NNV_ERR_UNSUPPORTED, "no one-launch Winograd layer for this shape");
    const int* status = nullptr;
    NNV_TRY(device_status_address(&status));
    WlDev g{x, w, bias, add, y, C, H, W, K, pad, OH, OW, TW, tiles, act, p.slices, p.quads, early ? 1 : 0, const_cast<int*>(status)};
    return m == 4 ? launch_wl<4, 2>(g, st) : p.T == 1 ? launch_wl<6, 1>(g, st) : launch_wl<6, 2>(g, st);
}

}  // namespace nnv

// Which kernels run an F(m,3) layer of `tiles` tiles, for the tests: the fp32 tile GEMM, a whole layer in one launch, that launch's tiles a block, slices
// and quads of input channels, and the tile GEMM's groups of output channels.
extern "C" void nnv_internal_wino_rule(int m, int C, int K, int tiles, int32_t* out) {
    const nnv::WlPlan p = nnv::wl_plan(m, C, K, tiles);
    const int32_t v[] = {nnv::wino_small_applies(m, tiles, (int)nnv::align_up(C, 8), K), p.use, p.T, p.slices, p.quads, nnv::wino_small_groups(m, C, K, tiles)};
    std::copy(std::begin(v), std::end(v), out);
}
