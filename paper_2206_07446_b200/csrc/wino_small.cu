// The Winograd tile GEMM of F(4x4,3x3) and F(6x6,3x3) on images of a few tiles, on the FP32 pipes:  M[b][t][k] = sum_c V[b][t][c] U[b][k][c].
//
// Bound: the bytes of U (36 or 64 times the channel pairs: 38 MB for 512 -> 512), each word of which meets T <= 12 words of V.  The tensor-core GEMM
// fills 128 rows whatever T is and splits every word of U into bf16 parts on its way through shared memory; here a word goes from memory
// into a register and is multiplied T times, in fp32.
//   - A block owns 64 output channels of one plane b; V's plane lies in shared memory.  Eight warps: four groups of 16 channels x two halves of the
//     input channels, or, where that leaves SMs idle and lone warps with long sums, two groups x quarters or one x eighths (below).  Eight lanes read 128 contiguous bytes of a channel's row, a warp four rows at a time, sixteen in all, so that a word of V
//     read from shared memory serves four rows of a lane.
//   - The lanes' sums are reduced by exchanging halves (3.5 T shuffles), the halves of the input channels through shared memory; the order is fixed,
//     and wino_layer.cu's is the same where it may run the layer: that has the same bits whether its weights come transformed or raw.  (Where that
//     kernel deals the channels to eight blocks, a half is summed as two quarters.)
// 512 -> 512 F(4,3) @7 in a model, U in the L2: 7.4 us against 11.3 on the tensor cores.
#include <algorithm>
#include <type_traits>

#include "nnv_internal.h"

namespace nnv {
namespace {

constexpr int WS_THREADS = 256;

// T: tiles, rounded up (tiles that do not exist have zeros in shared memory); UN: 32-channel blocks in flight; GROUPS: warps side by side, 16 output channels
// each, the others share out the input channels.
template <int T, int UN, int GROUPS>
__global__ void __launch_bounds__(WS_THREADS, 2)
wino_small_kernel(const float* __restrict__ V, const float* __restrict__ U, float* __restrict__ M, int tiles, int K, int Cp,
                  int quarters, unsigned long long* stamp) {
    constexpr int WS_K = 16 * GROUPS, PARTS = 8 / GROUPS;
    extern __shared__ __align__(16) float sv[];                // V's plane [T][pitch], later the partial sums [PARTS][WS_K][T + 1]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int cl = lane & 7, rl = lane >> 3, rg = warp % GROUPS, part = warp / GROUPS;
    const int b = blockIdx.y, k0 = blockIdx.x * WS_K;
    const int pitch = ((Cp + 31) & ~31) + 4;                   // (eight lanes read 128 bytes of a row: any pitch will do)
    const int blocks = (Cp + 31) / 32, i0 = blocks * part / PARTS, i1 = blocks * (part + 1) / PARTS;
    const int middle = T <= 4 && PARTS == 2 && quarters ? blocks * (2 * part + 1) / 4 : -1;    // where a sum of its own begins
    const float* const u = U + ((long long)b * K + k0 + rg * 16 + rl) * Cp + 4 * cl;
    const int rows = K - k0 - rg * 16 - rl;                    // rows 4 r of this lane that exist: 4 r < rows
    float acc[4][T];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int t = 0; t < T; ++t) acc[r][t] = 0.f;
    float first[4][T <= 4 ? T : 1];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int t = 0; t < (T <= 4 ? T : 1); ++t) first[r][t] = 0.f;
    float4 w[UN][4];
    auto fetch = [&](int i, float4 (&f)[4]) {
        const bool in = i < i1 && 32 * i + 4 * cl < Cp;
#pragma unroll
        for (int r = 0; r < 4; ++r)
            f[r] = in && 4 * r < rows ? __ldg(reinterpret_cast<const float4*>(u + (long long)(4 * r) * Cp + 32 * i)) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    pdl_enter();
    if (tid == 32) stamp_start(stamp);
#pragma unroll
    for (int n = 0; n < UN; ++n) fetch(i0 + n, w[n]);
    const float* const v = V + (long long)b * tiles * Cp;
    const int words = pitch / 4;
    for (int i = tid; i < T * words; i += WS_THREADS) {
        const int t = i / words, c = (i - t * words) * 4;
        *reinterpret_cast<float4*>(sv + t * pitch + c) = t < tiles && c < Cp ? __ldg(reinterpret_cast<const float4*>(v + (long long)t * Cp + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
#pragma unroll 1
    for (int i = i0; i < i1; i += UN) {
#pragma unroll
        for (int n = 0; n < UN; ++n) {
            float4 x[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) x[r] = w[n][r];
            fetch(i + UN + n, w[n]);
            // (a block beyond the half multiplies zeros with whatever V holds there: with V's own numbers, which may be infinite)
            if constexpr (T <= 4) {
                if (i + n == middle) {
#pragma unroll
                    for (int r = 0; r < 4; ++r)
#pragma unroll
                        for (int t = 0; t < T; ++t) { first[r][t] = acc[r][t]; acc[r][t] = 0.f; }
                }
            }
            if (i + n < i1) {
                const float* row = sv + 32 * (i + n) + 4 * cl;
#pragma unroll
                for (int t = 0; t < T; ++t) {
                    const float4 y = *reinterpret_cast<const float4*>(row + t * pitch);
#pragma unroll
                    for (int r = 0; r < 4; ++r) acc[r][t] = fmaf(x[r].w, y.w, fmaf(x[r].z, y.z, fmaf(x[r].y, y.y, fmaf(x[r].x, y.x, acc[r][t]))));
                }
            }
        }
    }
    if constexpr (T <= 4) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int t = 0; t < T; ++t) acc[r][t] = first[r][t] + acc[r][t];
    }
    // Eight lanes' sums: each exchange halves what a lane holds.  It ends up with row 2 (cl >> 2) + (cl >> 1 & 1) and half of the tiles.
    auto trade = [&](float keep_low, float keep_high, int bit) {
        const bool high = cl & bit;
        return (high ? keep_high : keep_low) + __shfl_xor_sync(0xffffffffu, high ? keep_low : keep_high, bit);
    };
    float s2[2][T], s1[T], s[T / 2];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int t = 0; t < T; ++t) s2[r][t] = trade(acc[r][t], acc[r + 2][t], 4);
#pragma unroll
    for (int t = 0; t < T; ++t) s1[t] = trade(s2[0][t], s2[1][t], 2);
#pragma unroll
    for (int t = 0; t < T / 2; ++t) s[t] = trade(s1[t], s1[t + T / 2], 1);
    __syncthreads();                                           // V is read no more
    {
        const int row = rg * 16 + rl + 4 * (2 * (cl >> 2) + (cl >> 1 & 1));
        float* dst = sv + (part * WS_K + row) * (T + 1) + (cl & 1) * (T / 2);
#pragma unroll
        for (int t = 0; t < T / 2; ++t) dst[t] = s[t];
    }
    __syncthreads();
    for (int i = tid; i < T * WS_K; i += WS_THREADS) {
        const int t = i / WS_K, k = i % WS_K;
        if (t >= tiles || k0 + k >= K) continue;
        float sum = sv[k * (T + 1) + t];
#pragma unroll
        for (int q = 1; q < PARTS; ++q) sum += sv[(q * WS_K + k) * (T + 1) + t];
        M[((long long)b * tiles + t) * K + k0 + k] = sum;
    }
    if (stamp) {
        __syncthreads();
        if (tid == 0) stamp_end(stamp);
    }
}

}  // namespace

// Where it is ahead of the tensor-core GEMM, weights from DRAM, whole layers in us, tensor cores / here: F(4,3) 256 -> 256 @3 8.5 / 6.3, @7 9.0 / 7.1,
// 512 -> 512 @7 16.4 / 15.3, F(6,3) 128 -> 128 @11 7.3 / 5.7, 256 -> 256 @11 11.7 / 9.5; with U of 67 MB (F(6,3) 512 -> 512 @11 21.9 / 23.0, F(4,3) 1024 -> 512
// @7 23.4 / 23.4) and beyond eight tiles (F(4,3) 128 -> 128 @11 6.8 / 6.7, 512 -> 512 @11 16.0 / 18.2) the other has caught up.
bool wino_small_applies(int m, int T, int Cp, int K) {
    const Tuning& tn = tuning();
    if (!tn.winosmall || tn.gemm_bn || tn.gemm_ring) return false;     // (overrides of the tensor cores' tile GEMM)
    const double bytes = 4.0 * (m + 2) * (m + 2) * K * Cp;
    return m != 2 && Cp <= 2048 && (T <= 8 ? bytes <= 40e6 : T <= 12 && bytes <= 5e6);
}

// Groups of 16 output channels a block: the fewest that leave at most two blocks an SM and no part of the input channels empty; four where wino_layer.cu
// sums the layer too.  us of a layer, tensor cores / four groups / as chosen: F(4,3) 960 -> 16 @12x16 10.6 / 16.1 / 10.4, 640 -> 48 @12 10.2 / 12.4 / 9.0, 1024 -> 256 @8x12
// 15.6 / 17.0 / 13.7, F(6,3) 448 -> 32 @18 9.6 / 13.2 / 8.8; over 563 layers of 16 - 1024 channels 0.904 of the time that four groups take everywhere (the best of
// the three forms 0.901), 7 of them more than 3 % behind the tensor cores (1024 outputs of up to 32 inputs on nine tiles or more).
int wino_small_groups(int m, int C, int K, int T) {
    if (wino_layer_parts(m, C, K, T)) return 4;
    for (int g = 1; g < 4; g *= 2)
        if (ceil_div(K, 16 * g) * (m + 2) * (m + 2) <= 2 * 148 && 8 / g <= ceil_div(C, 32)) return g;
    return 4;
}

nnv_status_t launch_wino_small(int m, const float* V, const float* U, float* M, int T, int K, int C, int Cp, cudaStream_t st) {
    unsigned long long* const stamp = next_stamp();
    next_stamp() = nullptr;
    const int quarters = wino_layer_parts(m, C, K, T) == 4;
    auto go = [&](auto tt, auto gg, auto kernel) -> cudaError_t {
        constexpr int TT = decltype(tt)::value, WS_K = 16 * decltype(gg)::value;
        const size_t smem = sizeof(float) * std::max((size_t)TT * (align_up(Cp, 32) + 4), (size_t)128 * (TT + 1));
        static const cudaError_t attr = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(sizeof(float) * TT * (2048 + 4)));
        if (attr != cudaSuccess) return attr;
        return launch_pdl(kernel, dim3(ceil_div(K, WS_K), (m + 2) * (m + 2)), dim3(WS_THREADS), smem, st, V, U, M, T, K, Cp, quarters, stamp);
    };
    auto pick = [&](auto gg) {
        constexpr int GG = decltype(gg)::value;
        const std::integral_constant<int, 4> t4;
        const std::integral_constant<int, 8> t8;
        const std::integral_constant<int, 12> t12;
        return T <= 4 ? go(t4, gg, wino_small_kernel<4, 3, GG>) : T <= 8 ? go(t8, gg, wino_small_kernel<8, 2, GG>) : go(t12, gg, wino_small_kernel<12, 2, GG>);
    };
    const int groups = wino_small_groups(m, C, K, T);
    NNV_CUDA(groups == 1 ? pick(std::integral_constant<int, 1>()) : groups == 2 ? pick(std::integral_constant<int, 2>()) : pick(std::integral_constant<int, 4>()));
    return NNV_OK;
}

}  // namespace nnv
