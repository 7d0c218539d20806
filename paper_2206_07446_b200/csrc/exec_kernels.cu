// Execution-side kernels that are not tensor-core contractions: im2col, the Winograd input and
// output transforms, fp32 direct and depthwise convolution, pooling and layout conversion.
// Activations are NHWC fp32 (batch 1).
#include <cuda_bf16.h>

#include <type_traits>

#include "nnv_internal.h"
#include "wino_tables.cuh"

namespace nnv {

__device__ __forceinline__ float apply_act(float v, int act) {
    if (act == 1) return fmaxf(v, 0.f);
    if (act == 2) return fminf(fmaxf(v, 0.f), 6.f);
    return v;
}

template <typename OutT> __device__ inline OutT to_out(float v);
template <> __device__ inline float to_out<float>(float v) { return v; }
template <> __device__ inline __nv_bfloat16 to_out<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// ---- im2col ---------------------------------------------------------------------------------
// Xcol[p][q], q = (r*S+s)*C + c; zero outside the image and for q >= R*S*C.
template <typename OutT>
__global__ void __launch_bounds__(256)
im2col_kernel(const float* __restrict__ x, OutT* __restrict__ col, int C, int H, int W, int R, int S, int stride,
              int pad, int OH, int OW, int Qp) {
    pdl_enter();
    const long long n = (long long)OH * OW * Qp;
    const int Q = R * S * C;
    for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < n; i += (long long)gridDim.x * 256) {
        const int p = (int)(i / Qp), q = (int)(i - (long long)p * Qp);
        float v = 0.f;
        if (q < Q) {
            const int rs = q / C, c = q - rs * C;
            const int r = rs / S, s = rs - r * S;
            const int oh = p / OW, ow = p - oh * OW;
            const int ih = oh * stride + r - pad, iw = ow * stride + s - pad;
            if (ih >= 0 && ih < H && iw >= 0 && iw < W) v = __ldg(x + ((long long)ih * W + iw) * C + c);
        }
        col[i] = to_out<OutT>(sizeof(OutT) == 4 ? round_tf32(v) : v);
    }
}

// The same matrix for small reductions (R*S*C up to IM2COL_TABLE entries: network stems with C = 3).  The
// (r, s, c) of every column q is worked out once per block into a shared-memory table; a warp then writes one
// pixel's row at a time, lane = q, so the inner loop has no division and the stores are contiguous.
constexpr int IM2COL_TABLE = 1024;
template <typename OutT>
__global__ void __launch_bounds__(256)
im2col_table_kernel(const float* __restrict__ x, OutT* __restrict__ col, int C, int H, int W, int R, int S, int stride,
                    int pad, int OH, int OW, int Qp) {
    pdl_enter();
    __shared__ int tab[IM2COL_TABLE];                           // (r << 20) | (s << 10) | c, or -1 for the zero padding q >= Q
    const int Q = R * S * C;
    for (int q = threadIdx.x; q < Qp; q += 256) {
        const int rs = q / C, c = q - rs * C;
        const int r = rs / S, sx = rs - r * S;
        tab[q] = q < Q ? ((r << 20) | (sx << 10) | c) : -1;
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int P = OH * OW;
    for (int p = blockIdx.x * 8 + warp; p < P; p += gridDim.x * 8) {
        const int oh = p / OW, ow = p - oh * OW;
        const int ih0 = oh * stride - pad, iw0 = ow * stride - pad;
        OutT* dst = col + (long long)p * Qp;
        for (int q = lane; q < Qp; q += 32) {
            const int e = tab[q];
            float v = 0.f;
            if (e >= 0) {
                const int ih = ih0 + (e >> 20), iw = iw0 + ((e >> 10) & 1023);
                if (ih >= 0 && ih < H && iw >= 0 && iw < W) v = __ldg(x + ((long long)ih * W + iw) * C + (e & 1023));
            }
            dst[q] = to_out<OutT>(sizeof(OutT) == 4 ? round_tf32(v) : v);
        }
    }
}

// Four consecutive q per thread; valid when C % 4 == 0 (a quad never straddles a filter tap).
template <typename OutT>
__global__ void __launch_bounds__(256)
im2col_vec4_kernel(const float* __restrict__ x, OutT* __restrict__ col, int C, int H, int W, int R, int S, int stride,
                   int pad, int OH, int OW, int Qp) {
    pdl_enter();
    const int Qv = Qp / 4;
    const long long n = (long long)OH * OW * Qv;
    const int Q = R * S * C;
    for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < n; i += (long long)gridDim.x * 256) {
        const int p = (int)(i / Qv), q = 4 * (int)(i - (long long)p * Qv);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (q < Q) {
            const int rs = q / C, c = q - rs * C;
            const int r = rs / S, s = rs - r * S;
            const int oh = p / OW, ow = p - oh * OW;
            const int ih = oh * stride + r - pad, iw = ow * stride + s - pad;
            if (ih >= 0 && ih < H && iw >= 0 && iw < W)
                v = __ldg(reinterpret_cast<const float4*>(x + ((long long)ih * W + iw) * C + c));
        }
        OutT* dst = col + (long long)p * Qp + q;
        if constexpr (sizeof(OutT) == 4) {
            *reinterpret_cast<float4*>(dst) = make_float4(round_tf32(v.x), round_tf32(v.y), round_tf32(v.z), round_tf32(v.w));
        } else {
            __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
            uint2 u;
            u.x = *reinterpret_cast<uint32_t*>(&a);
            u.y = *reinterpret_cast<uint32_t*>(&b);
            *reinterpret_cast<uint2*>(dst) = u;
        }
    }
}

nnv_status_t launch_im2col(bool bf16, const float* x, void* col, int C, int H, int W, int R, int S, int stride,
                           int pad, int OH, int OW, int Qp, cudaStream_t st) {
    const bool vec = (C % 4) == 0;
    const long long n = (long long)OH * OW * (vec ? Qp / 4 : Qp);
    const unsigned grid = (unsigned)std::min<long long>((n + 255) / 256, 148ll * 32);
    if (vec) {
        if (bf16) NNV_LAUNCH((im2col_vec4_kernel<__nv_bfloat16>), grid, 256, 0, st, x, (__nv_bfloat16*)col, C, H, W, R, S, stride, pad, OH, OW, Qp);
        else NNV_LAUNCH((im2col_vec4_kernel<float>), grid, 256, 0, st, x, (float*)col, C, H, W, R, S, stride, pad, OH, OW, Qp);
    } else if (Qp <= IM2COL_TABLE && C < 1024 && R < 1024 && S < 1024) {
        const unsigned g2 = (unsigned)std::min<long long>(((long long)OH * OW + 7) / 8, 148ll * 16);
        if (bf16) NNV_LAUNCH((im2col_table_kernel<__nv_bfloat16>), g2, 256, 0, st, x, (__nv_bfloat16*)col, C, H, W, R, S, stride, pad, OH, OW, Qp);
        else NNV_LAUNCH((im2col_table_kernel<float>), g2, 256, 0, st, x, (float*)col, C, H, W, R, S, stride, pad, OH, OW, Qp);
    } else {
        if (bf16) NNV_LAUNCH((im2col_kernel<__nv_bfloat16>), grid, 256, 0, st, x, (__nv_bfloat16*)col, C, H, W, R, S, stride, pad, OH, OW, Qp);
        else NNV_LAUNCH((im2col_kernel<float>), grid, 256, 0, st, x, (float*)col, C, H, W, R, S, stride, pad, OH, OW, Qp);
    }
    NNV_CUDA(cudaGetLastError());
    return NNV_OK;
}

// ---- Winograd data transforms ---------------------------------------------------------------
// Two forms of each data transform.  A thread per (tile, channel) loads A*A values, works through ~2 A*A*A multiply-adds and stores as
// many: on a layer of a few thousand of them (512 -> 512 @7, F(4,3): 16 blocks) a handful of warps do everything one after the other.
// So up to WT_BLOCKS blocks the work of a tile is dealt to A warps: a warp for every column of the tile and then, through shared memory,
// for every row of its transform, a lane a channel.  More blocks than that cost more than they spread.
// us a layer (three kernels, chained), a thread per tile and channel / a block per tile and 32 channels: F(4,3) 64 -> 64 @56 10.4 / 7.3,
// 128 -> 128 @28 9.9 / 7.6, 512 -> 512 @7 16.5 / 15.6, F(6,3) 128 -> 128 @28 15.0 / 8.0, 64 -> 128 @112 22.4 / 15.9; F(2,3) 64 -> 64 @200 38 / 59,
// F(4,3) 64 -> 64 @224 37.7 / 40.2.
template <int M_> struct WinoTileLimit { static constexpr long long BLOCKS = M_ == 4 ? 3000 : 2000; };
template <int M_> static bool wino_tile_blocks(int TH, int TW, int channels) {
    return (long long)TH * TW * ceil_div(channels, 32) <= WinoTileLimit<M_>::BLOCKS;
}

// What the transform writes.  V[(xi*A+nu)][t][cp]; SPLIT (Cp % 32 == 0): a block of 32 words holds its 32 elements as bf16 hi = rn(v), then
// lo = rn(v - hi), the operand of the compensated GEMM; neighbouring lanes swap halves, so that each stores one word.
template <bool SPLIT> __device__ __forceinline__ int wino_word(int c) { return SPLIT ? (c & ~31) + ((c & 1) << 4) + ((c & 31) >> 1) : c; }
template <int M_, typename OutT, bool SPLIT> __device__ __forceinline__ OutT wino_operand(float s, int c) {
    if constexpr (SPLIT) {
        const __nv_bfloat16 hi = __float2bfloat16_rn(s), lo = __float2bfloat16_rn(s - __bfloat162float(hi));
        const uint32_t own = (uint32_t)__bfloat16_as_ushort(hi) | (uint32_t)__bfloat16_as_ushort(lo) << 16;
        const uint32_t other = __shfl_xor_sync(0xffffffffu, own, 1);
        return __uint_as_float((c & 1) ? __byte_perm(other, own, 0x7632) : __byte_perm(own, other, 0x5410));
    } else {
        return to_out<OutT>((sizeof(OutT) == 4 && M_ == 2) ? round_tf32(s) : s);
    }
}

// One thread per (tile, padded channel); channel is the fastest index so that every load and
// store of a warp covers 32 consecutive channels: for layers with tiles enough to fill the GPU that way.
template <int M_, typename OutT, bool SPLIT>
__global__ void __launch_bounds__(128)
wino_input_kernel(const float* __restrict__ x, OutT* __restrict__ V, int C, int Cp, int H, int W, int pad, int TH,
                  int TW) {
    pdl_enter();
    constexpr int A = WinoBA<M_>::A;
    const long long T = (long long)TH * TW;
    const long long idx = (long long)blockIdx.x * 128 + threadIdx.x;
    if (idx >= T * Cp) return;
    const int t = (int)(idx / Cp), c = (int)(idx - (long long)t * Cp);
    const int th = t / TW, tw = t - th * TW;
    const int h0 = th * M_ - pad, w0 = tw * M_ - pad;
    float d[A][A];
#pragma unroll
    for (int i = 0; i < A; ++i) {
        const int h = h0 + i;
#pragma unroll
        for (int j = 0; j < A; ++j) {
            const int w = w0 + j;
            d[i][j] = (c < C && h >= 0 && h < H && w >= 0 && w < W) ? __ldg(x + ((long long)h * W + w) * C + c) : 0.f;
        }
    }
#pragma unroll
    for (int j = 0; j < A; ++j) {                                // B^T d
        float col[A], v[A];
#pragma unroll
        for (int i = 0; i < A; ++i) col[i] = d[i][j];
        wino_input(col, v);
#pragma unroll
        for (int i = 0; i < A; ++i) d[i][j] = v[i];
    }
    OutT* out = V + (long long)t * Cp + wino_word<SPLIT>(c);
#pragma unroll
    for (int i = 0; i < A; ++i) {                                // (B^T d) B
        float v[A];
        wino_input(d[i], v);
#pragma unroll
        for (int j = 0; j < A; ++j) out[(long long)(i * A + j) * T * Cp] = wino_operand<M_, OutT, SPLIT>(v[j], c);
    }
}

// A block takes one tile and 32 channels.
template <int M_, typename OutT, bool SPLIT>
__global__ void __launch_bounds__(32 * WinoBA<M_>::A)
wino_input_tile_kernel(const float* __restrict__ x, OutT* __restrict__ V, int C, int Cp, int H, int W, int pad, int TH,
                  int TW) {
    constexpr int A = WinoBA<M_>::A;
    __shared__ float tmp[A][A][32];                              // B^T d
    const int lane = threadIdx.x & 31, col = threadIdx.x >> 5;
    const int t = blockIdx.x, c = blockIdx.y * 32 + lane;
    const int th = t / TW, tw = t - th * TW;
    const int h0 = th * M_ - pad, w = tw * M_ - pad + col;
    const bool inside = c < C && w >= 0 && w < W;
    const float* src = x + ((long long)h0 * W + w) * C + c;
    const long long plane = (long long)TH * TW * Cp;
    OutT* out = V + (long long)(col * A) * plane + (long long)t * Cp + wino_word<SPLIT>(c);
    pdl_enter();
    float d[A];
#pragma unroll
    for (int l = 0; l < A; ++l) d[l] = inside && h0 + l >= 0 && h0 + l < H ? __ldg(src + (long long)l * W * C) : 0.f;
    float s[A];
    wino_input(d, s);
#pragma unroll
    for (int i = 0; i < A; ++i) tmp[i][col][lane] = s[i];
    __syncthreads();
#pragma unroll
    for (int l = 0; l < A; ++l) d[l] = tmp[col][l][lane];        // the warp's row
    wino_input(d, s);                                            // V = tmp B
#pragma unroll
    for (int j = 0; j < A; ++j) {
        const OutT v = wino_operand<M_, OutT, SPLIT>(s[j], c);   // (a shuffle: by all lanes)
        if (c < Cp) out[j * plane] = v;
    }
}

nnv_status_t launch_wino_input(int m, bool bf16, bool split, const float* x, void* V, int C, int Cp, int H, int W, int pad,
                               int TH, int TW, cudaStream_t st) {
    const long long n = (long long)TH * TW * Cp;
    auto go = [&](auto mm, auto zero, auto pre) {
        constexpr int M_ = decltype(mm)::value;
        using OutT = decltype(zero);
        constexpr bool S = decltype(pre)::value;
        if (wino_tile_blocks<M_>(TH, TW, Cp))
            return launch_pdl(wino_input_tile_kernel<M_, OutT, S>, dim3(TH * TW, ceil_div(Cp, 32)), dim3(32 * (M_ + 2)), 0, st, x, (OutT*)V, C, Cp, H, W, pad, TH, TW);
        return launch_stream(STREAM_RESIDENT, wino_input_kernel<M_, OutT, S>, dim3((unsigned)((n + 127) / 128)), dim3(128), 0, st, x, (OutT*)V, C, Cp, H, W, pad, TH, TW);
    };
    const std::integral_constant<int, 2> m2;
    const std::integral_constant<int, 4> m4;
    const std::integral_constant<int, 6> m6;
    const __nv_bfloat16 b{};
    if (m == 2) NNV_CUDA(bf16 ? go(m2, b, std::false_type()) : go(m2, 0.f, std::false_type()));
    else if (m == 4) NNV_CUDA(bf16 ? go(m4, b, std::false_type()) : split ? go(m4, 0.f, std::true_type()) : go(m4, 0.f, std::false_type()));
    else if (m == 6) NNV_CUDA(bf16 ? go(m6, b, std::false_type()) : split ? go(m6, 0.f, std::true_type()) : go(m6, 0.f, std::false_type()));
    else return fail(NNV_ERR_INVALID_ARG, "no Winograd tile size %d", m);
    return NNV_OK;
}

// One thread per (tile, output channel), channel fastest.  Y tile = A^T M A, then bias, residual
// addend and activation; pixels beyond the output grid are clipped.
template <int M_>
__global__ void __launch_bounds__(128)
wino_output_kernel(const float* __restrict__ Mt, float* __restrict__ y, const float* __restrict__ bias,
                   const float* __restrict__ add, int act, int K, int OH, int OW, int TH, int TW) {
    pdl_enter();
    constexpr int A = WinoBA<M_>::A;
    const long long T = (long long)TH * TW;
    const long long idx = (long long)blockIdx.x * 128 + threadIdx.x;
    if (idx >= T * K) return;
    const int t = (int)(idx / K), k = (int)(idx - (long long)t * K);
    const int th = t / TW, tw = t - th * TW;
    const float* src = Mt + (long long)t * K + k;
    // The residual's loads leave first and without a condition of their own (pixels beyond the grid read the tile's first
    // one): loaded one by one next to the stores they cost 8 us on a 64 -> 64 layer @56 that takes 5 without them.
    float av[M_][M_];
    if (add) {
#pragma unroll
        for (int i = 0; i < M_; ++i)
#pragma unroll
            for (int j = 0; j < M_; ++j) {
                const int oh = min(th * M_ + i, OH - 1), ow = min(tw * M_ + j, OW - 1);
                av[i][j] = __ldg(add + ((long long)oh * OW + ow) * K + k);
            }
    }
    float tmp[M_][A];                                            // tmp = A^T M, built one M row at a time
#pragma unroll
    for (int i = 0; i < M_; ++i)
#pragma unroll
        for (int j = 0; j < A; ++j) tmp[i][j] = 0.f;
#pragma unroll
    for (int l = 0; l < A; ++l) {
        float row[A];
#pragma unroll
        for (int j = 0; j < A; ++j) row[j] = __ldg(src + (long long)(l * A + j) * T * K);
#pragma unroll
        for (int i = 0; i < M_; ++i)
            if (WinoBA<M_>::at(i, l) != 0.f) {
#pragma unroll
                for (int j = 0; j < A; ++j) tmp[i][j] += WinoBA<M_>::at(i, l) * row[j];
            }
    }
    const float b = bias ? __ldg(bias + k) : 0.f;
#pragma unroll
    for (int i = 0; i < M_; ++i) {
        const int oh = th * M_ + i;
#pragma unroll
        for (int j = 0; j < M_; ++j) {
            const int ow = tw * M_ + j;
            float s = 0.f;
#pragma unroll
            for (int l = 0; l < A; ++l)
                if (WinoBA<M_>::at(j, l) != 0.f) s += tmp[i][l] * WinoBA<M_>::at(j, l);
            if (oh < OH && ow < OW) {
                const long long o = ((long long)oh * OW + ow) * K + k;
                s += b;
                if (add) s += av[i][j];
                y[o] = apply_act(s, act);
            }
        }
    }
}

// A block takes one tile and 32 output channels; its first M_ warps write a row of the output tile each.
template <int M_>
__global__ void __launch_bounds__(32 * WinoBA<M_>::A)
wino_output_tile_kernel(const float* __restrict__ Mt, float* __restrict__ y, const float* __restrict__ bias,
                   const float* __restrict__ add, int act, int K, int OH, int OW, int TH, int TW) {
    constexpr int A = WinoBA<M_>::A;
    __shared__ float tmp[M_][A][32];                             // A^T M
    const int lane = threadIdx.x & 31, col = threadIdx.x >> 5;
    const int t = blockIdx.x, k = blockIdx.y * 32 + lane;
    const int th = t / TW, tw = t - th * TW;
    const bool live = k < K;
    const long long plane = (long long)TH * TW * K;
    const float* src = Mt + (long long)col * plane + (long long)t * K + k;
    const int oh = th * M_ + col, ow = tw * M_;                  // the warp's row of the output tile (the last warps have none)
    const bool writes = live && col < M_ && oh < OH;
    const long long at = ((long long)oh * OW + ow) * K + k;
    pdl_enter();
    float v[A];
#pragma unroll
    for (int l = 0; l < A; ++l) v[l] = live ? __ldg(src + (long long)(l * A) * plane) : 0.f;
    float av[M_];                                                // the residual's loads leave with the others
    if (add) {
#pragma unroll
        for (int j = 0; j < M_; ++j) av[j] = writes && ow + j < OW ? __ldg(add + at + (long long)j * K) : 0.f;
    }
    const float b = bias && live ? __ldg(bias + k) : 0.f;
#pragma unroll
    for (int i = 0; i < M_; ++i) {
        float s = 0.f;
#pragma unroll
        for (int l = 0; l < A; ++l)
            if (WinoBA<M_>::at(i, l) != 0.f) s += WinoBA<M_>::at(i, l) * v[l];
        tmp[i][col][lane] = s;
    }
    __syncthreads();
    if (!writes) return;
#pragma unroll
    for (int l = 0; l < A; ++l) v[l] = tmp[col][l][lane];
#pragma unroll
    for (int j = 0; j < M_; ++j) {
        float s = 0.f;
#pragma unroll
        for (int l = 0; l < A; ++l)
            if (WinoBA<M_>::at(j, l) != 0.f) s += v[l] * WinoBA<M_>::at(j, l);
        if (ow + j < OW) {
            s += b;
            if (add) s += av[j];
            y[at + (long long)j * K] = apply_act(s, act);
        }
    }
}

nnv_status_t launch_wino_output(int m, const float* Mt, float* y, const float* bias, const float* add, int act,
                                int K, int OH, int OW, int TH, int TW, cudaStream_t st) {
    const long long n = (long long)TH * TW * K;
    auto go = [&](auto mm) {
        constexpr int M_ = decltype(mm)::value;
        if (wino_tile_blocks<M_>(TH, TW, K))
            return launch_pdl(wino_output_tile_kernel<M_>, dim3(TH * TW, ceil_div(K, 32)), dim3(32 * (M_ + 2)), 0, st, Mt, y, bias, add, act, K, OH, OW, TH, TW);
        return launch_stream(STREAM_RESIDENT, wino_output_kernel<M_>, dim3((unsigned)((n + 127) / 128)), dim3(128), 0, st, Mt, y, bias, add, act, K, OH, OW, TH, TW);
    };
    if (m == 2) NNV_CUDA(go(std::integral_constant<int, 2>()));
    else if (m == 4) NNV_CUDA(go(std::integral_constant<int, 4>()));
    else if (m == 6) NNV_CUDA(go(std::integral_constant<int, 6>()));
    else return fail(NNV_ERR_INVALID_ARG, "no Winograd tile size %d", m);
    return NNV_OK;
}

// ---- fp32 depthwise convolution -------------------------------------------------------------
// One thread per (output pixel, channel), channel fastest; raw weights W[c][r][s] are read as is.
__global__ void __launch_bounds__(256)
depthwise_kernel(const float* __restrict__ x, const float* __restrict__ w, const float* __restrict__ bias,
                 const float* __restrict__ add, float* __restrict__ y, int act, int C, int H, int W, int R, int S,
                 int stride, int pad, int OH, int OW) {
    pdl_enter();
    const long long n = (long long)OH * OW * C;
    for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < n; i += (long long)gridDim.x * 256) {
        const int p = (int)(i / C), c = (int)(i - (long long)p * C);
        const int oh = p / OW, ow = p - oh * OW;
        float acc = bias ? __ldg(bias + c) : 0.f;
        for (int r = 0; r < R; ++r) {
            const int ih = oh * stride + r - pad;
            if (ih < 0 || ih >= H) continue;
            for (int s = 0; s < S; ++s) {
                const int iw = ow * stride + s - pad;
                if (iw < 0 || iw >= W) continue;
                acc = fmaf(__ldg(x + ((long long)ih * W + iw) * C + c), __ldg(w + ((long long)c * R + r) * S + s), acc);
            }
        }
        if (add) acc += __ldg(add + i);
        y[i] = apply_act(acc, act);
    }
}

// 3x3 depthwise, stride 1 or 2, C % 4 == 0: one thread = four channels x PX neighbouring output pixels of a row (the input
// window is loaded once for them).  A block takes `cg` channel quads (consecutive threads: contiguous 16-byte accesses) and as
// many pixel groups as fill it; its raw weights W[c][r][s], one contiguous range, come through shared memory -- read by each
// thread for itself, nine loads 144 bytes apart, they cost more cache lines than the activation.
constexpr int DW_MAX_CG = 32;
template <int STRIDE, int PX>
__global__ void __launch_bounds__(256)
depthwise3x3_v4_kernel(const float* __restrict__ x, const float* __restrict__ w, const float* __restrict__ bias,
                       const float* __restrict__ add, float* __restrict__ y, int act, int C, int H, int W, int pad, int OH, int OW, int cg) {
    pdl_enter();
    constexpr int NCOL = (PX - 1) * STRIDE + 3;
    __shared__ __align__(16) float sw[DW_MAX_CG * 36];
    const int C4 = C >> 2, OWP = (OW + PX - 1) / PX;
    const int q0 = blockIdx.y * cg, nq = min(cg, C4 - q0);     // this block's channel quads
    const int ppb = 256 / cg, lc = threadIdx.x % cg, lp = threadIdx.x / cg;
    const int pg = blockIdx.x * ppb + lp;                      // pixel group
    const bool live = lp < ppb && lc < nq && pg < OH * OWP;
    const int oh = pg / OWP, ow0 = (pg - oh * OWP) * PX;
    const int c = (q0 + lc) * 4;
    const int ih0 = oh * STRIDE - pad, iw0 = ow0 * STRIDE - pad;
    float4 v[3][NCOL];
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int col = 0; col < NCOL; ++col) {
            const int ih = ih0 + r, iw = iw0 + col;
            v[r][col] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (live && ih >= 0 && ih < H && iw >= 0 && iw < W) v[r][col] = __ldg(reinterpret_cast<const float4*>(x + ((long long)ih * W + iw) * C + c));
        }
    for (int i = threadIdx.x; i < nq * 9; i += 256) reinterpret_cast<float4*>(sw)[i] = __ldg(reinterpret_cast<const float4*>(w + (long long)q0 * 36) + i);
    __syncthreads();
    if (!live) return;
    float wv[36];                                             // [channel 0..3][tap 0..8]
#pragma unroll
    for (int j = 0; j < 9; ++j) {
        const float4 t = *reinterpret_cast<const float4*>(sw + lc * 36 + 4 * j);
        wv[4 * j] = t.x; wv[4 * j + 1] = t.y; wv[4 * j + 2] = t.z; wv[4 * j + 3] = t.w;
    }
    const float4 b4 = bias ? __ldg(reinterpret_cast<const float4*>(bias + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int p = 0; p < PX; ++p) {
        const int ow = ow0 + p;
        if (ow >= OW) break;
        float4 o = b4;
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int sx = 0; sx < 3; ++sx) {
                const float4 t = v[r][p * STRIDE + sx];
                const int k = r * 3 + sx;
                o.x = fmaf(t.x, wv[k], o.x); o.y = fmaf(t.y, wv[9 + k], o.y);
                o.z = fmaf(t.z, wv[18 + k], o.z); o.w = fmaf(t.w, wv[27 + k], o.w);
            }
        const long long off = ((long long)oh * OW + ow) * C + c;
        if (add) {
            const float4 a4 = __ldg(reinterpret_cast<const float4*>(add + off));
            o.x += a4.x; o.y += a4.y; o.z += a4.z; o.w += a4.w;
        }
        o.x = apply_act(o.x, act); o.y = apply_act(o.y, act); o.z = apply_act(o.z, act); o.w = apply_act(o.w, act);
        *reinterpret_cast<float4*>(y + off) = o;
    }
}

nnv_status_t launch_depthwise(const float* x, const float* w, const float* bias, const float* add, float* y,
                              int act, int C, int H, int W, int R, int S, int stride, int pad, int OH, int OW,
                              cudaStream_t st) {
    const bool al16 = ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(w) | reinterpret_cast<uintptr_t>(y) |
                        reinterpret_cast<uintptr_t>(bias) | reinterpret_cast<uintptr_t>(add)) & 15) == 0;
    if (R == 3 && S == 3 && (stride == 1 || stride == 2) && (C % 4) == 0 && al16 && (long long)OH * OW < (1 << 24) && C <= (1 << 22)) {
        // Channel quads per block: even shares of at most 32.  Pixels per thread: four, fewer where that leaves SMs without a
        // block (10 x 10 x 384: 12 blocks of 256 threads with four, 39 with one).
        const int C4 = C / 4, cg = ceil_div(C4, ceil_div(C4, DW_MAX_CG)), ppb = 256 / cg;
        auto grid_of = [&](int px) { return dim3(ceil_div(OH * ceil_div(OW, px), ppb), ceil_div(C4, cg)); };
        int px = 4;
        while (px > 1 && (long long)grid_of(px).x * grid_of(px).y < 148) px /= 2;
        const dim3 grid = grid_of(px);
        auto go = [&](auto kernel) { return launch_stream(STREAM_SMALL, kernel, grid, dim3(256), 0, st, x, w, bias, add, y, act, C, H, W, pad, OH, OW, cg); };
        if (stride == 1) NNV_CUDA(px == 4 ? go(depthwise3x3_v4_kernel<1, 4>) : px == 2 ? go(depthwise3x3_v4_kernel<1, 2>) : go(depthwise3x3_v4_kernel<1, 1>));
        else NNV_CUDA(px == 4 ? go(depthwise3x3_v4_kernel<2, 4>) : px == 2 ? go(depthwise3x3_v4_kernel<2, 2>) : go(depthwise3x3_v4_kernel<2, 1>));
        return NNV_OK;
    }
    const long long n = (long long)OH * OW * C;
    const unsigned grid = (unsigned)std::min<long long>((n + 255) / 256, 148ll * 32);
    NNV_CUDA(launch_stream(STREAM_SMALL, depthwise_kernel, dim3(grid), dim3(256), 0, st, x, w, bias, add, y, act, C, H, W, R, S, stride, pad, OH, OW));
    return NNV_OK;
}

// ---- pooling and layout ---------------------------------------------------------------------
__global__ void __launch_bounds__(256)
maxpool_kernel(const float* __restrict__ x, float* __restrict__ y, int C, int H, int W, int R, int stride, int pad,
               int OH, int OW) {
    pdl_enter();
    const long long n = (long long)OH * OW * C;
    for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < n; i += (long long)gridDim.x * 256) {
        const int p = (int)(i / C), c = (int)(i - (long long)p * C);
        const int oh = p / OW, ow = p - oh * OW;
        float m = -INFINITY;
        for (int r = 0; r < R; ++r) {
            const int ih = oh * stride + r - pad;
            if (ih < 0 || ih >= H) continue;
            for (int s = 0; s < R; ++s) {
                const int iw = ow * stride + s - pad;
                if (iw < 0 || iw >= W) continue;
                m = fmaxf(m, __ldg(x + ((long long)ih * W + iw) * C + c));
            }
        }
        y[i] = m;
    }
}

// C % 4 == 0: four channels per thread.  R is 2 or 3 in practice; the window's loads do not depend on one another.
template <int R>
__global__ void __launch_bounds__(256)
maxpool_v4_kernel(const float4* __restrict__ x, float4* __restrict__ y, int C4, int H, int W, int stride, int pad, int OH, int OW) {
    pdl_enter();
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= OH * OW * C4) return;
    const int p = i / C4, c = i - p * C4;
    const int oh = p / OW, ow = p - oh * OW;
    const int h0 = oh * stride - pad, w0 = ow * stride - pad;
    float4 v[R][R];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int s = 0; s < R; ++s) {
            const int h = h0 + r, w = w0 + s;
            v[r][s] = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
            if (h >= 0 && h < H && w >= 0 && w < W) v[r][s] = __ldg(x + ((long long)h * W + w) * C4 + c);
        }
    float4 m = v[0][0];
#pragma unroll
    for (int q = 1; q < R * R; ++q) {
        const float4 t = v[q / R][q % R];
        m.x = fmaxf(m.x, t.x); m.y = fmaxf(m.y, t.y); m.z = fmaxf(m.z, t.z); m.w = fmaxf(m.w, t.w);
    }
    y[i] = m;
}

__global__ void __launch_bounds__(256)
gavgpool_kernel(const float* __restrict__ x, float* __restrict__ y, int C, int HW) {
    pdl_enter();
    const int c = blockIdx.x * 256 + threadIdx.x;
    if (c >= C) return;
    float s = 0.f;
    for (int p = 0; p < HW; ++p) s += __ldg(x + (long long)p * C + c);
    y[c] = s / (float)HW;
}

// Few channels (a model's image): a thread moves V neighbouring pixels, 4 V bytes from every channel plane, so that a read
// in place from pinned host memory asks for whole lines once.
template <int V>
__global__ void __launch_bounds__(256)
chw_to_hwc_few_kernel(const float* __restrict__ in, float* __restrict__ out, int C, int HW) {
    pdl_enter();
    const int p = (blockIdx.x * 256 + threadIdx.x) * V;
    if (p >= HW) return;
    float v[4][V];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        if (c >= C) break;
        if constexpr (V == 4) {
            const float4 q = __ldg(reinterpret_cast<const float4*>(in + (long long)c * HW + p));
            v[c][0] = q.x; v[c][1] = q.y; v[c][2] = q.z; v[c][3] = q.w;
        } else {
            v[c][0] = __ldg(in + (long long)c * HW + p);
        }
    }
#pragma unroll
    for (int j = 0; j < V; ++j)
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (c < C) out[(long long)(p + j) * C + c] = v[c][j];
}

// [R][Cn] -> [Cn][R] in tiles of 32 x 32 through shared memory: reads and writes are both contiguous along a warp.  With a
// status word given, one thread copies it to the host (the last kernel of a run; a copy of its own would cost more).
__global__ void __launch_bounds__(256)
transpose_kernel(const float* __restrict__ in, float* __restrict__ out, int R, int Cn, const int* status, int* h_status) {
    pdl_enter();
    __shared__ float tile[32][33];
    const int tiles_c = (Cn + 31) / 32;
    const int c0 = (int)(blockIdx.x % tiles_c) * 32, r0 = (int)(blockIdx.x / tiles_c) * 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = r0 + ty + 8 * i;
        if (r < R && c0 + tx < Cn) tile[ty + 8 * i][tx] = __ldg(in + (long long)r * Cn + c0 + tx);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int c = c0 + ty + 8 * i;
        if (c < Cn && r0 + tx < R) out[(long long)c * R + r0 + tx] = tile[tx][ty + 8 * i];
    }
    if (h_status && blockIdx.x == 0 && threadIdx.x == 0) *h_status = *reinterpret_cast<const volatile int*>(status);
}

static inline unsigned grid_for(long long n) { return (unsigned)std::min<long long>((n + 255) / 256, 148ll * 32); }

nnv_status_t launch_maxpool(const float* x, float* y, int C, int H, int W, int R, int stride, int pad, int OH,
                            int OW, cudaStream_t st) {
    if ((R == 2 || R == 3) && (C % 4) == 0 && ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y)) & 15) == 0 &&
        (long long)OH * OW * C < (1ll << 31)) {
        const dim3 grid(ceil_div(OH * OW * (C / 4), 256));
        const float4* x4 = reinterpret_cast<const float4*>(x);
        float4* y4 = reinterpret_cast<float4*>(y);
        if (R == 2) NNV_CUDA(launch_stream(STREAM_SMALL, maxpool_v4_kernel<2>, grid, dim3(256), 0, st, x4, y4, C / 4, H, W, stride, pad, OH, OW));
        else NNV_CUDA(launch_stream(STREAM_SMALL, maxpool_v4_kernel<3>, grid, dim3(256), 0, st, x4, y4, C / 4, H, W, stride, pad, OH, OW));
        return NNV_OK;
    }
    NNV_CUDA(launch_stream(STREAM_SMALL, maxpool_kernel, dim3(grid_for((long long)OH * OW * C)), dim3(256), 0, st, x, y, C, H, W, R, stride, pad, OH, OW));
    return NNV_OK;
}
nnv_status_t launch_gavgpool(const float* x, float* y, int C, int H, int W, cudaStream_t st) {
    NNV_LAUNCH((gavgpool_kernel), ceil_div(C, 256), 256, 0, st, x, y, C, H * W);
    NNV_CUDA(cudaGetLastError());
    return NNV_OK;
}
static nnv_status_t launch_transpose(const float* in, float* out, int R, int Cn, const int* status, int* h_status, cudaStream_t st) {
    const long long tiles = (long long)ceil_div(Cn, 32) * ceil_div(R, 32);
    NNV_REQUIRE(tiles < (1ll << 31), NNV_ERR_UNSUPPORTED, "image too large for the layout conversion");
    const dim3 grid((unsigned)tiles);
    NNV_CUDA(launch_pdl(transpose_kernel, grid, dim3(256), 0, st, in, out, R, Cn, status, h_status));
    return NNV_OK;
}
nnv_status_t launch_chw_to_hwc(const float* in, float* out, int C, int H, int W, cudaStream_t st) {
    const int HW = H * W;
    if (C <= 4 && (HW % 4) == 0 && (reinterpret_cast<uintptr_t>(in) & 15) == 0)
        NNV_CUDA(launch_pdl(chw_to_hwc_few_kernel<4>, dim3(ceil_div(HW, 1024)), dim3(256), 0, st, in, out, C, HW));
    else if (C <= 4)
        NNV_CUDA(launch_pdl(chw_to_hwc_few_kernel<1>, dim3(ceil_div(HW, 256)), dim3(256), 0, st, in, out, C, HW));
    else
        return launch_transpose(in, out, C, HW, nullptr, nullptr, st);
    return NNV_OK;
}
nnv_status_t launch_hwc_to_chw(const float* in, float* out, int C, int H, int W, cudaStream_t st, const int* status, int* h_status) {
    return launch_transpose(in, out, H * W, C, status, h_status, st);
}

}  // namespace nnv
