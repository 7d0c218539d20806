// Batched tensor-core GEMM for sm_100a:  D[b][M][N] = A[b][M][Kd] * B[b][N][Kd]^T.
//
// Both operands are K-major (row-major with the reduction index innermost), which is how the
// Winograd tile GEMM (V[xi,nu][T][C] x U[xi,nu][K][C]), the im2col GEMM (Xcol[P][Q] x P[K][Q])
// and the 1x1 GEMM (X[P][C] x W[K][C]) all present themselves.  Pixels / tiles sit on the MMA's
// M dimension (128 TMEM lanes), output channels on N.
//
// Structure of one CTA (one 128 x BN output tile, 256 threads):
//   warps 0, 7  TMA producers of A and B: cp.async.bulk.tensor loads of 128-byte-wide K slices into a ring of
//            shared-memory stages (128B swizzle), completion on "full" mbarriers
//   warps 1, 6  issue tcgen05.mma (one lane each) from shared-memory descriptors for alternate K blocks, each into its own
//            fp32 accumulator in TMEM, and release the stages that are refilled with tcgen05.commit on "empty" mbarriers (an
//            arrival that nobody waits for could meet a CTA that has left); warp 1 allocates TMEM
//   warps 4, 5  every other load of deep K loops; warps 2-5  the bias, and the conversion of operands
//   all eight  write out: tcgen05.ld the accumulators (each warp 32 TMEM lanes), apply bias / residual / activation, store fp32 rows
// These layers are latency-bound (5 - 10 dependent phases of ~0.1 - 0.5 us each); what bounds each phase was read from
// device-clock probes.  Two producers and two issuers: one thread pays 157 cycles per load and ~560 per K block of waiting,
// issuing four MMAs and committing, more than the fill (~320 cycles of 24 KB) or the tensor pipe need.  Their loops run under
// elect.sync, not "lane == 0": the operands then stay in uniform registers (a K block 340 -> 260 cycles).
// 1024 -> 256 1x1 @14 (64 CTAs, 8 splits) went from 9900 to 6200 cycles from the previous kernel's end, chained calls of
// 64 -> 64 3x3 @56 from 8.2 to 5.2 us, 256 -> 256 3x3 @14 from 9.1 to 5.6 us, 512 -> 2048 1x1 @7 from 6.2 to 4.3 us.
// Every mbarrier wait is bounded; a wait that gives up records NNV_ERR_TIMEOUT in a device status
// word and the CTA drains and exits instead of hanging.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <mutex>
#include <type_traits>

#include "nnv_internal.h"

namespace nnv {

__device__ int g_device_status = 0;

nnv_status_t read_device_status(int32_t* code) {
    NNV_CUDA(cudaDeviceSynchronize());
    int v = 0;
    NNV_CUDA(cudaMemcpyFromSymbol(&v, g_device_status, sizeof(int)));
    if (v != 0) {
        int zero = 0;
        NNV_CUDA(cudaMemcpyToSymbol(g_device_status, &zero, sizeof(int)));
    }
    *code = v;
    return NNV_OK;
}

__device__ unsigned long long g_stamps[2 * STAMP_SLOTS_PER_LAYER * STAMP_MAX_LAYERS];

unsigned long long*& next_stamp() {
    static thread_local unsigned long long* p = nullptr;
    return p;
}

nnv_status_t stamps_device_base(unsigned long long** base) {
    void* ptr = nullptr;
    NNV_CUDA(cudaGetSymbolAddress(&ptr, g_stamps));
    *base = static_cast<unsigned long long*>(ptr);
    return NNV_OK;
}

nnv_status_t device_status_address(const int** d) {
    void* ptr = nullptr;
    NNV_CUDA(cudaGetSymbolAddress(&ptr, g_device_status));
    *d = static_cast<const int*>(ptr);
    return NNV_OK;
}

namespace {

constexpr int BM = 128;                 // rows of A per tile = TMEM lanes
constexpr int BK_BYTES = 128;           // bytes of K per stage row = one 128B swizzle atom
constexpr int A_STAGE_BYTES = BM * BK_BYTES;
constexpr int GEMM_THREADS = 192;
// gemm_tc_kernel: a second MMA issuer and a second producer; splitting both operands (mode 2), gathering (modes 4 - 7) and rounding
// (mode 8) take four more warps
constexpr int gemm_tc_threads(int mode) { return mode == 2 || mode >= 4 ? 384 : 256; }   // (3: the write-out's warps convert)
constexpr int GATHER_WARPS = 8;
// Loading warps an operand has: in modes 0 and 1 a second one takes every other block of K loops of six blocks and more.
__host__ __device__ constexpr int gemm_loaders(int mode, int nkb, int stages) { return (mode == 0 || mode == 1) && nkb >= 6 && stages >= 2 ? 2 : 1; }
constexpr int GEMM_BAR_BYTES = 8 * (3 * 8 + 6) + 512;         // barriers, TMEM address, bias of the tile's columns
constexpr uint32_t WAIT_LIMIT = 1u << 20;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait: false when the limit ran out (the caller records a timeout and bails out).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    for (uint32_t i = 0; i < WAIT_LIMIT; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
        : "memory");
}

// im2col-mode load: `pixelsPerColumn` consecutive output pixels starting at the filter window whose
// top-left input coordinate is (w, h), each shifted by the tap offset (off_w, off_h); channels
// [c, c + channelsPerPixel).  Positions outside the image read as zero.
__device__ __forceinline__ void tma_load_im2col_4d(uint32_t dst, const CUtensorMap* map, int c, int w, int h, int n,
                                                   uint16_t off_w, uint16_t off_h, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.im2col.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6], {%7, %8};"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(c), "r"(w), "r"(h), "r"(n), "r"(bar), "h"(off_w), "h"(off_h)
        : "memory");
}

// Tile store shared -> global through the tensor map (rows / columns outside the tensor are clipped).
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, uint32_t src, int c0, int c1, int c2) {
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%2, %3, %4}], [%1];"
                 ::"l"(reinterpret_cast<uint64_t>(map)), "r"(src), "r"(c0), "r"(c1), "r"(c2)
                 : "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// All of this thread's tile stores have finished READING shared memory (the global writes complete with the grid).
__device__ __forceinline__ void tma_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

// Barrier over every thread of every CTA in the cluster (release / acquire), in one piece or as its two halves.
__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync_all() {
    cluster_arrive();
    cluster_wait();
}
__device__ __forceinline__ uint32_t cluster_addr(uint32_t local, int rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}
// Bulk copy of `bytes` (a multiple of 16) from this CTA's shared memory into a cluster CTA's, counted on the barrier there.
__device__ __forceinline__ void bulk_push(uint32_t remote_dst, uint32_t src, uint32_t bytes, uint32_t remote_bar) {
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(remote_dst), "r"(src), "r"(bytes), "r"(remote_bar) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, rows 128 bytes apart,
// 8-row groups 1024 bytes apart (stride byte offset), descriptor version 1.
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
    d |= (uint64_t)1 << 16;                     // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;           // stride byte offset
    d |= (uint64_t)1 << 46;                     // version
    d |= (uint64_t)2 << 61;                     // SWIZZLE_128B
    return d;
}

// The same with the 64-byte swizzle: rows 64 bytes apart (32 bf16), 8-row groups 512 bytes apart.
__device__ __forceinline__ uint64_t make_smem_desc64(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(512 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)4 << 61;                     // SWIZZLE_64B
    return d;
}

template <bool BF16>
__device__ __forceinline__ void umma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    if constexpr (BF16) {
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
            ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
    } else {
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}"
            ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
    }
}

__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// (A TMEM load is one instruction of the whole warp: lanes that came here by different ways meet first.)
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    __syncwarp();
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t (&r)[16]) {
    __syncwarp();
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld8_nowait(uint32_t taddr, uint32_t (&r)[8]) {
    __syncwarp();
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// One lane of a converged warp, picked by the hardware: code under this predicate may keep its operands in uniform registers.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}

__device__ __forceinline__ float4 lds128(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void sts128(uint32_t addr, const float4& v) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

struct GemmDev {
    unsigned long long* stamp;        // device-clock stamps of this launch, or null
    float* D;
    const float* bias;
    const float* addend;
    long long ldd, strideD;
    int M, N, Kd, BN, act, tmem_cols, splits, stages, issuers;
    int rows;                         // rows of A per tile, at most 128
    int z_tiles;                      // output map: 0 = {N, M, batch}; else {N, rows, tiles} with this many tiles per batch entry
    uint32_t bar_off;                 // byte offset (from the aligned base) of the barriers
    int chunk;                        // unsplit: columns of a staging sub-tile (16); 0: plain stores
    uint32_t recv_off;                // splits > 1: byte offset (from the aligned base) of the received partial rows
    uint32_t stage_off;               // byte offset (from the aligned base) of the dedicated staging tile; 0 = the idle ring
    // implicit im2col (A is the NHWC activation itself): 0 = off
    // (2: its tiles are whole image rows, fetched as plain boxes)
    int ic_on, ic_C, ic_cblk, ic_S, ic_OW, ic_stride, ic_pad;
    // modes 4 - 7: the activation, its size and the window's length R * S * C; magic numbers that divide by C and S
    const float* x;
    int ic_H, ic_W, ic_Q;
    uint32_t magic_c, magic_s;
};

__device__ __forceinline__ float act_fn(float v, int act) {
    if (act == 1) return fmaxf(v, 0.f);
    if (act == 2) return fminf(fmaxf(v, 0.f), 6.f);
    return v;
}

// Descriptor for the un-swizzled K-major layout used by the converted bf16 tiles: 8x16-byte core
// matrices, `lbo` bytes between core matrices adjacent in K, `sbo` bytes between 8-row groups.
__device__ __forceinline__ uint64_t make_smem_desc_plain(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;                     // version; layout type 0 = no swizzle
    return d;
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// Split eight fp32 values into bf16 hi = rn(x) and lo = rn(x - hi), packed as two 16-byte chunks.
__device__ __forceinline__ void split8(const float4& a, const float4& b, uint4& hi, uint4& lo) {
    auto split2 = [](float x, float y, uint32_t& h, uint32_t& l) {
        const __nv_bfloat162 p = __floats2bfloat162_rn(x, y);
        h = *reinterpret_cast<const uint32_t*>(&p);
        const __nv_bfloat162 q = __floats2bfloat162_rn(x - __uint_as_float(h << 16), y - __uint_as_float(h & 0xFFFF0000u));
        l = *reinterpret_cast<const uint32_t*>(&q);
    };
    split2(a.x, a.y, hi.x, lo.x); split2(a.z, a.w, hi.y, lo.y);
    split2(b.x, b.y, hi.z, lo.z); split2(b.z, b.w, hi.w, lo.w);
}

__device__ __forceinline__ uint4 pack8_bf16(const float4& a, const float4& b) {
    const __nv_bfloat162 p0 = __floats2bfloat162_rn(a.x, a.y), p1 = __floats2bfloat162_rn(a.z, a.w);
    const __nv_bfloat162 p2 = __floats2bfloat162_rn(b.x, b.y), p3 = __floats2bfloat162_rn(b.z, b.w);
    return make_uint4(*reinterpret_cast<const uint32_t*>(&p0), *reinterpret_cast<const uint32_t*>(&p1),
                      *reinterpret_cast<const uint32_t*>(&p2), *reinterpret_cast<const uint32_t*>(&p3));
}

// Converts chunk c (8 of the 32 elements) of row r of a staged fp32 tile (TMA, 128-byte swizzle) into bf16 tiles in the
// un-swizzled core-matrix layout, `rows` rows tall: hi and lo, or (SPLIT = false) one tile rounded to nearest even.
template <bool SPLIT>
__device__ __forceinline__ void convert_chunk(const uint8_t* src_tile, uint8_t* hi_tile, uint8_t* lo_tile, int r, int c, int rows) {
    const uint8_t* src = src_tile + r * 128;
    const float4 v0 = *reinterpret_cast<const float4*>(src + (((2 * c) ^ (r & 7)) << 4));
    const float4 v1 = *reinterpret_cast<const float4*>(src + (((2 * c + 1) ^ (r & 7)) << 4));
    const int off = (c * rows + r) * 16;
    if constexpr (SPLIT) {
        uint4 hi, lo;
        split8(v0, v1, hi, lo);
        *reinterpret_cast<uint4*>(hi_tile + off) = hi;
        *reinterpret_cast<uint4*>(lo_tile + off) = lo;
    } else {
        *reinterpret_cast<uint4*>(hi_tile + off) = pack8_bf16(v0, v1);
    }
}

// MODE 3: A is fp32 (the activation itself, direct or through the TMA's im2col mode) and is rounded to bf16 by the
// epilogue warps on its way through shared memory; B is the bf16 packed weight, fetched with the 64-byte swizzle.
// MODE 0: TF32 operands (fp32 words), 1: BF16 operands, 2: fp32 operands multiplied as
// hi*hi + lo*hi + hi*lo of their bf16 splits (error-compensated, fp32-class accuracy).
// MODE 4 - 7: A is gathered from the filter windows of the activation by eight warps, element by element (4: TF32, 5: BF16) or
// four channels at a time (6, 7), and rounded to nearest even on the way; B as in mode 0 or 1.
// MODE 8: TF32 on the boxes of a small image (below 128 KiB), whose tiles warps 2-5 and 8-11 round to nearest even where they lie;
// the tensor core would truncate them, an error of 4.3e-4 a layer against 2.9e-4.  The two groups of warps take the K blocks in
// turn, as the issuers do: all eight on every block take 5 % longer, four 20 %.  Bound: the pass through shared memory (25 KB a
// block of 98 rows) behind each load.  us, gathered / this / truncated: 64 -> 64 3x3 @14 4.2 / 3.9 / 3.6, 160 -> 160 @14 6.6 / 5.4 / 4.3,
// 256 -> 256 @7 6.0 / 4.8 / 4.2, 320 -> 320 @10 8.4 / 6.4 / 5.1.
constexpr int ROUNDED = 8;
// MODE 9: mode 2 on an A that is split already: a row's block of 32 words holds its elements' bf16 hi parts, then their lo parts (the
// Winograd input transform writes it so where the channels come in whole blocks), and only B's rows are split here, a third of the work
// or less.  The same products in the same order as mode 2.
constexpr int SPLIT_A = 9;
__host__ __device__ constexpr bool x3_mode(int mode) { return mode == 2 || mode == SPLIT_A; }
__host__ __device__ constexpr bool gather_mode(int mode) { return mode >= 4 && mode <= 7; }
__host__ __device__ constexpr bool converting_mode(int mode) { return x3_mode(mode) || mode == 3 || mode == ROUNDED; }
__host__ __device__ constexpr bool bf16_mode(int mode) { return mode == 1 || mode == 5 || mode == 7; }   // both operands staged as bf16
template <int MODE> struct ModeTraits {
    static constexpr int BKE = bf16_mode(MODE) ? 64 : 32;      // K elements per stage
};
// n / d for n * d < 2^32, with magic = ceil(2^32 / d)
__device__ __forceinline__ int div_magic(int n, int d, uint32_t magic) { return d == 1 ? n : (int)__umulhi((uint32_t)n, magic); }

// A stage holds the `rows` rows of A that are loaded (the MMA's other rows read whatever follows and are never written out)
// and BN rows of B, 128 bytes each; the conversion modes add the bf16 tiles, `pad8(rows)` rows tall: A (hi, lo), B (hi, lo) in
// mode 2; A in mode 3, whose B arrives as bf16.
__host__ __device__ constexpr int pad8(int rows) { return (rows + 7) & ~7; }
__host__ __device__ constexpr uint32_t a_stage_of(int rows) { return ((uint32_t)rows * BK_BYTES + 1023u) & ~1023u; }
template <int MODE>
__host__ __device__ constexpr uint32_t stage_bytes_of(int BN, int rows) {
    const uint32_t a = a_stage_of(rows), b = (uint32_t)(BN * BK_BYTES);
    if (MODE == 3) return (a + (uint32_t)(pad8(rows) * 64) + b / 2 + 1023u) & ~1023u;
    if (MODE == 2) return (a + b + (uint32_t)(pad8(rows) * 128) + b + 1023u) & ~1023u;
    if (MODE == SPLIT_A) return (a + 2 * b + 1023u) & ~1023u;
    return a + b;
}

// (Four CTAs to an SM, 64 registers a thread, for unsplit launches without conversion, whose grids may be many waves of short K loops:
// 17 -> 24 F(2,3) @180 BF16 20.3 us with three, 18.5 with four.)
template <int MODE, bool SPLIT>
__global__ void __launch_bounds__(gemm_tc_threads(MODE), MODE == 2 || MODE >= 4 ? 2 : MODE == 3 || SPLIT ? 3 : 4)
gemm_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
               const __grid_constant__ CUtensorMap tmAdd, const GemmDev g) {
    extern __shared__ uint8_t smem_raw[];
    const int STAGES = g.stages;                              // depth of the shared-memory ring (2..8)
    constexpr int MAXS = 8;
    constexpr int BKE = ModeTraits<MODE>::BKE;
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const int BN = g.BN;
    const uint32_t b_stage_bytes = (uint32_t)BN * BK_BYTES;
    const uint32_t b_bytes = MODE == 3 ? (uint32_t)BN * 64u : b_stage_bytes, a_bytes = (uint32_t)g.rows * BK_BYTES;
    const uint32_t a_stage = a_stage_of(g.rows);
    const int rp = pad8(g.rows);
    const uint32_t stage_bytes = stage_bytes_of<MODE>(BN, g.rows);
    const uint32_t bars = sbase + g.bar_off;                  // behind the ring       // full[S], empty[S], conv[S], tmem_full, holder
    auto full_bar = [&](int s) { return bars + 8u * s; };
    auto empty_bar = [&](int s) { return bars + 8u * (MAXS + s); };
    auto conv_bar = [&](int s) { return bars + 8u * (2 * MAXS + s); };
    const uint32_t tmem_full_bar = bars + 8u * (3 * MAXS);
    const uint32_t holder = bars + 8u * (3 * MAXS + 1);
    const uint32_t addend_bar = bars + 8u * (3 * MAXS + 2);
    const uint32_t recv_bar = bars + 8u * (3 * MAXS + 3);
    const uint32_t bias_bar = bars + 8u * (3 * MAXS + 4);
    const uint32_t sbias = bars + 8u * (3 * MAXS + 6);        // the tile's BN bias values (zeros without a bias)
    // Write-out through shared memory (g.chunk): the tile is staged as [16-column chunk][warp quarter] sub-tiles of 32 rows, their
    // 16-byte words in the 64-byte swizzle.  With a residual addend the sub-tiles live in their own region and the addend is loaded
    // INTO them while the K loop runs, so the write-out adds in place; without one they reuse the ring, which is idle by then.
    // (The width is a launch parameter although it is always 16: as a constant it let the compiler rearrange the loop, 256 -> 1024 1x1
    // @14 3.14 us against 3.05, 24 -> 144 @40 2.38 against 2.32.)
    const int CW = g.chunk;
    const uint32_t chunk_bytes = 32u * (uint32_t)CW * 4u;
    const uint32_t stg0 = sbase + g.stage_off;
    const int quarters = (g.rows + 31) >> 5;                  // 32-row sub-tiles of the tile
    const int y0 = g.z_tiles ? 0 : (int)blockIdx.x * g.rows;  // output map: first row and third coordinate of the tile
    volatile uint32_t* holder_ptr = reinterpret_cast<volatile uint32_t*>(smem_raw + (holder - smem_u32(smem_raw)));

    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    // blockIdx.z = batch * splits + split; the `splits` CTAs of one output tile form a thread-block
    // cluster, each reducing its own contiguous range of K blocks.
    const int splits = SPLIT ? g.splits : 1;
    const int sp = (int)blockIdx.z % splits, b = (int)blockIdx.z / splits;
    const int zd = g.z_tiles ? b * g.z_tiles + (int)blockIdx.x : b;
    const int m0 = blockIdx.x * g.rows, n0 = blockIdx.y * BN;
    const int nkb_all = g.ic_on ? g.Kd : (g.Kd + BKE - 1) / BKE;  // implicit mode: Kd already counts K blocks
    const int kb0 = (nkb_all * sp) / splits;                  // K blocks number a few thousand at most: 32-bit is enough
    const int nkb = (nkb_all * (sp + 1)) / splits - kb0;
    // Split K: rank `sp` of the cluster owns the tile's rows [sp * rows_per, ...); only rows that exist are reduced.
    const int live = min(g.rows, g.M - m0);
    const int rows_per = (live + splits - 1) / splits;
    const int my_rows = max(0, min(rows_per, live - sp * rows_per));

    if (warp == 0 && lane == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmA)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmB)) : "memory");
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full_bar(s), gather_mode(MODE) ? GATHER_WARPS + 1 : 2);
            mbar_init(empty_bar(s), 1);
            mbar_init(conv_bar(s), x3_mode(MODE) ? 8 : 4);
        }
        mbar_init(tmem_full_bar, (uint32_t)g.issuers);
        mbar_init(addend_bar, 1);
        mbar_init(recv_bar, 1);
        mbar_init(bias_bar, 4);
        if (CW && g.addend) asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmAdd)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(holder), "r"((uint32_t)g.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // One K block: operand tiles of iteration `it` into ring slot `s` (= it mod STAGES; the loops carry
    // slot and phase along instead of dividing: STAGES is a run-time value and these single-thread
    // loops are latency-bound, every instruction in them is on the critical path).
    // Implicit mode: K runs over (filter tap, channel block).  The tile's first output pixel and the K
    // position of the next block are kept as running values: the producer issues blocks in order, and a
    // division per block would sit on the latency path of the very first loads.
    int ic_w0 = 0, ic_h0 = 0, ic_cb = 0, ic_fs = 0, ic_fr = 0, ic_tap = 0;
    if (g.ic_on) {
        const int p0 = m0 / g.ic_OW, q0 = m0 - p0 * g.ic_OW;
        ic_w0 = q0 * g.ic_stride - g.ic_pad;
        ic_h0 = p0 * g.ic_stride - g.ic_pad;
        ic_tap = kb0 / g.ic_cblk;
        ic_cb = kb0 - ic_tap * g.ic_cblk;
        ic_fr = ic_tap / g.ic_S;
        ic_fs = ic_tap - ic_fr * g.ic_S;
    }
    auto issue_a = [&](int it, int s) {
        mbar_expect_tx(full_bar(s), a_bytes);
        const uint32_t a_dst = sbase + s * stage_bytes;
        if (g.ic_on) {
            // A comes straight from the activation: the block is channel block ic_cb of tap (ic_fr, ic_fs)
            if (g.ic_on == 2) tma_load_3d(a_dst, &tmA, ic_cb * BKE, ic_w0 + ic_fs, ic_h0 + ic_fr, full_bar(s));
            else tma_load_im2col_4d(a_dst, &tmA, ic_cb * BKE, ic_w0, ic_h0, 0, (uint16_t)ic_fs, (uint16_t)ic_fr, full_bar(s));
            if (++ic_cb == g.ic_cblk) {
                ic_cb = 0;
                if (++ic_fs == g.ic_S) { ic_fs = 0; ++ic_fr; }
            }
        } else {
            tma_load_3d(a_dst, &tmA, (kb0 + it) * BKE, m0, b, full_bar(s));
        }
    };
    auto issue_b = [&](int it, int s) {
        int q = (kb0 + it) * BKE;                             // the block's first position in the packed weight rows
        if (g.ic_on) {
            q = ic_tap * g.ic_C + ic_cb * BKE;
            if (++ic_cb == g.ic_cblk) { ic_cb = 0; ++ic_tap; }
        }
        mbar_expect_tx(full_bar(s), b_bytes);
        const uint32_t b_dst = sbase + s * stage_bytes + a_stage;
        // MODE 3: BN rows of 32 bf16 with the 64-byte swizzle, staged after the fp32 and the bf16 A tile
        tma_load_3d(MODE == 3 ? b_dst + rp * 64 : b_dst, &tmB, q, n0, b, full_bar(s));
    };
    // Gather modes: {byte offset of the first element, taps inside the image} of the window of each of the tile's output pixels;
    // the taps as a bit for every filter row (0 - 15) and every filter column (16 - 30).  No bits: the pixel does not exist.
    uint2* const windows = reinterpret_cast<uint2*>(smem_raw + (sbias - smem_u32(smem_raw)) + 512);
    if constexpr (gather_mode(MODE)) {
        if (threadIdx.x < BM) {
            const int m = m0 + (int)threadIdx.x, oh = m / g.ic_OW;
            const int ih = oh * g.ic_stride - g.ic_pad, iw = (m - oh * g.ic_OW) * g.ic_stride - g.ic_pad;
            auto inside = [](int first, int size, int most) {  // bits i < most with 0 <= first + i < size
                const int lo = min(max(-first, 0), most), hi = min(max(size - first, 0), most);
                return hi > lo ? (1u << hi) - (1u << lo) : 0u;
            };
            const uint32_t taps = inside(ih, g.ic_H, 16) | inside(iw, g.ic_W, 15) << 16;
            windows[threadIdx.x] = make_uint2((uint32_t)((ih * g.ic_W + iw) * g.ic_C) * 4u, (int)threadIdx.x < live ? taps : 0u);
        }
    }
    // What the write-out needs besides the accumulator is worked out here, where it costs nothing: a warp that has its scheduler to
    // itself pays 5 - 30 cycles for every dependent instruction.  (The pins keep the compiler from moving it behind the waits.)
    auto pin = [](auto& v) {
        if constexpr (sizeof(v) == 8) asm volatile("" : "+l"(v));
        else asm volatile("" : "+r"(v));
    };
    int quarter = warp & 3, grp = warp >= 2 && warp <= 5 ? 0 : 1, t = grp * 128 + quarter * 32 + lane;
    uint32_t tacc_off = (uint32_t)(quarter * 32) << 16;
    pin(t); pin(tacc_off);
    int rows_live = live - quarter * 32;                      // unsplit: rows of this warp's quarter, its first sub-tile, its lane's first word in memory
    uint32_t out_sub = 0;
    float* out_dst = nullptr;
    // split: see below
    int nch = 0, rot0 = 0, qstep = 0, rstep = 0, rot_step = 0, rr = 0, cc = 0, rot = 0, vec = 0;
    uint32_t prow = 0, push_dst = 0, push_bar = 0, push_src = 0, push_bytes = 0;
    float* dbase = nullptr;
    const float* abase = nullptr;
    if constexpr (!SPLIT) {
        out_sub = stg0 + (uint32_t)(grp * quarters + quarter) * chunk_bytes;
        out_dst = g.D + (long long)b * g.strideD + (long long)(m0 + quarter * 32 + (lane >> 2)) * g.ldd + n0 + grp * 16 + (lane & 3) * 4;
        pin(rows_live); pin(out_sub); pin(out_dst);
    } else {
        const int r0 = sp * rows_per, q0 = quarter * 32;
        nch = BN / 4;
        rot0 = (q0 + lane) % nch;
        prow = sbase + (uint32_t)(q0 + lane) * (uint32_t)BN * 4u;
        const int a0 = max(q0, lane * rows_per), a1 = min(min(q0 + 32, live), (lane + 1) * rows_per);
        if (grp == 0 && lane < splits && a1 > a0) {
            push_dst = cluster_addr(sbase + g.recv_off + (uint32_t)((r0 + a0 - lane * rows_per) * BN) * 4u, lane);
            push_bar = cluster_addr(recv_bar, lane);
            push_src = sbase + (uint32_t)(a0 * BN) * 4u;
            push_bytes = (uint32_t)((a1 - a0) * BN) * 4u;
        }
        vec = ((g.ldd & 3) == 0) && ((g.N & 3) == 0) && ((reinterpret_cast<uintptr_t>(g.D) & 15) == 0) &&
              (!g.addend || (reinterpret_cast<uintptr_t>(g.addend) & 15) == 0);
        // thread t walks the (row, 4-column group) grid of its CTA's rows in steps of 256
        qstep = 256 / nch; rstep = 256 - qstep * nch;
        rr = t / nch; cc = t - rr * nch; rot = (r0 + rr) % nch;
        rot_step = qstep % nch;
        dbase = g.D + (long long)b * g.strideD + (long long)(m0 + r0) * g.ldd + n0;
        abase = g.addend ? g.addend + (long long)(m0 + r0) * g.ldd + n0 : nullptr;
        pin(nch); pin(rot0); pin(prow); pin(push_dst); pin(push_bar); pin(push_src); pin(push_bytes); pin(vec);
        pin(qstep); pin(rstep); pin(rr); pin(cc); pin(rot); pin(rot_step); pin(dbase); pin(abase);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if constexpr (SPLIT) {
        if (threadIdx.x == 64 && my_rows) mbar_expect_tx(recv_bar, (uint32_t)(splits * my_rows * BN) * 4u);
        __syncwarp();
        cluster_arrive_relaxed();                             // this CTA's (fenced) barriers may be signalled from here on
    }
    const uint32_t tmem_base = *holder_ptr;
    pdl_wait();                                               // set-up above overlaps the previous kernel's tail
    pdl_trigger();
    if (threadIdx.x == 32) stamp_start(g.stamp);

    // Operand conversion (modes 2, 3 and 8), by warps 2-5 (and 8-11 in modes 2 and 8): MODE 3 rounds A to bf16 (the weights arrive as
    // bf16), MODE 8 to TF32 in place, MODE 2 splits both operands into bf16 hi / lo tiles.  The work of a stage is dealt to the warps in pieces of
    // 32 rows x 8 elements: a thread that converted whole rows of A and B alone paid ~3400 cycles a K block in dependent
    // instructions, most of the kernel's time (512 -> 512 F(4,3) @7, whole layer: 38.7 -> 23.5 us).
    auto convert_stages = [&](int cw) -> bool {
        uint8_t* const sm0 = smem_raw + (sbase - smem_u32(smem_raw));
        const int ga = (g.rows + 31) >> 5, gb = (BN + 31) >> 5;
        int s = 0;
        uint32_t ph = 0;
        for (int it = 0; it < nkb; ++it, s = (s + 1 == STAGES ? 0 : s + 1), ph ^= (s == 0 ? 1u : 0u)) {
            if (MODE == ROUNDED && (g.issuers == 2 ? it & 1 : 0) != cw >> 2) continue;
            if (!mbar_wait(full_bar(s), ph)) return false;
            uint8_t* const st = sm0 + s * stage_bytes;
            uint8_t* const cv = st + a_stage + (x3_mode(MODE) ? b_stage_bytes : 0u);      // converted tiles: A hi, A lo, B hi, B lo
            if constexpr (MODE == 3) {
                const int r = cw * 32 + lane;                 // a row of A per thread
                if (r < g.rows) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) convert_chunk<false>(st, cv, cv, r, c, rp);
                }
            } else if constexpr (MODE == ROUNDED) {
                const int r = (cw & 3) * 32 + lane;           // a row of A per thread, its words in another order for each of eight lanes
                if (r < g.rows) {
                    float4 v[8];                              // all loads first: the compiler keeps them behind earlier stores
#pragma unroll
                    for (int c = 0; c < 8; ++c) v[c] = *reinterpret_cast<const float4*>(st + r * 128 + ((c ^ (r & 7)) << 4));
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        *reinterpret_cast<float4*>(st + r * 128 + ((c ^ (r & 7)) << 4)) =
                            make_float4(round_tf32(v[c].x), round_tf32(v[c].y), round_tf32(v[c].z), round_tf32(v[c].w));
                }
            } else if constexpr (MODE == SPLIT_A) {
                for (int i = cw; i < 4 * gb; i += 8) {
                    const int r = (i >> 2) * 32 + lane;
                    if (r < BN) convert_chunk<true>(st + a_stage, cv, cv + b_stage_bytes / 2, r, i & 3, BN);
                }
            } else {
#pragma unroll 2
                for (int i = cw; i < 4 * (ga + gb); i += 8) {
                    const int grp = i >> 2, c = i & 3;
                    if (grp < ga) {
                        const int r = grp * 32 + lane;
                        if (r < g.rows) convert_chunk<true>(st, cv, cv + rp * 64, r, c, rp);
                    } else {
                        const int r = (grp - ga) * 32 + lane;
                        uint8_t* const bh = cv + rp * 128;
                        if (r < BN) convert_chunk<true>(st + a_stage, bh, bh + b_stage_bytes / 2, r, c, BN);
                    }
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes -> visible to the MMA's reads
            __syncwarp();
            if (lane == 0) mbar_arrive(conv_bar(s));
        }
        return true;
    };
    // Gather modes: A's tile of every K block, by eight warps.  A lane keeps its place in the row (and so its filter tap and channel)
    // for the whole block and walks the rows: reads are contiguous along the window, the swizzled row is written in one piece.
    // Issue slots bound it (per row a window, a test of the tap, an address, a load, the rounding, a store), and it replaces a pass
    // that writes the R*S-fold matrix to memory and one that reads it back: 7x7 stem of a 224 x 224 image 10.5 -> 7.6 us (bf16
    // 10.6 -> 6.5), its 3x3 one 6.0 -> 4.0, 3x3 stride-1 stem 12.1 -> 8.9; 37 -> 64 3x3 @56 10.9 -> 7.0 (bf16 8.2 -> 5.7).
    auto gather_stages = [&](int gw) -> bool {
        constexpr bool BF = bf16_mode(MODE);
        constexpr int V = MODE >= 6 ? 4 : 1;                  // consecutive channels of one load
        constexpr int E = V == 4 ? 4 : BF ? 2 : 1;            // elements of a row a lane writes
        constexpr int LPR = BKE / E, RPS = 32 / LPR;          // lanes to a row, rows a warp writes at a time
        constexpr int PITCH = GATHER_WARPS * RPS;             // rows all warps write at a time: a multiple of 8
        constexpr int STEPS = BM / (2 * PITCH);               // half a tile's rows at a time: all loads of the half, then its stores
        const int r0 = gw * RPS + lane / LPR, ql = (lane % LPR) * E;
        const uint32_t byte = (uint32_t)(ql * (BF ? 2 : 4));  // of the row: its 16-byte word is swizzled by the row
        const uint32_t dst0 = (uint32_t)r0 * 128u + (((byte >> 4) ^ (uint32_t)(r0 & 7)) << 4) + (byte & 15u);
        const char* const x = reinterpret_cast<const char*>(g.x);
        uint8_t* const sm0 = smem_raw + (sbase - smem_u32(smem_raw));
        int s = 0;
        uint32_t ph = 0;
        for (int it = 0; it < nkb; ++it, s = (s + 1 == STAGES ? 0 : s + 1), ph ^= (s == 0 ? 1u : 0u)) {
            uint32_t off[E / V], tap[E / V];
#pragma unroll
            for (int e = 0; e < E / V; ++e) {
                const int q = (kb0 + it) * BKE + ql + e, t = div_magic(q, g.ic_C, g.magic_c), c = q - t * g.ic_C;
                const int fr = div_magic(t, g.ic_S, g.magic_s), fs = t - fr * g.ic_S;
                off[e] = (uint32_t)((fr * g.ic_W + fs) * g.ic_C + c) * 4u;
                tap[e] = q < g.ic_Q ? (1u << fr | 0x10000u << fs) : 0x80000000u;   // (the row's padding reads as zero)
            }
            if (it >= STAGES && !mbar_wait(empty_bar(s), ph ^ 1u)) return false;
            const uint2* win = windows + r0;
            uint8_t* dst = sm0 + s * stage_bytes + dst0;
#pragma unroll 1
            for (int r = r0; r < g.rows; r += BM / 2, win += BM / 2, dst += BM / 2 * 128) {
                float v[STEPS][E];
#pragma unroll
                for (int u = 0; u < STEPS; ++u) {
                    const uint2 w = win[u * PITCH];
#pragma unroll
                    for (int e = 0; e < E / V; ++e) {
                        const bool in = (w.y & tap[e]) == tap[e];
                        const char* src = x + (w.x + off[e]);
                        if constexpr (V == 4) {
                            const float4 f = in ? __ldg(reinterpret_cast<const float4*>(src)) : make_float4(0.f, 0.f, 0.f, 0.f);
                            v[u][0] = f.x; v[u][1] = f.y; v[u][2] = f.z; v[u][3] = f.w;
                        } else {
                            v[u][e] = in ? __ldg(reinterpret_cast<const float*>(src)) : 0.f;
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < STEPS; ++u) {
                    if (r + u * PITCH >= g.rows) continue;
                    uint8_t* const d = dst + u * PITCH * 128;
                    if constexpr (BF) {
                        __nv_bfloat162 h[E / 2];
#pragma unroll
                        for (int e = 0; e < E / 2; ++e) h[e] = __floats2bfloat162_rn(v[u][2 * e], v[u][2 * e + 1]);
                        if constexpr (E == 4) *reinterpret_cast<uint2*>(d) = make_uint2(*reinterpret_cast<uint32_t*>(&h[0]), *reinterpret_cast<uint32_t*>(&h[1]));
                        else *reinterpret_cast<__nv_bfloat162*>(d) = h[0];
                    } else if constexpr (E == 4) {
                        *reinterpret_cast<float4*>(d) = make_float4(round_tf32(v[u][0]), round_tf32(v[u][1]), round_tf32(v[u][2]), round_tf32(v[u][3]));
                    } else {
                        *reinterpret_cast<float*>(d) = round_tf32(v[u][0]);
                    }
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes -> visible to the MMA's reads
            __syncwarp();
            if (lane == 0) mbar_arrive(full_bar(s));
        }
        return true;
    };
    // One place that runs the gathering, for the epilogue's warps and the extra ones alike: a second copy of the code for the second
    // group is fetched cold by every launch.  (The bias is fetched before it: 1x1 205 -> 96 @40 6.0 us against 6.7.)
    bool gathered = true;
    float early_bias = 0.f;
    if constexpr (gather_mode(MODE)) {
        if (warp >= 8 || (warp >= 2 && warp <= 5)) {
            const int t = (int)threadIdx.x - 64;
            if (g.bias && t < BN && n0 + t < g.N) early_bias = __ldg(g.bias + n0 + t);
            gathered = gather_stages(warp >= 8 ? warp - 4 : warp - 2);
            if (!gathered && lane == 0) atomicExch(&g_device_status, (int)NNV_ERR_TIMEOUT);
            __syncwarp();
        }
    }
    // Producers.  A load costs the thread that issues it ~165 cycles whatever its size, more than the copy engine needs for it (1.1
    // cycles a row of 128 bytes) or the MMAs of its K block: the activation's and the weights' loads come from a warp each, and where
    // warps 4 and 5 have nothing to convert they take every other block (us in a replayed graph, two loading warps / four: 64 -> 64 3x3
    // @56, 18 blocks a CTA, 5.85 / 4.56, 320 -> 1280 1x1 @7, ten, 3.34 / 3.03, 128 -> 128 3x3 @28, nine, 4.82 / 4.57, 2048 -> 512 1x1 @7,
    // eight, 4.10 / 4.14; with five and fewer the same within a few per cent either way: 160 -> 1280 @7 2.62 / 2.46, 512 -> 128 @28
    // 3.53 / 3.53, 1024 -> 256 @14 3.95 / 4.00).
    constexpr bool FOUR = MODE == 0 || MODE == 1;
    const int step = gemm_loaders(MODE, nkb, STAGES);
    auto produce = [&](bool is_a, int first_it) {
        bool ok = true;
        int s = first_it;                                     // (a ring that two loaders share has two slots or more; a slot's next block is one phase on, whosever it is)
        uint32_t ph = 0;
        const int first = min(nkb, STAGES);
        auto skip = [&]() {                                   // the other warp's block
            if (!g.ic_on || ++ic_cb != g.ic_cblk) return;
            ic_cb = 0;
            ++ic_tap;
            if (++ic_fs == g.ic_S) { ic_fs = 0; ++ic_fr; }
        };
        if (first_it) skip();
        for (int it = first_it; it < nkb; it += step) {
            if (it >= STAGES) ok = mbar_wait(empty_bar(s), ph ^ 1u);
            if (!ok) break;
            if (is_a) {
                issue_a(it, s);
            } else {
                issue_b(it, s);
                if (first_it == 0 && it < first && it + step >= first && CW && g.addend) {   // straight into the staging sub-tiles
                    const int nch = BN / CW;
                    mbar_expect_tx(addend_bar, (uint32_t)(nch * quarters) * chunk_bytes);
                    for (int j = 0; j < nch; ++j)             // (a box is as high as the tile's sub-tiles together)
                        tma_load_3d(stg0 + (uint32_t)(j * quarters) * chunk_bytes, &tmAdd, n0 + j * CW, y0, zd, addend_bar);
                }
            }
            if (FOUR && step == 2) skip();
            s += step;
            if (s >= STAGES) { s -= STAGES; ph ^= 1u; }
        }
        if (!ok) {
            atomicExch(&g_device_status, (int)NNV_ERR_TIMEOUT);
            for (int i = 0; i < 1000; ++i) __nanosleep(1000);       // let loads already in flight land
        }
    };
    if (warp == 0 || warp == 7) {
        if (!(gather_mode(MODE) && warp == 0) && elect_one()) produce(warp == 0, 0);
    } else if (warp >= 8) {
        if constexpr (x3_mode(MODE) || MODE == ROUNDED) {
            if (!convert_stages(warp - 4) && lane == 0) atomicExch(&g_device_status, (int)NNV_ERR_TIMEOUT);
        }
        __syncwarp();
        if constexpr (SPLIT) cluster_wait();
    } else if (warp == 1 || warp == 6) {
        // MMA issuers.  One thread that waits for a stage, issues its four MMAs into one accumulator and commits takes
        // ~560 cycles a K block (device-clock probes), several times what the tensor pipe needs at these tile widths, so
        // `g.issuers` warps take the K blocks in turn, each into an accumulator of its own; the epilogue adds them.
        const int iss = warp == 1 ? 0 : warp - 5;
        if (iss < g.issuers && elect_one()) {
            // instruction descriptor: fp32 accumulate, A/B format, both K-major, N, M = 128
            const uint32_t fmt = (MODE == 0 || MODE == 4 || MODE == 6 || MODE == ROUNDED) ? 2u : 1u;
            const uint32_t idesc = (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
            const uint32_t acc = tmem_base + (uint32_t)(iss * BN);
            bool ok = true;
            int s = iss % STAGES;
            uint32_t ph = (uint32_t)(iss / STAGES) & 1u;
            for (int it = iss; it < nkb; it += g.issuers) {
                ok = mbar_wait(converting_mode(MODE) ? conv_bar(s) : full_bar(s), ph);
                if (!ok) break;
                tc_fence_after();
                const uint32_t first = it != iss ? 1u : 0u;     // 0: the accumulator's first MMA overwrites it
                const uint32_t a_src = sbase + s * stage_bytes;
                if constexpr (MODE == 2) {
                    // converted tiles follow the staged ones: A_hi, A_lo (64 bytes a row), B_hi, B_lo
                    const uint32_t a_hi = a_src + a_stage + b_stage_bytes, a_lo = a_hi + rp * 64;
                    const uint32_t b_hi = a_lo + rp * 64, b_lo = b_hi + b_stage_bytes / 2;
                    const uint32_t lbo_a = (uint32_t)rp * 16u, lbo_b = (uint32_t)BN * 16u;
#pragma unroll
                    for (int kk = 0; kk < 2; ++kk) {            // 2 K-steps of 16 bf16 = 2 core matrices each
                        const uint64_t ah = make_smem_desc_plain(a_hi + kk * 2 * lbo_a, lbo_a, 128);
                        const uint64_t al = make_smem_desc_plain(a_lo + kk * 2 * lbo_a, lbo_a, 128);
                        const uint64_t bh = make_smem_desc_plain(b_hi + kk * 2 * lbo_b, lbo_b, 128);
                        const uint64_t bl = make_smem_desc_plain(b_lo + kk * 2 * lbo_b, lbo_b, 128);
                        umma<true>(acc, al, bh, idesc, kk ? 1u : first);   // small terms first
                        umma<true>(acc, ah, bl, idesc, 1u);
                        umma<true>(acc, ah, bh, idesc, 1u);
                    }
                } else if constexpr (MODE == SPLIT_A) {
                    const uint32_t b_hi = a_src + a_stage + b_stage_bytes, b_lo = b_hi + b_stage_bytes / 2, lbo_b = (uint32_t)BN * 16u;
                    const uint64_t adesc = make_smem_desc(a_src);      // a row: 64 bytes of hi, 64 of lo
#pragma unroll
                    for (int kk = 0; kk < 2; ++kk) {
                        const uint64_t ah = adesc + (uint64_t)(kk * 2), al = adesc + (uint64_t)(4 + kk * 2);
                        const uint64_t bh = make_smem_desc_plain(b_hi + kk * 2 * lbo_b, lbo_b, 128);
                        const uint64_t bl = make_smem_desc_plain(b_lo + kk * 2 * lbo_b, lbo_b, 128);
                        umma<true>(acc, al, bh, idesc, kk ? 1u : first);   // small terms first
                        umma<true>(acc, ah, bl, idesc, 1u);
                        umma<true>(acc, ah, bh, idesc, 1u);
                    }
                } else if constexpr (MODE == 3) {
                    const uint32_t a_bf = a_src + a_stage, lbo_a = (uint32_t)rp * 16u;
                    const uint64_t bdesc = make_smem_desc64(a_bf + rp * 64);
#pragma unroll
                    for (int kk = 0; kk < 2; ++kk)             // 2 K-steps of 16 bf16 = 2 core matrices (32 bytes) each
                        umma<true>(acc, make_smem_desc_plain(a_bf + kk * 2 * lbo_a, lbo_a, 128), bdesc + (uint64_t)(kk * 2), idesc,
                                   kk ? 1u : first);
                } else {
                    const uint64_t adesc = make_smem_desc(a_src);
                    const uint64_t bdesc = make_smem_desc(a_src + a_stage);
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)             // 4 MMAs of 32 bytes of K each
                        umma<bf16_mode(MODE)>(acc, adesc + (uint64_t)(kk * 2), bdesc + (uint64_t)(kk * 2), idesc, kk ? 1u : first);
                }
                if (it + STAGES < nkb) umma_commit(empty_bar(s));
                s += g.issuers;
                while (s >= STAGES) { s -= STAGES; ph ^= 1u; }
            }
            if (ok) umma_commit(tmem_full_bar);
            else atomicExch(&g_device_status, (int)NNV_ERR_TIMEOUT);
        }
    } else {
        const int c = (int)threadIdx.x - 64;
        float bias = early_bias;
        if constexpr (!gather_mode(MODE)) bias = (g.bias && c < BN && n0 + c < g.N) ? __ldg(g.bias + n0 + c) : 0.f;
        if constexpr (FOUR)
            if (step == 2 && warp >= 4 && elect_one()) produce(warp == 4, 1);
        __syncwarp();
        if constexpr (converting_mode(MODE)) gathered = convert_stages(warp - 2);
        if (c < BN) *reinterpret_cast<float*>(smem_raw + (sbias - smem_u32(smem_raw)) + 4 * c) = bias;
        __syncwarp();
        if (lane == 0) mbar_arrive(bias_bar);
    }
    __syncwarp();
    if (warp < 8) {
        // Write-out, by the eight warps that led here: the TMEM lanes a warp may read are those of its number modulo four, so each
        // quarter of the tile's rows has two (one of warps 2-5, one of the producers and issuers, whose work is done by then),
        // which take the column chunks in turn.
        bool ok = gathered;
        auto act4 = [&](float4& v) {
            if (g.act) {
                const float hi = g.act == 2 ? 6.f : INFINITY;
                v.x = fminf(fmaxf(v.x, 0.f), hi); v.y = fminf(fmaxf(v.y, 0.f), hi);
                v.z = fminf(fmaxf(v.z, 0.f), hi); v.w = fminf(fmaxf(v.w, 0.f), hi);
            }
        };
        auto wait_acc = [&]() {
            ok = ok && mbar_wait(bias_bar, 0) && mbar_wait(tmem_full_bar, 0);
            if constexpr (!SPLIT)
                if (g.addend && CW) ok = ok && mbar_wait(addend_bar, 0);
            tc_fence_after();
            if (!ok && lane == 0) atomicExch(&g_device_status, (int)NNV_ERR_TIMEOUT);
            ok = __all_sync(0xffffffffu, ok);
        };
        const uint32_t tacc = tmem_base + tacc_off;
        const bool two = min(g.issuers, nkb) > 1;
        // 16 accumulator columns of this lane's row, the issuers' accumulators added in order
        auto acc16 = [&](int c0, float (&v)[16]) {
            uint32_t r[16], q[16];
            tmem_ld16_nowait(tacc + (uint32_t)c0, r);
            tmem_ld16_nowait(tacc + (uint32_t)(two ? BN + c0 : c0), q);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = two ? __uint_as_float(r[i]) + __uint_as_float(q[i]) : __uint_as_float(r[i]);
        };
        if constexpr (!SPLIT) {
            // Per 16 columns: lane = one accumulator row, TMEM -> registers -> (+ bias, + addend from the staging sub-tile, activation) ->
            // staging sub-tile; then its rows from there to memory, 64 bytes each.  (One compact loop: code that a launch runs once
            // costs more to fetch than to execute.)  Large outputs of two K blocks and no residual were faster by tiled stores of 32 columns
            // (us, those / this: 32 -> 256 1x1 @112 BF16 5.2 / 6.2, 64 -> 640 @80 7.8 / 8.5, F(2,3) 32 -> 480 @113x120 56.7 / 58.5), with a residual
            // slower (64 -> 256 @180 TF32 21.3 / 17.9).  Whole lines stored by a quarter's two warps together give half of it back and cost
            // small layers 1 - 5 % (resident ResNet-18-shaped inference, F(4,3), 214 -> 220).
            if (CW && grp * 16 < BN) {
                wait_acc();
                if (ok && rows_live > 0) {
                    const uint32_t sub_step = 2u * (uint32_t)quarters * chunk_bytes;
#pragma unroll 1
                    for (int c0 = grp * 16; c0 < BN; c0 += 32, out_sub += sub_step, out_dst += 32) {
                        float v[16];
                        acc16(c0, v);
                        const uint32_t row0 = out_sub + (uint32_t)lane * 64u, swz = (uint32_t)((lane >> 1) & 3) << 4;
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const float4 bb = lds128(sbias + (uint32_t)(c0 + 4 * c) * 4u);
                            v[c * 4] += bb.x; v[c * 4 + 1] += bb.y; v[c * 4 + 2] += bb.z; v[c * 4 + 3] += bb.w;
                        }
                        if (g.addend) {
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                const float4 aa = lds128(row0 + (((uint32_t)c << 4) ^ swz));
                                v[c * 4] += aa.x; v[c * 4 + 1] += aa.y; v[c * 4 + 2] += aa.z; v[c * 4 + 3] += aa.w;
                            }
                        }
                        if (g.act) {
                            const float hi = g.act == 2 ? 6.f : INFINITY;
#pragma unroll
                            for (int c = 0; c < 16; ++c) v[c] = fminf(fmaxf(v[c], 0.f), hi);
                        }
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            sts128(row0 + (((uint32_t)c << 4) ^ swz), make_float4(v[c * 4], v[c * 4 + 1], v[c * 4 + 2], v[c * 4 + 3]));
                        __syncwarp();
                        const int r1 = lane >> 2, w1 = lane & 3;
                        const uint32_t src = out_sub + (uint32_t)r1 * 64u + (uint32_t)((w1 ^ ((r1 >> 1) & 3)) << 4);
                        if (n0 + c0 + 4 * w1 < g.N) {
                            float4 q[4];
#pragma unroll
                            for (int i = 0; i < 4; ++i) q[i] = lds128(src + (uint32_t)i * 512u);
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                if (r1 + i * 8 < rows_live) *reinterpret_cast<float4*>(out_dst + (long long)(i * 8) * g.ldd) = q[i];
                        }
                    }
                }
            } else if (!CW) {
                wait_acc();
                if (ok) {
                    const int m = m0 + quarter * 32 + lane;
                    float* drow = g.D + (long long)b * g.strideD + (long long)m * g.ldd;
                    const float* arow = g.addend ? g.addend + (long long)m * g.ldd : nullptr;
                    const bool row_live = quarter * 32 + lane < live;
#pragma unroll 1
                    for (int c0 = grp * 16; c0 < BN; c0 += (c0 & 8) ? 24 : 8) {
                        uint32_t r[8], q[8];
                        tmem_ld8_nowait(tacc + (uint32_t)c0, r);
                        tmem_ld8_nowait(tacc + (uint32_t)(two ? BN + c0 : c0), q);
                        tmem_wait_ld();
                        float aa[8];                          // eight addends at a time: one by one, behind the stores, each would wait for memory
#pragma unroll
                        for (int j = 0; j < 8; ++j) aa[j] = arow && row_live && n0 + c0 + j < g.N ? __ldg(arow + n0 + c0 + j) : 0.f;
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const int n = n0 + c0 + j;
                            if (row_live && n < g.N) {
                                float bb;
                                asm volatile("ld.shared.f32 %0, [%1];" : "=f"(bb) : "r"(sbias + (uint32_t)(c0 + j) * 4u) : "memory");
                                const float v = two ? __uint_as_float(r[j]) + __uint_as_float(q[j]) : __uint_as_float(r[j]);
                                drow[n] = act_fn(arow ? v + bb + aa[j] : v + bb, g.act);
                            }
                        }
                    }
                }
            }
        } else {
            // Split K, sender: park the partial tile in the stage ring (idle by then) as rows of BN words, the 16-byte words
            // of a row rotated by its index so that the lanes' stores meet different banks, and let the copy engine push
            // every owner its rows of this quarter's 32.  Owner: the rows arrive from every CTA of the cluster (its own
            // included); they are added in rank order (a fixed order: the result does not depend on timing), bias /
            // residual / activation are applied and row-contiguous 128-bit words are stored.
            const int q0 = quarter * 32;
            cluster_wait();                                   // every CTA's barriers are initialised
            wait_acc();
            if (ok && q0 < live) {
#pragma unroll 1
                for (int c0 = grp * 16; c0 < BN; c0 += 32) {
                    float v[16];
                    acc16(c0, v);
                    int pos = rot0 + (c0 >> 2);
                    if (pos >= nch) pos -= nch;
#pragma unroll
                    for (int j = 0; j < 16; j += 4) {
                        if (q0 + lane < live) sts128(prow + (uint32_t)pos * 16u, make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]));
                        pos = pos + 1 == nch ? 0 : pos + 1;
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes -> visible to the bulk copies
            }
            __syncwarp();
            asm volatile("barrier.sync %0, 64;" ::"r"(2 + quarter) : "memory");    // both warps' columns of these rows are parked
            if (ok && push_bytes) bulk_push(push_dst, push_src, push_bytes, push_bar);
            int total = my_rows * nch;
            // (the residual's words are fetched one step ahead, the first ones while the rows are on their way)
            auto fetch_addend = [&](int idx) {
                return vec && abase && idx < total && n0 + cc * 4 < g.N ? __ldg(reinterpret_cast<const float4*>(abase + (long long)rr * g.ldd + cc * 4))
                                                                        : make_float4(0.f, 0.f, 0.f, 0.f);
            };
            float4 ahead = fetch_addend(t);
            if (my_rows && !mbar_wait(recv_bar, 0)) {
                if (lane == 0) atomicExch(&g_device_status, (int)NNV_ERR_TIMEOUT);
                total = 0;
            }
            __syncwarp();
            cluster_arrive_relaxed();                         // this CTA's rows have arrived: their senders may leave
            const uint32_t recv = sbase + g.recv_off, part_stride = (uint32_t)(rows_per * BN) * 4u;
            auto reduce = [&](auto nsplits) {
                constexpr int NS = decltype(nsplits)::value;
#pragma unroll 1
                for (int idx = t; idx < total; idx += 256) {
                    const int p = cc + rot >= nch ? cc + rot - nch : cc + rot;
                    const uint32_t src = recv + (uint32_t)(rr * BN) * 4u + (uint32_t)p * 16u;
                    constexpr int NB = NS < 8 ? NS : 8;       // loads in flight
                    float4 v[NB];
#pragma unroll
                    for (int rk = 0; rk < NB; ++rk) v[rk] = lds128(src + (uint32_t)rk * part_stride);
                    float4 o = lds128(sbias + (uint32_t)cc * 16u);
                    const int n = cc * 4;
                    const long long off = (long long)rr * g.ldd + n;
                    const float4 aa = ahead;
                    rr += qstep; cc += rstep; rot += rot_step;
                    if (cc >= nch) { cc -= nch; ++rr; ++rot; }
                    if (rot >= nch) rot -= nch;
                    ahead = fetch_addend(idx + 256);
                    float4 a = v[0];
#pragma unroll
                    for (int rk = 1; rk < NB; ++rk) { a.x += v[rk].x; a.y += v[rk].y; a.z += v[rk].z; a.w += v[rk].w; }
                    if constexpr (NS > 8) {
#pragma unroll
                        for (int rk = 0; rk < 8; ++rk) v[rk] = lds128(src + (uint32_t)(rk + 8) * part_stride);
#pragma unroll
                        for (int rk = 0; rk < 8; ++rk) { a.x += v[rk].x; a.y += v[rk].y; a.z += v[rk].z; a.w += v[rk].w; }
                    }
                    o.x += a.x; o.y += a.y; o.z += a.z; o.w += a.w;
                    if (n0 + n < g.N) {
                        if (vec) {
                            if (abase) { o.x += aa.x; o.y += aa.y; o.z += aa.z; o.w += aa.w; }
                            act4(o);
                            *reinterpret_cast<float4*>(dbase + off) = o;
                        } else {
                            const float vv[4] = {o.x, o.y, o.z, o.w};
                            for (int j = 0; j < 4 && n0 + n + j < g.N; ++j)
                                dbase[off + j] = act_fn(abase ? vv[j] + __ldg(abase + off + j) : vv[j], g.act);
                        }
                    }
                }
            };
            if (splits == 16) reduce(std::integral_constant<int, 16>());
            else if (splits == 8) reduce(std::integral_constant<int, 8>());
            else if (splits == 4) reduce(std::integral_constant<int, 4>());
            else reduce(std::integral_constant<int, 2>());
        }
    }
    __syncwarp();
    if constexpr (SPLIT) {
        if (warp >= 8) cluster_arrive_relaxed();
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

#include "conv3x3_tc.cuh"
#include "conv3x3_bf16.cuh"
#include "gemm_sp.cuh"
#include "wino_fused.cuh"
#include "inverted_bottleneck.cuh"

// ---- host side --------------------------------------------------------------------------------
PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
PFN_cuTensorMapEncodeIm2col_v12000 g_encode_im2col = nullptr;
std::once_flag g_encode_once;
cudaError_t g_encode_err = cudaSuccess;

nnv_status_t get_encoder() {
    std::call_once(g_encode_once, [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        g_encode_err = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q);
        if (g_encode_err == cudaSuccess && q == cudaDriverEntryPointSuccess) g_encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
        void* fn2 = nullptr;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeIm2col", &fn2, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            g_encode_im2col = (PFN_cuTensorMapEncodeIm2col_v12000)fn2;
    });
    NNV_REQUIRE(g_encode != nullptr, NNV_ERR_CUDA, "cuTensorMapEncodeTiled is not available from this driver");
    return NNV_OK;
}

// 3-D map over a K-major operand: dims {Kd, rows, batch}, box {128 bytes of K, box_rows, 1}.
nnv_status_t encode_operand(CUtensorMap* map, const void* base, bool bf16, int Kd, int rows, int batch, int64_t ld,
                            int64_t batch_stride, int box_rows) {
    const uint64_t es = bf16 ? 2 : 4;
    NNV_REQUIRE((reinterpret_cast<uintptr_t>(base) & 15) == 0, NNV_ERR_INVALID_ARG, "GEMM operand is not 16-byte aligned");
    NNV_REQUIRE((ld * es) % 16 == 0 && (batch_stride * es) % 16 == 0, NNV_ERR_INVALID_ARG,
                "GEMM operand strides must be multiples of 16 bytes");
    cuuint64_t dims[3] = {(cuuint64_t)Kd, (cuuint64_t)rows, (cuuint64_t)batch};
    cuuint64_t strides[2] = {(cuuint64_t)(ld * es), (cuuint64_t)(batch_stride * es)};
    cuuint32_t box[3] = {(cuuint32_t)(BK_BYTES / es), (cuuint32_t)box_rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = g_encode(map, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3,
                          const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                          CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    NNV_REQUIRE(r == CUDA_SUCCESS, NNV_ERR_CUDA, "cuTensorMapEncodeTiled failed with code %d", (int)r);
    return NNV_OK;
}

// 3-D map over the residual addend (the output's geometry): dims {N, M, batch}, boxes of 16 columns, 64-byte swizzle, x `box_rows`
// rows: what a column chunk's staging sub-tiles hold together.
nnv_status_t encode_addend_tiles(CUtensorMap* map, const void* base, int N, int M, int batch, int64_t ld, int64_t batch_stride, int box_rows) {
    cuuint64_t dims[3] = {(cuuint64_t)N, (cuuint64_t)M, (cuuint64_t)batch};    // or {N, rows of a tile, tiles}
    cuuint64_t strides[2] = {(cuuint64_t)(ld * 4), (cuuint64_t)(batch_stride * 4)};
    cuuint32_t box[3] = {16, (cuuint32_t)box_rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(base), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    NNV_REQUIRE(r == CUDA_SUCCESS, NNV_ERR_CUDA, "cuTensorMapEncodeTiled (residual tiles) failed with code %d", (int)r);
    return NNV_OK;
}

// 4-D im2col map over an NHWC fp32 activation {C, W, H, 1}: 32 channels x `pixels` output pixels per load.
nnv_status_t encode_im2col_operand(CUtensorMap* map, const void* base, int C, int H, int W, int R, int S, int stride,
                                   int pad, int pixels) {
    NNV_REQUIRE(g_encode_im2col != nullptr, NNV_ERR_CUDA, "cuTensorMapEncodeIm2col is not available from this driver");
    NNV_REQUIRE((reinterpret_cast<uintptr_t>(base) & 15) == 0 && (C % 4) == 0, NNV_ERR_INVALID_ARG,
                "implicit-GEMM activation must be 16-byte aligned with C a multiple of 4");
    cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)H, 1};
    cuuint64_t strides[3] = {(cuuint64_t)C * 4, (cuuint64_t)W * C * 4, (cuuint64_t)H * W * C * 4};
    int lower[2] = {-pad, -pad};
    int upper[2] = {pad - (S - 1), pad - (R - 1)};
    cuuint32_t estr[4] = {1, (cuuint32_t)stride, (cuuint32_t)stride, 1};
    CUresult r = g_encode_im2col(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<void*>(base), dims, strides, lower,
                                 upper, 32, pixels, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                 CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    NNV_REQUIRE(r == CUDA_SUCCESS, NNV_ERR_CUDA, "cuTensorMapEncodeIm2col failed with code %d", (int)r);
    return NNV_OK;
}

// 3-D tiled map over an NHWC fp32 activation {C, W, H}: boxes of 32 channels x `box_w` pixels x `box_h`
// rows (the halo boxes of conv3x3_tc_kernel); coordinates outside the image read as zero.
nnv_status_t encode_halo_operand(CUtensorMap* map, const void* base, int C, int H, int W, int box_h, int box_w = 8) {
    NNV_REQUIRE((reinterpret_cast<uintptr_t>(base) & 15) == 0 && (C % 4) == 0, NNV_ERR_INVALID_ARG,
                "activation must be 16-byte aligned with C a multiple of 4");
    cuuint64_t dims[3] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)H};
    cuuint64_t strides[2] = {(cuuint64_t)C * 4, (cuuint64_t)W * C * 4};
    cuuint32_t box[3] = {32, (cuuint32_t)box_w, (cuuint32_t)box_h};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(base), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    NNV_REQUIRE(r == CUDA_SUCCESS, NNV_ERR_CUDA, "cuTensorMapEncodeTiled (halo boxes) failed with code %d", (int)r);
    return NNV_OK;
}

// Shared memory of a cluster's CTA is at least the share of the SM's 228 KB (1 KB of it the system's) that its TMEM columns are of
// 512, so that CTAs that fit an SM find their columns free, whichever launches they come from.  tcgen05.alloc waits without a limit:
// where more CTAs fit than have columns, each of three clusters may hold columns on some SMs and wait for them on another.
// (A CTA without a cluster waits for nobody else once it has its columns and needs no such rule.)
constexpr size_t tmem_share_bytes(int cols) { return (size_t)228 * 1024 * cols / 512 - 1024; }

// Tiling of conv3x3_tc_kernel for one layer.
struct ConvTiling { int MT, BN, splits, na, nb, tmem_cols; size_t smem; };

// Bytes of one halo-box slot and one weight-tile slot.
size_t conv_a_slot(int MT) { return (size_t)(16 * MT + 2) * 1024; }
size_t conv_b_slot(int BN) { return (size_t)BN * BK_BYTES; }

size_t conv_smem_bytes(int MT, int BN, int na, int nb) {
    return (size_t)1024 + (size_t)na * conv_a_slot(MT) + (size_t)nb * conv_b_slot(BN) + 8 * (2 * CONV_MAX_NA + 2 * CONV_MAX_NB + 2);
}

// Fills in ring depths (unless given), shared-memory size and TMEM columns; false if the tiling does
// not fit (shared memory, or room to park the partial tiles of a K split).
bool finish_conv_tiling(ConvTiling* t) {
    const size_t park = t->splits > 1 ? (size_t)t->MT * BM * (t->BN + 4) * 4 : 0;
    auto rings = [&] { return (size_t)t->na * conv_a_slot(t->MT) + (size_t)t->nb * conv_b_slot(t->BN); };
    if (t->na <= 0 || t->nb <= 0) {
        t->na = 2; t->nb = 3;
        while (rings() < park && t->nb < CONV_MAX_NB) ++t->nb;      // deeper rings only to make room for the parked tiles
        while (rings() < park && t->na < CONV_MAX_NA) ++t->na;
    }
    t->tmem_cols = 32;
    while (t->tmem_cols < t->MT * t->BN) t->tmem_cols *= 2;
    t->smem = conv_smem_bytes(t->MT, t->BN, t->na, t->nb);
    if (t->splits > 1) t->smem = std::max(t->smem, tmem_share_bytes(t->tmem_cols));
    return t->smem <= 200u * 1024u && rings() >= park;
}

// CTAs that run at once in clusters of `splits`, `occ` to an SM: whole clusters must find room inside one GPC (as
// cudaOccupancyMaxActiveClusters reports).
int cluster_slots(int splits, int occ) {
    static constexpr int slots[5][3] = {{148, 296, 444}, {148, 296, 444}, {132, 284, 416}, {120, 264, 384}, {112, 224, 336}};
    return slots[splits == 16 ? 4 : splits == 8 ? 3 : splits == 4 ? 2 : splits - 1][std::min(occ, 3) - 1];
}

uint32_t gemm_stage_bytes(int mode, int bn, int rows) {
    return mode == GEMM_X3 ? stage_bytes_of<2>(bn, rows) : mode == SPLIT_A ? stage_bytes_of<SPLIT_A>(bn, rows) : mode == GEMM_BF16_CVT ? stage_bytes_of<3>(bn, rows) : stage_bytes_of<0>(bn, rows);
}

// Ring depth: 8 stages when every CTA has an SM to itself (a lone CTA needs that many loads in flight on weights that come
// cold from HBM), 4 when several share one, and no more than the K blocks a CTA walks: the shared memory left over lets
// the next kernel's CTAs in early (warm ResNet-50-shaped inference 426 -> 415 us).
int gemm_ring(int mode, int bn, int rows, long long ctas, int nkb) {
    const int sb = (int)gemm_stage_bytes(mode, bn, rows);
    // (X3 stages are twice as large: as many as fit one CTA, or two CTAs on an SM)
    if (x3_mode(mode)) return std::max(2, std::min({4, (ctas <= 148 ? 200 : 104) * 1024 / sb, nkb}));
    const int most = (ctas <= 148 && 8 * sb <= 200 * 1024) ? 8 : 4;
    return std::max(2, std::min(most, nkb));
}

// Tiling of gemm_tc_kernel: waves x (K blocks per CTA x time per block + start and write-out).  A K block costs a CTA the issue of
// its MMAs (or the wait for its conversion) whatever BN <= 128 is, or the fill of its shared memory (per SM, and from L2 over all
// SMs); a split adds the pushes of the partial rows.  Constants (microseconds) fitted to sweeps of every BN and split, chained
// launches, by the excess of the chosen tilings over the best measured ones: TF32 1.3 % over 213 layers (the former constants 2.1 %),
// BF16 operands 0.4 % over 28 (1.8 %), BF16 math on fp32 activations 1.3 % over 79 (3.7 %).
// A gather mode's K block takes the eight warps time for every row, most of it in steps of half a tile; a second CTA on the SM adds
// `share` of it.  Its tiles may be lower than 128 rows (any height that divides M), which spreads the rows over more SMs.  Fitted the
// same way over 33 shapes: the chosen tilings are 3 % above the best measured ones on average.
// X3's K block waits for the split of its operands (by pieces of 32 rows), most of which a second CTA on the SM overlaps: fitted over
// 106 F(4,3) / F(6,3) layers with A split already, 0.2 % above the best measured tilings on average, and 23 without, 1.3 %.
// Mode 8's K block waits for the rounding; CTAs that share an SM count by the clusters that fit (clusters of 16 put 128 CTAs on 112
// places): fitted to 34 layers, 0.6 % above the best measured tilings (the TF32 constants: 5.6 %).
// Output rows that are no multiple of 16 bytes are stored word by word from the accumulator's layout, a line for every row and word, by
// unsplit launches (split ones store what they have added row by row): 0.1 us a column of 128 rows and resident CTA, fitted to 56 layers
// with and without a residual.  The chosen tilings are 2.8 % above the best measured ones on average, 7.5 % without: 24 -> 67 3x3/2 @69
// with a residual 7.6 us unsplit, 4.6 in two splits.  (Not the tile GEMMs of Winograd layers, whose many short CTAs hide the stores:
// 160 -> 410 F(4,3) @81 64 us unsplit, 83 in splits.)
struct TilingCost { double fixed, block, sm_rate, l2_rate, start, column, shared_column, split, split_word; };
constexpr TilingCost tiling_cost(int mode) {
    return gather_mode(mode) ? TilingCost{0.87, 0.146, 108e3, 10.9e6, 1.85, 0.0093, 0.0, 0.28, 1.22e-4}
           : mode == SPLIT_A ? TilingCost{1.87, 0.434, 28.2e3, 7.4e6, 0.0, 0.0098, 0.0, 1.46, 2.4e-5}
           : mode == 2       ? TilingCost{1.87, 0.91, 27.2e3, 6.9e6, 0.0, 0.0188, 0.0, 1.47, 0.9e-5}
           : mode == ROUNDED ? TilingCost{1.87, 0.146, 108e3, 10.9e6, 0.80, 0.0093, 0.0, 0.26, 1.22e-4}
           : mode == 1       ? TilingCost{1.87, 0.366, 26.8e3, 2.9e6, 0.0, 0.0022, 0.0, 0.0, 2.32e-3}
           : mode == 3       ? TilingCost{1.87, 0.372, 48.9e3, 5.02e6, 0.0, 0.0065, 0.0, 0.67, 1.53e-4}
                             : TilingCost{1.87, 0.10, 114e3, 11.8e6, 2.97, 0.010, 0.0247, 0.546, 1.69e-4};
}
struct GemmTiling { int BN, splits, rows, waves; };
GemmTiling search_gemm_tiling(int mode, int M, int N, int batch, int nkb) {
    constexpr struct { double row_us, share; } gather[4] = {{0.0064, 0.36}, {0.0054, 0.60}, {0.0025, 0.81}, {0.0042, 0.40}};   // modes 4 - 7
    const bool x3 = x3_mode(mode);
    const bool rounded = mode == ROUNDED;
    const TilingCost c = tiling_cost(mode);
    const int least = ceil_div(M, BM);
    const int most = gather_mode(mode) ? std::max(least, std::min(M / 16, 296)) : least;
    GemmTiling best{16, 1, gemm_rows(M), 1};
    double best_t = 1e30;
    for (int m_tiles = least; m_tiles <= most; ++m_tiles) {
        if (m_tiles != least && M % m_tiles != 0) continue;
        const int rows = M % m_tiles == 0 ? M / m_tiles : BM;
        for (int bn = 16; bn <= std::min(128, ceil_div(N, 16) * 16); bn += bn < 64 ? 16 : 32) {
            const double kb_bytes = (double)(rows * BK_BYTES + bn * BK_BYTES);
            for (int sp = 1; sp <= 16 && sp <= nkb; sp *= 2) {
                const long long ctas = (long long)m_tiles * ceil_div(N, bn) * batch * sp;
                const int nk = ceil_div(nkb, sp), ring = gemm_ring(mode, bn, rows, ctas, nk);
                int tmem = 32;
                while (tmem < 2 * bn) tmem *= 2;
                const double smem = 2048.0 + (double)ring * gemm_stage_bytes(mode, bn, rows) + (sp > 1 ? 4.0 * rows * bn : 0.0);
                const int occ = std::max(1, std::min({mode == 2 || mode >= 4 ? 2 : 3, (int)(226.0 * 1024.0 / smem), 512 / tmem}));
                const long long slots = cluster_slots(sp, occ);
                const double waves = (double)((ctas + slots - 1) / slots);
                const int lone = rounded ? cluster_slots(sp, 1) : 148;
                const double res = (double)std::min<long long>(occ, (ctas + lone - 1) / lone);
                double kb = std::max({c.block * res, kb_bytes * res / c.sm_rate, kb_bytes * (double)std::min(ctas, slots) / c.l2_rate});
                if (x3) kb = std::max(kb, (0.40 + 0.07 * ((mode == 2 ? ceil_div(rows, 32) : 0) + ceil_div(bn, 32))) * (1 + 0.15 * (res - 1)));
                if (gather_mode(mode))
                    kb = std::max(kb, (0.2 + gather[mode & 3].row_us * (0.65 * 64 * ceil_div(rows, 64) + 0.35 * rows)) * (1 + gather[mode & 3].share * (res - 1)));
                if (rounded) kb = std::max(kb, (0.25 + 0.0005 * rows) * (1 + 0.8 * (res - 1)));
                const double split = sp > 1 ? c.split + c.split_word * bn * rows * res : 0.0;
                const double ragged = sp == 1 && batch == 1 && (N & 3) ? 0.1 * res * std::min(bn, N) * rows / BM : 0.0;
                const double t = c.fixed + waves * (nk * kb + c.start + (c.column + c.shared_column * (res - 1)) * bn + split + ragged);
                if (t < best_t - 1e-9) { best_t = t; best = GemmTiling{bn, sp, rows, (int)waves}; }
            }
        }
    }
    return best;
}

// The search takes the host longer than the rest of a launch: a thread remembers its latest answers.
GemmTiling pick_gemm_tiling(int mode, int M, int N, int batch, int nkb) {
    struct Entry { int mode = -1, M, N, batch, nkb; GemmTiling t; };
    static thread_local Entry table[128];
    const uint32_t h = ((uint32_t)M * 2654435761u) ^ ((uint32_t)N * 40503u) ^ ((uint32_t)nkb * 9176u) ^ (uint32_t)(batch * 31 + mode);
    Entry& e = table[(h ^ (h >> 15)) & 127u];
    if (e.mode != mode || e.M != M || e.N != N || e.batch != batch || e.nkb != nkb)
        e = Entry{mode, M, N, batch, nkb, search_gemm_tiling(mode, M, N, batch, nkb)};
    return e.t;
}

// The TF32 halo kernel's tiling, if it is to be used: one MMA tile per CTA, channel tiles of up to 128, two or one box slots and three
// weight tiles (two or three CTAs then share an SM, and one CTA's fill and write-out overlap another's MMAs).  It moves fewer operand
// bytes than the implicit GEMM but has one issuing thread where that has two, and its K split is dear.  Of the tilings the one with
// the least estimated time (us), if that is below the GEMM's: waves x (channel blocks per CTA x time per block + start and write-out).
// A block's time depends on the CTAs that share the SM and on the box slots, 2.4 with an SM to itself, 3.1 for two (2.7 at 64 columns),
// 5.2 for three on one slot; an even spread is not to be had with room for three CTAs to an SM or in clusters of eight.  A K block of
// the GEMM is 0.155 at 64 columns, 0.235 at 128, 0.32 with two CTAs to an SM.  Where the GEMM's tiles need a second wave the halo kernel
// is always ahead.  A K split runs in one wave of whole clusters or not at all: a second one costs as much as the first (72 clusters of
// four on 71 places: 384 -> 512 @48 34.7 us, with one box slot and three CTAs to an SM 27.4).
// The halo kernel's figures are fitted to 240 layers (64 - 768 channels, 28 - 224 pixels a side), the GEMM's to 20.  Measured, halo kernel
// / implicit GEMM: 64 -> 64 @224 12.1 / 16.3, 128 -> 256 @112 18.1 / 20.4, 512 -> 512 @72 54 / 74, 768 -> 64 @112 29.8 / 34.6, 512 -> 256
// @56 23.0 / 22.7; the GEMM's: 128 -> 128 @112 13.6 / 11.6, 256 -> 256 @56 16.9 / 14.7, 384 -> 512 @48 21.6 / 18.9, 192 -> 192 @96 17.1 / 13.9,
// 512 -> 512 @28 15.7 / 14.0.
double halo_us(const ConvTiling& t, long long tiles, int cblk) {
    const int occ = std::max(1, std::min({(int)(227u * 1024u / (t.smem + 1024)), 512 / t.tmem_cols, 3}));
    const long long ctas = tiles * t.splits, slots = cluster_slots(t.splits, occ);
    if (t.splits > 1 && ctas > slots) return 1e30;
    const int r = t.splits == 8 ? occ : (int)std::min<double>(occ, std::ceil((double)ctas / cluster_slots(t.splits, 1) + (occ == 3 ? 0.3 : 0.0)));
    const double bn = t.BN;
    const double block = t.na >= 2 ? (r == 1 ? 2.44 : r == 2 ? std::max(2.44, 2.25 + 0.00625 * bn) : std::max(2.6, 2.6 + 0.0164 * bn))
                                   : (r == 1 ? 2.6 + 0.0057 * bn : r == 2 ? 2.5 + 0.0125 * bn : 5.2);
    const double rest = t.splits == 1 ? 3.5 + 0.0155 * bn : t.splits == 2 ? 5.4 + 0.06 * bn : t.splits == 4 ? 5.0 + 0.045 * bn : 5.8 + 0.045 * bn;
    return (double)((ctas + slots - 1) / slots) * (ceil_div(cblk, t.splits) * block + rest);
}
bool pick_conv_tiling(int C, int H, int W, int N, const GemmTiling& gemm, ConvTiling* out) {
    const int cblk = ceil_div(C, 32), BN = std::min(128, ceil_div(N, 16) * 16);
    const long long tiles = (long long)ceil_div(H, 16) * ceil_div(W, 8) * ceil_div(N, BN);
    double best = 1e30;
    if (gemm.waves == 1) {
        const long long ctas = (long long)ceil_div(H * W, gemm.rows) * ceil_div(N, gemm.BN) * gemm.splits;
        best = ceil_div(9 * cblk, gemm.splits) * (ctas <= 148 ? 0.075 + 0.00125 * gemm.BN : 0.324) + 1.98 + 0.023 * gemm.BN +
               (gemm.splits == 1 ? 0.0 : gemm.splits == 2 ? 0.64 + 0.0137 * gemm.BN : 1.02 + 0.0021 * gemm.BN);
    }
    bool found = false;
    for (int splits = 1; splits <= 8 && splits <= cblk; splits *= 2)
        for (int na = 2; na >= 1; --na) {
            ConvTiling c{};
            c.MT = 1; c.BN = BN; c.splits = splits; c.na = na; c.nb = 3;
            if (!finish_conv_tiling(&c)) continue;
            const double t = halo_us(c, tiles, cblk);
            if (t < best - 1e-9) { best = t; *out = c; found = true; }
        }
    return found;
}

// Ring, issuers and shared-memory layout of one launch of gemm_tc_kernel (host arithmetic only; `mode` is the kernel's).
struct GemmShape {
    int BN, splits, rows, m_tiles, issuers, ring, tmem_cols;
    uint32_t bar_off, recv_off, stage_off;
    size_t smem_bytes;
};

nnv_status_t gemm_shape(int mode, const GemmTiling& tile, int M, int N, int batch, int nkb, bool staged, bool addend, GemmShape* out) {
    GemmShape g{};
    const Tuning& tn = tuning();
    g.BN = tile.BN; g.splits = tile.splits; g.rows = tile.rows;
    g.m_tiles = ceil_div(M, g.rows);
    if (tn.gemm_bn && tn.gemm_splits <= nkb) { g.BN = tn.gemm_bn; g.splits = tn.gemm_splits; }   // override (nnv_tuning_set)
    // (BF16 on fp32 activations: two MMAs a K block wait for the conversion, not for their issuer; one accumulator then adds the
    // blocks in order, and 3x3/2 256 -> 512 @28 takes 8.4 us against 8.5, 5x5 64 -> 64 @56 8.8 against 8.9)
    g.issuers = mode == GEMM_BF16_CVT ? 1 : 2;
    g.tmem_cols = 32;
    while (g.tmem_cols < g.BN * g.issuers) g.tmem_cols *= 2;
    const bool split = g.splits > 1;
    const size_t sb = gemm_stage_bytes(mode, g.BN, g.rows), bars = GEMM_BAR_BYTES + (gather_mode(mode) ? BM * 8 : 0);
    const int nkb_cta = ceil_div(nkb, g.splits);
    g.ring = gemm_ring(mode, g.BN, g.rows, (long long)g.m_tiles * ceil_div(N, g.BN) * batch * g.splits, nkb_cta);
    if (tn.gemm_ring && (size_t)tn.gemm_ring * sb <= 210u * 1024u) g.ring = tn.gemm_ring;
    // Write-out through swizzled staging tiles when the output rows are 16-byte multiples (else plain stores), in
    // the ring once that is idle; with a residual addend, which is loaded while the ring works, in a place of their own.
    const size_t staging = (size_t)ceil_div(g.rows, 32) * 32 * g.BN * 4;
    // Split K: room to park the partial tile in the ring, and for the rows this CTA receives (its share from every CTA).
    const size_t park = split ? (size_t)g.rows * g.BN * 4 : (staged && !addend) ? staging : 0;
    const size_t behind = split ? (size_t)g.splits * ceil_div(g.rows, g.splits) * g.BN * 4 : (staged && addend) ? staging + 1024 : 0;
    while (g.ring < 8 && g.ring * sb < park) ++g.ring;
    while (g.ring > 1 && 2048 + g.ring * sb + bars + behind > 226u * 1024u && (g.ring - 1) * sb >= park) --g.ring;
    // Two issuers take alternate K blocks, so in a ring of odd depth the blocks of one slot go to one and the other in turn.  A wait
    // by parity only tells neighbouring phases apart: an issuer that is through with block i - 2 takes the slot of block i for full
    // while the load of its former block, i - depth, is still on its way (loads may land in any order).  It would multiply what
    // is there and release the slot; the producers then arrive at a barrier whose phase already has all its arrivals, and loads
    // land in a CTA that has gone.  So a ring that is refilled has an even depth: an issuer then has its slots for itself.
    // (X3's issuers wait for eight warps that convert the blocks in order: block i - 2 converted means block i - depth is, from
    // two slots on.  Mode 8's two groups of warps take the blocks in turn like the issuers; with one issuer one group takes all.)
    if (g.issuers == 2 && nkb_cta > g.ring && (x3_mode(mode) ? g.ring == 1 : (g.ring & 1) == 1)) {
        if (g.ring > 1 && (g.ring - 1) * sb >= park) --g.ring;
        else g.issuers = 1;
    }
    g.bar_off = (uint32_t)(g.ring * sb);
    const size_t ring_and_bars = g.ring * sb + bars;
    g.recv_off = (uint32_t)align_up(ring_and_bars, 128);
    g.stage_off = addend ? (uint32_t)align_up(ring_and_bars, 1024) : 0;
    g.smem_bytes = (size_t)1024 + (split ? g.recv_off + behind : (staged && addend) ? g.stage_off + staging : ring_and_bars);
    // the MMAs read 128 rows of A from every stage, the last one included
    g.smem_bytes = std::max(g.smem_bytes, (size_t)1024 + (g.ring - 1) * sb + A_STAGE_BYTES);
    if (split) g.smem_bytes = std::max(g.smem_bytes, tmem_share_bytes(g.tmem_cols));
    NNV_REQUIRE(g.smem_bytes <= 226u * 1024u, NNV_ERR_UNSUPPORTED, "GEMM tiling does not fit shared memory");
    *out = g;
    return NNV_OK;
}

std::once_flag g_attr_once;

// [kernel mode][K split over a cluster]
constexpr decltype(&gemm_tc_kernel<0, false>) gemm_kernels[10][2] = {
    {gemm_tc_kernel<0, false>, gemm_tc_kernel<0, true>}, {gemm_tc_kernel<1, false>, gemm_tc_kernel<1, true>},
    {gemm_tc_kernel<2, false>, gemm_tc_kernel<2, true>}, {gemm_tc_kernel<3, false>, gemm_tc_kernel<3, true>},
    {gemm_tc_kernel<4, false>, gemm_tc_kernel<4, true>}, {gemm_tc_kernel<5, false>, gemm_tc_kernel<5, true>},
    {gemm_tc_kernel<6, false>, gemm_tc_kernel<6, true>}, {gemm_tc_kernel<7, false>, gemm_tc_kernel<7, true>},
    {gemm_tc_kernel<ROUNDED, false>, gemm_tc_kernel<ROUNDED, true>}, {gemm_tc_kernel<SPLIT_A, false>, gemm_tc_kernel<SPLIT_A, true>}};
// [BF16 math][patches shared by a cluster]
constexpr decltype(&inverted_bottleneck_kernel<false, false>) ib_kernels[2][2] = {
    {inverted_bottleneck_kernel<false, false>, inverted_bottleneck_kernel<false, true>},
    {inverted_bottleneck_kernel<true, false>, inverted_bottleneck_kernel<true, true>}};
static_assert(GEMM_TF32 == 0 && GEMM_BF16 == 1 && GEMM_X3 == 2 && GEMM_BF16_CVT == 3, "the table's order");

}  // namespace

nnv_status_t gemm_tc_init() {
    NNV_TRY(get_encoder());
    std::call_once(g_attr_once, [] {
        for (auto& forms : gemm_kernels)
            for (auto* kernel : forms) {
                cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
                cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
            }
        cudaFuncSetAttribute(conv3x3_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
        cudaFuncSetAttribute(conv3x3_bf16_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
        cudaFuncSetAttribute(conv3x3_bf16_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
        cudaFuncSetAttribute(gemm_sp_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
        cudaFuncSetAttribute(conv3x3_tc_persistent_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
        cudaFuncSetAttribute(wino_f2_fused_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
        cudaFuncSetAttribute(conv3x3_tc_ws_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
        for (auto& forms : ib_kernels)
            for (auto* kernel : forms) {
                cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
                cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
            }
    });
    return NNV_OK;
}

// bf16 packed weights [N][ld]: boxes of 32 elements (64 bytes, 64-byte swizzle) x BN rows.  (Boxes of 16-byte pieces, which would
// land un-swizzled, cost the copy engine as much per piece as one of 64 or 128 bytes does.)
static nnv_status_t encode_bf16_weights(CUtensorMap* map, const void* base, int64_t ld, int Kd, int N, int BN) {
    NNV_REQUIRE((ld % 8) == 0 && (reinterpret_cast<uintptr_t>(base) & 15) == 0, NNV_ERR_INVALID_ARG, "bf16 weight rows must be 16-byte multiples");
    cuuint64_t dims[3] = {(cuuint64_t)Kd, (cuuint64_t)N, 1};
    cuuint64_t strides[2] = {(cuuint64_t)ld * 2, (cuuint64_t)ld * 2 * N};
    cuuint32_t box[3] = {32, (cuuint32_t)BN, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    NNV_REQUIRE(r == CUDA_SUCCESS, NNV_ERR_CUDA, "cuTensorMapEncodeTiled (bf16 weights) failed with code %d", (int)r);
    return NNV_OK;
}

// 3-D tiled map over the NHWC fp32 output {K, W, H}: boxes of `cw` channels x 8 pixels x 4 rows (what one warp of the
// 3x3 kernel holds), in the swizzled layout the epilogue writes.
static nnv_status_t encode_conv_output(CUtensorMap* map, const void* base, int K, int H, int W, int cw) {
    cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)W, (cuuint64_t)H};
    cuuint64_t strides[2] = {(cuuint64_t)K * 4, (cuuint64_t)W * K * 4};
    cuuint32_t box[3] = {(cuuint32_t)cw, 8, 4};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(base), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, cw == 32 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    NNV_REQUIRE(r == CUDA_SUCCESS, NNV_ERR_CUDA, "cuTensorMapEncodeTiled (3x3 output boxes) failed with code %d", (int)r);
    return NNV_OK;
}

// BF16 math: K splits and column tile of conv3x3_bf16_kernel.
// The pair with the least estimated time (microseconds): fixed cost + waves x (channel blocks per CTA + write-out).  Beside a split's
// receive buffer for 128 columns shared memory holds two weight boxes, which costs 0.7 us against what 96 and 112 columns (three or
// four boxes) lead one to expect (mean over 112 tilings).  Over 171 layers of 32 - 1024 channels on 7 - 224 pixels a side the chosen
// tilings are 0.3 % above the best measured ones on average (0.5 % without that term: 512 -> 512 @28 on 128 columns in four splits
// 12.0 us, on 64 in two 10.8); furthest off are 320 -> 64 @45, 7.4 us on 16 columns where 64 in four splits take 6.5, and 640 -> 640
// @9x12, 4 %.
struct ConvBTiling { int BN, splits; double t; };

static ConvBTiling pick_conv_bf16_tiling(int C, int H, int W, int N) {
    ConvBTiling best{16, 1, 1e30};
    const int patches = ceil_div(H, 16) * ceil_div(W, 8), cblk = C / 32;
    for (int bn = 16; bn <= std::min(128, ceil_div(N, 16) * 16); bn += 16) {
        for (int sp = 1; sp <= 8 && sp <= cblk; sp *= 2) {
            const long long ctas = (long long)patches * ceil_div(N, bn) * sp;
            // capacity of one CTA per SM in clusters of 1 / 2, 4 and 8
            const int slots = sp <= 2 ? 148 : sp == 4 ? 132 : 120;
            const double waves = (double)((ctas + slots - 1) / slots);
            const int blocks = ceil_div(cblk, sp);
            const double two_boxes = sp > 1 && bn > 112 && blocks > 1 ? 0.7 : 0.0;
            const double t = 2.39 + waves * (blocks * (0.72 + 0.0018 * bn) + 0.25 + 0.019 * bn + (sp > 1 ? 0.0184 * bn : 0.0) + two_boxes);
            if (t < best.t - 1e-9) best = ConvBTiling{bn, sp, t};
        }
    }
    return best;
}

// Rings, issuers and shared-memory layout of one launch of conv3x3_bf16_kernel.
struct ConvBShape {
    int splits, na, nb, issuers, tmem_cols;
    uint32_t b_off, bar_off, recv_off;
    size_t smem_bytes;
};

static nnv_status_t conv_bf16_shape(int C, int BN, int splits, ConvBShape* out) {
    ConvBShape g{};
    g.splits = splits;
    g.tmem_cols = 32;
    while (g.tmem_cols < 2 * BN) g.tmem_cols *= 2;
    // two channel blocks of weights in flight where they fit (three filter rows each)
    const size_t recv = splits > 1 ? (size_t)128 * BN * 4 : 0;
    // boxes in flight: as many as the channel blocks, where six weight boxes still fit (and at least two, whose room the write-out uses)
    const int ncb = ceil_div(C / 32, splits);
    g.na = std::max(2, std::min(CB_MAX_NA, ncb));
    auto b_off = [&](int na) { return (uint32_t)align_up((size_t)na * CB_A32 + 2 * CB_ABF, 1024); };
    while (g.na > 2 && b_off(g.na) + CB_BAR_BYTES + 256 + recv + (size_t)6 * BN * 192 > 225u * 1024u) --g.na;
    g.b_off = b_off(g.na);
    const int stages = 3 * ncb;
    g.nb = std::min({6, stages, (int)((225u * 1024u - g.b_off - CB_BAR_BYTES - 256 - recv) / ((size_t)BN * 192))});
    // (two issuers take alternate filter rows: a ring that is refilled has an even depth, as in gemm_tc_kernel)
    g.issuers = 2;
    if (stages > g.nb && (g.nb & 1)) {
        if (g.nb > 1) --g.nb;
        else g.issuers = 1;
    }
    g.bar_off = (uint32_t)align_up(g.b_off + (size_t)g.nb * BN * 192, 16);
    g.recv_off = (uint32_t)align_up(g.bar_off + CB_BAR_BYTES, 128);
    g.smem_bytes = std::max((size_t)1024 + g.recv_off + recv, splits > 1 ? tmem_share_bytes(g.tmem_cols) : 0);
    NNV_REQUIRE(g.nb >= 1 && g.smem_bytes <= 226u * 1024u, NNV_ERR_UNSUPPORTED, "3x3 tiling does not fit shared memory");
    *out = g;
    return NNV_OK;
}

static nnv_status_t launch_conv3x3_bf16(const GemmArgs& a, int BN, int splits, cudaStream_t st) {
    ConvBDev g{};
    ConvBShape sh;
    NNV_TRY(conv_bf16_shape(a.ic.C, BN, splits, &sh));
    CUtensorMap tmA, tmB;
    const int C = a.ic.C, H = a.ic.H, W = a.ic.W;
    NNV_REQUIRE(a.ldd == a.N, NNV_ERR_INVALID_ARG, "the 3x3 kernel writes a dense NHWC output");
    NNV_TRY(encode_halo_operand(&tmA, a.A, C, H, W, 18, 10));
    {
        // packed bf16 rows [N][9 taps][C] seen as {C, N rows, 9 taps}: one box holds a filter row's three taps x 32 channels
        NNV_REQUIRE((a.ldb % 8) == 0 && (reinterpret_cast<uintptr_t>(a.B) & 15) == 0, NNV_ERR_INVALID_ARG, "bf16 weight rows must be 16-byte multiples");
        cuuint64_t dims[3] = {(cuuint64_t)C, (cuuint64_t)a.N, 9};
        cuuint64_t strides[2] = {(cuuint64_t)a.ldb * 2, (cuuint64_t)C * 2};
        cuuint32_t box[3] = {32, (cuuint32_t)BN, 3};
        cuuint32_t estr[3] = {1, 1, 1};
        CUresult r = g_encode(&tmB, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(a.B), dims, strides, box, estr,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        NNV_REQUIRE(r == CUDA_SUCCESS, NNV_ERR_CUDA, "cuTensorMapEncodeTiled (bf16 filter taps) failed with code %d", (int)r);
    }
    g.stamp = next_stamp();
    next_stamp() = nullptr;
    g.D = a.D; g.bias = a.bias; g.addend = a.addend;
    g.C = C; g.H = H; g.W = W; g.K = a.N;
    g.BN = BN; g.act = a.act; g.splits = splits;
    g.cblk = C / 32; g.tiles_w = ceil_div(W, 8);
    g.tmem_cols = sh.tmem_cols; g.na = sh.na; g.nb = sh.nb; g.issuers = sh.issuers;
    g.b_off = sh.b_off; g.bar_off = sh.bar_off; g.recv_off = sh.recv_off;
    const dim3 grid(ceil_div(H, 16) * g.tiles_w, ceil_div(a.N, BN), splits);
    NNV_REQUIRE(grid.y <= 65535, NNV_ERR_UNSUPPORTED, "convolution grid too large");
    NNV_CUDA(launch_pdl_cluster(splits > 1 ? conv3x3_bf16_kernel<true> : conv3x3_bf16_kernel<false>, grid, dim3(CB_THREADS), sh.smem_bytes, st, splits, tmA, tmB, g));
    return NNV_OK;
}

static nnv_status_t launch_conv3x3_tc(const GemmArgs& a, const ConvTiling& ct, cudaStream_t st) {
    CUtensorMap tmA, tmB, tmD;
    NNV_TRY(encode_halo_operand(&tmA, a.A, a.ic.C, a.ic.H, a.ic.W, 16 * ct.MT + 2));
    NNV_TRY(encode_operand(&tmB, a.B, false, a.Kd, a.N, 1, a.ldb, a.strideB, ct.BN));
    ConvDev g;
    g.stamp = next_stamp();
    next_stamp() = nullptr;
    g.D = a.D; g.bias = a.bias; g.addend = a.addend;
    g.C = a.ic.C; g.H = a.ic.H; g.W = a.ic.W; g.K = a.N;
    g.BN = ct.BN; g.MT = ct.MT; g.act = a.act; g.tmem_cols = ct.tmem_cols; g.splits = ct.splits; g.na = ct.na; g.nb = ct.nb;
    g.cblk = ceil_div(a.ic.C, 32); g.tiles_w = ceil_div(a.ic.W, 8);
    NNV_REQUIRE(a.ldd == a.N, NNV_ERR_INVALID_ARG, "the 3x3 kernel writes a dense NHWC output");
    // Write-out by TMA when nothing is added after the K loop but the bias, the output rows are 16-byte multiples and
    // the staged tile fits into the (then idle) rings; else plain stores.
    g.tma_out = 0;
    const size_t rings = (size_t)ct.na * conv_a_slot(ct.MT) + (size_t)ct.nb * conv_b_slot(ct.BN);
    if (ct.splits == 1 && !a.addend && (a.N % 4) == 0 && (reinterpret_cast<uintptr_t>(a.D) & 15) == 0 &&
        (!a.bias || (reinterpret_cast<uintptr_t>(a.bias) & 15) == 0) && (size_t)ct.MT * BM * ct.BN * 4 <= rings) {
        g.tma_out = (ct.BN % 32) == 0 ? 32 : 16;
        NNV_TRY(encode_conv_output(&tmD, a.D, a.N, a.ic.H, a.ic.W, g.tma_out));
    } else {
        tmD = tmA;                                               // unused by the kernel, but a kernel parameter must hold a valid object
    }
    dim3 grid(ceil_div(a.ic.H, 16 * ct.MT) * g.tiles_w, ceil_div(a.N, ct.BN), ct.splits);
    NNV_REQUIRE(grid.y <= 65535, NNV_ERR_UNSUPPORTED, "convolution grid too large");
    (void)launch_pdl_cluster(conv3x3_tc_kernel, grid, dim3(GEMM_THREADS), ct.smem, st, ct.splits, tmA, tmB, tmD, g);
    NNV_CUDA(cudaGetLastError());
    return NNV_OK;
}

// 3-D tiled map over an NHWC fp32 activation {C, W, H} whose box is 32 channels of `box_h` whole image rows.
static nnv_status_t encode_image_operand(CUtensorMap* map, const void* base, int C, int H, int W, int box_h) {
    NNV_REQUIRE((reinterpret_cast<uintptr_t>(base) & 15) == 0 && (C % 4) == 0 && W <= 256 && H <= 256, NNV_ERR_INVALID_ARG,
                "activation must be 16-byte aligned with C a multiple of 4 and at most 256 pixels a side");
    cuuint64_t dims[3] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)H};
    cuuint64_t strides[2] = {(cuuint64_t)C * 4, (cuuint64_t)W * C * 4};
    cuuint32_t box[3] = {32, (cuuint32_t)W, (cuuint32_t)box_h};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(base), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    NNV_REQUIRE(r == CUDA_SUCCESS, NNV_ERR_CUDA, "cuTensorMapEncodeTiled (whole-image boxes) failed with code %d", (int)r);
    return NNV_OK;
}

nnv_status_t launch_gemm_sp(const nnv_layer_desc_t& L, const LayerGeom& geo, const SmallPPlan& sp, const float* x, const float* wt,
                            const float* bias, const float* addend, float* y, void* ws, cudaStream_t st) {
    NNV_TRY(gemm_tc_init());
    NNV_REQUIRE(sp.splits == 1 || ws, NNV_ERR_INVALID_ARG, "the K split needs its scratch");
    CUtensorMap tmW, tmX;
    NNV_TRY(encode_operand(&tmW, wt, false, geo.Qp, L.K, 1, geo.Qp, (int64_t)L.K * geo.Qp, BM));
    NNV_TRY(encode_image_operand(&tmX, x, L.C, L.H, L.W, L.H));
    SpDev g;
    g.stamp = next_stamp();
    next_stamp() = nullptr;
    g.D = y; g.part = (float*)ws; g.bias = bias; g.addend = addend;
    g.P = geo.P; g.K = L.K; g.C = L.C; g.S = L.S; g.pad = L.pad; g.Npad = sp.Npad; g.act = L.act;
    g.tmem_cols = 32;
    while (g.tmem_cols < sp.Npad) g.tmem_cols *= 2;
    g.splits = sp.splits; g.stages = sp.stages; g.cblk = L.C / 32; g.nkb_all = sp.nkb;
    g.b_slot_bytes = sp.b_slot_bytes; g.b_tx_bytes = (uint32_t)(L.H * L.W) * 128u;
    const size_t smem = (size_t)1024 + (size_t)sp.stages * (A_STAGE_BYTES + sp.b_slot_bytes) + 8 * (2 * SP_MAX_STAGES + 2);
    dim3 grid(ceil_div(L.K, BM), sp.splits);
    (void)launch_pdl(gemm_sp_kernel, grid, dim3(GEMM_THREADS), smem, st, tmW, tmX, g);
    NNV_CUDA(cudaGetLastError());
    if (sp.splits > 1) {
        const long long n4 = (long long)geo.P * L.K / 4;
        const unsigned blocks = (unsigned)((n4 + 31) / 32);
        (void)launch_pdl(splitk_reduce_kernel, dim3(blocks), dim3(256), 0, st, (const float*)ws, y, bias, addend, geo.P, L.K, sp.splits,
                         L.act, g.stamp);
        NNV_CUDA(cudaGetLastError());
    }
    return NNV_OK;
}

nnv_status_t launch_wino_f2_fused(const nnv_layer_desc_t& L, const LayerGeom& geo, const float* x, const float* U, const float* bias,
                                  const float* addend, float* y, cudaStream_t st) {
    NNV_TRY(gemm_tc_init());
    NNV_REQUIRE((reinterpret_cast<uintptr_t>(x) & 15) == 0 && (reinterpret_cast<uintptr_t>(U) & 15) == 0 &&
                    (reinterpret_cast<uintptr_t>(y) & 15) == 0 && (!bias || (reinterpret_cast<uintptr_t>(bias) & 15) == 0) &&
                    (!addend || (reinterpret_cast<uintptr_t>(addend) & 15) == 0),
                NNV_ERR_INVALID_ARG, "the fused Winograd kernel needs 16-byte aligned buffers");
    WfDev g;
    g.stamp = next_stamp();
    next_stamp() = nullptr;
    g.x = x; g.y = y; g.bias = bias; g.addend = addend;
    g.C = L.C; g.H = L.H; g.W = L.W; g.K = L.K; g.pad = L.pad; g.OH = geo.OH; g.OW = geo.OW;
    g.TW = ceil_div(geo.OW, 2);
    g.T = ceil_div(geo.OH, 2) * g.TW;
    g.act = L.act;
    // 32 output channels per CTA (all 512 TMEM columns) when that still gives every other SM a CTA, else 16
    const int row_tiles = ceil_div(g.T, BM);
    g.BN = ((L.K % 32) == 0 && (long long)row_tiles * (L.K / 32) >= 74) ? 32 : 16;
    g.tmem_cols = 16 * g.BN;
    g.nsteps = L.C / 8;
    g.stages = std::min(WF_MAX_STAGES, std::max(1, g.nsteps));
    const uint32_t b_stage = 2u * 16u * (uint32_t)g.BN * 16u;
    while (g.stages > 1 && (size_t)1024 + (size_t)g.stages * (WF_A_STAGE + b_stage) + 8 * (3 * WF_MAX_STAGES + 2) > 220u * 1024u) --g.stages;
    const size_t smem = (size_t)1024 + (size_t)g.stages * (WF_A_STAGE + b_stage) + 8 * (3 * WF_MAX_STAGES + 2);
    CUtensorMap tmU;
    {
        cuuint64_t dims[3] = {(cuuint64_t)geo.Cp, (cuuint64_t)L.K, 16};
        cuuint64_t strides[2] = {(cuuint64_t)geo.Cp * 4, (cuuint64_t)L.K * geo.Cp * 4};
        cuuint32_t box[3] = {4, (cuuint32_t)g.BN, 16};
        cuuint32_t estr[3] = {1, 1, 1};
        CUresult r = g_encode(&tmU, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(U), dims, strides, box, estr,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        NNV_REQUIRE(r == CUDA_SUCCESS, NNV_ERR_CUDA, "cuTensorMapEncodeTiled (transformed filters) failed with code %d", (int)r);
    }
    dim3 grid(row_tiles, ceil_div(L.K, g.BN));
    (void)launch_pdl(wino_f2_fused_kernel, grid, dim3(GEMM_THREADS), smem, st, tmU, g);
    NNV_CUDA(cudaGetLastError());
    return NNV_OK;
}

// The weights-stationary form; `fits` tells whether the layer's weight slice and the kernel's other buffers fit.
static size_t convw_smem_bytes(int cblk, int BN) {
    return (size_t)1024 + (size_t)9 * cblk * BN * BK_BYTES + (size_t)CONVW_NA * 18 * 1024 + 4 * 4096 + 8 * (CONVW_MAX_WT + 2 * CONVW_NA + 5);
}
static bool convw_fits(const GemmArgs& a, int* BN_out) {
    const int cblk = ceil_div(a.ic.C, 32);
    const int BN = std::min(128, ceil_div(a.N, 16) * 16);
    if (9 * cblk > CONVW_MAX_WT || (BN % 16) != 0 || a.addend || (a.N % 4) != 0 || a.ldd != a.N) return false;
    if ((reinterpret_cast<uintptr_t>(a.D) & 15) != 0 || (a.bias && (reinterpret_cast<uintptr_t>(a.bias) & 15) != 0)) return false;
    // the widest channel tile (a multiple of 16, at most 128) whose weight slice fits
    for (int bn = BN; bn >= 16; bn -= 16) {
        if (convw_smem_bytes(cblk, bn) <= 226u * 1024u) { *BN_out = bn; return true; }
    }
    return false;
}
static nnv_status_t launch_conv3x3_ws(const GemmArgs& a, int BN, cudaStream_t st) {
    CUtensorMap tmA, tmB, tmD;
    NNV_TRY(encode_halo_operand(&tmA, a.A, a.ic.C, a.ic.H, a.ic.W, 18));
    NNV_TRY(encode_operand(&tmB, a.B, false, a.Kd, a.N, 1, a.ldb, a.strideB, BN));
    ConvWDev g;
    g.stamp = next_stamp();
    next_stamp() = nullptr;
    g.bias = a.bias;
    g.C = a.ic.C; g.H = a.ic.H; g.W = a.ic.W; g.K = a.N;
    g.BN = BN; g.act = a.act;
    g.cblk = ceil_div(a.ic.C, 32); g.tiles_w = ceil_div(a.ic.W, 8);
    g.patches = ceil_div(a.ic.H, 16) * g.tiles_w;
    g.cw = (BN % 32) == 0 ? 32 : 16;
    g.tmem_cols = 32;
    while (g.tmem_cols < 2 * BN) g.tmem_cols *= 2;
    NNV_TRY(encode_conv_output(&tmD, a.D, a.N, a.ic.H, a.ic.W, g.cw));
    const int n_tiles = ceil_div(a.N, BN);
    const int ctas_x = std::max(1, std::min(g.patches, 148 / n_tiles));
    const size_t smem = convw_smem_bytes(g.cblk, BN);
    (void)launch_pdl(conv3x3_tc_ws_kernel, dim3(ctas_x, n_tiles), dim3(GEMM_THREADS), smem, st, tmA, tmB, tmD, g);
    NNV_CUDA(cudaGetLastError());
    return NNV_OK;
}

// The persistent form: BN channels per tile, `per_sm` CTAs per SM, ring depths na / nb.
static nnv_status_t launch_conv3x3_persistent(const GemmArgs& a, int BN, int per_sm, int na, int nb, cudaStream_t st) {
    CUtensorMap tmA, tmB;
    NNV_TRY(encode_halo_operand(&tmA, a.A, a.ic.C, a.ic.H, a.ic.W, 18));
    NNV_TRY(encode_operand(&tmB, a.B, false, a.Kd, a.N, 1, a.ldb, a.strideB, BN));
    ConvPDev g;
    g.stamp = next_stamp();
    next_stamp() = nullptr;
    g.D = a.D; g.bias = a.bias; g.addend = a.addend;
    g.C = a.ic.C; g.H = a.ic.H; g.W = a.ic.W; g.K = a.N;
    g.BN = BN; g.act = a.act; g.na = na; g.nb = nb;
    g.cblk = ceil_div(a.ic.C, 32); g.tiles_w = ceil_div(a.ic.W, 8);
    g.n_tiles = ceil_div(a.N, BN);
    g.tiles_total = ceil_div(a.ic.H, 16) * g.tiles_w * g.n_tiles;
    g.tmem_cols = 32;
    while (g.tmem_cols < 2 * BN) g.tmem_cols *= 2;
    NNV_REQUIRE(a.ldd == a.N, NNV_ERR_INVALID_ARG, "the 3x3 kernel writes a dense NHWC output");
    const size_t smem = (size_t)1024 + (size_t)na * 18 * 1024 + (size_t)nb * BN * BK_BYTES + 4 * 32 * 36 * 4 +
                        8 * (2 * CONV_MAX_NA + 2 * CONV_MAX_NB + 5);
    NNV_REQUIRE(smem <= 220u * 1024u, NNV_ERR_UNSUPPORTED, "persistent 3x3 tiling does not fit shared memory");
    const int ctas = std::min(g.tiles_total, 148 * per_sm);
    (void)launch_pdl(conv3x3_tc_persistent_kernel, dim3(ctas), dim3(GEMM_THREADS), smem, st, tmA, tmB, g);
    NNV_CUDA(cudaGetLastError());
    return NNV_OK;
}

nnv_status_t launch_gemm_tc(const GemmArgs& a, cudaStream_t st) {
    NNV_REQUIRE(a.M > 0 && a.N > 0 && a.Kd > 0 && a.batch > 0, NNV_ERR_INVALID_ARG, "empty GEMM");
    NNV_TRY(gemm_tc_init());
    // Tiling: column tile BN and K splits (a thread-block cluster of up to 16 CTAs) with the least estimated time.
    const int bke = (a.mode == GEMM_BF16) ? 64 : 32;
    const bool gather = a.ic.on && a.ic.gather;
    // an activation below 128 KiB comes as boxes of whole image rows
    const bool boxes = a.ic.on && !gather && 4ull * a.ic.C * a.ic.H * a.ic.W < 131072ull &&
                       image_row_boxes(a.ic.H, a.ic.W, a.ic.R, a.ic.S, a.ic.stride, a.ic.pad);
    const int mode = gather ? (a.mode == GEMM_BF16 ? 5 : 4) + ((a.ic.C % 4) == 0 ? 2 : 0)
                            : boxes && a.mode == GEMM_TF32 ? ROUNDED : a.mode == GEMM_X3 && a.split_a ? SPLIT_A : a.mode;   // the kernel's
    const int nkb_all = a.ic.on && !gather ? a.ic.R * a.ic.S * ceil_div(a.ic.C, 32) : ceil_div(a.Kd, bke);
    const GemmTiling tile = pick_gemm_tiling(mode, a.M, a.N, a.batch, nkb_all);
    const Tuning& tn = tuning();
    // A 3x3 / stride 1 / pad 1 layer large enough to fill the GPU runs on the halo-resident kernel,
    // which moves fewer operand bytes through L2 and shared memory.
    if (a.ic.on && !gather && (a.mode == GEMM_TF32 || a.mode == GEMM_BF16_CVT) && a.batch == 1 && a.ic.R == 3 && a.ic.S == 3 && a.ic.stride == 1 &&
        a.ic.pad == 1 && (a.ic.C % 32) == 0) {
        if (a.mode == GEMM_BF16_CVT) {
            ConvBTiling ct = pick_conv_bf16_tiling(a.ic.C, a.ic.H, a.ic.W, a.N);
            if (tn.conv3x3 == 2 && tn.conv_splits <= a.ic.C / 32) ct = ConvBTiling{tn.conv_bn, tn.conv_splits, 0.0};
            if (tn.conv3x3 != 1) return launch_conv3x3_bf16(a, ct.BN, ct.splits, st);
        } else {
        ConvTiling ct;
        bool use = pick_conv_tiling(a.ic.C, a.ic.H, a.ic.W, a.N, tile, &ct);
        if (tn.conv3x3 == 1) {
            use = false;
        } else if (tn.conv3x3 == 2) {
            ConvTiling f{};
            f.MT = tn.conv_mt; f.BN = tn.conv_bn; f.splits = tn.conv_splits; f.na = tn.conv_na; f.nb = tn.conv_nb;
            if (f.splits <= ceil_div(a.ic.C, 32) && finish_conv_tiling(&f)) {
                ct = f;
                use = true;
            }
        }
        // The persistent form runs only on request.  Measured on B200 (L2 flushed): one resident
        // CTA per SM reaches 152 TFLOP/s on 64 -> 64 @ 224 and two reach 205, against 328 for two or three
        // one-tile CTAs per SM: inside one CTA the single MMA-issuing thread (about 82 cycles per tcgen05.mma
        // against 32 cycles of execution at N = 64) bounds the tile rate, and independent CTAs, each with its own
        // issuing thread, lift that bound where a second accumulator does not.
        // The weights-stationary form runs only on request.  Measured on B200 (64 -> 64, L2 flushed or not): 20.4 us on
        // a 224 x 224 image against 11.3 for the one-tile kernel, and 5.4 us for every further patch of a CTA.  One thread
        // issues one tcgen05.mma per ~82 cycles whatever N is, so the 72 MMAs (N = 64) of a patch take 3 us of issue time
        // alone where the tensor pipe needs 1.2; three one-tile CTAs per SM issue from three threads, and the resident
        // weights leave room for only three halo boxes in flight.
        int wbn = 0;
        if (tn.convw == 2 && convw_fits(a, &wbn)) return launch_conv3x3_ws(a, wbn, st);
        if (tn.convp == 2 && (size_t)tn.convp_bn <= (size_t)ceil_div(a.N, 16) * 16)
            return launch_conv3x3_persistent(a, tn.convp_bn, tn.convp_per_sm, tn.convp_na ? tn.convp_na : 2, tn.convp_nb ? tn.convp_nb : 4, st);
        if (use) return launch_conv3x3_tc(a, ct, st);
        }
    }
    const bool vec_ok = (a.N % 4) == 0 && (a.ldd % 4) == 0 && (a.strideD % 4) == 0 && (reinterpret_cast<uintptr_t>(a.D) & 15) == 0 &&
                        (!a.addend || ((reinterpret_cast<uintptr_t>(a.addend) & 15) == 0 && a.batch == 1));
    GemmShape sh;
    NNV_TRY(gemm_shape(mode, tile, a.M, a.N, a.batch, nkb_all, vec_ok, a.addend != nullptr, &sh));
    const int BN = sh.BN, splits = sh.splits, rows = sh.rows, m_tiles = sh.m_tiles;
    const bool staged = vec_ok && splits == 1;

    const bool bf16 = a.mode == GEMM_BF16;
    CUtensorMap tmA, tmB, tmAdd;
    GemmDev g;
    g.stamp = next_stamp();
    next_stamp() = nullptr;
    g.D = a.D; g.bias = a.bias; g.addend = a.addend;
    g.ldd = a.ldd; g.strideD = a.strideD;
    g.M = a.M; g.N = a.N; g.Kd = a.Kd; g.BN = BN; g.act = a.act; g.tmem_cols = sh.tmem_cols; g.splits = splits; g.stages = sh.ring; g.issuers = sh.issuers;
    g.rows = rows; g.bar_off = sh.bar_off; g.recv_off = sh.recv_off; g.stage_off = sh.stage_off;
    g.chunk = staged ? 16 : 0;
    g.ic_on = 0; g.ic_C = g.ic_cblk = g.ic_S = g.ic_OW = g.ic_stride = g.ic_pad = 0;
    g.x = nullptr; g.ic_H = g.ic_W = g.ic_Q = 0; g.magic_c = g.magic_s = 0;
    if (gather) {
        g.x = static_cast<const float*>(a.A);
        g.ic_C = a.ic.C; g.ic_S = a.ic.S; g.ic_OW = a.ic.OW; g.ic_stride = a.ic.stride; g.ic_pad = a.ic.pad;
        g.ic_H = a.ic.H; g.ic_W = a.ic.W; g.ic_Q = a.ic.R * a.ic.S * a.ic.C;
        g.magic_c = 0xFFFFFFFFu / (uint32_t)a.ic.C + 1u;
        g.magic_s = 0xFFFFFFFFu / (uint32_t)a.ic.S + 1u;
    } else if (a.ic.on) {
        NNV_REQUIRE((a.mode == GEMM_TF32 || a.mode == GEMM_BF16_CVT) && a.batch == 1, NNV_ERR_INVALID_ARG,
                    "implicit im2col needs fp32 activations (TF32 or converting BF16 mode) and one batch");
        if (boxes) NNV_TRY(encode_image_operand(&tmA, a.A, a.ic.C, a.ic.H, a.ic.W, rows / a.ic.W));
        else NNV_TRY(encode_im2col_operand(&tmA, a.A, a.ic.C, a.ic.H, a.ic.W, a.ic.R, a.ic.S, a.ic.stride, a.ic.pad, rows));
        g.ic_on = boxes ? 2 : 1; g.ic_C = a.ic.C; g.ic_cblk = ceil_div(a.ic.C, 32); g.ic_S = a.ic.S; g.ic_OW = a.ic.OW;
        g.ic_stride = a.ic.stride; g.ic_pad = a.ic.pad;
        g.Kd = a.ic.R * a.ic.S * g.ic_cblk;                       // number of K blocks
    } else {
        NNV_TRY(encode_operand(&tmA, a.A, bf16, a.Kd, a.M, a.batch, a.lda, a.strideA, rows));
    }
    if (a.mode == GEMM_BF16_CVT) {
        NNV_REQUIRE(a.batch == 1, NNV_ERR_INVALID_ARG, "the converting BF16 mode needs one batch");
        NNV_TRY(encode_bf16_weights(&tmB, a.B, a.ldb, (int)a.ldb, a.N, BN));
    } else {
        NNV_TRY(encode_operand(&tmB, a.B, bf16, a.Kd, a.N, a.batch, a.ldb, a.strideB, BN));
    }
    if (gather) tmA = tmB;                                       // unused by the kernel, but a kernel parameter must hold a valid object

    // equal tiles: the output is addressed as {N, rows, tiles}, so that the hardware clips a tile's last 32-row box
    const bool equal = a.M == m_tiles * rows && (a.batch == 1 || a.strideD == (int64_t)a.M * a.ldd);
    NNV_REQUIRE(equal || rows == BM, NNV_ERR_INVALID_ARG, "batched GEMM outputs must be dense");
    g.z_tiles = equal ? m_tiles : 0;
    auto encode_addend = [&](CUtensorMap* map, const void* base) {
        const int box_rows = ceil_div(rows, 32) * 32;
        if (equal) return encode_addend_tiles(map, base, a.N, rows, m_tiles * a.batch, a.ldd, (int64_t)rows * a.ldd, box_rows);
        return encode_addend_tiles(map, base, a.N, a.M, a.batch, a.ldd, a.batch > 1 ? a.strideD : (int64_t)a.M * a.ldd, box_rows);
    };
    if (staged && a.addend) NNV_TRY(encode_addend(&tmAdd, a.addend));
    else tmAdd = tmA;

    dim3 grid(m_tiles, ceil_div(a.N, BN), a.batch * splits);
    NNV_REQUIRE(grid.y <= 65535 && grid.z <= 65535, NNV_ERR_UNSUPPORTED, "GEMM grid too large");
    NNV_REQUIRE(a.mode >= GEMM_TF32 && a.mode <= GEMM_BF16_CVT, NNV_ERR_INVALID_ARG, "unknown GEMM mode %d", a.mode);
    (void)launch_pdl_cluster(gemm_kernels[mode][splits > 1], grid, dim3(gemm_tc_threads(mode)), sh.smem_bytes, st, splits, tmA, tmB, tmAdd, g);
    NNV_CUDA(cudaGetLastError());
    return NNV_OK;
}

// ---- inverted bottleneck: shape of a launch -----------------------------------------------------
namespace {

// The channel blocks of every CTA that shares a patch, in the order of the projection's own launch: its `splits` ranges of the n blocks,
// whole (`both`: two accumulators, or with one issuer one) or an accumulator's blocks each.
bool ib_ranks(int n, int splits, int issuers, bool unit, IbShape* s) {
    s->ranks = 0; s->pairs = 0; s->nb_most = 0; s->splits = splits;
    s->both = issuers == 2 && !unit;
    s->step = issuers == 2 && unit ? 2 : 1;
    for (int sp = 0; sp < splits; ++sp) {
        const int k0 = n * sp / splits, k1 = n * (sp + 1) / splits;
        for (int par = 0; par < s->step; ++par) {
            const int count = ceil_div(k1 - k0 - par, s->step);
            if (count <= 0) continue;
            if (s->ranks == IB_MAX_RANKS || count > IB_MAX_NB) return false;
            if (par == 1) s->pairs |= 1u << sp;
            s->first[s->ranks] = (uint16_t)(k0 + par);
            s->count[s->ranks] = (uint8_t)count;
            s->nb_most = std::max(s->nb_most, count);
            ++s->ranks;
        }
    }
    return true;
}

// Shared memory of a launch; false where it does not fit.
bool ib_layout(bool bf16, int nkb1, IbShape* s) {
    const size_t xs = a_stage_of(s->rows), ds = bf16 ? (size_t)pad8(s->px) * 64 : a_stage_of(s->px);
    const size_t conv = bf16 ? (size_t)nkb1 * pad8(s->rows) * 64 : 0;
    const size_t w1 = (size_t)nkb1 * s->nb_most * (bf16 ? 2048 : 4096), w2 = (size_t)s->nb_most * s->BN2 * (bf16 ? 64 : 128);
    const size_t recv = s->ranks > 1 ? (size_t)s->ranks * ceil_div(s->px, s->ranks) * s->BN2 * 4 : 0;
    s->w1_off = (uint32_t)(nkb1 * xs);
    s->conv_off = (uint32_t)align_up(s->w1_off + w1, 1024);
    // first the operands of the expansion, then its output, then the rows received; behind them those of the projection, then its rows
    const size_t r0 = align_up(std::max({(size_t)s->conv_off + conv, (size_t)s->nb_most * s->rows * IB_PITCH, recv}), 1024);
    s->d_off = (uint32_t)r0;
    s->w2_off = (uint32_t)align_up(r0 + s->nb_most * ds, 1024);
    const size_t r1 = std::max((size_t)s->w2_off + w2, r0 + (size_t)s->px * s->BN2 * 4);
    s->bar_off = (uint32_t)align_up(r1, 128);
    s->par_off = (uint32_t)align_up(s->bar_off + IB_BAR_BYTES, 16);
    s->smem_bytes = 1024 + s->par_off + 4 * ((size_t)s->nb_most * (64 + 288) + s->BN2);
    // an MMA reads 128 rows of A, the last block's included
    s->smem_bytes = std::max({s->smem_bytes, (size_t)1024 + (nkb1 - 1) * xs + A_STAGE_BYTES, (size_t)1024 + s->d_off + (s->nb_most - 1) * ds + A_STAGE_BYTES,
                              (size_t)1024 + s->conv_off + conv + A_STAGE_BYTES / 2});
    s->tmem_cols = 32;
    while (s->tmem_cols < std::max(s->issuers * s->nb_most * 32, (s->both ? 2 : 1) * s->BN2)) s->tmem_cols *= 2;
    if (s->ranks > 1) s->smem_bytes = std::max(s->smem_bytes, std::min((size_t)226 * 1024, tmem_share_bytes(s->tmem_cols)));   // (226 KB: an SM of its own)
    return s->smem_bytes <= 226u * 1024u && s->tmem_cols <= 512;
}

// Clusters that find SMs of their own.
int ib_lone(int ranks) {
    static constexpr int lone[10] = {148, 148, 74, 48, 33, 24, 24, 15, 15, 14};
    return ranks < 10 ? lone[ranks] : 7;
}
// Estimated time of a launch, us: waves of clusters x (start and phases of fixed length, the pixels' loads, the passes over accumulators
// and pixels), plus the bytes from L2 over all CTAs.  A cluster of more than nine CTAs finds one place in a GPC; a second CTA on an SM adds half.
// Fitted to 1867 launches of 78 blocks (TF32, 96 - 224 pixels): the chosen shapes are 1.1 % above the best measured ones on average (BF16,
// 67 blocks: 1.5 %).
int ib_occupancy(const IbShape& s) { return std::max(1, std::min({(int)(227u * 1024u / (s.smem_bytes + 1024)), 512 / s.tmem_cols, 2})); }
double ib_us(const IbShape& s, bool bf16, int nkb1, int stride, int occ) {
    const int one = ib_lone(s.ranks), clusters = s.tiles_h * s.tiles_w;
    const int waves = ceil_div(clusters, one * occ), resident = std::min(occ, ceil_div(clusters, one));
    const double weights = (bf16 ? 0.5 : 1.0) * s.nb_most * (nkb1 * 4096.0 + s.BN2 * 128.0), pixels = nkb1 * s.rows * 128.0;
    const double phases = 8.4e-5 * pixels + 0.5 * s.nb_most + (stride == 2 ? 0.69 : 0.5) * ceil_div(s.nb_most * s.px, IB_THREADS / 16) +
                          0.06 * ceil_div(ceil_div(s.px, s.ranks) * s.BN2, IB_THREADS);
    return waves * (1.69 + phases * (0.5 + 0.5 * resident)) + 3.85e-8 * (weights + pixels) * clusters * s.ranks + (occ == 1 ? 0.29 : 0.0);
}

IbShape search_ib(bool bf16, int C, int E, int K, int OH, int OW, int stride, int splits, int issuers) {
    const int nkb1 = ceil_div(C, 32);
    IbShape best{};
    best.t = 1e30;
    // The patch heights and widths there are: the least of every number of rows, while a halo of three columns fits the rows of an MMA.
    int heights[BM], widths[BM];
    auto sizes = [&](int n, int* out) {
        int count = 0;
        for (int v = std::min(n, (BM / 3 - 3) / stride + 1); v >= 1; --v)
            if (ceil_div(n, ceil_div(n, v)) == v) out[count++] = v;
        return count;
    };
    const int nh = sizes(OH, heights), nw = sizes(OW, widths);
    for (int unit = 0; unit < (issuers == 2 ? 2 : 1); ++unit) {
        IbShape s{};
        s.BN2 = ceil_div(K, 16) * 16;
        s.issuers = issuers;
        if (!ib_ranks(ceil_div(E, 32), splits, issuers, unit != 0, &s)) continue;
        if (s.BN2 > (s.both ? 256 : 512)) continue;
        // Patches of the least height and width for their numbers of rows and columns, no more than four times as long as wide unless as long as the
        // image.
        for (int h = 0; h < nh; ++h) {
            const int ph = heights[h], hh = (ph - 1) * stride + 3;
            for (int w = 0; w < nw; ++w) {
                const int pw = widths[w], hw = (pw - 1) * stride + 3;
                if (hh * hw > BM) continue;
                if ((ph > 4 * pw && ph < OH) || (pw > 4 * ph && pw < OW)) continue;
                s.ph = ph; s.pw = pw; s.hw = hw; s.rows = hh * hw; s.px = ph * pw;
                s.tiles_h = ceil_div(OH, ph); s.tiles_w = ceil_div(OW, pw);
                if (ib_us(s, bf16, nkb1, stride, 2) >= best.t || !ib_layout(bf16, nkb1, &s)) continue;
                s.t = ib_us(s, bf16, nkb1, stride, ib_occupancy(s));
                if (s.t < best.t - 1e-9) best = s;
            }
        }
    }
    return best;
}

}  // namespace

// The block's launch, if it is to be one: 1x1 expansion (TF32 or BF16 GEMM), 3x3 depthwise and 1x1 projection of the same math, whose
// activations the GEMMs read in place.
static bool ib_shape(const nnv_layer_desc_t& a, const nnv_layer_desc_t& d, const nnv_layer_desc_t& p, int math, IbShape* out) {
    const int mode = math == NNV_MATH_BF16 ? GEMM_BF16_CVT : GEMM_TF32, align = math == NNV_MATH_BF16 ? 8 : 4;
    const Tuning& tn = tuning();
    if (tn.gemm_bn || tn.gemm_ring || tn.smallp_splits || (math == NNV_MATH_BF16 && !tn.bf16cvt)) return false;   // overrides of the GEMMs' launches
    if (a.R != 1 || a.S != 1 || a.stride != 1 || a.pad != 0 || a.groups != 1 || p.R != 1 || p.S != 1 || p.stride != 1 || p.pad != 0 || p.groups != 1) return false;
    if (d.R != 3 || d.S != 3 || d.pad != 1 || (d.stride != 1 && d.stride != 2) || d.groups != d.C || d.K != d.C || d.C != a.K || p.C != d.K) return false;
    if (a.act == 0 || d.act == 0) return false;                // (a clamp would turn the NaNs of a linear layer into numbers)
    if (a.C % align || a.K % align || p.K % 4 || a.C > 32 * IB_MAX_KB || a.K > 32 * 255 || p.K > 512) return false;
    const int OH = (a.H - 1) / d.stride + 1, OW = (a.W - 1) / d.stride + 1, nkb1 = ceil_div(a.C, 32), nkb2 = ceil_div(a.K, 32);
    if ((double)a.H * a.W * a.K >= 2.0e9 || (double)OH * OW * p.K >= 2.0e9) return false;         // 32-bit places in the outputs
    const GemmTiling t1 = pick_gemm_tiling(mode, a.H * a.W, a.K, 1, nkb1), t2 = pick_gemm_tiling(mode, OH * OW, p.K, 1, nkb2);
    if (t1.splits != 1) return false;
    GemmShape g1, g2;
    if (gemm_shape(mode, t1, a.H * a.W, a.K, 1, nkb1, true, false, &g1) != NNV_OK) return false;
    if (gemm_shape(mode, t2, OH * OW, p.K, 1, nkb2, true, p.in1 >= 0, &g2) != NNV_OK) return false;
    if (g1.issuers != g2.issuers) return false;
    *out = search_ib(math == NNV_MATH_BF16, a.C, a.K, p.K, OH, OW, d.stride, g2.splits, g2.issuers);
    return out->t < 1e29;
}

// Searches for the shape of a block and launches of one so far, for the tests.
static std::atomic<uint64_t> g_ib_searches{0}, g_ib_launches{0};

const IbShape* inverted_bottleneck_shape(const nnv_layer_desc_t& a, const nnv_layer_desc_t& d, const nnv_layer_desc_t& p, int math, IbEntry* e) {
    const Tuning& tn = tuning();
    if (!e->known || e->tuning != tn.generation) {
        g_ib_searches.fetch_add(1, std::memory_order_relaxed);
        e->use = ib_shape(a, d, p, math, &e->shape);
        e->tuning = tn.generation;
        e->known = true;
    }
    return e->use ? &e->shape : nullptr;
}

nnv_status_t launch_inverted_bottleneck(const nnv_layer_desc_t& a, const nnv_layer_desc_t& d, const nnv_layer_desc_t& p, int math, const IbShape& shape,
                                        const IbBuffers& io, cudaStream_t st) {
    NNV_TRY(gemm_tc_init());
    const IbShape* const s = &shape;
    const bool bf16 = math == NNV_MATH_BF16;
    const int Qp1 = (a.C + 7) / 8 * 8, Qp2 = (p.C + 7) / 8 * 8;
    CUtensorMap tmX, tmW1, tmW2;
    const int w2_boxes = s->BN2 > 256 ? 2 : 1;
    NNV_TRY(encode_halo_operand(&tmX, io.x, a.C, a.H, a.W, s->rows / s->hw, s->hw));
    if (bf16) {
        NNV_TRY(encode_bf16_weights(&tmW1, io.w1, Qp1, Qp1, a.K, 32));
        NNV_TRY(encode_bf16_weights(&tmW2, io.w2, Qp2, Qp2, p.K, s->BN2 / w2_boxes));
    } else {
        NNV_TRY(encode_operand(&tmW1, io.w1, false, a.C, a.K, 1, Qp1, (int64_t)a.K * Qp1, 32));
        NNV_TRY(encode_operand(&tmW2, io.w2, false, p.C, p.K, 1, Qp2, (int64_t)p.K * Qp2, s->BN2 / w2_boxes));
    }
    IbDev g{};
    g.early = io.early;
    g.e = io.e; g.d = io.d; g.y = io.y; g.b1 = io.b1; g.b2 = io.b2; g.b3 = io.b3; g.addend = io.addend; g.wd = io.wd;
    g.E = a.K; g.K = p.K; g.H = a.H; g.W = a.W; g.OH = p.H; g.OW = p.W; g.stride = d.stride;
    g.most1 = a.act == 2 ? 6.f : INFINITY; g.most2 = d.act == 2 ? 6.f : INFINITY; g.act3 = p.act;
    g.ph = s->ph; g.pw = s->pw; g.hw = s->hw; g.rows = s->rows; g.px = s->px; g.tiles_w = s->tiles_w;
    g.nkb1 = ceil_div(a.C, 32); g.nb_most = s->nb_most; g.step = s->step; g.both = s->both; g.ranks = s->ranks; g.splits = s->splits; g.BN2 = s->BN2;
    g.w2_boxes = w2_boxes; g.issuers = s->issuers; g.tmem_cols = s->tmem_cols;
    g.magic_hw = 0xFFFFFFFFu / (uint32_t)s->hw + 1u; g.magic_pw = 0xFFFFFFFFu / (uint32_t)s->pw + 1u;
    g.magic_nch = 0xFFFFFFFFu / (uint32_t)(s->BN2 / 4) + 1u; g.magic_n = 0xFFFFFFFFu / (uint32_t)s->BN2 + 1u; g.magic_px = 0xFFFFFFFFu / (uint32_t)s->px + 1u;
    g.w1_off = s->w1_off; g.conv_off = s->conv_off; g.d_off = s->d_off; g.w2_off = s->w2_off; g.bar_off = s->bar_off; g.par_off = s->par_off;
    std::copy(std::begin(s->first), std::end(s->first), g.first);
    std::copy(std::begin(s->count), std::end(s->count), g.count);
    g.pairs = s->pairs;
    const dim3 grid(s->tiles_h * s->tiles_w, 1, s->ranks);
    g_ib_launches.fetch_add(1, std::memory_order_relaxed);
    NNV_CUDA(launch_pdl_cluster(ib_kernels[bf16][s->ranks > 1], grid, dim3(IB_THREADS), s->smem_bytes, st, s->ranks, tmX, tmW1, tmW2, g));
    return NNV_OK;
}

}  // namespace nnv

// Host-side launch shape of gemm_tc_kernel for the tests (kernel mode, K blocks of 128 bytes).
extern "C" int nnv_internal_gemm_shape(int mode, int M, int N, int batch, int nkb, int staged, int addend, int32_t* out) {
    using namespace nnv;
    GemmShape s;
    const nnv_status_t st = gemm_shape(mode, pick_gemm_tiling(mode, M, N, batch, nkb), M, N, batch, nkb, staged != 0, addend != 0, &s);
    if (st != NNV_OK) return st;
    const int32_t v[] = {s.BN, s.splits, s.rows, s.m_tiles, s.issuers, s.ring, s.tmem_cols, (int32_t)s.bar_off, (int32_t)s.recv_off,
                         (int32_t)s.stage_off, (int32_t)s.smem_bytes, (int32_t)gemm_stage_bytes(mode, s.BN, s.rows), gemm_tc_threads(mode)};
    std::copy(std::begin(v), std::end(v), out);
    return NNV_OK;
}

// The launch shape of an inverted-residual block C -> E -> K on an H x W image, for the tests; 1: the layers run as launches of their own.
extern "C" int nnv_internal_ib_shape(int bf16, int C, int E, int K, int H, int W, int stride, int residual, int32_t* out) {
    using namespace nnv;
    nnv_layer_desc_t a{}, d{}, p{};
    a.op = d.op = p.op = NNV_OP_CONV;
    a.act = d.act = 1;
    a.C = C; a.K = E; a.R = a.S = 1; a.stride = 1; a.groups = 1; a.H = H; a.W = W; a.in1 = -1;
    d.C = d.K = d.groups = E; d.R = d.S = 3; d.stride = stride; d.pad = 1; d.H = H; d.W = W; d.in1 = -1;
    p.C = E; p.K = K; p.R = p.S = 1; p.stride = 1; p.groups = 1; p.H = (H - 1) / stride + 1; p.W = (W - 1) / stride + 1; p.in1 = residual ? 0 : -1;
    IbEntry entry;
    const IbShape* s = inverted_bottleneck_shape(a, d, p, bf16 ? NNV_MATH_BF16 : NNV_MATH_TF32, &entry);
    if (!s) return 1;
    const int32_t v[] = {s->ph, s->pw, s->hw, s->rows, s->px, s->tiles_h, s->tiles_w, s->ranks, s->both, s->step, s->nb_most, s->BN2, s->issuers,
                         s->tmem_cols, (int32_t)s->w1_off, (int32_t)s->conv_off, (int32_t)s->d_off, (int32_t)s->w2_off, (int32_t)s->bar_off,
                         (int32_t)s->par_off, (int32_t)s->smem_bytes, (int32_t)s->pairs};
    std::copy(std::begin(v), std::end(v), out);
    for (int r = 0; r < IB_MAX_RANKS; ++r) { out[24 + 2 * r] = r < s->ranks ? s->first[r] : -1; out[25 + 2 * r] = r < s->ranks ? s->count[r] : 0; }
    return 0;
}

extern "C" uint64_t nnv_internal_ib_launches() { return nnv::g_ib_launches.load(std::memory_order_relaxed); }
extern "C" uint64_t nnv_internal_ib_searches() { return nnv::g_ib_searches.load(std::memory_order_relaxed); }

extern "C" int nnv_internal_gemm_loaders(int mode, int nkb, int ring) { return nnv::gemm_loaders(mode, nkb, ring); }

// The 3x3 halo kernel's tiling for a TF32 layer, for the tests; out[0] = 0: the implicit GEMM takes the layer.
extern "C" int nnv_internal_conv3x3_shape(int C, int H, int W, int N, int32_t* out) {
    using namespace nnv;
    ConvTiling t{};
    const GemmTiling gemm = pick_gemm_tiling(GEMM_TF32, H * W, N, 1, 9 * ceil_div(C, 32));
    const bool use = pick_conv_tiling(C, H, W, N, gemm, &t);
    const int32_t v[] = {use, t.MT, t.BN, t.splits, t.na, t.nb, t.tmem_cols, (int32_t)t.smem, gemm.waves};
    std::copy(std::begin(v), std::end(v), out);
    return NNV_OK;
}

// The BF16 3x3 kernel's launch shape, for the tests; BN = 0: the tiling that the library picks.
extern "C" int nnv_internal_conv3x3_bf16_shape(int C, int H, int W, int N, int BN, int splits, int32_t* out) {
    using namespace nnv;
    if (BN == 0) {
        const ConvBTiling t = pick_conv_bf16_tiling(C, H, W, N);
        BN = t.BN; splits = t.splits;
    }
    ConvBShape s;
    const nnv_status_t st = conv_bf16_shape(C, BN, splits, &s);
    if (st != NNV_OK) return st;
    const int32_t v[] = {BN, s.splits, s.na, s.nb, s.issuers, s.tmem_cols, (int32_t)s.b_off, (int32_t)s.bar_off, (int32_t)s.recv_off, (int32_t)s.smem_bytes};
    std::copy(std::begin(v), std::end(v), out);
    return NNV_OK;
}
