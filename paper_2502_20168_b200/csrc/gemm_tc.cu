#include <type_traits>
// bf16 projections on the 5th-generation tensor cores (tcgen05.mma, accumulators in tensor
// memory, operands staged in shared memory by TMA).  The kernels:
//
//  * gemm_tc_tn_pair_kernel: out[m, n] = sum_k A[m, k] * W[n, k]  (both operands K-contiguous).  Persistent
//    clusters of two CTAs walking 256 x 256 accumulator tiles (problems with fewer tiles than CTA pairs:
//    gemm_tc_small.cu).  A = activations or states [B*T, K]; W = packed parameters.  With kSplitW
//    the 256 accumulator columns of a tile hold the products with the high and the low bf16 halves of 128
//    weight rows, summed in the epilogue (weights then carry ~16 mantissa bits; see
//    pack_params_kernel).  With a product schedule the accumulator sums several products of bf16
//    planes of both operands (fp32-accurate results, see gemm_tc_small.cu).  Epilogues: fp32 store; bf16
//    acc + diag * skip; the same with column sums of skip * dot; fp32 store with a gated bf16 result.
//  * gemm_scan_fwd_kernel / gemm_scan_bwd_kernel: the pair kernel with the scan of Sec. III-B (and its
//    adjoint) in the epilogue, so that Bu and g_x never reach memory.  The CTAs of a pair take two
//    sequences, or (kTPair) alternate tiles of one.
//  * gemm_tc_nt_kernel / gemm_tc_nt_pair_kernel: part[s, i, j] = sum_{m in slice s} A[m, i] * Bm[m, j]
//    (both operands contiguous in the output index, i.e. MN-major), split over the B*T rows: the weight
//    gradients.
//
// Warp roles in all: warp 0 issues TMA loads, warp 1 owns tensor memory and issues the MMAs, the other
// warps drain accumulators (each may read one TMEM lane quarter).  Every mbarrier wait is bounded; a wait
// that gives up raises a CTA-wide abort flag, the status word of the workspace header is set, tensor
// memory is released and the kernel returns.
#include <algorithm>
#include <utility>

#include "kernels.h"
#include "tcgen05.cuh"

namespace ssm {
namespace tc {
using namespace tma;

constexpr int BN = 256;   // accumulator columns per tile
constexpr int kStages = 4;      // shared-memory stages of the NT kernel (and size of the barrier arrays)
constexpr int kABytes = BM * BK * 2;
constexpr int kBBytes = BN * BK * 2;
constexpr int kStageBytes = kABytes + kBBytes;
// NT kernels: producer, MMA and epilogue warps; slices of several segments (nt_epilogue) take two warps per TMEM lane quarter
__host__ __device__ constexpr int nt_epi_warps(bool segs) { return segs ? 8 : 4; }
__host__ __device__ constexpr int nt_threads(bool segs) { return 64 + 32 * nt_epi_warps(segs); }
__host__ __device__ constexpr int nt_epi_cols(bool segs) { return BN / 2 * 4 / nt_epi_warps(segs); }   // columns of a warp
constexpr int kTnEpiWarps = 8;     // TN kernel: two epilogue warps per TMEM lane quarter
constexpr int kTnThreads = 64 + 32 * kTnEpiWarps;
constexpr int kTmemCols = 512;  // two accumulator buffers of BN columns
constexpr int kStagingBytes = kTnEpiWarps * 32 * 32 * 4;  // per epilogue warp: 32 rows x 32 fp32 columns
constexpr int kMaxDiag = 4096;                  // widest output whose diagonal fits the shared copy
constexpr int kSkipBytes = kTnEpiWarps * 2 * 32 * 32 * 2;   // two 32 x 32 bf16 skip tiles per epilogue warp
// Epilogues of the TN kernels: 0 = fp32 result; 1 = bf16(acc + diag * skip); 2 = fp32 result AND
// a gated bf16 result skip * sigmoid(acc) (needs a staging buffer for each); 3 = epilogue 1 AND the
// column sums of skip * dot over the rows this CTA drains (a second operand tile beside every skip
// tile, per-warp sums in shared memory): CTA pairs only, outputs of at most kDotMaxN columns.
constexpr int kDotMaxN = 1024;
__host__ __device__ constexpr int tn_skip_bytes(int epi) { return epi == 0 ? 0 : (epi == 3 ? 2 * kSkipBytes : kSkipBytes); }
__host__ __device__ constexpr int tn_diag_bytes(int epi) {
    return epi == 1 ? kMaxDiag * 4 : (epi == 3 ? kDotMaxN * 4 + kTnEpiWarps * (kDotMaxN / 2) * 4 : 0);
}
__host__ __device__ constexpr int tn_staging_bytes(int epi) { return epi == 2 ? kStagingBytes + kStagingBytes / 2 : kStagingBytes; }
constexpr size_t kNtSmemBytes = (size_t)kStages * kStageBytes + 1024 + 256;

struct Smem {
    uint8_t* tiles;       // 1024-byte aligned
    uint8_t* staging;     // epilogue transpose buffers
    float* diag;          // copy of the epilogue's diagonal
    uint8_t* skipbuf;     // bf16 epilogue: per epilogue warp two 32 x 32 bf16 tiles of the skip operand
    // mbarriers of a kind sit 8 bytes apart: their addresses are computed, so that no array is indexed at
    // run time (that would put this struct into local memory)
    uint32_t full0, empty0, tmem_full0, tmem_empty0, skip_full0;
    __device__ __forceinline__ uint32_t full(int i) const { return full0 + 8u * (uint32_t)i; }
    __device__ __forceinline__ uint32_t empty(int i) const { return empty0 + 8u * (uint32_t)i; }
    __device__ __forceinline__ uint32_t tmem_full(int i) const { return tmem_full0 + 8u * (uint32_t)i; }
    __device__ __forceinline__ uint32_t tmem_empty(int i) const { return tmem_empty0 + 8u * (uint32_t)i; }
    __device__ __forceinline__ uint32_t skip_full(int i) const { return skip_full0 + 8u * (uint32_t)i; }
    uint32_t tmem_slot;   // where tcgen05.alloc writes the base address
    volatile int* abort_flag;
    // Kernels whose epilogue warps meet at barriers: a wait of one of those warps gave up.  Written before their barrier and
    // read after it, so that all of them leave or none (the load and MMA warps may raise abort_flag between two reads).
    // It takes the first skip slot, which these kernels do not use, so that one base address serves both flags.
    __device__ __forceinline__ volatile int* epi_abort() const { return abort_flag + 1; }
    volatile uint32_t* tmem_slot_ptr;
};

// Layout: [stages][epilogue staging][skip tiles][diag copy][barriers]; the NT kernel has none of the
// epilogue buffers.
__device__ __forceinline__ Smem carve_smem(uint8_t* raw, int stages, int staging_bytes, int diag_bytes,
                                           int stage_bytes = kStageBytes, int skip_bytes = 0) {
    Smem s;
    uintptr_t base = (reinterpret_cast<uintptr_t>(raw) + 1023) & ~(uintptr_t)1023;
    s.tiles = reinterpret_cast<uint8_t*>(base);
    s.staging = s.tiles + (size_t)stages * stage_bytes;
    s.skipbuf = s.staging + staging_bytes;
    s.diag = reinterpret_cast<float*>(s.skipbuf + skip_bytes);
    uint8_t* bars = s.skipbuf + skip_bytes + diag_bytes;
    s.full0 = smem_u32(bars);
    s.empty0 = smem_u32(bars + 8 * kStages);
    s.tmem_full0 = smem_u32(bars + 8 * (2 * kStages));
    s.tmem_empty0 = smem_u32(bars + 8 * (2 * kStages + 2));
    s.tmem_slot_ptr = reinterpret_cast<volatile uint32_t*>(bars + 8 * (2 * kStages + 4));
    s.tmem_slot = smem_u32(bars + 8 * (2 * kStages + 4));
    s.abort_flag = reinterpret_cast<volatile int*>(bars + 8 * (2 * kStages + 4) + 4);
    s.skip_full0 = smem_u32(bars + 8 * (2 * kStages + 5));
    return s;
}

// Common prologue: barriers, tensor memory.  Returns the TMEM base address.
__device__ __forceinline__ uint32_t prologue(const Smem& s, int warp, int lane, int epilogue_threads) {
    if (threadIdx.x == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(s.full(i), 1);
            mbar_init(s.empty(i), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(s.tmem_full(i), 1);
            mbar_init(s.tmem_empty(i), epilogue_threads);
        }
        for (int i = 0; i < 2 * kTnEpiWarps; ++i) mbar_init(s.skip_full(i), 1);
        *s.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(s.tmem_slot, kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    (void)lane;
    return *s.tmem_slot_ptr;
}

__device__ __forceinline__ void epilogue_exit(const Smem& s, int warp, uint32_t tmem_base, WsHeader* hdr) {
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) {
        __syncwarp();
        tmem_dealloc(tmem_base, kTmemCols);
    }
    if (threadIdx.x == 0 && *s.abort_flag && hdr) hdr->status = SSM_ERR_TIMEOUT;
}

// ---------------------------------------------------------------------------------------------
// TN kernel
// ---------------------------------------------------------------------------------------------
struct TnParams {
    int M;            // rows of A / out
    int n_tiles;      // accumulator tiles along N (each BN columns of W rows)
    int k_blocks;     // K / BK
    int ldo;          // leading dimension of out (and skip): the number of output columns
    const float* diag;
    WsHeader* hdr;
    const char* a_base;   // A as bytes; rows are K * 2 bytes apart and contiguous
    int a_row_bytes;
    float* dot_part;      // epilogue 3: [CTAs, ldo] column sums of skip * dot, one row per CTA
    // Sum of several products in one accumulator (operands split into bf16 planes laid side by side along K:
    // plane a of A in columns [a Kp, (a + 1) Kp), likewise W): k-block kb belongs to product kb / kpp, which
    // takes plane (pa >> 4 j) & 15 of A and plane (pb >> 4 j) & 15 of W.  kpp = 0: one product, planes 0.
    int kpp;              // k-blocks per product (Kp / BK)
    uint32_t pa, pb;
    __device__ __forceinline__ int a_col(int kb) const {
        if (kpp == 0) return kb * BK;
        const int j = kb / kpp;
        return (int)((pa >> (4 * j)) & 15u) * kpp * BK + (kb - j * kpp) * BK;
    }
    __device__ __forceinline__ int w_col(int kb) const {
        if (kpp == 0) return kb * BK;
        const int j = kb / kpp;
        return (int)((pb >> (4 * j)) & 15u) * kpp * BK + (kb - j * kpp) * BK;
    }
};

// sums[c] += sum over the 32 rows of a[row][c] * b[row][c], c < 32, for two 32 x 32 bf16 tiles in shared memory (64-byte
// rows, 64-byte swizzle).  The sums are the diagonal of a^T b: eight 16 x 8 x 16 matrix instructions, of whose results one
// element in 16 is used.  (On the CUDA cores a lane holds a row, so that the products have to be turned round: 32 products
// and a butterfly of 31 shuffles, about 190 instructions a tile against 40: du and dD of 16384 x 512 x 512
// 24.9 -> 20.9 us.)
__device__ __forceinline__ void add_column_dots(uint32_t a, uint32_t b, int lane, float* sums) {
    const int g = lane >> 2, t = lane & 3;
    float d[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) d[j][e] = 0.f;
    // 8 x 8 blocks, transposed on the way: lanes 8 i .. 8 i + 7 point at the rows of block i of four
    const int r8 = lane & 7, blk = lane >> 3;
    auto addr = [&](uint32_t base, int row, int chunk) { return base + (uint32_t)(row * 64 + ((chunk ^ ((row >> 1) & 3)) << 4)); };
    auto load4 = [](uint32_t p, uint32_t (&f)[4]) {
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                     : "=r"(f[0]), "=r"(f[1]), "=r"(f[2]), "=r"(f[3]) : "r"(p) : "memory");
    };
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            uint32_t fa[4], fb[4];   // fa: (chunk, rows) = (2i, lo), (2i + 1, lo), (2i, hi), (2i + 1, hi); fb: (2i, lo), (2i, hi), ...
            load4(addr(a, 16 * k + 8 * (blk >> 1) + r8, 2 * i + (blk & 1)), fa);
            load4(addr(b, 16 * k + 8 * (blk & 1) + r8, 2 * i + (blk >> 1)), fb);
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                float(&c)[4] = d[2 * i + j];
                asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                             : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                             : "r"(fa[0]), "r"(fa[1]), "r"(fa[2]), "r"(fa[3]), "r"(fb[2 * j]), "r"(fb[2 * j + 1]));
            }
        }
    // column 8 j + g of block j is element (g, g) of its half of the results: with the lanes whose t is g / 2
    if (t == (g >> 1)) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int e = 2 * (j & 1);
            sums[8 * j + g] += (g & 1) ? d[j][e + 1] : d[j][e];
        }
    }
}

// One epilogue warp's share of a finished accumulator tile: rows m0 + 32 (warp % 4) .. + 31, one half
// of the tile's output columns (from n_out0), in slabs of 32 columns; a lane holds one row of a slab.
// Waits for the tile's MMAs; false when aborting.
//  kEpi 0: fp32 results.  The slab goes through a 128-byte-swizzled staging buffer and leaves as
//          one TMA store of a 32 x 32 box (rows past M are clipped by the unit).
//  kEpi 1: out = bf16(acc + diag[n] * skip[m, n]).  The skip slab arrives by TMA (two buffers per
//          warp, fetched two slabs ahead, the first ones while the tile's MMAs still run) and the
//          bf16 slab leaves by TMA, both as 32 x 32 boxes with the 64-byte swizzle, so a lane reads
//          and writes its own 64-byte row without bank conflicts and nothing passes through the
//          load/store path to global memory.  `skip_phase`: the warp's barrier parities (bit b).
//          With next_m0 >= 0 (the tile this warp drains next) a buffer that has been read is refilled with the next
//          tile's first slabs, so that they have arrived when that tile starts; *skip_ahead says whether the
//          tile now starting found its first slabs requested already.
template <int kEpi, bool kSplitW, int kCols = BN>
__device__ __forceinline__ bool tn_drain_tile(const Smem& s, const TnParams& p, const CUtensorMap* tmOut,
                                              const CUtensorMap* tmSkip, const CUtensorMap* tmGate, int warp, int lane,
                                              int m0, int n_out0, int acc, uint32_t acc_phase, uint32_t tmem_base,
                                              uint32_t& skip_phase, int next_m0 = -1, int next_n_out0 = 0,
                                              bool* skip_ahead = nullptr) {
    constexpr int kOutCols = kSplitW ? BN / 2 : kCols;
    const int q = warp & 3;             // TMEM lane quarter this warp may read
    const int half = (warp - 2) >> 2;   // which half of the tile's columns this warp drains
    const int row0 = m0 + q * 32;       // first of this warp's 32 rows
    constexpr int kSlabs = kOutCols / 32 / 2;
    const int slab0 = half * kSlabs;    // this warp's slabs: slab0 .. slab0 + kSlabs - 1
    const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * BN);
    uint8_t* stg_bytes = s.staging + (size_t)(warp - 2) * (tn_staging_bytes(kEpi) / kTnEpiWarps);

    if (kEpi == 0) {
        if (!mbar_wait(s.tmem_full(acc), acc_phase, s.abort_flag)) return false;
        tc_fence_after();
        float4* stg = reinterpret_cast<float4*>(stg_bytes);
#pragma unroll
        for (int sl = 0; sl < kSlabs; ++sl) {
            const int c = (slab0 + sl) * 32;
            uint32_t r[32], r2[32];
            tmem_ld32(t_row + (uint32_t)c, r);
            if (kSplitW) tmem_ld32(t_row + (uint32_t)(BN / 2 + c), r2);
            tmem_ld_wait();
            if (elect_one()) tma_store_wait_read();   // the previous slab has left the staging buffer
            __syncwarp();
            // 16-byte chunk j of row `lane` sits at chunk j ^ (lane & 7): the 128-byte swizzle
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                float4 v = make_float4(__uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1]),
                                       __uint_as_float(r[4 * j + 2]), __uint_as_float(r[4 * j + 3]));
                if (kSplitW) {
                    v.x += __uint_as_float(r2[4 * j]);
                    v.y += __uint_as_float(r2[4 * j + 1]);
                    v.z += __uint_as_float(r2[4 * j + 2]);
                    v.w += __uint_as_float(r2[4 * j + 3]);
                }
                stg[lane * 8 + (j ^ (lane & 7))] = v;
            }
            fence_async_smem();
            __syncwarp();
            if (row0 < p.M && n_out0 + c < p.ldo && elect_one()) tma_store_2d(tmOut, smem_u32(stg), n_out0 + c, row0);
        }
        return true;
    }

    // ---- kEpi == 1, 2, 3: the skip operand arrives by TMA (kEpi 3: and the dot operand beside it)
    constexpr bool kDot = kEpi == 3;
    const int w = warp - 2;
    uint8_t* skb = s.skipbuf + (size_t)w * (kDot ? 8192 : 4096);   // two 2 KB skip tiles (then two dot tiles)
    const uint32_t sbar[2] = {s.skip_full(2 * w), s.skip_full(2 * w + 1)};
    const int swz = (lane >> 1) & 3;               // 64-byte swizzle: chunk c of row `lane` sits at chunk c ^ swz
    auto fetch_skip_at = [&](int sl, int n_first, int row_first) {
        const int b = sl & 1;
        mbar_expect_tx(sbar[b], kDot ? 4096 : 2048);
        tma_load_2d(smem_u32(skb + b * 2048), tmSkip, sbar[b], n_first + (slab0 + sl) * 32, row_first);
        if (kDot) tma_load_2d(smem_u32(skb + 4096 + b * 2048), tmGate, sbar[b], n_first + (slab0 + sl) * 32, row_first);
    };
    auto fetch_skip = [&](int sl) { fetch_skip_at(sl, n_out0, row0); };
    static_assert(kSlabs % 2 == 0, "slab s of the next tile takes the buffer of slab s of this one");
    const bool ahead = skip_ahead && *skip_ahead;   // this tile's first two slabs were requested while the last one was drained
    const bool prefetch_next = kEpi != 2 && skip_ahead && next_m0 >= 0;
    if (skip_ahead) *skip_ahead = prefetch_next;
    if (!ahead && elect_one()) {
        fence_async_smem();   // (the lanes' reads of the previous tile's last slabs: fenced and joined there)
        fetch_skip(0);
        if (kSlabs > 1) fetch_skip(1);
    }
    if (!mbar_wait(s.tmem_full(acc), acc_phase, s.abort_flag)) return false;
    tc_fence_after();
    if (kEpi == 2) {
        // z = acc goes out in fp32, skip * sigmoid(z) in bf16; one staging buffer each
        float4* stg = reinterpret_cast<float4*>(stg_bytes);
        uint8_t* ob = stg_bytes + 4096;
#pragma unroll
        for (int sl = 0; sl < kSlabs; ++sl) {
            const int c = (slab0 + sl) * 32, b = sl & 1;
            uint32_t r[32], r2[32];
            tmem_ld32(t_row + (uint32_t)c, r);
            if (kSplitW) tmem_ld32(t_row + (uint32_t)(BN / 2 + c), r2);
            if (!mbar_wait(sbar[b], (skip_phase >> b) & 1u, s.abort_flag)) return false;
            skip_phase ^= 1u << b;
            uint4 sk[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) sk[j] = *reinterpret_cast<const uint4*>(skb + b * 2048 + lane * 64 + ((j ^ swz) << 4));
            tmem_ld_wait();
            // The refill below is a write of the async proxy over what these lanes have just read through the
            // generic proxy: without the proxy fences it can land before a lane's read has been served.
            fence_async_smem();
            __syncwarp();
            if (sl + 2 < kSlabs && elect_one()) {
                fence_async_smem();
                fetch_skip(sl + 2);
            }
            if (elect_one()) tma_store_wait_read();   // the previous slab has left both staging buffers
            __syncwarp();
            uint4 o[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const __nv_bfloat162* s2 = reinterpret_cast<const __nv_bfloat162*>(&sk[j]);
                __nv_bfloat162* o2 = reinterpret_cast<__nv_bfloat162*>(&o[j]);
                float z[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) z[e] = __uint_as_float(r[8 * j + e]) + (kSplitW ? __uint_as_float(r2[8 * j + e]) : 0.f);
                stg[lane * 8 + ((2 * j) ^ (lane & 7))] = make_float4(z[0], z[1], z[2], z[3]);
                stg[lane * 8 + ((2 * j + 1) ^ (lane & 7))] = make_float4(z[4], z[5], z[6], z[7]);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 sf = __bfloat1622float2(s2[e]);
                    o2[e] = __floats2bfloat162_rn(sf.x * sigmoid_f<__nv_bfloat16>(z[2 * e]), sf.y * sigmoid_f<__nv_bfloat16>(z[2 * e + 1]));
                }
                *reinterpret_cast<uint4*>(ob + lane * 64 + ((j ^ swz) << 4)) = o[j];
            }
            fence_async_smem();
            __syncwarp();
            if (row0 < p.M && n_out0 + c < p.ldo && elect_one()) {
                tma_store_2d(tmOut, smem_u32(stg), n_out0 + c, row0);
                tma_store_2d(tmGate, smem_u32(ob), n_out0 + c, row0);
            }
        }
        return true;
    }
#pragma unroll
    for (int sl = 0; sl < kSlabs; ++sl) {
        const int c = (slab0 + sl) * 32, b = sl & 1;
        uint32_t r[32];
        tmem_ld32(t_row + (uint32_t)c, r);
        if (!mbar_wait(sbar[b], (skip_phase >> b) & 1u, s.abort_flag)) return false;
        skip_phase ^= 1u << b;
        uint4 sk[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) sk[j] = *reinterpret_cast<const uint4*>(skb + b * 2048 + lane * 64 + ((j ^ swz) << 4));
        if (kDot) {
            const uint32_t dots = smem_u32(skb + b * 2048);
            float* acc_cols = s.diag + kDotMaxN + (size_t)w * (kDotMaxN / 2) + (n_out0 / kCols) * (kCols / 2) + sl * 32;
            add_column_dots(dots, dots + 4096, lane, acc_cols);   // (rows outside M were read as zero)
        }
        tmem_ld_wait();
        // Every lane has asked for its skip row; the buffer takes the slab after next.  That refill is a
        // write of the async proxy over data just read through the generic proxy: the proxy fences order the
        // two (without them the refill was seen to land before a lane's read had been served, when another
        // kernel shared the SMs and the skip rows came from L2).
        fence_async_smem();
        __syncwarp();
        if (elect_one()) {
            if (sl + 2 < kSlabs) {
                fence_async_smem();
                fetch_skip(sl + 2);
            } else if (prefetch_next) {   // the next tile's slab sl + 2 - kSlabs (0 or 1) into the buffer just read
                fence_async_smem();
                fetch_skip_at(sl + 2 - kSlabs, next_n_out0, next_m0 + q * 32);
            }
        }
        uint4 o[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 d0 = *reinterpret_cast<const float4*>(s.diag + n_out0 + c + 8 * j);
            const float4 d1 = *reinterpret_cast<const float4*>(s.diag + n_out0 + c + 8 * j + 4);
            const float dd[8] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y, d1.z, d1.w};
            const __nv_bfloat162* s2 = reinterpret_cast<const __nv_bfloat162*>(&sk[j]);
            __nv_bfloat162* o2 = reinterpret_cast<__nv_bfloat162*>(&o[j]);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float2 sf = __bfloat1622float2(s2[e]);
                o2[e] = __floats2bfloat162_rn(fmaf(dd[2 * e], sf.x, __uint_as_float(r[8 * j + 2 * e])),
                                              fmaf(dd[2 * e + 1], sf.y, __uint_as_float(r[8 * j + 2 * e + 1])));
            }
        }
        uint8_t* ob = stg_bytes + b * 2048;
        if (elect_one()) tma_store_wait_read_n<1>();   // the store from this buffer two slabs ago has read it
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 4; ++j) *reinterpret_cast<uint4*>(ob + lane * 64 + ((j ^ swz) << 4)) = o[j];
        fence_async_smem();
        __syncwarp();
        if (row0 < p.M && n_out0 + c < p.ldo && elect_one()) tma_store_2d(tmOut, smem_u32(ob), n_out0 + c, row0);
    }
    return true;
}

// ---------------------------------------------------------------------------------------------
// TN kernel on CTA pairs
// ---------------------------------------------------------------------------------------------
// kEpi: see tn_drain_tile.  kSplitW: columns [0,128) and [128,256) of the accumulator tile are the hi and lo weight
// halves of the same 128 output columns.  A cluster of two CTAs works on a 256 x 256 accumulator tile:
// CTA r holds rows m0 + 128 r .. of A and rows n0 + 128 r .. of the W tile, so every CTA brings
// in 32 KB per k-block instead of 48 KB for the same number of tensor-core cycles (operand
// delivery into the SM, not the tensor pipe, bounds a single-CTA kernel).  The leader (CTA 0)
// issues the MMAs; its `full` barriers count the bytes of both CTAs' loads; its commits arrive
// on the `empty` / `tmem_full` barriers of both CTAs; both CTAs' epilogue warps arrive on the
// leader's `tmem_empty` barriers.
constexpr int kPairStages = 4;
// (the epilogue with the column sums gives one operand stage up for its second operand tiles and its sums)
#ifndef SSM_PAIR_STAGES_BF16_EPILOGUE
#define SSM_PAIR_STAGES_BF16_EPILOGUE 4
#endif
__host__ __device__ constexpr int pair_stages(int epi) { return epi == 3 ? 3 : (epi == 1 ? SSM_PAIR_STAGES_BF16_EPILOGUE : kPairStages); }
__host__ __device__ constexpr int pair_stage_bytes(int cols) { return kABytes + cols / 2 * BK * 2; }
constexpr size_t pair_smem_bytes(int epi, int cols = BN) {
    return (size_t)pair_stages(epi) * pair_stage_bytes(cols) + tn_staging_bytes(epi) + tn_skip_bytes(epi) + tn_diag_bytes(epi) + 1024 +
           256;
}

// kCols: columns of a tile, BN, or BN / 2 for the bf16 epilogues where wider tiles leave pairs without work (narrow_tiles).
template <int kEpi, bool kSplitW, int kCols = BN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kTnThreads, 1)
gemm_tc_tn_pair_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmWh,
                       const __grid_constant__ CUtensorMap tmOut, const __grid_constant__ CUtensorMap tmSkip,
                       const __grid_constant__ CUtensorMap tmGate, TnParams p) {
    extern __shared__ uint8_t smem_raw[];
    constexpr int kSt = pair_stages(kEpi);
    constexpr int kStBytes = pair_stage_bytes(kCols);
    const Smem s = carve_smem(smem_raw, kSt, tn_staging_bytes(kEpi), tn_diag_bytes(kEpi), kStBytes,
                              tn_skip_bytes(kEpi));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    // barriers and tensor memory (both CTAs), then the whole pair meets
    if (threadIdx.x == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(s.full(i), 1);
            mbar_init(s.empty(i), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(s.tmem_full(i), 1);
            mbar_init(s.tmem_empty(i), 2 * 32 * kTnEpiWarps);
        }
        for (int i = 0; i < 2 * kTnEpiWarps; ++i) mbar_init(s.skip_full(i), 1);
        *s.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();
    if (warp == 1) tmem_alloc_pair(s.tmem_slot, kTmemCols);
    tc_fence_before();
    cluster_sync_all();
    tc_fence_after();
    const uint32_t tmem_base = *s.tmem_slot_ptr;
    grid_dep_wait();   // the set-up above ran beside the end of the kernel before this one
    grid_dep_launch();
    if (kEpi == 1 || kEpi == 3)   // (zero where the last tile reaches past the output's columns)
        for (int i = threadIdx.x; i < p.n_tiles * kCols; i += kTnThreads) s.diag[i] = i < p.ldo ? p.diag[i] : 0.f;
    if (kEpi == 3)   // the epilogue warps' column sums start at zero
        for (int i = threadIdx.x; i < kTnEpiWarps * (kDotMaxN / 2); i += kTnThreads) s.diag[kDotMaxN + i] = 0.f;
    if (kEpi == 1 || kEpi == 3) __syncthreads();

    const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
    const int m_pairs = (p.M + 2 * BM - 1) / (2 * BM);
    const int total = m_pairs * p.n_tiles;
    constexpr int kOutCols = kSplitW ? BN / 2 : kCols;

    if (warp == 0) {
        if (elect_one()) {
            prefetch_tmap(&tmA);
            prefetch_tmap(&tmWh);
        }
        const uint32_t leader_full0 = map_to_cta(s.full(0), 0);   // (the leader's barriers are 8 bytes apart there too)
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        // The 128 rows of A a tile needs are one contiguous range: have L2 fetch the next tile's
        // range in one piece, so that DRAM sees long bursts instead of 128-byte row pieces.
        auto prefetch_a = [&](int tile) {
            if (tile >= total) return;
            const int m0 = (tile / p.n_tiles) * (2 * BM) + (int)rank * BM;
            const int rows = min(BM, p.M - m0);
            if (rows > 0 && elect_one()) l2_prefetch_bulk(p.a_base + (size_t)m0 * p.a_row_bytes, (uint32_t)rows * p.a_row_bytes);
            // (asking L2 for the epilogue's operand rows as well made the bf16-epilogue kernels 15 - 30 % slower)
        };
        prefetch_a(pair);
        for (int tile = pair; tile < total && ok; tile += npairs) {
            const int m0 = (tile / p.n_tiles) * (2 * BM) + (int)rank * BM;
            const int n0 = (tile % p.n_tiles) * kCols + (int)rank * (kCols / 2);
            prefetch_a(tile + npairs);
            for (int kb = 0; kb < p.k_blocks; ++kb) {
                if (!(ok = mbar_wait_warp(s.empty(stage), phase ^ 1u, s.abort_flag))) break;
                if (elect_one()) {
                    if (rank == 0) mbar_expect_tx(s.full(stage), 2 * kStBytes);
                    const uint32_t a_dst = smem_u32(s.tiles + (size_t)stage * kStBytes);
                    tma_load_2d_pair(a_dst, &tmA, leader_full0 + 8u * stage, p.a_col(kb), m0);
                    tma_load_2d_pair(a_dst + kABytes, &tmWh, leader_full0 + 8u * stage, p.w_col(kb), n0);
                }
                if (++stage == kSt) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
        }
    } else if (warp == 1) {
        if (rank == 0) {
            constexpr uint32_t idesc = instr_desc(2 * BM, kCols, 0, 0);
            int stage = 0, acc = 0;
            uint32_t phase = 0, acc_phase = 0;
            bool ok = true;
            for (int tile = pair; tile < total && ok; tile += npairs) {
                if (!(ok = mbar_wait_warp(s.tmem_empty(acc), acc_phase ^ 1u, s.abort_flag))) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + (uint32_t)(acc * BN);
                for (int kb = 0; kb < p.k_blocks; ++kb) {
                    if (!(ok = mbar_wait_warp(s.full(stage), phase, s.abort_flag))) break;
                    tc_fence_after();
                    const uint32_t a_addr = smem_u32(s.tiles + (size_t)stage * kStBytes);
                    const uint64_t adesc = smem_desc_kmajor(a_addr);
                    const uint64_t bdesc = smem_desc_kmajor(a_addr + kABytes);
                    if (elect_one()) {
#pragma unroll
                        for (int k = 0; k < BK / UK; ++k)
                            umma_bf16_pair(d_tmem, adesc + (uint64_t)(2 * k), bdesc + (uint64_t)(2 * k), idesc,
                                           (uint32_t)((kb | k) != 0));
                        umma_commit_pair(s.empty(stage));
                    }
                    if (++stage == kSt) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
                if (!ok) break;
                if (elect_one()) umma_commit_pair(s.tmem_full(acc));
                if ((acc ^= 1) == 0) acc_phase ^= 1u;
            }
        }
    } else {
        const uint32_t leader_empty0 = map_to_cta(s.tmem_empty(0), 0);
        int acc = 0;
        uint32_t acc_phase = 0, skip_phase = 0;
        bool ok = true;
        bool skip_ahead = false;
        for (int tile = pair; tile < total && ok; tile += npairs) {
            const int m0 = (tile / p.n_tiles) * (2 * BM) + (int)rank * BM, n_out0 = (tile % p.n_tiles) * kOutCols;
            const int nxt = tile + npairs;
            const int next_m0 = nxt < total ? (nxt / p.n_tiles) * (2 * BM) + (int)rank * BM : -1;
            if (!(ok = tn_drain_tile<kEpi, kSplitW, kCols>(s, p, &tmOut, &tmSkip, &tmGate, warp, lane, m0, n_out0, acc, acc_phase, tmem_base,
                                                    skip_phase, next_m0, nxt < total ? (nxt % p.n_tiles) * kOutCols : 0, &skip_ahead)))
                break;
            tc_fence_before();
            mbar_arrive_cluster(leader_empty0 + 8u * acc);
            if ((acc ^= 1) == 0) acc_phase ^= 1u;
        }
        if (elect_one()) tma_store_wait_all();
        if (kEpi == 3) {
            // this CTA's column sums: the four warps that drain a column half added in a fixed order, one row
            // of p.dot_part per CTA (the sum over the CTAs follows in another kernel)
            asm volatile("bar.sync 1, %0;" ::"n"(32 * kTnEpiWarps) : "memory");
            const float* sums = s.diag + kDotMaxN;
            for (int n = threadIdx.x - 64; n < p.ldo; n += 32 * kTnEpiWarps) {
                const int half = (n % kCols) / (kCols / 2), idx = (n / kCols) * (kCols / 2) + n % (kCols / 2);
                float t = 0.f;
#pragma unroll
                for (int q = 0; q < 4; ++q) t += sums[(size_t)(4 * half + q) * (kDotMaxN / 2) + idx];
                p.dot_part[(size_t)blockIdx.x * p.ldo + n] = t;
            }
        }
    }
    // nobody leaves (or frees tensor memory) while the other CTA may still signal or compute
    tc_fence_before();
    __syncwarp();
    cluster_sync_all();
    tc_fence_after();
    if (warp == 1) tmem_dealloc_pair(tmem_base, kTmemCols);
    if (threadIdx.x == 0 && *s.abort_flag && p.hdr) p.hdr->status = SSM_ERR_TIMEOUT;
}

// ---------------------------------------------------------------------------------------------
// Input projection and forward scan in one kernel (CTA pairs)
// ---------------------------------------------------------------------------------------------
// x_t = keep_t Abar x_{t-1} + Bbar u_t without Bu ever reaching HBM: the accumulator tile of the
// projection (128 consecutive steps of one sequence x 64 states, weights hi + lo) is scanned by
// the epilogue and leaves as the two bf16 planes of x.  To make that possible a CTA walks the
// tiles of one (sequence, 64 states) chain in time order and keeps the state between tiles; the
// two CTAs of a pair take different sequences (the rows of an MMA need not be neighbours) and the
// same weight tile.  Epilogue per tile, 256 threads: (1) accumulators (hi + lo) into a
// 128 x 128 fp32 tile in shared memory, 128-byte swizzled; the weight rows are packed so that the
// columns of two neighbouring states come out as (re, re, im, im); (2) thread (pair of states,
// eighth of the rows) reads its 16 rows into registers and folds them with packed fp32x2
// multiply-adds - the first group from the carried state, the others from zero - and the groups
// are joined as in the streaming scan kernels; (3) it folds again and writes the hi and lo bf16
// halves of its results into its row group's part of the tile (everybody has read the tile by
// then), which one lane per row group hands to the TMA unit (8-byte global stores from the
// threads themselves measured 5 % slower).
// T = 16, 32 or 64: a tile holds 128 / T whole sequences, a chain is one tile, and every row group that
// begins a sequence starts from that sequence's initial state.
// kTPair (few long sequences): both CTAs of a pair walk ONE sequence, CTA 0 its
// even tiles and CTA 1 its odd ones, which gives twice the chains at the full tile size.  Every row
// group then folds from zero; the last row group joins the groups' results into the tile's own
// contribution, waits for the state that enters the tile (written into this CTA's shared memory by
// the peer, two slots and two barriers in turn), adds Abar^128 times that state unless a flag cuts
// it off, and stores the result into the peer's shared memory: one multiply-add per tile and CTA
// lies between receiving a state and passing it on.
struct FsParams {
    int B, T, P;
    int n_tiles;      // state groups: P / kS
    int k_blocks;     // H / 64
    int tblocks;      // tiles a CTA walks per chain: T / 128 rounded up, or 1; kTPair: T / 256 rounded up
    int unit_rows;    // rows of a chain: T, or 128 when T < 128
    int n_units;      // chains per state group: B, or ceil(B * T / 128)
    int gps;          // row groups per sequence inside a tile: 8, or T / 16
    int nchains;      // n_tiles * ceil(n_units / 2); kTPair: n_tiles * B
    const float2* Abar;
    const float4* Apow;   // [2][P / 2]: Abar^16 and Abar^128 of two neighbouring states (re, re, im, im)
    const uint8_t* done;
    const float2* x0;
    float2* xT;
    uint32_t* x_hi;   // plane of high halves, one 32-bit word (re, im as bf16) per state: [B*T, P]
    size_t plane;     // words from the hi plane to the lo plane
    WsHeader* hdr;
};

// Sizes of the kernels that scan in their epilogue, for chains of kS states (64, or 32 where 64-state
// chains would leave CTA pairs without work): the MMA tile is 256 rows x 4 kS columns (re / im of kS states,
// hi | lo weight halves), a CTA holds 2 kS weight rows, the fp32 tile it scans is 128 rows x 2 kS columns,
// and kS / 2 scanning threads (two states each) share a group of 16 rows.
constexpr int kFsRows = 16;                  // rows per scanning thread; 8 row groups per tile
static_assert(kFsRows == 16 && BM == 128, "the powers of Abar that pack_params_kernel stores");
template <int kS>
struct FsCfg {
    static_assert(kS == 64 || kS == 32, "chains of 64 or 32 states");
    static constexpr int kPairs = kS / 2;              // state pairs of a tile = scanning threads per row group
    static constexpr int kN = 4 * kS;                  // accumulator columns of a tile
    static constexpr int kCols = 2 * kS;               // fp32 columns after hi + lo
    static constexpr int kChunks = kCols / 4;          // 16-byte chunks per row of the fp32 tile
    static constexpr int kWRows = 2 * kS;              // weight rows per CTA
    static constexpr int kEpiWarps = kS / 8;           // 8 (two per TMEM lane quarter; 16 measured slower) or 4
    static constexpr int kEpiThreads = 32 * kEpiWarps;
    static constexpr int kThreads = 64 + kEpiThreads;
    static constexpr int kTileBytes = BM * kCols * 4;
    static constexpr int kStageBytes = kABytes + kWRows * BK * 2;
    static constexpr int kGroupBytes = 2 * kFsRows * kPairs * 8;   // both planes of one row group's results
    static constexpr size_t kSmemBytes = (size_t)kPairStages * kStageBytes + kTileBytes + 1024 + 256;
};

// Two fp32 values in one 64-bit register pair, and the packed multiply-add on them: the scan of
// the epilogue advances two states per instruction.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
struct C2 {
    f32x2 re, im;   // two complex numbers: (re, re), (im, im)
};
// a * x + b for two states at once (nai = -Im a)
__device__ __forceinline__ f32x2 neg2(f32x2 a) { return a ^ 0x8000000080000000ull; }
// 16 bytes from global to shared memory without a register in between; complete after cp_async_wait.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ C2 cstep2(f32x2 ar, f32x2 ai, f32x2 nai, C2 x, C2 b) {
    C2 r;
    r.re = fma2(ar, x.re, fma2(nai, x.im, b.re));
    r.im = fma2(ar, x.im, fma2(ai, x.re, b.im));
    return r;
}

template <int kThreadsN>
__device__ __forceinline__ void epi_sync_n() { asm volatile("bar.sync 1, %0;" ::"n"(kThreadsN) : "memory"); }

template <int kS, bool kTPair, bool kRagged>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(FsCfg<kS>::kThreads, 1)
gemm_scan_fwd_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmWh,
                     const __grid_constant__ CUtensorMap tmX, FsParams p) {
    using Cfg = FsCfg<kS>;
    constexpr int kPairs = Cfg::kPairs, kChunks = Cfg::kChunks, kFsEpiThreads = Cfg::kEpiThreads, kFsEpiWarps = Cfg::kEpiWarps;
    constexpr int kStageB = Cfg::kStageBytes;
    auto epi_sync = [] { epi_sync_n<Cfg::kEpiThreads>(); };
    extern __shared__ uint8_t smem_raw[];
    __shared__ float4 agg_e[kFsEpiThreads], carry_s[kPairs];   // (re, re, im, im) of two neighbouring states
    __shared__ __align__(16) float4 pow_s[2][kTPair ? 2 : 1][kPairs];   // powers of Abar: chains alternate between two slots
    __shared__ uint32_t masks[4];
    __shared__ float4 carry_ring[2][kTPair ? kPairs : 1];   // kTPair: the state handed over by the peer CTA, two slots in turn
    __shared__ __align__(8) uint64_t carry_bar[2];           // kTPair: slot i has arrived (one arrival per sending thread)
    static_assert(!kTPair || kPairs == 32, "the last row group of a tile is one warp");
    const Smem s = carve_smem(smem_raw, kPairStages, Cfg::kTileBytes, 0, kStageB, 0);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    if (threadIdx.x == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(s.full(i), 1);
            mbar_init(s.empty(i), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(s.tmem_full(i), 1);
            mbar_init(s.tmem_empty(i), 2 * kFsEpiThreads);
            mbar_init(smem_u32(&carry_bar[i]), kPairs);
        }
        *s.abort_flag = *s.epi_abort() = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (threadIdx.x < 4) masks[threadIdx.x] = 0u;
    __syncwarp();
    if (warp == 1) tmem_alloc_pair(s.tmem_slot, kTmemCols);
    tc_fence_before();
    cluster_sync_all();
    tc_fence_after();
    const uint32_t tmem_base = *s.tmem_slot_ptr;
    grid_dep_wait();   // the set-up above ran beside the end of the kernel before this one
    grid_dep_launch();

    const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
    const int M = p.B * p.T;
    // chain -> (64 states, this CTA's sequence or, for short sequences, tile of rows); tile tb of a chain -> first row
    // kTPair: both CTAs of the pair walk ONE sequence, tile 2 tb on CTA 0 and tile 2 tb + 1 on CTA 1.
    auto seq_of = [&](int chain) { return kTPair ? chain / p.n_tiles : 2 * (chain / p.n_tiles) + (int)rank; };
    auto row_of = [&](int chain, int tb) {
        const int b = seq_of(chain);
        if (kTPair) return b * p.unit_rows + (2 * tb + (int)rank) * BM;
        return b < p.n_units ? b * p.unit_rows + tb * BM : M;   // nothing left for this CTA: rows past the end read as zero
    };

    if (warp == 0) {
        if (elect_one()) {
            prefetch_tmap(&tmA);
            prefetch_tmap(&tmWh);
        }
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int chain = pair; chain < p.nchains && ok; chain += npairs) {
            const int n0 = (chain % p.n_tiles) * Cfg::kN + (int)rank * Cfg::kWRows;
            for (int tb = 0; tb < p.tblocks && ok; ++tb) {
                const int m0 = row_of(chain, tb);
                // (no L2 prefetch of the next tile's rows here: with it the kernel ran 7 % slower)
                for (int kb = 0; kb < p.k_blocks; ++kb) {
                    if (!(ok = mbar_wait_warp(s.empty(stage), phase ^ 1u, s.abort_flag))) break;
                    const uint32_t leader_full = map_to_cta(s.full(stage), 0);
                    if (elect_one()) {
                        if (rank == 0) mbar_expect_tx(s.full(stage), 2 * kStageB);
                        const uint32_t a_dst = smem_u32(s.tiles + (size_t)stage * kStageB);
                        tma_load_2d_pair(a_dst, &tmA, leader_full, kb * BK, m0);
                        tma_load_2d_pair(a_dst + kABytes, &tmWh, leader_full, kb * BK, n0);
                    }
                    if (++stage == kPairStages) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (rank == 0) {
            constexpr uint32_t idesc = instr_desc(2 * BM, Cfg::kN, 0, 0);
            int stage = 0, acc = 0;
            uint32_t phase = 0, acc_phase = 0;
            bool ok = true;
            for (int chain = pair; chain < p.nchains && ok; chain += npairs) {
                for (int tb = 0; tb < p.tblocks && ok; ++tb) {
                    if (!(ok = mbar_wait_warp(s.tmem_empty(acc), acc_phase ^ 1u, s.abort_flag))) break;
                    tc_fence_after();
                    const uint32_t d_tmem = tmem_base + (uint32_t)(acc * Cfg::kN);
                    for (int kb = 0; kb < p.k_blocks; ++kb) {
                        if (!(ok = mbar_wait_warp(s.full(stage), phase, s.abort_flag))) break;
                        tc_fence_after();
                        const uint32_t a_addr = smem_u32(s.tiles + (size_t)stage * kStageB);
                        const uint64_t adesc = smem_desc_kmajor(a_addr);
                        const uint64_t bdesc = smem_desc_kmajor(a_addr + kABytes);
                        if (elect_one()) {
#pragma unroll
                            for (int k = 0; k < BK / UK; ++k)
                                umma_bf16_pair(d_tmem, adesc + (uint64_t)(2 * k), bdesc + (uint64_t)(2 * k), idesc,
                                               (uint32_t)((kb | k) != 0));
                            umma_commit_pair(s.empty(stage));
                        }
                        if (++stage == kPairStages) {
                            stage = 0;
                            phase ^= 1u;
                        }
                    }
                    if (!ok) break;
                    if (elect_one()) umma_commit_pair(s.tmem_full(acc));
                    if ((acc ^= 1) == 0) acc_phase ^= 1u;
                }
            }
        }
    } else {
        volatile int* epi_flag = s.epi_abort();
        const uint32_t leader_empty0 = map_to_cta(s.tmem_empty(0), 0);
        constexpr int R = kFsRows, nsl = BM / kFsRows;   // rows per thread; groups of rows
        const int te = threadIdx.x - 64;            // 0 .. kFsEpiThreads - 1
        const int q = warp & 3, grp = (warp - 2) >> 2;   // drain role: TMEM lane quarter, 32-column group
        const int sp = te % kPairs, sl = te / kPairs;   // scan role: pair of states of the tile, group of its rows
        // the lane that talks to the TMA unit for its row group (always the same one)
        auto group_leader = [&] { return kPairs == 32 ? elect_one() : lane % kPairs == 0; };
        const int prow = q * 32 + lane;             // drain role: row of the tile
        float4* T4 = reinterpret_cast<float4*>(s.staging);
        const C2 zero = {0ull, 0ull};
        int acc = 0;
        uint32_t acc_phase = 0;
        uint32_t n_recv = 0, n_send = 0;            // kTPair: states received from / handed to the peer so far
        const uint32_t peer_ring = map_to_cta(smem_u32(&carry_ring[0][0]), rank ^ 1u);
        const uint32_t peer_bar = map_to_cta(smem_u32(&carry_bar[0]), rank ^ 1u);
        bool ok = true;
        // The flag of this thread's row, loaded one tile ahead (the load's latency would otherwise stand at the
        // head of every tile).
        auto flag_of = [&](int chain, int tb) {
            if (!p.done || te >= BM || chain >= p.nchains) return false;
            const int m = row_of(chain, tb) + te;
            return seq_of(chain) < p.n_units && m < M && p.done[(size_t)m] != 0;
        };
        bool flag_next = flag_of(pair, 0);
        // The chain's multipliers are loaded one chain ahead as well (a chain is a single tile when the sequences are short).
        auto abar_of = [&](int chain, int k) {
            return chain < p.nchains ? p.Abar[(chain % p.n_tiles) * kS + 2 * sp + k] : make_float2(0.f, 0.f);
        };
        float2 a0_next = abar_of(pair, 0), a1_next = abar_of(pair, 1);
        int chain_par = 0;
        for (int chain = pair; chain < p.nchains && ok; chain += npairs) {
            const int n_tile = chain % p.n_tiles, b = seq_of(chain);
            const bool has_seq = b < p.n_units;
            const bool short_seq = !kTPair && !kRagged && p.T < BM;        // then b counts tiles of rows, not sequences
            const int g0 = sl - sl % p.gps;         // the first row group of this group's sequence in the tile
            const bool from_carry = !kTPair && sl == g0;   // (kTPair: the carried state arrives late; every group joins)
            const int pg = n_tile * kS + 2 * sp;    // the first of this thread's two states
            const float2 a0 = a0_next, a1 = a1_next;
            a0_next = abar_of(chain + npairs, 0);
            a1_next = abar_of(chain + npairs, 1);
            const f32x2 ar = pack2(a0.x, a1.x), ai = pack2(a0.y, a1.y), nai = pack2(-a0.y, -a1.y);
            // Abar^R, what a row group does to the state that enters it, and for kTPair Abar^128, what a tile does: on their way
            // while the first tile's MMAs run.  (Squared up from the rounded Abar in fp32, every step of a long sequence
            // carried that rounding: xT of 60 x 3000 steps 4.1e-5 off, with these 9.0e-6.)
            chain_par ^= 1;
            if (te < kPairs) {
                const float4* src = p.Apow + (n_tile * kS) / 2 + te;
                cp_async16(smem_u32(&pow_s[chain_par][0][te]), src);
                if (kTPair) cp_async16(smem_u32(&pow_s[chain_par][kTPair ? 1 : 0][te]), src + p.P / 2);
            }
            C2 cin = zero;      // kTPair: the state that enters this CTA's tile
            if (kTPair && rank == 0 && p.x0) {
                const float2 c0 = p.x0[(size_t)b * p.P + pg], c1 = p.x0[(size_t)b * p.P + pg + 1];
                cin.re = pack2(c0.x, c1.x);
                cin.im = pack2(c0.y, c1.y);
            }
            if (sl == 0 && !short_seq && !kTPair) {   // the carried state, as (re, re, im, im) of the two states
                float2 c0 = make_float2(0.f, 0.f), c1 = c0;
                if (p.x0 && has_seq) {
                    c0 = p.x0[(size_t)b * p.P + pg];
                    c1 = p.x0[(size_t)b * p.P + pg + 1];
                }
                carry_s[sp] = make_float4(c0.x, c1.x, c0.y, c1.y);
            }
            for (int tb = 0; tb < p.tblocks; ++tb) {
                const int m0 = row_of(chain, tb);
                if (p.done && te < BM) {
                    const uint32_t mk = __ballot_sync(0xffffffffu, flag_next);
                    if (lane == 0) masks[te >> 5] = mk;
                }
                flag_next = tb + 1 < p.tblocks ? flag_of(chain, tb + 1) : flag_of(chain + npairs, 0);
                (void)mbar_wait(s.tmem_full(acc), acc_phase, epi_flag);
                cp_async_wait();
                if (group_leader()) tma_store_wait_read();   // this row group's results of the previous tile have left shared memory
                epi_sync();   // flags visible, tile free (nobody reads the previous one any more); also:
                              // the 256 threads leave together or not at all
                if (*epi_flag) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                // (1) accumulators -> shared-memory tile: 16-byte chunk j of a 128-byte group sits at j ^ (row & 7)
                const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * Cfg::kN);
#pragma unroll
                for (int g = grp; g < Cfg::kCols / 32; g += kFsEpiWarps / 4) {   // 32 columns = one 128-byte group of the row
                    uint32_t r[32], r2[32];
                    tmem_ld32(t_row + (uint32_t)(g * 32), r);
                    tmem_ld32(t_row + (uint32_t)(Cfg::kCols + g * 32), r2);
                    tmem_ld_wait();
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        T4[prow * kChunks + g * 8 + (j ^ (prow & 7))] =
                            make_float4(__uint_as_float(r[4 * j]) + __uint_as_float(r2[4 * j]),
                                        __uint_as_float(r[4 * j + 1]) + __uint_as_float(r2[4 * j + 1]),
                                        __uint_as_float(r[4 * j + 2]) + __uint_as_float(r2[4 * j + 2]),
                                        __uint_as_float(r[4 * j + 3]) + __uint_as_float(r2[4 * j + 3]));
                }
                tc_fence_before();
                mbar_arrive_cluster(leader_empty0 + 8u * acc);
                if ((acc ^= 1) == 0) acc_phase ^= 1u;
                epi_sync();
                // (2) scan: this thread's two states over its R rows.  The flags of a row group are the
                // same for the whole warp: a group without flags takes loops without the tests.
                const int r0 = sl * R;
                // kRagged: rows of the tile that lie inside the sequence (the others hold rows of the next one: nothing that
                // is kept depends on them); else the last tile of short sequences may be ragged
                const int left = p.T - (kTPair ? 2 * tb + (int)rank : tb) * BM;
                const bool grp_valid = has_seq && (kRagged ? r0 < left : m0 + r0 < M);
                const int b_grp = short_seq ? (m0 + r0) / p.T : b;      // this group's sequence
                uint32_t gflags = 0;   // bit g: row group g has a flag
                if (p.done) {
#pragma unroll
                    for (int w = 0; w < 4; ++w) {
                        const uint32_t mk = masks[w];
#pragma unroll
                        for (int h = 0; h < 32 / R; ++h)
                            if ((mk >> (h * R)) & ((1u << R) - 1u)) gflags |= 1u << (w * (32 / R) + h);
                    }
                }
                const uint32_t mask = p.done ? (masks[r0 >> 5] >> (r0 & 31)) & ((1u << R) - 1u) : 0u;
                C2 v[R];
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    const int row = r0 + i;
                    const float4 t = T4[row * kChunks + ((sp & ~7) | ((sp & 7) ^ (row & 7)))];   // (re, re, im, im)
                    v[i].re = pack2(t.x, t.y);
                    v[i].im = pack2(t.z, t.w);
                }
                C2 e = zero;
                if (from_carry) {   // from the carried or the initial state: these results are final
                    float4 c;
                    if (!short_seq) {
                        c = carry_s[sp];
                    } else if (p.x0 && grp_valid) {
                        const float2 c0 = p.x0[(size_t)b_grp * p.P + pg], c1 = p.x0[(size_t)b_grp * p.P + pg + 1];
                        c = make_float4(c0.x, c1.x, c0.y, c1.y);
                    } else {
                        c = make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                    C2 x = {pack2(c.x, c.y), pack2(c.z, c.w)};
                    if (mask == 0u) {
#pragma unroll
                        for (int i = 0; i < R; ++i) v[i] = x = cstep2(ar, ai, nai, x, v[i]);
                    } else {
#pragma unroll
                        for (int i = 0; i < R; ++i) {
                            if ((mask >> i) & 1u) x = zero;
                            v[i] = x = cstep2(ar, ai, nai, x, v[i]);
                        }
                    }
                    e = x;
                } else if (mask == 0u) {
#pragma unroll
                    for (int i = 0; i < R; ++i) e = cstep2(ar, ai, nai, e, v[i]);
                } else {
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        if ((mask >> i) & 1u) e = zero;
                        e = cstep2(ar, ai, nai, e, v[i]);
                    }
                }
                {
                    float e0, e1, e2, e3;
                    unpack2(e.re, e0, e1);
                    unpack2(e.im, e2, e3);
                    agg_e[te] = make_float4(e0, e1, e2, e3);
                }
                epi_sync();   // group results visible; every thread has its rows in registers
                const float4 pw = pow_s[chain_par][0][sp];
                const f32x2 pr = pack2(pw.x, pw.y), pi = pack2(pw.z, pw.w), npi = neg2(pi);
                C2 x = e;
                if (kTPair) {
                    // The state that enters the tile comes from the peer CTA (the tile before this one), except for
                    // the sequence's first tile.  The last row group passes the tile's end state on as soon as it
                    // can: the tile's own contribution (the groups' results joined from zero) is ready before the
                    // peer's state arrives, so the hand-over costs one multiply-add per tile and CTA.
                    const bool first = rank == 0 && tb == 0, last = rank == 1 && tb == p.tblocks - 1;
                    C2 tile = zero;
                    const float4 tw = pow_s[chain_par][kTPair ? 1 : 0][sp];
                    if (sl == nsl - 1 && !last) {
#pragma unroll
                        for (int g = 0; g < nsl - 1; ++g) {
                            const float4 c = agg_e[g * kPairs + sp];
                            const C2 eg = {pack2(c.x, c.y), pack2(c.z, c.w)};
                            tile = (g == 0 || ((gflags >> g) & 1u)) ? eg : cstep2(pr, pi, npi, tile, eg);
                        }
                        tile = ((gflags >> (nsl - 1)) & 1u) ? e : cstep2(pr, pi, npi, tile, e);
                    }
                    if (!first) {
                        (void)mbar_wait_acquire_cluster(smem_u32(&carry_bar[n_recv & 1u]), (n_recv >> 1) & 1u, epi_flag);
                        const float4 c = carry_ring[n_recv & 1u][sp];
                        cin.re = pack2(c.x, c.y);
                        cin.im = pack2(c.z, c.w);
                        ++n_recv;
                    }
                    if (sl == nsl - 1 && !last) {
                        const f32x2 tr = pack2(tw.x, tw.y), ti = pack2(tw.z, tw.w);
                        const C2 out = gflags == 0u ? cstep2(tr, ti, neg2(ti), cin, tile) : tile;
                        float o0, o1, o2, o3;
                        unpack2(out.re, o0, o1);
                        unpack2(out.im, o2, o3);
                        st_cluster_f4(peer_ring + (uint32_t)(((n_send & 1u) * kPairs + sp) * sizeof(float4)), make_float4(o0, o1, o2, o3));
                        mbar_arrive_release_cluster(peer_bar + 8u * (n_send & 1u));
                        ++n_send;
                    }
                    x = cin;
#pragma unroll
                    for (int g = 0; g < nsl - 1; ++g) {
                        if (g < sl) {
                            const float4 c = agg_e[g * kPairs + sp];
                            const C2 eg = {pack2(c.x, c.y), pack2(c.z, c.w)};
                            x = ((gflags >> g) & 1u) ? eg : cstep2(pr, pi, npi, x, eg);
                        }
                    }
                } else if (!from_carry) {   // state before this group's first row
                    {
                        const float4 c = agg_e[g0 * kPairs + sp];
                        x.re = pack2(c.x, c.y);
                        x.im = pack2(c.z, c.w);
                    }
#pragma unroll
                    for (int g = 1; g < nsl - 1; ++g) {
                        if (g > g0 && g < sl) {
                            const float4 c = agg_e[g * kPairs + sp];
                            const C2 eg = {pack2(c.x, c.y), pack2(c.z, c.w)};
                            x = ((gflags >> g) & 1u) ? eg : cstep2(pr, pi, npi, x, eg);
                        }
                    }
                }
                // (3) fold again; results as hi / lo bf16 halves into this warp's part of the tile (everybody
                // has its rows in registers by now): [plane][row][64 states], which the warp hands to the TMA unit
                uint8_t* warp_out = s.staging + sl * Cfg::kGroupBytes;
                uint2* out = reinterpret_cast<uint2*>(warp_out) + sp;
                auto emit = [&](int i, C2 xv) {
                    float re0, re1, im0, im1;
                    unpack2(xv.re, re0, re1);
                    unpack2(xv.im, im0, im1);
                    const __nv_bfloat162 h0 = __floats2bfloat162_rn(re0, im0), h1 = __floats2bfloat162_rn(re1, im1);
                    const float2 f0 = __bfloat1622float2(h0), f1 = __bfloat1622float2(h1);
                    const __nv_bfloat162 l0 = __floats2bfloat162_rn(re0 - f0.x, im0 - f0.y);
                    const __nv_bfloat162 l1 = __floats2bfloat162_rn(re1 - f1.x, im1 - f1.y);
                    out[i * kPairs] = make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1));
                    out[(R + i) * kPairs] = make_uint2(*reinterpret_cast<const uint32_t*>(&l0), *reinterpret_cast<const uint32_t*>(&l1));
                };
                C2 xend = zero;   // kRagged: the state after the sequence's last row, in the group that holds it
                const int iend = left - 1 - r0;
                if (from_carry) {
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        emit(i, v[i]);
                        if (kRagged && i == iend) xend = v[i];
                    }
                } else if (mask == 0u) {
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        emit(i, x = cstep2(ar, ai, nai, x, v[i]));
                        if (kRagged && i == iend) xend = x;
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        if ((mask >> i) & 1u) x = zero;
                        emit(i, x = cstep2(ar, ai, nai, x, v[i]));
                        if (kRagged && i == iend) xend = x;
                    }
                }
                fence_async_smem();
                __syncwarp();
                if (grp_valid && group_leader()) {
                    if (kRagged) tma_store_4d_nocommit(&tmX, smem_u32(warp_out), n_tile * kS, p.T - left + r0, b, 0);   // clipped at T
                    else tma_store_3d_nocommit(&tmX, smem_u32(warp_out), n_tile * kS, m0 + r0, 0);
                    tma_commit_group();
                }
                if (kRagged && p.xT && has_seq && iend >= 0 && iend < R) {
                    float x0r, x1r, x0i, x1i;
                    unpack2(xend.re, x0r, x1r);
                    unpack2(xend.im, x0i, x1i);
                    p.xT[(size_t)b * p.P + pg] = make_float2(x0r, x0i);
                    p.xT[(size_t)b * p.P + pg + 1] = make_float2(x1r, x1i);
                }
                if (short_seq ? (sl - g0 == p.gps - 1) : (sl == nsl - 1)) {   // the group that ends a sequence or the tile
                    float x0r, x1r, x0i, x1i;
                    unpack2(x.re, x0r, x1r);
                    unpack2(x.im, x0i, x1i);
                    // (not after the chain's last tile: by then the first group may already have set up the next chain)
                    if (kTPair) {
                        if (!kRagged && rank == 1 && tb == p.tblocks - 1 && p.xT) {
                            p.xT[(size_t)b * p.P + pg] = make_float2(x0r, x0i);
                            p.xT[(size_t)b * p.P + pg + 1] = make_float2(x1r, x1i);
                        }
                    } else if (!short_seq && tb < p.tblocks - 1) {
                        carry_s[sp] = make_float4(x0r, x1r, x0i, x1i);
                    } else if (!kRagged && p.xT && grp_valid) {
                        p.xT[(size_t)b_grp * p.P + pg] = make_float2(x0r, x0i);
                        p.xT[(size_t)b_grp * p.P + pg + 1] = make_float2(x1r, x1i);
                    }
                }
            }
        }
        if (group_leader()) tma_store_wait_all();
    }
    tc_fence_before();
    __syncwarp();
    cluster_sync_all();
    tc_fence_after();
    if (warp == 1) tmem_dealloc_pair(tmem_base, kTmemCols);
    if (threadIdx.x == 0 && (*s.abort_flag || *s.epi_abort()) && p.hdr) p.hdr->status = SSM_ERR_TIMEOUT;
}

// ---------------------------------------------------------------------------------------------
// g_x projection and reverse scan in one kernel (CTA pairs)
// ---------------------------------------------------------------------------------------------
// s_t = g_x,t + keep_{t+1} conj(Abar) s_{t+1} without g_x ever reaching HBM, and the sums
// gAbar = sum_t keep_t s_t conj(x_{t-1}).  The kernel is gemm_scan_fwd_kernel run backwards: a CTA
// walks the tiles of a chain from the last to the first, the last row group starts from the carried
// value, rows are folded from the last to the first, and the reset that acts between rows i and
// i + 1 is the flag of row i + 1.  What is new is x_{t-1}: once a warp has its 16 rows of g_x in
// registers, its part of the shared-memory tile is free, and one lane has the TMA unit copy the
// rows m - 1 ... m + 14 of both planes of x there (one row early; the row before a sequence's first
// is replaced by x0).  In the second pass a thread reads its two states' x_{t-1}, adds
// s_t conj(x_{t-1}) to its sums and writes the hi / lo halves of s_t to the same place, which
// then leaves through the TMA unit as in the forward kernel.  The sums stay in registers for the
// whole chain and are added over the row groups at its end: one entry of gA_part per (sequence,
// state), each written once.  T as for the forward kernel.  kTPair as there, run backwards: CTA 1
// holds the later tile of a pair of tiles, the first row group passes s of the tile's first row
// on, and each CTA writes its own row of gA_part (two per sequence).
struct FbParams {
    int B, T, P;
    int n_tiles;      // state groups: P / kS
    int k_blocks;     // H / 64
    int tblocks;      // tiles a CTA walks per chain: T / 128 rounded up, or 1; kTPair: T / 256 rounded up
    int unit_rows;    // rows of a chain: T, or 128 when T < 128 (a tile then holds 128 / T whole sequences)
    int n_units;      // chains per state group: B, or ceil(B * T / 128)
    int gps;          // row groups per sequence inside a tile: 8, or T / 16
    int nchains;      // n_tiles * ceil(n_units / 2); kTPair: n_tiles * B
    const float2* Abar;
    const float4* Apow;   // [2][P / 2]: Abar^16 and Abar^128 of two neighbouring states (re, re, im, im)
    const uint8_t* done;
    const float2* x0;     // [B, P] or NULL
    const float2* gxT;    // [B, P] or NULL
    float2* gA_part;      // [n_units, P]: one row of sums per chain; kTPair: [2 B, P], row 2 b + CTA rank
    float2* gx0;          // [B, P] or NULL
    WsHeader* hdr;
};

template <int kS, bool kTPair, bool kRagged>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(FsCfg<kS>::kThreads, 1)
gemm_scan_bwd_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmWh,
                     const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmS, FbParams p) {
    using Cfg = FsCfg<kS>;
    constexpr int kPairs = Cfg::kPairs, kChunks = Cfg::kChunks, kFsEpiThreads = Cfg::kEpiThreads, kFsEpiWarps = Cfg::kEpiWarps;
    constexpr int kStageB = Cfg::kStageBytes;
    auto epi_sync = [] { epi_sync_n<Cfg::kEpiThreads>(); };
    extern __shared__ uint8_t smem_raw[];
    __shared__ float4 agg_e[kFsEpiThreads], carry_s[kPairs];   // (re, re, im, im) of two neighbouring states
    __shared__ __align__(16) float4 pow_s[2][kTPair ? 2 : 1][kPairs];   // powers of Abar: chains alternate between two slots
    __shared__ uint32_t masks[8];   // [0, 4): flags of the rows one later (the resets of the reverse scan); [4, 8): of the rows
    __shared__ __align__(8) uint64_t xbar[BM / kFsRows];   // one per row group: its rows of x have arrived
    __shared__ float4 carry_ring[2][kTPair ? kPairs : 1];   // kTPair: the value handed over by the peer CTA, two slots in turn
    __shared__ __align__(8) uint64_t carry_bar[2];           // kTPair: slot i has arrived (one arrival per sending thread)
    static_assert(!kTPair || kPairs == 32, "the first row group of a tile is one warp");
    const Smem s = carve_smem(smem_raw, kPairStages, Cfg::kTileBytes, 0, kStageB, 0);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    if (threadIdx.x == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(s.full(i), 1);
            mbar_init(s.empty(i), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(s.tmem_full(i), 1);
            mbar_init(s.tmem_empty(i), 2 * kFsEpiThreads);
            mbar_init(smem_u32(&carry_bar[i]), kPairs);
        }
        for (int i = 0; i < BM / kFsRows; ++i) mbar_init(smem_u32(&xbar[i]), 1);
        *s.abort_flag = *s.epi_abort() = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (threadIdx.x < 8) masks[threadIdx.x] = 0u;
    __syncwarp();
    if (warp == 1) tmem_alloc_pair(s.tmem_slot, kTmemCols);
    tc_fence_before();
    cluster_sync_all();
    tc_fence_after();
    const uint32_t tmem_base = *s.tmem_slot_ptr;
    grid_dep_wait();   // the set-up above ran beside the end of the kernel before this one
    grid_dep_launch();

    const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
    const int M = p.B * p.T;
    // kTPair: both CTAs of the pair walk ONE sequence, tile 2 tb on CTA 0 and tile 2 tb + 1 on CTA 1.
    auto seq_of = [&](int chain) { return kTPair ? chain / p.n_tiles : 2 * (chain / p.n_tiles) + (int)rank; };
    auto row_of = [&](int chain, int tb) {
        const int b = seq_of(chain);
        if (kTPair) return b * p.unit_rows + (2 * tb + (int)rank) * BM;
        return b < p.n_units ? b * p.unit_rows + tb * BM : M;   // nothing for this CTA: rows past the end read as zero
    };

    if (warp == 0) {
        if (elect_one()) {
            prefetch_tmap(&tmA);
            prefetch_tmap(&tmWh);
        }
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int chain = pair; chain < p.nchains && ok; chain += npairs) {
            const int n0 = (chain % p.n_tiles) * Cfg::kN + (int)rank * Cfg::kWRows;
            for (int tb = p.tblocks - 1; tb >= 0 && ok; --tb) {
                const int m0 = row_of(chain, tb);
                for (int kb = 0; kb < p.k_blocks; ++kb) {
                    if (!(ok = mbar_wait_warp(s.empty(stage), phase ^ 1u, s.abort_flag))) break;
                    const uint32_t leader_full = map_to_cta(s.full(stage), 0);
                    if (elect_one()) {
                        if (rank == 0) mbar_expect_tx(s.full(stage), 2 * kStageB);
                        const uint32_t a_dst = smem_u32(s.tiles + (size_t)stage * kStageB);
                        tma_load_2d_pair(a_dst, &tmA, leader_full, kb * BK, m0);
                        tma_load_2d_pair(a_dst + kABytes, &tmWh, leader_full, kb * BK, n0);
                    }
                    if (++stage == kPairStages) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
            }
        }
    } else if (warp == 1) {
        if (rank == 0) {
            constexpr uint32_t idesc = instr_desc(2 * BM, Cfg::kN, 0, 0);
            int stage = 0, acc = 0;
            uint32_t phase = 0, acc_phase = 0;
            bool ok = true;
            for (int chain = pair; chain < p.nchains && ok; chain += npairs) {
                for (int tb = 0; tb < p.tblocks && ok; ++tb) {
                    if (!(ok = mbar_wait_warp(s.tmem_empty(acc), acc_phase ^ 1u, s.abort_flag))) break;
                    tc_fence_after();
                    const uint32_t d_tmem = tmem_base + (uint32_t)(acc * Cfg::kN);
                    for (int kb = 0; kb < p.k_blocks; ++kb) {
                        if (!(ok = mbar_wait_warp(s.full(stage), phase, s.abort_flag))) break;
                        tc_fence_after();
                        const uint32_t a_addr = smem_u32(s.tiles + (size_t)stage * kStageB);
                        const uint64_t adesc = smem_desc_kmajor(a_addr);
                        const uint64_t bdesc = smem_desc_kmajor(a_addr + kABytes);
                        if (elect_one()) {
#pragma unroll
                            for (int k = 0; k < BK / UK; ++k)
                                umma_bf16_pair(d_tmem, adesc + (uint64_t)(2 * k), bdesc + (uint64_t)(2 * k), idesc,
                                               (uint32_t)((kb | k) != 0));
                            umma_commit_pair(s.empty(stage));
                        }
                        if (++stage == kPairStages) {
                            stage = 0;
                            phase ^= 1u;
                        }
                    }
                    if (!ok) break;
                    if (elect_one()) umma_commit_pair(s.tmem_full(acc));
                    if ((acc ^= 1) == 0) acc_phase ^= 1u;
                }
            }
        }
    } else {
        volatile int* epi_flag = s.epi_abort();
        const uint32_t leader_empty0 = map_to_cta(s.tmem_empty(0), 0);
        constexpr int R = kFsRows, nsl = BM / kFsRows;   // rows per thread; groups of rows
        const int te = threadIdx.x - 64;            // 0 .. kFsEpiThreads - 1
        const int q = warp & 3, grp = (warp - 2) >> 2;   // drain role: TMEM lane quarter, 32-column group
        const int sp = te % kPairs, sl = te / kPairs;   // scan role: pair of states of the tile, group of its rows
        // the lane that talks to the TMA unit for its row group (always the same one)
        auto group_leader = [&] { return kPairs == 32 ? elect_one() : lane % kPairs == 0; };
        const int prow = q * 32 + lane;             // drain role: row of the tile
        const bool short_seq = !kTPair && !kRagged && p.T < BM;            // then a chain is one tile of 128 / T whole sequences
        const int g0 = sl - sl % p.gps;             // first and last row group of this group's sequence in the tile
        const int gl = g0 + p.gps - 1;
        const bool from_carry = !kTPair && sl == gl;           // the last rows come first (kTPair: the carried value arrives late; every group joins)
        uint32_t n_recv = 0, n_send = 0;            // kTPair: values received from / handed to the peer so far
        const uint32_t peer_ring = map_to_cta(smem_u32(&carry_ring[0][0]), rank ^ 1u);
        const uint32_t peer_bar = map_to_cta(smem_u32(&carry_bar[0]), rank ^ 1u);
        float4* T4 = reinterpret_cast<float4*>(s.staging);
        uint8_t* warp_buf = s.staging + sl * Cfg::kGroupBytes;   // this row group's rows of the tile; later x_{t-1}, then s
        uint2* xs = reinterpret_cast<uint2*>(warp_buf) + sp;
        const uint32_t xb = smem_u32(&xbar[sl]);
        uint32_t xphase = 0;
        const C2 zero = {0ull, 0ull};
        int acc = 0;
        uint32_t acc_phase = 0;
        bool ok = true;
        // The flags of this thread's row of a tile, loaded one tile ahead: bit 0 a row's own flag, bit 1 the flag of the row
        // after it if that row belongs to the same sequence.
        auto flags_of = [&](int chain, int tb) -> uint32_t {
            if (!p.done || te >= BM || chain >= p.nchains || seq_of(chain) >= p.n_units) return 0u;
            const int m = row_of(chain, tb) + te, tix = kTPair ? 2 * tb + (int)rank : tb;   // tix: the tile's place in its sequence
            const bool next_in_seq = short_seq ? ((te + 1) % p.T != 0 && m + 1 < M) : (tix * BM + te + 1 < p.T);
            return (m < M && p.done[(size_t)m] != 0 ? 1u : 0u) | (next_in_seq && p.done[(size_t)m + 1] != 0 ? 2u : 0u);
        };
        uint32_t flags_next = flags_of(pair, p.tblocks - 1);
        // The chain's multipliers are loaded one chain ahead (a chain is a single tile when the sequences are short).
        auto abar_of = [&](int chain, int k) {
            return chain < p.nchains ? p.Abar[(chain % p.n_tiles) * kS + 2 * sp + k] : make_float2(0.f, 0.f);
        };
        float2 a0_next = abar_of(pair, 0), a1_next = abar_of(pair, 1);
        int chain_par = 0;
        for (int chain = pair; chain < p.nchains && ok; chain += npairs) {
            const int n_tile = chain % p.n_tiles, b = seq_of(chain);
            const bool has_seq = b < p.n_units;
            const int pg = n_tile * kS + 2 * sp;    // the first of this thread's two states
            const float2 a0 = cconj(a0_next), a1 = cconj(a1_next);
            a0_next = abar_of(chain + npairs, 0);
            a1_next = abar_of(chain + npairs, 1);
            const f32x2 ar = pack2(a0.x, a1.x), ai = pack2(a0.y, a1.y), nai = pack2(-a0.y, -a1.y);
            chain_par ^= 1;   // Abar^R and, for kTPair, Abar^128: as in the forward kernel
            if (te < kPairs) {
                const float4* src = p.Apow + (n_tile * kS) / 2 + te;
                cp_async16(smem_u32(&pow_s[chain_par][0][te]), src);
                if (kTPair) cp_async16(smem_u32(&pow_s[chain_par][kTPair ? 1 : 0][te]), src + p.P / 2);
            }
            C2 cin = zero;      // kTPair: s of the row after this CTA's tile (nothing after the sequence's last row)
            C2 g = zero;        // this thread's part of the chain's sums s_t conj(x_{t-1})
            f32x2 gim_neg = 0ull;   // the part of Im g that enters with a minus sign, summed apart
            C2 xinit = zero;    // x0: what stands before the sequence's first row
            if (!short_seq && sl == 0 && p.x0 && has_seq && (!kTPair || rank == 0)) {
                const float2 c0 = p.x0[(size_t)b * p.P + pg], c1 = p.x0[(size_t)b * p.P + pg + 1];
                xinit.re = pack2(c0.x, c1.x);
                xinit.im = pack2(c0.y, c1.y);
            }
            if (from_carry) carry_s[sp] = make_float4(0.f, 0.f, 0.f, 0.f);   // nothing follows the last row
            for (int tb = p.tblocks - 1; tb >= 0; --tb) {
                const int m0 = row_of(chain, tb);
                if (p.done && te < BM) {
                    const uint32_t mk0 = __ballot_sync(0xffffffffu, flags_next & 1u), mk1 = __ballot_sync(0xffffffffu, flags_next & 2u);
                    if (lane == 0) {
                        masks[te >> 5] = mk1;
                        masks[4 + (te >> 5)] = mk0;
                    }
                }
                flags_next = tb > 0 ? flags_of(chain, tb - 1) : flags_of(chain + npairs, p.tblocks - 1);
                (void)mbar_wait(s.tmem_full(acc), acc_phase, epi_flag);
                tc_fence_after();
                // (1) accumulators -> shared-memory tile: 16-byte chunk j of a 128-byte group sits at j ^ (row & 7).
                // A warp drains two groups of 32 columns (hi + lo halves each): the first group's loads are in
                // flight while it waits for the tile to be free, the second group's while it stores the first.
                constexpr int kGrpStep = kFsEpiWarps / 4;   // a warp drains the 32-column groups grp and grp + kGrpStep
                static_assert(Cfg::kCols / 32 == 2 * kGrpStep, "two 32-column groups per warp");
                const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * Cfg::kN);
                uint32_t ra[32], ra2[32], rb[32], rb2[32];
                tmem_ld32(t_row + (uint32_t)(grp * 32), ra);
                tmem_ld32(t_row + (uint32_t)(Cfg::kCols + grp * 32), ra2);
                cp_async_wait();
                if (group_leader()) tma_store_wait_read();   // this row group's results of the previous tile have left shared memory
                epi_sync();   // flags visible, tile free (nobody reads the previous one any more); also:
                              // the 256 threads leave together or not at all
                tmem_ld_wait();
                if (*epi_flag) {
                    ok = false;
                    break;
                }
                tmem_ld32(t_row + (uint32_t)((grp + kGrpStep) * 32), rb);
                tmem_ld32(t_row + (uint32_t)(Cfg::kCols + (grp + kGrpStep) * 32), rb2);
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    T4[prow * kChunks + grp * 8 + (j ^ (prow & 7))] =
                        make_float4(__uint_as_float(ra[4 * j]) + __uint_as_float(ra2[4 * j]),
                                    __uint_as_float(ra[4 * j + 1]) + __uint_as_float(ra2[4 * j + 1]),
                                    __uint_as_float(ra[4 * j + 2]) + __uint_as_float(ra2[4 * j + 2]),
                                    __uint_as_float(ra[4 * j + 3]) + __uint_as_float(ra2[4 * j + 3]));
                tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    T4[prow * kChunks + (grp + kGrpStep) * 8 + (j ^ (prow & 7))] =
                        make_float4(__uint_as_float(rb[4 * j]) + __uint_as_float(rb2[4 * j]),
                                    __uint_as_float(rb[4 * j + 1]) + __uint_as_float(rb2[4 * j + 1]),
                                    __uint_as_float(rb[4 * j + 2]) + __uint_as_float(rb2[4 * j + 2]),
                                    __uint_as_float(rb[4 * j + 3]) + __uint_as_float(rb2[4 * j + 3]));
                tc_fence_before();
                mbar_arrive_cluster(leader_empty0 + 8u * acc);
                if ((acc ^= 1) == 0) acc_phase ^= 1u;
                epi_sync();
                // (2) this thread's two states over its R rows, last row first
                const int r0 = sl * R;
                const int left = p.T - (kTPair ? 2 * tb + (int)rank : tb) * BM;   // kRagged: rows of the tile inside the sequence
                const bool grp_valid = has_seq && (kRagged ? r0 < left : m0 + r0 < M);   // (short sequences: the last tile may be ragged)
                const int b_grp = short_seq ? (m0 + r0) / p.T : b;      // this group's sequence
                uint32_t gflags = 0;   // bit g: a reset acts inside or right after row group g
                uint32_t mask = 0u, mask0 = 0u;
                if (p.done) {
#pragma unroll
                    for (int w = 0; w < 4; ++w) {
                        const uint32_t mk = masks[w];
#pragma unroll
                        for (int h = 0; h < 32 / R; ++h)
                            if ((mk >> (h * R)) & ((1u << R) - 1u)) gflags |= 1u << (w * (32 / R) + h);
                    }
                    mask = (masks[r0 >> 5] >> (r0 & 31)) & ((1u << R) - 1u);
                    mask0 = (masks[4 + (r0 >> 5)] >> (r0 & 31)) & ((1u << R) - 1u);
                }
                C2 v[R];
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    const int row = r0 + i;
                    const float4 t = T4[row * kChunks + ((sp & ~7) | ((sp & 7) ^ (row & 7)))];   // (re, re, im, im)
                    v[i].re = pack2(t.x, t.y);
                    v[i].im = pack2(t.z, t.w);
                }
                if (kRagged && left < r0 + R) {   // rows of the next sequence: nothing may come from them
#pragma unroll
                    for (int i = 0; i < R; ++i)
                        if (r0 + i >= left) v[i] = zero;
                }
                if (kRagged && p.gxT && has_seq && left > r0 && left <= r0 + R) {   // the gradient of the final state
                    const float2 c0 = p.gxT[(size_t)b * p.P + pg], c1 = p.gxT[(size_t)b * p.P + pg + 1];
                    const C2 add = {pack2(c0.x, c1.x), pack2(c0.y, c1.y)};
#pragma unroll
                    for (int i = 0; i < R; ++i)
                        if (r0 + i == left - 1) v[i].re = add2(v[i].re, add.re), v[i].im = add2(v[i].im, add.im);
                }
                if (!kRagged && sl == gl && tb == p.tblocks - 1 && (!kTPair || rank == 1) && p.gxT && grp_valid) {   // the gradient of the final state
                    const float2 c0 = p.gxT[(size_t)b_grp * p.P + pg], c1 = p.gxT[(size_t)b_grp * p.P + pg + 1];
                    float v0, v1, v2, v3;
                    unpack2(v[R - 1].re, v0, v1);
                    unpack2(v[R - 1].im, v2, v3);
                    v[R - 1].re = pack2(v0 + c0.x, v1 + c1.x);
                    v[R - 1].im = pack2(v2 + c0.y, v3 + c1.y);
                }
                // the warp has its rows: rows m - 1 ... m + R - 2 of x (both planes) into its part of the tile
                fence_async_smem();
                __syncwarp();
                if (group_leader()) {
                    mbar_expect_tx(xb, Cfg::kGroupBytes);
                    tma_load_3d(smem_u32(warp_buf), &tmX, xb, n_tile * kS, m0 + r0 - 1, 0);
                    // and the same rows of the tile before this one into L2, where the next load will find them
                    if (tb > 0) tma_prefetch_3d(&tmX, n_tile * kS, m0 - (kTPair ? 2 : 1) * BM + r0 - 1, 0);
                }
                C2 e = zero;
                if (from_carry) {   // from the carried value (nothing, for a sequence inside the tile): these results are final
                    const float4 c = short_seq ? make_float4(0.f, 0.f, 0.f, 0.f) : carry_s[sp];
                    C2 x = {pack2(c.x, c.y), pack2(c.z, c.w)};
                    if (mask == 0u) {
#pragma unroll
                        for (int i = R - 1; i >= 0; --i) v[i] = x = cstep2(ar, ai, nai, x, v[i]);
                    } else {
#pragma unroll
                        for (int i = R - 1; i >= 0; --i) {
                            if ((mask >> i) & 1u) x = zero;
                            v[i] = x = cstep2(ar, ai, nai, x, v[i]);
                        }
                    }
                    e = x;
                } else if (mask == 0u) {
#pragma unroll
                    for (int i = R - 1; i >= 0; --i) e = cstep2(ar, ai, nai, e, v[i]);
                } else {
#pragma unroll
                    for (int i = R - 1; i >= 0; --i) {
                        if ((mask >> i) & 1u) e = zero;
                        e = cstep2(ar, ai, nai, e, v[i]);
                    }
                }
                {
                    float e0, e1, e2, e3;
                    unpack2(e.re, e0, e1);
                    unpack2(e.im, e2, e3);
                    agg_e[te] = make_float4(e0, e1, e2, e3);
                }
                epi_sync();   // group results visible
                const float4 pw = pow_s[chain_par][0][sp];
                const f32x2 pr = pack2(pw.x, pw.y), npi = pack2(pw.z, pw.w), pi = neg2(npi);   // (conjugate)
                C2 x = e;
                if (kTPair) {
                    // The value that enters the tile (s of the row after it) comes from the peer CTA, which holds the
                    // tile after this one, except for the sequence's last tile.  The first row group passes s of the
                    // tile's first row on as soon as it can: the tile's own contribution (the groups' results joined
                    // from zero) is ready before the peer's value arrives.
                    const bool first = rank == 1 && tb == p.tblocks - 1, last = rank == 0 && tb == 0;
                    C2 tile = zero;
                    const float4 tw = pow_s[chain_par][kTPair ? 1 : 0][sp];
                    if (sl == 0 && !last) {
#pragma unroll
                        for (int gq = nsl - 1; gq >= 1; --gq) {
                            const float4 c = agg_e[gq * kPairs + sp];
                            const C2 eg = {pack2(c.x, c.y), pack2(c.z, c.w)};
                            tile = (gq == nsl - 1 || ((gflags >> gq) & 1u)) ? eg : cstep2(pr, pi, npi, tile, eg);
                        }
                        tile = (gflags & 1u) ? e : cstep2(pr, pi, npi, tile, e);
                    }
                    if (!first) {
                        (void)mbar_wait_acquire_cluster(smem_u32(&carry_bar[n_recv & 1u]), (n_recv >> 1) & 1u, epi_flag);
                        const float4 c = carry_ring[n_recv & 1u][sp];
                        cin.re = pack2(c.x, c.y);
                        cin.im = pack2(c.z, c.w);
                        ++n_recv;
                    } else {
                        cin = zero;
                    }
                    if (sl == 0 && !last) {
                        const f32x2 tr = pack2(tw.x, tw.y), nti = pack2(tw.z, tw.w);
                        const C2 out = gflags == 0u ? cstep2(tr, neg2(nti), nti, cin, tile) : tile;
                        float o0, o1, o2, o3;
                        unpack2(out.re, o0, o1);
                        unpack2(out.im, o2, o3);
                        st_cluster_f4(peer_ring + (uint32_t)(((n_send & 1u) * kPairs + sp) * sizeof(float4)), make_float4(o0, o1, o2, o3));
                        mbar_arrive_release_cluster(peer_bar + 8u * (n_send & 1u));
                        ++n_send;
                    }
                    x = cin;
#pragma unroll
                    for (int gq = nsl - 1; gq >= 1; --gq) {
                        if (gq > sl) {
                            const float4 c = agg_e[gq * kPairs + sp];
                            const C2 eg = {pack2(c.x, c.y), pack2(c.z, c.w)};
                            x = ((gflags >> gq) & 1u) ? eg : cstep2(pr, pi, npi, x, eg);
                        }
                    }
                } else if (!from_carry) {   // s of the row after this group's last
                    {
                        const float4 c = agg_e[gl * kPairs + sp];
                        x.re = pack2(c.x, c.y);
                        x.im = pack2(c.z, c.w);
                    }
#pragma unroll
                    for (int gq = nsl - 2; gq >= 1; --gq) {
                        if (gq > sl && gq < gl) {
                            const float4 c = agg_e[gq * kPairs + sp];
                            const C2 eg = {pack2(c.x, c.y), pack2(c.z, c.w)};
                            x = ((gflags >> gq) & 1u) ? eg : cstep2(pr, pi, npi, x, eg);
                        }
                    }
                }
                // (3) fold again, with x_{t-1} at hand: sums for gAbar, s as hi / lo bf16 halves in place of x
                if (!mbar_wait(xb, xphase, epi_flag)) {
                    // (the wait gave up: the flag is set, everybody leaves at the next barrier)
                }
                xphase ^= 1u;
                if (kRagged && left >= r0 && left < r0 + R) {
                    // the row after the sequence's last: its s is 0, its x is the sequence's final state, which enters no
                    // product and may be infinite
                    xs[(left - r0) * kPairs] = xs[(R + left - r0) * kPairs] = make_uint2(0u, 0u);
                }
                const bool seq_start = tb == 0 && sl == g0 && (!kTPair || rank == 0);   // row 0 of this group is the sequence's first row
                if (short_seq && seq_start) {                // the state before that row: this sequence's x0
                    xinit = zero;
                    if (p.x0 && grp_valid) {
                        const float2 c0 = p.x0[(size_t)b_grp * p.P + pg], c1 = p.x0[(size_t)b_grp * p.P + pg + 1];
                        xinit.re = pack2(c0.x, c1.x);
                        xinit.im = pack2(c0.y, c1.y);
                    }
                }
                // A tile without flags (the common case) takes the loop without the per-row tests.
                auto fold_rows = [&](auto with_flags) {
                    constexpr bool kFlags = decltype(with_flags)::value;
#pragma unroll
                    for (int i = R - 1; i >= 0; --i) {
                        C2 sv = v[i];
                        if (!from_carry) {
                            if (kFlags && ((mask >> i) & 1u)) x = zero;
                            sv = x = cstep2(ar, ai, nai, x, v[i]);
                        }
                        if (!kFlags || !((mask0 >> i) & 1u)) {
                            C2 xp;
                            if (seq_start && i == 0) {
                                xp = xinit;
                            } else {
                                const uint2 xh = xs[i * kPairs], xl = xs[(R + i) * kPairs];
                                xp.re = add2(pack2(__uint_as_float(xh.x << 16), __uint_as_float(xh.y << 16)),
                                             pack2(__uint_as_float(xl.x << 16), __uint_as_float(xl.y << 16)));
                                xp.im = add2(pack2(__uint_as_float(xh.x & 0xffff0000u), __uint_as_float(xh.y & 0xffff0000u)),
                                             pack2(__uint_as_float(xl.x & 0xffff0000u), __uint_as_float(xl.y & 0xffff0000u)));
                            }
                            // g += s conj(x):  re += s.re x.re + s.im x.im,  im += s.im x.re - s.re x.im (two sums)
                            g.re = fma2(sv.re, xp.re, fma2(sv.im, xp.im, g.re));
                            g.im = fma2(sv.im, xp.re, g.im);
                            gim_neg = fma2(sv.re, xp.im, gim_neg);
                        }
                        float re0, re1, im0, im1;
                        unpack2(sv.re, re0, re1);
                        unpack2(sv.im, im0, im1);
                        const __nv_bfloat162 h0 = __floats2bfloat162_rn(re0, im0), h1 = __floats2bfloat162_rn(re1, im1);
                        const uint32_t hb0 = *reinterpret_cast<const uint32_t*>(&h0), hb1 = *reinterpret_cast<const uint32_t*>(&h1);
                        const f32x2 lre = sub2(sv.re, pack2(__uint_as_float(hb0 << 16), __uint_as_float(hb1 << 16)));
                        const f32x2 lim = sub2(sv.im, pack2(__uint_as_float(hb0 & 0xffff0000u), __uint_as_float(hb1 & 0xffff0000u)));
                        float lr0, lr1, li0, li1;
                        unpack2(lre, lr0, lr1);
                        unpack2(lim, li0, li1);
                        const __nv_bfloat162 l0 = __floats2bfloat162_rn(lr0, li0), l1 = __floats2bfloat162_rn(lr1, li1);
                        xs[i * kPairs] = make_uint2(hb0, hb1);
                        xs[(R + i) * kPairs] = make_uint2(*reinterpret_cast<const uint32_t*>(&l0), *reinterpret_cast<const uint32_t*>(&l1));
                    }
                };
                if ((mask | mask0) == 0u)
                    fold_rows(std::false_type{});
                else
                    fold_rows(std::true_type{});
                fence_async_smem();
                __syncwarp();
                if (grp_valid && group_leader()) {
                    if (kRagged) tma_store_4d_nocommit(&tmS, smem_u32(warp_buf), n_tile * kS, p.T - left + r0, b, 0);   // clipped at T
                    else tma_store_3d_nocommit(&tmS, smem_u32(warp_buf), n_tile * kS, m0 + r0, 0);
                    tma_commit_group();
                }
                if (sl == g0) {   // x is s of the first row of the tile (of the sequence, when it lies inside the tile)
                    float x0r, x1r, x0i, x1i;
                    unpack2(x.re, x0r, x1r);
                    unpack2(x.im, x0i, x1i);
                    if (kTPair && !(rank == 0 && tb == 0)) {
                        // (handed to the peer above)
                    } else if (tb > 0) {
                        carry_s[sp] = make_float4(x0r, x1r, x0i, x1i);
                    } else if (p.gx0 && grp_valid) {   // what reaches the initial state: keep_0 conj(Abar) s_0
                        const bool cut = (mask0 & 1u) != 0u;
                        const float2 z = make_float2(0.f, 0.f);
                        p.gx0[(size_t)b_grp * p.P + pg] = cut ? z : cfma(a0, make_float2(x0r, x0i), z);
                        p.gx0[(size_t)b_grp * p.P + pg + 1] = cut ? z : cfma(a1, make_float2(x1r, x1i), z);
                    }
                }
            }
            if (!ok) break;
            // the chain's sums over the row groups (agg_e is free: everybody is past the last tile's join)
            epi_sync();
            {
                float g0, g1, g2, g3;
                unpack2(g.re, g0, g1);
                unpack2(sub2(g.im, gim_neg), g2, g3);
                agg_e[te] = make_float4(g0, g1, g2, g3);
            }
            epi_sync();
            if (sl == 0 && has_seq) {
                float4 sum = agg_e[sp];
#pragma unroll
                for (int gq = 1; gq < nsl; ++gq) {
                    const float4 c = agg_e[gq * kPairs + sp];
                    sum.x += c.x, sum.y += c.y, sum.z += c.z, sum.w += c.w;
                }
                const size_t part_row = kTPair ? 2 * (size_t)b + rank : (size_t)b;   // kTPair: each CTA has half of the sequence's rows
                p.gA_part[part_row * p.P + pg] = make_float2(sum.x, sum.z);
                p.gA_part[part_row * p.P + pg + 1] = make_float2(sum.y, sum.w);
            }
        }
        if (group_leader()) tma_store_wait_all();
    }
    tc_fence_before();
    __syncwarp();
    cluster_sync_all();
    tc_fence_after();
    if (warp == 1) tmem_dealloc_pair(tmem_base, kTmemCols);
    if (threadIdx.x == 0 && (*s.abort_flag || *s.epi_abort()) && p.hdr) p.hdr->status = SSM_ERR_TIMEOUT;
}

// ---------------------------------------------------------------------------------------------
// NT kernel (weight gradients): one 128 x 256 output tile and one slice of the rows per CTA
// ---------------------------------------------------------------------------------------------
struct NtParams {
    int K;              // rows of A and Bm (the reduction index)
    int J;              // columns of Bm = leading dimension of a partial
    int I;              // columns of A
    int j_tiles;        // J / (BN / 2)
    int blocks_per_split;  // k-blocks (of BK rows) per slice
    int first;          // the product blockIdx.z = 0 stands for
    float* part[2];     // [splits, I, J] each
    WsHeader* hdr;
};
struct NtMaps {
    CUtensorMap a[2], hi[2], lo[2];   // per product
};

// The tensor core truncates its fp32 accumulator at every addition: a chain of n of them is about n 2^-25 2/3 off its sum.
// So a slice of more than kNtSegment k-blocks (64 additions) is multiplied in segments of that length, alternately into the
// two halves of tensor memory, and the epilogue warps add a finished segment to their registers while the next one runs
// (16384 rows x 1024 x 1024 in one chain: dB 1.9e-5 off, in segments 4.8e-6; 323.9 and 322.3 us for the pass).  Shorter
// slices take the kernels without that (kSegs = false): with its registers the next kernel finds no room on the SM before
// this one ends (6400 rows at 256, 128: 55.0 / 57.4 us for the pass).
constexpr int kNtSegment = 16;

// What an epilogue warp does with a slice: adds its segments, both planes of Bm each, and stores its 32 rows x nt_epi_cols
// columns (dst: this lane's row).  `leader_empty0`: the tmem_empty barriers of the CTA that issues the MMAs, as a cluster
// address where kPair.
template <bool kPair, bool kSegs>
__device__ __forceinline__ void nt_epilogue(const Smem& s, float* dst, bool row_ok, int nkb, int warp, int lane, uint32_t tmem_base,
                                            uint32_t leader_empty0) {
    constexpr int kCols = nt_epi_cols(kSegs);
    const uint32_t t_row = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(((warp - 2) >> 2) * kCols);
    if (!kSegs) {
        if (nkb > 0) {
            if (!mbar_wait_warp(s.tmem_full(0), 0, s.abort_flag)) return;
            tc_fence_after();
        }
#pragma unroll 1
        for (int c = 0; c < kCols; c += 32) {
            uint32_t r[32], r2[32];
            if (nkb > 0) {
                tmem_ld32(t_row + (uint32_t)c, r);
                tmem_ld32(t_row + (uint32_t)(BN / 2 + c), r2);
                tmem_ld_wait();
            } else {
#pragma unroll
                for (int i = 0; i < 32; ++i) r[i] = r2[i] = 0u;
            }
            if (row_ok)
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    reinterpret_cast<float4*>(dst + c)[i] =
                        make_float4(__uint_as_float(r[4 * i]) + __uint_as_float(r2[4 * i]),
                                    __uint_as_float(r[4 * i + 1]) + __uint_as_float(r2[4 * i + 1]),
                                    __uint_as_float(r[4 * i + 2]) + __uint_as_float(r2[4 * i + 2]),
                                    __uint_as_float(r[4 * i + 3]) + __uint_as_float(r2[4 * i + 3]));
        }
        return;
    }
    float sum[kCols];
#pragma unroll
    for (int i = 0; i < kCols; ++i) sum[i] = 0.f;
    const int segs = (nkb + kNtSegment - 1) / kNtSegment;
#pragma unroll 1
    for (int seg = 0; seg < segs; ++seg) {
        const int buf = seg & 1;
        if (!mbar_wait_warp(s.tmem_full(buf), (uint32_t)(seg >> 1) & 1u, s.abort_flag)) return;
        tc_fence_after();
#pragma unroll
        for (int c = 0; c < kCols; c += 16) {   // (16 columns at a time: registers)
            uint32_t r[16], r2[16];
            tmem_ld16(t_row + (uint32_t)(buf * BN + c), r);
            tmem_ld16(t_row + (uint32_t)(buf * BN + BN / 2 + c), r2);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 16; ++i) sum[c + i] += __uint_as_float(r[i]) + __uint_as_float(r2[i]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
            if (kPair) mbar_arrive_cluster(leader_empty0 + 8u * (uint32_t)buf);
            else mbar_arrive(s.tmem_empty(buf));
        }
    }
    if (row_ok) {
#pragma unroll
        for (int i = 0; i < kCols / 4; ++i)
            reinterpret_cast<float4*>(dst)[i] = make_float4(sum[4 * i], sum[4 * i + 1], sum[4 * i + 2], sum[4 * i + 3]);
    }
}

// The 256 accumulator columns are 128 output columns times the two planes (hi, lo) of Bm, added in the epilogue.
template <bool kSegs>
__global__ void __launch_bounds__(nt_threads(kSegs), 1)
gemm_tc_nt_kernel(const __grid_constant__ NtMaps maps, const __grid_constant__ NtParams p) {
    const int z = (int)blockIdx.z + p.first;
    const CUtensorMap &tmA = maps.a[z], &tmBhi = maps.hi[z], &tmBlo = maps.lo[z];
    extern __shared__ uint8_t smem_raw[];
    const Smem s = carve_smem(smem_raw, kStages, 0, 0);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t tmem_base = prologue(s, warp, lane, nt_epi_warps(kSegs));
    grid_dep_wait();   // the set-up above ran beside the end of the kernel before this one
    grid_dep_launch();
    const int tile = blockIdx.x, split = blockIdx.y;
    constexpr int kOutCols = BN / 2;   // accumulator columns [0,128): hi plane, [128,256): lo plane
    const int i0 = (tile / p.j_tiles) * BM, j0 = (tile % p.j_tiles) * kOutCols;
    const int total_blocks = (p.K + BK - 1) / BK;
    const int kb0 = split * p.blocks_per_split;
    const int kb1 = min(total_blocks, kb0 + p.blocks_per_split);
    const int nkb = max(0, kb1 - kb0);

    if (warp == 0) {
        if (elect_one()) {
            prefetch_tmap(&tmA);
            prefetch_tmap(&tmBhi);
            prefetch_tmap(&tmBlo);
        }
        int stage = 0;
        uint32_t phase = 0;
        for (int kb = 0; kb < nkb; ++kb) {
            if (!mbar_wait_warp(s.empty(stage), phase ^ 1u, s.abort_flag)) break;
            if (elect_one()) {
                mbar_expect_tx(s.full(stage), kStageBytes);
                const uint32_t a_dst = smem_u32(s.tiles + (size_t)stage * kStageBytes);
                const int row = (kb0 + kb) * BK;
#pragma unroll
                for (int h = 0; h < BM / 64; ++h) tma_load_2d(a_dst + h * (BK * 128), &tmA, s.full(stage), i0 + 64 * h, row);
#pragma unroll
                for (int h = 0; h < BN / 128; ++h) {
                    tma_load_2d(a_dst + kABytes + h * (BK * 128), &tmBhi, s.full(stage), j0 + 64 * h, row);
                    tma_load_2d(a_dst + kABytes + (BN / 128 + h) * (BK * 128), &tmBlo, s.full(stage), j0 + 64 * h, row);
                }
            }
            if (++stage == kStages) {
                stage = 0;
                phase ^= 1u;
            }
        }
    } else if (warp == 1) {
        if (nkb > 0) {
            constexpr uint32_t idesc = instr_desc(BM, BN, 1, 1);
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int kb = 0; kb < nkb; ++kb) {
                const int seg = kSegs ? kb / kNtSegment : 0, buf = seg & 1, in_seg = kSegs ? kb % kNtSegment : kb;
                if (kSegs && in_seg == 0 && seg >= 2) {   // the epilogue has taken segment seg - 2 out of this half of tensor memory
                    if (!(ok = mbar_wait_warp(s.tmem_empty(buf), (uint32_t)((seg >> 1) - 1) & 1u, s.abort_flag))) break;
                    tc_fence_after();
                }
                if (!(ok = mbar_wait_warp(s.full(stage), phase, s.abort_flag))) break;
                tc_fence_after();
                const uint32_t a_addr = smem_u32(s.tiles + (size_t)stage * kStageBytes);
                const uint64_t adesc = smem_desc_mnmajor(a_addr);
                const uint64_t bdesc = smem_desc_mnmajor(a_addr + kABytes);
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < BK / UK; ++k) {
                        // 16 k-rows of 128 bytes further: +2048 bytes = +128 in the address field
                        umma_bf16(tmem_base + (uint32_t)(buf * BN), adesc + (uint64_t)(128 * k), bdesc + (uint64_t)(128 * k), idesc,
                                  (uint32_t)((in_seg | k) != 0));
                    }
                    umma_commit(s.empty(stage));
                    if (kb + 1 == nkb || (kSegs && in_seg + 1 == kNtSegment)) umma_commit(s.tmem_full(buf));
                }
                if (++stage == kStages) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
        }
    } else {
        const int row = i0 + (warp & 3) * 32 + lane, col = j0 + ((warp - 2) >> 2) * nt_epi_cols(kSegs);
        nt_epilogue<false, kSegs>(s, p.part[z] + ((size_t)split * p.I + row) * p.J + col, row < p.I, nkb, warp, lane, tmem_base, 0);
    }
    epilogue_exit(s, warp, tmem_base, p.hdr);
}

// ---------------------------------------------------------------------------------------------
// NT kernel on CTA pairs
// ---------------------------------------------------------------------------------------------
// The same product on clusters of two CTAs: one MMA spans a 256 x 256 accumulator tile, CTA r holding
// output rows i0 + 128 r .. (its 128 columns of A) and one plane of Bm (r = 0: the high halves, r = 1: the low
// halves; the MMA takes half of its B columns from each CTA).  Every CTA then brings in 32 KB per k-block
// instead of 48 KB for the same tensor-core cycles, which is what bounds the single-CTA kernel (96 KB through
// shared memory per 512 tensor-core cycles).  Barriers as in the TN pair kernel: the leader's `full` barriers
// count both CTAs' bytes, its commits arrive in both CTAs.  One tile and one slice of the rows per pair.
constexpr int kNtPairStages = 6;
constexpr int kNtPairStageBytes = kABytes + kBBytes / 2;   // 32 KB
constexpr size_t kNtPairSmemBytes = (size_t)kNtPairStages * kNtPairStageBytes + 1024 + 256;

template <bool kSegs>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(nt_threads(kSegs), 1)
gemm_tc_nt_pair_kernel(const __grid_constant__ NtMaps maps, const __grid_constant__ NtParams p) {
    const int z = (int)blockIdx.z + p.first;
    const CUtensorMap &tmA = maps.a[z], &tmBhi = maps.hi[z], &tmBlo = maps.lo[z];
    extern __shared__ uint8_t smem_raw[];
    const Smem s = carve_smem(smem_raw, kNtPairStages, 0, 0, kNtPairStageBytes, 0);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    // barriers of the ring: more stages than the common layout has slots for, so they take the skip slots
    auto rfull = [&](int i) { return s.skip_full(i); };
    auto rempty = [&](int i) { return s.skip_full(kNtPairStages + i); };
    if (threadIdx.x == 0) {
        for (int i = 0; i < kNtPairStages; ++i) {
            mbar_init(rfull(i), 1);
            mbar_init(rempty(i), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(s.tmem_full(i), 1);
            mbar_init(s.tmem_empty(i), 2 * nt_epi_warps(kSegs));
        }
        *s.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();
    if (warp == 1) tmem_alloc_pair(s.tmem_slot, kSegs ? kTmemCols : BN);
    tc_fence_before();
    cluster_sync_all();
    tc_fence_after();
    const uint32_t tmem_base = *s.tmem_slot_ptr;
    grid_dep_wait();   // the set-up above ran beside the end of the kernel before this one
    grid_dep_launch();

    const int tile = blockIdx.x >> 1, split = blockIdx.y;
    constexpr int kOutCols = BN / 2;
    const int i0 = (tile / p.j_tiles) * (2 * BM) + (int)rank * BM, j0 = (tile % p.j_tiles) * kOutCols;
    const int total_blocks = (p.K + BK - 1) / BK;
    const int kb0 = split * p.blocks_per_split;
    const int nkb = max(0, min(total_blocks, kb0 + p.blocks_per_split) - kb0);

    if (warp == 0) {
        if (elect_one()) {
            prefetch_tmap(&tmA);
            prefetch_tmap(rank == 0 ? &tmBhi : &tmBlo);
        }
        const CUtensorMap* tmB = rank == 0 ? &tmBhi : &tmBlo;
        int stage = 0;
        uint32_t phase = 0;
        for (int kb = 0; kb < nkb; ++kb) {
            if (!mbar_wait_warp(rempty(stage), phase ^ 1u, s.abort_flag)) break;
            const uint32_t leader_full = map_to_cta(rfull(stage), 0);
            if (elect_one()) {
                if (rank == 0) mbar_expect_tx(rfull(stage), 2 * kNtPairStageBytes);
                const uint32_t a_dst = smem_u32(s.tiles + (size_t)stage * kNtPairStageBytes);
                const int row = (kb0 + kb) * BK;
#pragma unroll
                for (int h = 0; h < BM / 64; ++h) tma_load_2d_pair(a_dst + h * (BK * 128), &tmA, leader_full, i0 + 64 * h, row);
#pragma unroll
                for (int h = 0; h < kOutCols / 64; ++h)
                    tma_load_2d_pair(a_dst + kABytes + h * (BK * 128), tmB, leader_full, j0 + 64 * h, row);
            }
            if (++stage == kNtPairStages) {
                stage = 0;
                phase ^= 1u;
            }
        }
    } else if (warp == 1) {
        if (rank == 0 && nkb > 0) {
            constexpr uint32_t idesc = instr_desc(2 * BM, BN, 1, 1);
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int kb = 0; kb < nkb; ++kb) {
                const int seg = kSegs ? kb / kNtSegment : 0, buf = seg & 1, in_seg = kSegs ? kb % kNtSegment : kb;
                if (kSegs && in_seg == 0 && seg >= 2) {   // both CTAs' epilogues have taken segment seg - 2 out of this half of tensor memory
                    if (!(ok = mbar_wait_warp(s.tmem_empty(buf), (uint32_t)((seg >> 1) - 1) & 1u, s.abort_flag))) break;
                    tc_fence_after();
                }
                if (!(ok = mbar_wait_warp(rfull(stage), phase, s.abort_flag))) break;
                tc_fence_after();
                const uint32_t a_addr = smem_u32(s.tiles + (size_t)stage * kNtPairStageBytes);
                const uint64_t adesc = smem_desc_mnmajor(a_addr);
                const uint64_t bdesc = smem_desc_mnmajor(a_addr + kABytes);
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < BK / UK; ++k)
                        umma_bf16_pair(tmem_base + (uint32_t)(buf * BN), adesc + (uint64_t)(128 * k), bdesc + (uint64_t)(128 * k), idesc,
                                       (uint32_t)((in_seg | k) != 0));
                    umma_commit_pair(rempty(stage));
                    if (kb + 1 == nkb || (kSegs && in_seg + 1 == kNtSegment)) umma_commit_pair(s.tmem_full(buf));
                }
                if (++stage == kNtPairStages) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
        }
    } else {
        const int row = i0 + (warp & 3) * 32 + lane, col = j0 + ((warp - 2) >> 2) * nt_epi_cols(kSegs);
        nt_epilogue<true, kSegs>(s, p.part[z] + ((size_t)split * p.I + row) * p.J + col, row < p.I, nkb, warp, lane, tmem_base,
                          map_to_cta(s.tmem_empty(0), 0));
    }
    // nobody leaves (or frees tensor memory) while the other CTA may still signal or compute
    tc_fence_before();
    __syncwarp();
    cluster_sync_all();
    tc_fence_after();
    if (warp == 1) tmem_dealloc_pair(tmem_base, kSegs ? kTmemCols : BN);
    if (threadIdx.x == 0 && *s.abort_flag && p.hdr) p.hdr->status = SSM_ERR_TIMEOUT;
}

// ---------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------
static int sm_count() { return device_sm_count(); }

// How many CTA pairs of `kernel` the current device runs at the same time.
int resident_pairs(const void* kernel, size_t smem_bytes, int threads) {
    return std::max(0, resident_clusters(kernel, 2, smem_bytes, threads));
}

template <typename K>
static bool set_smem(K kernel, size_t bytes) {
    return set_max_dynamic_smem(reinterpret_cast<const void*>(kernel), bytes);
}

}  // namespace tc

int tc_max_n() { return tc::kMaxDiag; }

bool tc_tn_supported(int M, int N_out, int K, bool split_w) {
    const int out_cols = split_w ? tc::BN / 2 : tc::BN;
    // Outputs are a multiple of 128 columns wide; a last tile of the 256-column kind may be half empty (its
    // weight rows past N_out read as zero and its results past N_out are clipped by the TMA stores).
    (void)out_cols;
    return M >= 1 && K >= tc::BK && (K % tc::BK) == 0 && (N_out % (tc::BN / 2)) == 0 && N_out <= tc::kMaxDiag;
}

static int pair_tiles_of(int M, int n_tiles) { return ((M + 2 * tc::BM - 1) / (2 * tc::BM)) * n_tiles; }

// Whether a projection has enough 256 x 256 tiles for the kernel on CTA pairs; the others take gemm_tc_small.cu.
// us back to back, pairs / few tiles, by number of tiles (products of planes: below):
//   acc + diag * skip:         24 tiles 9.3 / 9.5, 32: 12.2 / 12.4, 48: 9.7 / 11.6, 64: 12.7 / 14.6
//   the same with column sums: 32: 11.5 / 10.1, 48: 12.0 / 14.2 (the pair kernel keeps the sums of kDotMaxN columns)
//   hi + lo weights:           32: 6.6 / 5.9 and 10.4 / 11.9, 48: 7.9 / 8.9, 128: 17.4 / 25.0
// Six products of planes, whose planes the few-tile kernel loads once, stay there at every size.
enum { kEpiStore = 0, kEpiDiag = 1, kEpiGate = 2, kEpiDot = 3 };
static int epi_of(const GemmTcTN& g) { return g.gate_out ? kEpiGate : (g.store_f32 && !g.diag ? kEpiStore : (g.dot ? kEpiDot : kEpiDiag)); }
// Whether the kernel on pairs takes tiles of 128 columns instead of 256 (acc + diag * skip): where the shorter last round, or a
// last tile of 128 columns that would be half empty, is worth reading A twice as often.  A round of narrow tiles takes
// 0.7 of a wide one, 0.62 with the column sums, whose epilogue is the longer part.  us incl. 4 of events, wide / narrow, rows x
// columns: y 4100 x 512 14.8 / 13.1, 9600 x 384 17.1 / 14.7, 30000 x 384 25.0 / 24.8, 12800 x 512 18.9 / 20.6; du 9600 x 384 20.9 / 16.8,
// 30000 x 384 35.0 / 31.2, 64000 x 384 51.4 / 47.5, 12800 x 512 24.5 / 23.0, 30000 x 512 41.1 / 44.1.  Contractions above 512: never
// (6400 x 1024 x 1024 25.0 / 27.1 and 31.0 / 33.6).
static bool narrow_tiles(const GemmTcTN& g) {
    const int epi = epi_of(g);
    if ((epi != kEpiDiag && epi != kEpiDot) || g.n_products > 0 || g.K > 512) return false;
    const int pairs = std::max(1, tc::sm_count() / 2);
    auto rounds = [&](int cols) { return (pair_tiles_of(g.M, (g.N_out + cols - 1) / cols) + pairs - 1) / pairs; };
    return rounds(tc::BN / 2) * (epi == kEpiDot ? 0.62 : 0.7) < rounds(tc::BN);
}
static bool use_pairs(const GemmTcTN& g) {
    if (g.n_products > 3 || g.a_f32 || g.scan || g.add || (g.diag && g.store_f32)) return false;
    const int out_cols = g.split_w ? tc::BN / 2 : tc::BN, tiles = pair_tiles_of(g.M, (g.N_out + out_cols - 1) / out_cols);
    const int epi = epi_of(g);
    if (epi == kEpiDot && g.N_out > tc::kDotMaxN) return false;
    // Products of planes, which the few-tile kernel (CTA pairs there too) loads once: us of the gate's forward / backward call,
    // few tiles / pairs, rows x H: 6400 x 1024 (100 tiles) 64.7 / 69.4 and 104.3 / 105.7, 12800 x 1024 102.6 / 106.0 and
    // 179.6 / 181.0, 32768 x 1024 232.0 / 235.5 and 451.1 / 454.6; 16384 x 512 (128 tiles) 58.7 / 60.8 and 99.7 / 94.4,
    // 32768 x 512 105.1 / 100.9 and 185.4 / 179.9, 262144 x 512 736.6 / 697.2 and 1395 / 1300.
    if (g.n_products > 0) return tiles >= (g.K >= 1024 ? 600 : (epi == kEpiGate ? 160 : 80));
    // (in narrow tiles that run in one round already from 24: 2000 x 768 14.7 us on the few-tile kernel, 12.7)
    return tiles >= (epi == kEpiDiag ? (narrow_tiles(g) ? 24 : 32) : 40);
}
// Whether acc + diag * skip also leaves the column sums of skip * dot: not for many rows of very wide outputs, which the
// pair kernel takes faster without than the few-tile kernel with them.
bool tc_tn_dot_supported(int M, int N_out) { return N_out <= tc::kDotMaxN || pair_tiles_of(M, (N_out + tc::BN - 1) / tc::BN) < 32; }
// Most rows of column sums a projection leaves.
int tc_tn_dot_max_rows(int M) { return std::max(tc_tn_small_max_dot_rows(M), 2 * tc::sm_count()); }

int launch_gemm_tc_tn(const GemmTcTN& g, cudaStream_t st) {
    using namespace tc;
    if (!use_pairs(g)) return launch_gemm_tc_tn_small(g, st);
    const int epi = epi_of(g);
    const bool narrow = narrow_tiles(g);
    const int out_cols = g.split_w || narrow ? BN / 2 : BN;
    const int n_tiles = (g.N_out + out_cols - 1) / out_cols;
    if ((epi == 1 || epi == 3) && (g.split_w || !g.diag || !g.skip)) return SSM_ERR_SHAPE;
    if (epi == 3 && (!g.dot_part || !g.dot_rows)) return SSM_ERR_SHAPE;
    if (epi == 2 && (g.split_w || !g.store_f32 || !g.skip)) return SSM_ERR_SHAPE;
    CUtensorMap ma, mw, mo, ms, mg;
    // with a product schedule the operands are planes_a / planes_w bf16 planes of K columns each, side by side
    const int n_prod = g.n_products > 0 ? g.n_products : 1;
    const uint64_t a_cols = (uint64_t)g.K * (g.n_products > 0 ? g.planes_a : 1);
    const uint64_t w_cols = (uint64_t)g.K * (g.n_products > 0 ? g.planes_w : 1);
    if (g.n_products > 8) return SSM_ERR_SHAPE;
    if (!make_map(&ma, g.A, (uint64_t)g.M, a_cols, BK, BM)) return SSM_ERR_CUDA;
    if (g.store_f32) {   // fp32 result, stored by the TMA unit in boxes of 32 rows x 32 columns
        if (!make_map(&mo, g.out, (uint64_t)g.M, (uint64_t)g.N_out, 32, 32, true)) return SSM_ERR_CUDA;
    } else {             // bf16 result: 32 x 32 boxes, 64-byte rows
        if (!make_map(&mo, g.out, (uint64_t)g.M, (uint64_t)g.N_out, 32, 32, false, CU_TENSOR_MAP_SWIZZLE_64B)) return SSM_ERR_CUDA;
    }
    ms = mo;             // unused unless there is a skip operand
    mg = mo;             // unused unless there is a gated result
    if (epi != 0 && !make_map(&ms, g.skip, (uint64_t)g.M, (uint64_t)g.N_out, 32, 32, false, CU_TENSOR_MAP_SWIZZLE_64B))
        return SSM_ERR_CUDA;
    if (epi == 2 && !make_map(&mg, g.gate_out, (uint64_t)g.M, (uint64_t)g.N_out, 32, 32, false, CU_TENSOR_MAP_SWIZZLE_64B))
        return SSM_ERR_CUDA;
    if (epi == 3 && !make_map(&mg, g.dot, (uint64_t)g.M, (uint64_t)g.N_out, 32, 32, false, CU_TENSOR_MAP_SWIZZLE_64B))
        return SSM_ERR_CUDA;   // (the dot operand travels in the map slot of the gated result)
    TnParams p{g.M, n_tiles, n_prod * (g.K / BK), g.N_out, g.diag, g.hdr, (const char*)g.A, (int)a_cols * 2, g.dot_part,
               g.n_products > 0 ? g.K / BK : 0, g.prod_a, g.prod_w};
    const int pair_tiles = pair_tiles_of(g.M, n_tiles);
    // rows of the packed weight matrix that exist (tiles may reach past them: those rows read as zero)
    const uint64_t w_rows = g.split_w ? (uint64_t)2 * g.N_out : (uint64_t)g.N_out;
    bool ok = true;
    if (!make_map(&mw, g.W, w_rows, w_cols, BK, narrow ? BN / 4 : BN / 2)) return SSM_ERR_CUDA;
    count_launch();
    // The kernel is persistent: its grid is the number of CTA pairs the device can hold at once
    // (not every SM has a partner that a cluster may use).
#define SSM_LAUNCH_PAIR(EPI, SPLIT, COLS)                                                                  \
do {                                                                                                   \
    auto kern = gemm_tc_tn_pair_kernel<EPI, SPLIT, COLS>;                                              \
    constexpr size_t smem = pair_smem_bytes(EPI, COLS);                                                \
    ok = set_smem(kern, smem);                                                                         \
    const int pairs = ok ? resident_pairs(reinterpret_cast<const void*>(kern), smem, kTnThreads) : 0;              \
    ok = ok && pairs > 0;                                                                              \
    if (ok) launch_dep(kern, 2 * min(pairs, pair_tiles), kTnThreads, smem, st, ma, mw, mo, ms, mg, p);         \
    if (ok && g.dot_rows) *g.dot_rows = 2 * min(pairs, pair_tiles);                                    \
} while (0)
    if (epi == 3 && narrow) SSM_LAUNCH_PAIR(3, false, BN / 2);
    else if (epi == 3) SSM_LAUNCH_PAIR(3, false, BN);
    else if (epi == 2) SSM_LAUNCH_PAIR(2, false, BN);
    else if (epi == 1 && narrow) SSM_LAUNCH_PAIR(1, false, BN / 2);
    else if (epi == 1) SSM_LAUNCH_PAIR(1, false, BN);
    else if (g.split_w) SSM_LAUNCH_PAIR(0, true, BN);
    else SSM_LAUNCH_PAIR(0, false, BN);
#undef SSM_LAUNCH_PAIR
    return ok ? SSM_OK : SSM_ERR_CUDA;
}

// The two bf16 planes of a state tensor as [2, B*T, P] 32-bit words, in boxes of `states` states x kFsRows rows x both planes.
static bool make_plane_map(CUtensorMap* map, const void* planes, int M, int P, int states) {
    PFN_cuTensorMapEncodeTiled fn = tc::encode_fn();
    if (!fn) return false;
    cuuint64_t dims[3] = {(cuuint64_t)P, (cuuint64_t)M, 2};
    cuuint64_t strides[2] = {(cuuint64_t)P * 4, (cuuint64_t)M * P * 4};
    cuuint32_t box[3] = {(cuuint32_t)states, (cuuint32_t)tc::kFsRows, 2};
    cuuint32_t estr[3] = {1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT32, 3, const_cast<void*>(planes), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The same planes as [2, B, T, P] words, in boxes of one sequence: rows past a sequence's end are clipped.
static bool make_plane_map4(CUtensorMap* map, const void* planes, int B, int T, int P, int states) {
    PFN_cuTensorMapEncodeTiled fn = tc::encode_fn();
    if (!fn) return false;
    const cuuint64_t row = (cuuint64_t)P * 4;
    cuuint64_t dims[4] = {(cuuint64_t)P, (cuuint64_t)T, (cuuint64_t)B, 2};
    cuuint64_t strides[3] = {row, row * T, row * T * B};
    cuuint32_t box[4] = {(cuuint32_t)states, (cuuint32_t)tc::kFsRows, 1, 2};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT32, 4, const_cast<void*>(planes), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Fewest (sequence, state group) chain pairs for which the kernels that scan in the epilogue of a projection
// are taken: below it too many CTA pairs would idle while a few walk their chains tile by tile.  us per forward and backward
// pass, separate / fused, at H, P = 512, 256 unless stated: 30 chains 10 x 16384 (384, 192) 968 / 931; 28: 7 x 1000 120 / 103;
// 24: 6 x 4096 287 / 271, 12 x 1024 (256, 128) 103 / 86; 20: 5 x 2048 168 / 151, 5 x 16384 826 / 854; 18: 9 x 512 (256, 128)
// 72 / 63; 16: 2 x 4096 the separate kernels.
static int fused_min_pairs(int T) { return T <= 4096 ? 18 : 24; }

// Sequences whose rows do not fall on tile boundaries: a sequence's last tile is then partly empty.
static bool fs_ragged(int T) { return !(T % tc::BM == 0 || T == 16 || T == 32 || T == 64); }
static int fs_tiles(int T) { return (T + tc::BM - 1) / tc::BM; }   // tiles of a sequence (T a multiple of BM, or ragged)
// Chains per state group: the sequences, or, when a 128-row tile holds several whole sequences, the tiles.
static int fs_units(int B, int T) { return T >= tc::BM || fs_ragged(T) ? B : (B * T + tc::BM - 1) / tc::BM; }

// How the kernels that scan in their epilogue take a problem: chains of 64 states, of 32 (few sequences: twice
// the chains, half the tile), or not at all (group 0); and, for few long sequences, both CTAs of a pair on one
// sequence (time pairs: CTA 0 has the even tiles, CTA 1 the odd ones, the state passes from one to the other
// through shared memory), which doubles the chains without halving the tile.
struct FusedMode {
    int group;
    bool time_pairs;
};
static FusedMode fused_mode(int B, int T, int H, int P) {
    if (H % tc::BK != 0 || P % 64 != 0) return {0, false};
    const bool ragged = fs_ragged(T);
    const int pairs64 = (P / 64) * ((fs_units(B, T) + 1) / 2);
    const int np = tc::sm_count() / 2;
    // A tile of 32 states takes about 0.8 of the time of a tile of 64 (measured), so halving the chains pays only
    // where the second half of the CTA pairs would otherwise idle: 16 x 16384 at P = 256 1.88 -> 1.78 ms per step,
    // 16 x 1024 0.242 -> 0.229; with 64 of 74 pairs busy (32 sequences) it costs 30 - 50 % in these kernels.
    // Time pairs double the chains at the full tile: 16 x 16384 1.76 -> 1.48 ms, 16 x 1024 0.228 -> 0.212.
    const int narrow_below = tc::sm_count() / 4 + 1;
    const bool tp_ok = (T % (2 * tc::BM) == 0 || (ragged && T > tc::BM));
    // Rounds of chains x tiles per chain: what the kernels' time goes with.
    const int tiles = T >= tc::BM || ragged ? fs_tiles(T) : 1, tp_tiles = (T + 2 * tc::BM - 1) / (2 * tc::BM);
    const int steps = (pairs64 + np - 1) / np * tiles;
    const int tp_chains = (P / 64) * B, tp_steps = (tp_chains + np - 1) / np * tp_tiles;
    FusedMode m{0, false};
    if (pairs64 >= narrow_below) {
        // Enough chains either way.  Time pairs give twice the chains at half the length, which fills the last
        // round of chains better when there are only a few rounds (48 sequences at P = 256: 96 chains take two
        // rounds on 74 CTA pairs, 192 half-length chains three half-rounds).
        m = {64, tp_ok && tp_steps < steps};
    } else if (tp_ok && tp_chains >= fused_min_pairs(T)) {
        m = {64, true};
    } else if (pairs64 >= fused_min_pairs(T)) {
        m = {32, false};
    }
    // A ragged length costs the empty rows of each sequence's last tile (empty = rows of its tiles / T).  us per forward and
    // backward pass, separate / fused, at H, P = 512, 256 unless stated:
    //   empty 1.02: 16 x 1000 165 / 136, 60 x 3000 1248 / 1020;  1.1: 9 x 2500 (H 256) 202 / 174, 30 x 1100 (256, 128) 146 / 126
    //   1.28: 16 x 100 69.5 / 60.5, 64 x 100 99 / 85, 150 x 200 (384, 192) 198 / 191;  1.42: 700 x 90 (256, 128) 219 / 211
    //   1.6: 100 x 80 106 / 97;  1.78: 1000 x 72 508 / 523;  1.94: 200 x 66 153 / 146;  2.6: 500 x 50 235 / 262;  3.2: 2000 x 40 561 / 786
    // With few rounds the time is latency, which empty rows do not lengthen.
    const int empty16 = ragged ? 16 * tc::BM * fs_tiles(T) / T : 16;
    if (empty16 > 26 && !(empty16 <= 32 && (m.time_pairs ? tp_steps : steps) <= 8)) return {0, false};
    return m;
}
int tc_gemm_scan_group(int B, int T, int H, int P) { return fused_mode(B, T, H, P).group; }
bool tc_gemm_scan_time_pairs(int B, int T, int H, int P) { return fused_mode(B, T, H, P).time_pairs; }
bool tc_gemm_scan_fwd_supported(int B, int T, int H, int P) { return tc_gemm_scan_group(B, T, H, P) != 0; }
bool tc_gemm_scan_bwd_supported(int B, int T, int H, int P) { return tc_gemm_scan_group(B, T, H, P) != 0; }

template <int kS, bool kTPair, bool kRagged>
static int launch_gemm_scan_fwd_s(const GemmScanFwd& g, cudaStream_t st) {
    using namespace tc;
    using Cfg = FsCfg<kS>;
    const int M = g.B * g.T;
    CUtensorMap ma, mw, mx;
    if (!make_map(&ma, g.u, (uint64_t)M, (uint64_t)g.H, BK, BM)) return SSM_ERR_CUDA;
    if (!make_map(&mw, g.Wsplit, (uint64_t)4 * g.P, (uint64_t)g.H, BK, Cfg::kWRows)) return SSM_ERR_CUDA;
    if (!(kRagged ? make_plane_map4(&mx, g.x_planes, g.B, g.T, g.P, kS) : make_plane_map(&mx, g.x_planes, M, g.P, kS))) return SSM_ERR_CUDA;
    const int units = fs_units(g.B, g.T), n_tiles = g.P / kS;
    FsParams p{g.B, g.T, g.P, n_tiles, g.H / BK, kRagged ? fs_tiles(g.T) : (g.T >= BM ? g.T / BM : 1),
               kRagged || g.T >= BM ? g.T : BM, units, kRagged || g.T >= BM ? BM / kFsRows : g.T / kFsRows, n_tiles * ((units + 1) / 2),
               g.Abar, (const float4*)g.Apow, g.done, g.x0, g.xT, (uint32_t*)g.x_planes, (size_t)M * g.P, g.hdr};
    if (kTPair) {   // a chain is one sequence; each CTA has every other tile
        p.tblocks = (g.T + 2 * BM - 1) / (2 * BM);
        p.nchains = n_tiles * g.B;
    }
    count_launch();
    auto kern = gemm_scan_fwd_kernel<kS, kTPair, kRagged>;
    if (!set_smem(kern, Cfg::kSmemBytes)) return SSM_ERR_CUDA;
    const int pairs = resident_pairs(reinterpret_cast<const void*>(kern), Cfg::kSmemBytes, Cfg::kThreads);
    if (pairs <= 0) return SSM_ERR_CUDA;
    launch_dep(kern, 2 * min(pairs, p.nchains), Cfg::kThreads, Cfg::kSmemBytes, st, ma, mw, mx, p);
    return SSM_OK;
}

template <bool kRagged>
static int launch_gemm_scan_fwd_r(const GemmScanFwd& g, const FusedMode& m, cudaStream_t st) {
    if (m.group == 64)
        return m.time_pairs ? launch_gemm_scan_fwd_s<64, true, kRagged>(g, st) : launch_gemm_scan_fwd_s<64, false, kRagged>(g, st);
    if (m.group == 32) return launch_gemm_scan_fwd_s<32, false, kRagged>(g, st);
    return SSM_ERR_SHAPE;
}
int launch_gemm_scan_fwd(const GemmScanFwd& g, cudaStream_t st) {
    const FusedMode m = fused_mode(g.B, g.T, g.H, g.P);
    return fs_ragged(g.T) ? launch_gemm_scan_fwd_r<true>(g, m, st) : launch_gemm_scan_fwd_r<false>(g, m, st);
}

// Rows of gA_part that launch_gemm_scan_bwd writes: one per chain of a state group (two per sequence where both
// CTAs of a pair share a sequence).
int tc_gemm_scan_bwd_part_rows(int B, int T, int H, int P) {
    return fused_mode(B, T, H, P).time_pairs ? 2 * B : fs_units(B, T);
}

template <int kS, bool kTPair, bool kRagged>
static int launch_gemm_scan_bwd_s(const GemmScanBwd& g, cudaStream_t st) {
    using namespace tc;
    using Cfg = FsCfg<kS>;
    const int M = g.B * g.T;
    CUtensorMap ma, mw, mx, ms;
    if (!make_map(&ma, g.gy, (uint64_t)M, (uint64_t)g.H, BK, BM)) return SSM_ERR_CUDA;
    if (!make_map(&mw, g.Wsplit, (uint64_t)4 * g.P, (uint64_t)g.H, BK, Cfg::kWRows)) return SSM_ERR_CUDA;
    if (!make_plane_map(&mx, g.x_planes, M, g.P, kS)) return SSM_ERR_CUDA;
    if (!(kRagged ? make_plane_map4(&ms, g.s_planes, g.B, g.T, g.P, kS) : make_plane_map(&ms, g.s_planes, M, g.P, kS))) return SSM_ERR_CUDA;
    const int units = fs_units(g.B, g.T), n_tiles = g.P / kS;
    FbParams p{g.B, g.T, g.P, n_tiles, g.H / BK, kRagged ? fs_tiles(g.T) : (g.T >= BM ? g.T / BM : 1),
               kRagged || g.T >= BM ? g.T : BM, units, kRagged || g.T >= BM ? BM / kFsRows : g.T / kFsRows, n_tiles * ((units + 1) / 2),
               g.Abar, (const float4*)g.Apow, g.done, g.x0, g.gxT, g.gA_part, g.gx0, g.hdr};
    if (kTPair) {
        p.tblocks = (g.T + 2 * BM - 1) / (2 * BM);
        p.nchains = n_tiles * g.B;
    }
    count_launch();
    auto kern = gemm_scan_bwd_kernel<kS, kTPair, kRagged>;
    if (!set_smem(kern, Cfg::kSmemBytes)) return SSM_ERR_CUDA;
    const int pairs = resident_pairs(reinterpret_cast<const void*>(kern), Cfg::kSmemBytes, Cfg::kThreads);
    if (pairs <= 0) return SSM_ERR_CUDA;
    launch_dep(kern, 2 * min(pairs, p.nchains), Cfg::kThreads, Cfg::kSmemBytes, st, ma, mw, mx, ms, p);
    return SSM_OK;
}

template <bool kRagged>
static int launch_gemm_scan_bwd_r(const GemmScanBwd& g, const FusedMode& m, cudaStream_t st) {
    if (m.group == 64)
        return m.time_pairs ? launch_gemm_scan_bwd_s<64, true, kRagged>(g, st) : launch_gemm_scan_bwd_s<64, false, kRagged>(g, st);
    if (m.group == 32) return launch_gemm_scan_bwd_s<32, false, kRagged>(g, st);
    return SSM_ERR_SHAPE;
}
int launch_gemm_scan_bwd(const GemmScanBwd& g, cudaStream_t st) {
    const FusedMode m = fused_mode(g.B, g.T, g.H, g.P);
    return fs_ragged(g.T) ? launch_gemm_scan_bwd_r<true>(g, m, st) : launch_gemm_scan_bwd_r<false>(g, m, st);
}

bool tc_nt_supported(int I, int J) { return (I % tc::BM) == 0 && (J % (tc::BN / 2)) == 0; }

// Both products of a pair in one launch where the slices then still are short (a launch costs about 5 us of ramp and
// drain that the next one hides only partly; 0.35 us per k-block and CTA), else one launch each with twice the slices.
struct NtPlan {
    bool pairs, together;
    int splits;
};
static NtPlan nt_plan(int K, int I, int J) {
    const bool pairs = I % (2 * tc::BM) == 0;
    const int tiles = (pairs ? I / (2 * tc::BM) : I / tc::BM) * (J / (tc::BN / 2));
    const int slots = pairs ? tc::sm_count() / 2 : tc::sm_count();
    const int blocks = (K + tc::BK - 1) / tc::BK;
    auto clamp = [&](int s) { return std::max(1, std::min(std::min(s, blocks), 64)); };
    const int one = clamp(slots / tiles), two = clamp(slots / (2 * tiles));
    auto rounds = [&](int units) { return (units + slots - 1) / slots; };
    const double t_one = 2.0 * (rounds(tiles * one) * ((blocks + one - 1) / one) * 0.35 + 5.0);
    const double t_two = rounds(2 * tiles * two) * ((blocks + two - 1) / two) * 0.35 + 7.0;
    return t_two < t_one ? NtPlan{pairs, true, two} : NtPlan{pairs, false, one};
}
int tc_nt_splits(int K, int I, int J) { return nt_plan(K, I, J).splits; }

int launch_gemm_tc_nt2(int K, int I, int J, int splits, const GemmTcNT& g0, const GemmTcNT& g1, WsHeader* hdr, cudaStream_t st) {
    using namespace tc;
    const NtPlan plan = nt_plan(K, I, J);
    if (splits != plan.splits) return SSM_ERR_SHAPE;
    NtMaps maps;
    const GemmTcNT* g[2] = {&g0, &g1};
    for (int z = 0; z < 2; ++z) {
        if (!make_map(&maps.a[z], g[z]->A, (uint64_t)K, (uint64_t)I, 64, BK, false, CU_TENSOR_MAP_SWIZZLE_128B, (uint64_t)g[z]->lda))
            return SSM_ERR_CUDA;
        if (!make_map(&maps.hi[z], g[z]->Bm_hi, (uint64_t)K, (uint64_t)J, 64, BK)) return SSM_ERR_CUDA;
        if (!make_map(&maps.lo[z], g[z]->Bm_lo, (uint64_t)K, (uint64_t)J, 64, BK)) return SSM_ERR_CUDA;
    }
    const int blocks = (K + BK - 1) / BK, j_tiles = J / (BN / 2);
    NtParams p{K, J, I, j_tiles, (blocks + splits - 1) / splits, 0, {g0.part, g1.part}, hdr};
    for (; p.first < 2; p.first += plan.together ? 2 : 1) {
        const unsigned nz = plan.together ? 2 : 1;
        count_launch();
        auto run = [&](auto kern, unsigned ctas, size_t smem, int threads) {
            return set_smem(kern, smem) && launch_dep(kern, dim3(ctas * j_tiles, splits, nz), threads, smem, st, maps, p);
        };
        const unsigned pairs = 2 * (I / (2 * BM)), singles = I / BM;   // 256 x 256 tiles on CTA pairs, or 128 x 256
        bool ok;
        if (p.blocks_per_split > kNtSegment)
            ok = plan.pairs ? run(gemm_tc_nt_pair_kernel<true>, pairs, kNtPairSmemBytes, nt_threads(true)) : run(gemm_tc_nt_kernel<true>, singles, kNtSmemBytes, nt_threads(true));
        else
            ok = plan.pairs ? run(gemm_tc_nt_pair_kernel<false>, pairs, kNtPairSmemBytes, nt_threads(false)) : run(gemm_tc_nt_kernel<false>, singles, kNtSmemBytes, nt_threads(false));
        if (!ok) return SSM_ERR_CUDA;
    }
    return SSM_OK;
}

}  // namespace ssm
