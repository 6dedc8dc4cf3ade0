// Projections of fp32 layers with many tiles: out[m, n] = sum_k A[m, k] W[n, k] as six products of the three bf16 planes
// of both operands, with the layer's epilogue (fp32 store, or out = acc + diag * skip (+ add) and the column sums of
// skip * dot).
//
// Persistent, CTA pairs on 256 x 128 tiles: a CTA holds its 128 rows of A and 64 rows of W and brings in every plane of
// 32 columns of K once (36 KB, five stages), one thread of the pair issues the 12 MMAs of a stage, and eight warps of
// each CTA run the epilogue of its half of one tile out of one half of tensor memory while the MMAs of the next fill the
// other.  The one-tile-per-CTA kernel of gemm_tc_small.cu, which
// splits an fp32 operand itself and is better for few tiles, alternates on large problems between waiting for memory
// and multiplying, and splits every row once per column tile: 64000 x 512 x 512 with the skip term and the column sums
// 329 us there, 149 us here and 52 us for the planes (they serve the weight gradients as well).
// A 128 x 128 x 16 MMA of one CTA takes 97 cycles, of which 64 are the tensor core's (the operands come from shared
// memory: 8 KB), a 256 x 128 x 16 MMA of a pair 70 for twice the work.  64000 x 512 x 512 in a layer's passes,
// one CTA per 128 x 128 tile / pairs: 175 / 136 us, with the skip term and the column sums 189 / 149.
// hi hi has an accumulator of its own (see gemm_tc_small.cu).
// The tensor core truncates its accumulator at every addition.  A tile of more than kPlSegment stages of K is multiplied in
// that many segments of equal length, which take the two halves of tensor memory in turn like tiles of their own: the
// epilogue warps add a finished segment to their registers while the next one runs.  40000 rows, K = 384, errors of a layer's y and
// du against float64: 1.8e-7 and 1.2e-7 in one chain, 1.2e-7 and 0.7e-7 in two (CUDA cores: 1.6e-7 and 0.9e-7).  It costs 2 % of
// 64000 x 512 x 512, 4 to 9 % with the skip term and the column sums, whose epilogue then holds only one half of
// tensor memory's lead (194 to 198, 205 to 213, 214 to 233 us).  A short last segment: the same time, 1.27e-7 and 0.77e-7 off.
// Emptying the last segment before the epilogue's operands are requested (registers): du 248 us.
#include <algorithm>

#include "kernels.h"
#include "small_tile.cuh"

namespace ssm {
namespace tc {

constexpr int kPlBN = 128;
constexpr int kPlBK = 32;      // K extent of an operand stage: 64-byte rows
constexpr int kPlStages = 5;
constexpr int kPlATile = BM * kPlBK * 2, kPlWTile = kPlBN / 2 * kPlBK * 2;   // one plane, of a CTA
constexpr int kPlStageBytes = 3 * kPlATile + 3 * kPlWTile;
constexpr int kPlSegment = 8;  // stages of a segment at most: 16 additions per accumulator
constexpr int kPlEpiWarps = 8;
constexpr int kPlThreads = 64 + 32 * kPlEpiWarps;
constexpr int kPlSlabBytes = 32 * 32 * 4;
constexpr size_t kPlSmem = (size_t)kPlStages * kPlStageBytes + kPlEpiWarps * kPlSlabBytes + 1024;

struct PlanesArgs {
    int M, N, K, n_tiles, tiles, k_blocks;
    int segs, seg_blocks;      // segments of a tile, stages of a segment (the last one may have fewer)
    int planes_a, n_prod;      // planes of A (3, or 1: a bf16 operand), products of the schedule (see GemmTcTN)
    uint32_t pa, pw;
    void* out;
    const float* diag;
    const void *skip, *dot;
    const float* add;
    float* dot_part;           // four rows per 128 rows of A
    bool out_bf16, skip_bf16, dot_bf16;
    WsHeader* hdr;
};

struct PlanesBars {
    uint64_t full[kPlStages], empty[kPlStages], done[2], free[2];
    uint32_t tmem;
    int abort_flag;
};

template <bool kDiag, bool kSegs>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPlThreads, 1)
gemm_tc_planes_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmW, const __grid_constant__ PlanesArgs p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ PlanesBars bars;
    uint8_t* stages = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    volatile int* abort_flag = &bars.abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rank = (int)cluster_ctarank();
    const int pair = (int)blockIdx.x >> 1, npairs = (int)gridDim.x >> 1;
    if (threadIdx.x == 0) {
        for (int i = 0; i < kPlStages; ++i) {
            mbar_init(smem_u32(&bars.full[i]), 1);
            mbar_init(smem_u32(&bars.empty[i]), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&bars.done[i]), 1);
            mbar_init(smem_u32(&bars.free[i]), 2 * kPlEpiWarps);
        }
        bars.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        prefetch_tmap(&tmA);
        prefetch_tmap(&tmW);
    }
    __syncwarp();
    if (warp == 1) tmem_alloc_pair(smem_u32(&bars.tmem), 512);
    tc_fence_before();
    cluster_sync_all();
    tc_fence_after();
    const uint32_t tmem_base = bars.tmem;
    grid_dep_wait();
    grid_dep_launch();

    if (warp == 0) {
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int tile = pair; tile < p.tiles && ok; tile += npairs) {
            const int m0 = (2 * (tile / p.n_tiles) + rank) * BM, n0 = (tile % p.n_tiles) * kPlBN + rank * (kPlBN / 2);
            for (int kb = 0; kb < p.k_blocks; ++kb) {
                if (!(ok = mbar_wait_warp(smem_u32(&bars.empty[stage]), phase ^ 1u, abort_flag))) break;
                const uint32_t full = map_to_cta(smem_u32(&bars.full[stage]), 0);   // the leader counts both CTAs' loads
                const uint32_t dst = smem_u32(stages) + (uint32_t)stage * kPlStageBytes;
                if (elect_one()) {
                    if (rank == 0) mbar_expect_tx(smem_u32(&bars.full[stage]), 2u * (uint32_t)(p.planes_a * kPlATile + 3 * kPlWTile));
                    for (int q = 0; q < p.planes_a; ++q) tma_load_2d_pair(dst + q * kPlATile, &tmA, full, q * p.K + kb * kPlBK, m0);
#pragma unroll
                    for (int q = 0; q < 3; ++q)
                        tma_load_2d_pair(dst + 3 * kPlATile + q * kPlWTile, &tmW, full, q * p.K + kb * kPlBK, n0);
                }
                if (++stage == kPlStages) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
        }
    } else if (warp == 1) {
        if (rank == 0) {
            constexpr uint32_t idesc = instr_desc(2 * BM, kPlBN, 0, 0);
            const int n_prod = p.n_prod;
            const uint32_t pa = p.pa, pw = p.pw;
            int stage = 0, n = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int tile = pair; tile < p.tiles && ok; tile += npairs)
            for (int seg = 0; seg < (kSegs ? p.segs : 1) && ok; ++seg, ++n) {   // n: segments so far
                const int buf = n & 1, kb_first = kSegs ? seg * p.seg_blocks : 0, kb_end = kSegs ? min(p.k_blocks, kb_first + p.seg_blocks) : p.k_blocks;
                if (n >= 2) {   // the epilogue has taken segment n - 2 out of this half of tensor memory
                    if (!(ok = mbar_wait_warp(smem_u32(&bars.free[buf]), (uint32_t)((n >> 1) - 1) & 1u, abort_flag))) break;
                    tc_fence_after();
                }
                for (int kb = kb_first; kb < kb_end; ++kb) {
                    if (!(ok = mbar_wait_warp(smem_u32(&bars.full[stage]), phase, abort_flag))) break;
                    tc_fence_after();
                    const uint32_t base = smem_u32(stages) + (uint32_t)stage * kPlStageBytes;
                    if (elect_one()) {
                        for (int j = 0; j < n_prod; ++j) {
                            const bool small = j < n_prod - 1;
                            const uint32_t d_tmem = tmem_base + 256u * (uint32_t)buf + (small ? 128u : 0u);
                            const uint64_t ad = smem_desc_kmajor64(base + ((pa >> (4 * j)) & 15u) * kPlATile);
                            const uint64_t wd = smem_desc_kmajor64(base + 3 * kPlATile + ((pw >> (4 * j)) & 15u) * kPlWTile);
#pragma unroll
                            for (int k = 0; k < kPlBK / UK; ++k)
                                umma_bf16_pair(d_tmem, ad + (uint64_t)(2 * k), wd + (uint64_t)(2 * k), idesc,
                                          (uint32_t)!(kb == kb_first && k == 0 && (j == 0 || !small)));
                        }
                        umma_commit_pair(smem_u32(&bars.empty[stage]));
                    }
                    if (++stage == kPlStages) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
                if (ok && elect_one()) umma_commit_pair(smem_u32(&bars.done[buf]));
            }
        }
    } else {
        // A warp drains 32 rows x 64 columns of a tile in slabs of 32 x 32.  A slab is turned round in the warp's 4 KB of
        // shared memory (16-byte chunk j of row r at j ^ (r & 7)), after which a lane holds 4 columns of every fourth
        // row, and 8 lanes move 128 contiguous bytes of a row.
        const int ew = warp - 2, q = warp & 3, half = ew >> 2;
        float4* slab = reinterpret_cast<float4*>(stages + (size_t)kPlStages * kPlStageBytes + (size_t)ew * kPlSlabBytes);
        const int c = lane & 7, rr = lane >> 3;
        const uint32_t leader_free = map_to_cta(smem_u32(&bars.free[0]), 0);
        int n = 0;
        for (int tile = pair; tile < p.tiles; tile += npairs, ++n) {
            const int m_tile = 2 * (tile / p.n_tiles) + rank, m0 = m_tile * BM + 32 * q, n0 = (tile % p.n_tiles) * kPlBN + 64 * half;
            const uint32_t t_warp = tmem_base + ((uint32_t)(q * 32) << 16) + 64u * (uint32_t)half;
            bool ok = true;
            float sum[kSegs ? 64 : 1];   // this lane's row and the warp's 64 columns, all segments but the last
            if (kSegs) {
#pragma unroll
                for (int j = 0; j < (kSegs ? 64 : 1); ++j) sum[j] = 0.f;
#pragma unroll 1
                for (int seg = 0; seg + 1 < p.segs; ++seg, ++n) {
                    const int buf = n & 1;
                    if (!(ok = mbar_wait_warp(smem_u32(&bars.done[buf]), (uint32_t)(n >> 1) & 1u, abort_flag))) break;
                    tc_fence_after();
#pragma unroll
                    for (int c0 = 0; c0 < (kSegs ? 64 : 0); c0 += 16) {
                        uint32_t v[16], w[16];
                        tmem_ld16(t_warp + 256u * (uint32_t)buf + (uint32_t)c0, v);
                        tmem_ld16(t_warp + 256u * (uint32_t)buf + 128u + (uint32_t)c0, w);
                        tmem_ld_wait();
#pragma unroll
                        for (int j = 0; j < 16; ++j) sum[kSegs ? c0 + j : 0] += __uint_as_float(v[j]) + __uint_as_float(w[j]);
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(leader_free + 8u * (uint32_t)buf);
                }
                if (!ok) break;
            }
            const int buf = n & 1;
#pragma unroll(kSegs ? 2 : 1)
            for (int sl = 0; sl < 2; ++sl) {
                const int col = n0 + 32 * sl + 4 * c;
                const bool n_ok = col < p.N;
                Raw4<false> sk[8], dt[8];
                {   // the epilogue's operands come from far
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int m = m0 + rr + 4 * i;
                        if (kDiag && n_ok && m < p.M) {
                            sk[i].load(p.skip, p.skip_bf16, (size_t)m * p.N + col);
                            if (p.dot) dt[i].load(p.dot, p.dot_bf16, (size_t)m * p.N + col);
                        }
                    }
                }
                if (sl == 0) {
                    if (!(ok = mbar_wait_warp(smem_u32(&bars.done[buf]), (uint32_t)(n >> 1) & 1u, abort_flag))) break;
                    tc_fence_after();
                }
                const uint32_t t = t_warp + 256u * (uint32_t)buf + 32u * (uint32_t)sl;
#pragma unroll
                for (int h = 0; h < 2; ++h) {   // 16 columns at a time (registers)
                    uint32_t v[16], w[16];
                    tmem_ld16(t + 16u * (uint32_t)h, v);
                    tmem_ld16(t + 128u + 16u * (uint32_t)h, w);
                    tmem_ld_wait();
                    if (kSegs)
#pragma unroll
                        for (int j = 0; j < 16; ++j) v[j] = __float_as_uint(__uint_as_float(v[j]) + sum[kSegs ? 32 * sl + 16 * h + j : 0]);
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        slab[lane * 8 + ((4 * h + j) ^ (lane & 7))] =
                            make_float4(__uint_as_float(v[4 * j]) + __uint_as_float(w[4 * j]),
                                        __uint_as_float(v[4 * j + 1]) + __uint_as_float(w[4 * j + 1]),
                                        __uint_as_float(v[4 * j + 2]) + __uint_as_float(w[4 * j + 2]),
                                        __uint_as_float(v[4 * j + 3]) + __uint_as_float(w[4 * j + 3]));
                }
                if (sl == 1) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(leader_free + 8u * (uint32_t)buf);
                }
                __syncwarp();
                float4 dg = make_float4(0.f, 0.f, 0.f, 0.f), dsum = dg;
                if (kDiag && n_ok) dg = *reinterpret_cast<const float4*>(p.diag + col);
                {
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int r = rr + 4 * i, m = m0 + r;
                        if (m >= p.M || !n_ok) continue;
                        float4 v = slab[r * 8 + (c ^ (r & 7))];
                        const size_t e = (size_t)m * p.N + col;
                        if (kDiag) {
                            const float4 s4 = sk[i].get(p.skip_bf16);
                            if (p.add) {
                                const float4 a4 = *reinterpret_cast<const float4*>(p.add + e);
                                v.x += a4.x, v.y += a4.y, v.z += a4.z, v.w += a4.w;
                            }
                            v.x = fmaf(dg.x, s4.x, v.x);
                            v.y = fmaf(dg.y, s4.y, v.y);
                            v.z = fmaf(dg.z, s4.z, v.z);
                            v.w = fmaf(dg.w, s4.w, v.w);
                            if (p.dot) {
                                const float4 d4 = dt[i].get(p.dot_bf16);
                                dsum.x = fmaf(s4.x, d4.x, dsum.x);
                                dsum.y = fmaf(s4.y, d4.y, dsum.y);
                                dsum.z = fmaf(s4.z, d4.z, dsum.z);
                                dsum.w = fmaf(s4.w, d4.w, dsum.w);
                            }
                            store4_io(p.out, p.out_bf16, e, v);
                        } else {
                            *reinterpret_cast<float4*>(reinterpret_cast<float*>(p.out) + e) = v;
                        }
                    }
                }
                if (kDiag && p.dot) {   // the warp's 32 rows: one row of partial sums per warp and tile row
#pragma unroll
                    for (int o = 8; o <= 16; o *= 2) {
                        dsum.x += __shfl_xor_sync(0xffffffffu, dsum.x, o);
                        dsum.y += __shfl_xor_sync(0xffffffffu, dsum.y, o);
                        dsum.z += __shfl_xor_sync(0xffffffffu, dsum.z, o);
                        dsum.w += __shfl_xor_sync(0xffffffffu, dsum.w, o);
                    }
                    if (rr == 0 && n_ok && m_tile * BM < p.M)
                        *reinterpret_cast<float4*>(p.dot_part + (size_t)(4 * m_tile + q) * p.N + col) = dsum;
                }
                __syncwarp();   // the slab is free
            }
            if (!ok) break;
        }
    }
    // nobody leaves (or frees tensor memory) while the other CTA may still signal or compute
    tc_fence_before();
    __syncwarp();
    cluster_sync_all();
    tc_fence_after();
    if (warp == 1) tmem_dealloc_pair(tmem_base, 512);
    if (threadIdx.x == 0 && *abort_flag && p.hdr) p.hdr->status = SSM_ERR_TIMEOUT;
}

}  // namespace tc

// Many tiles: from about 100 (us back to back, this kernel with the split of A / the few-tile kernel: 4000 x 256, 64 tiles,
// 10.4 / 10.0, 4000 x 512, 128 tiles, 15.4 / 18.0; with skip term and column sums 13.2 / 11.6 and 18.1 / 22.0).
bool tc_planes_many_tiles(int M, int N_out) {
    return ((M + tc::BM - 1) / tc::BM) * ((N_out + tc::kPlBN - 1) / tc::kPlBN) >= 100;
}

int launch_gemm_tc_planes(const GemmTcTN& g, cudaStream_t st) {
    using namespace tc;
    if (g.a_f32 || g.n_products < 2 || g.n_products > 8 || g.planes_a > 3 || g.planes_w != 3 || g.K % BK != 0 || g.N_out % 32 != 0 || g.gate_out) return SSM_ERR_SHAPE;
    PlanesArgs p{};
    p.M = g.M, p.N = g.N_out, p.K = g.K, p.k_blocks = g.K / kPlBK;
    p.planes_a = g.planes_a, p.n_prod = g.n_products, p.pa = g.prod_a, p.pw = g.prod_w;
    p.segs = (p.k_blocks + kPlSegment - 1) / kPlSegment;
    p.seg_blocks = (p.k_blocks + p.segs - 1) / p.segs;
    p.n_tiles = (g.N_out + kPlBN - 1) / kPlBN;
    const int m_tiles = (g.M + BM - 1) / BM;
    p.tiles = (m_tiles + 1) / 2 * p.n_tiles;
    p.out = g.out, p.diag = g.diag, p.skip = g.skip, p.dot = g.dot, p.add = g.add, p.dot_part = g.dot_part;
    p.out_bf16 = !g.store_f32, p.skip_bf16 = g.skip_bf16, p.dot_bf16 = g.dot_bf16, p.hdr = g.hdr;
    if (g.dot_rows) *g.dot_rows = 4 * m_tiles;
    CUtensorMap ma, mw;
    if (!make_map(&ma, g.A, (uint64_t)g.M, (uint64_t)g.planes_a * g.K, kPlBK, BM, false, CU_TENSOR_MAP_SWIZZLE_64B)) return SSM_ERR_CUDA;
    if (!make_map(&mw, g.W, (uint64_t)g.N_out, 3 * (uint64_t)g.K, kPlBK, kPlBN / 2, false, CU_TENSOR_MAP_SWIZZLE_64B)) return SSM_ERR_CUDA;
    count_launch();
    auto run = [&](auto kern) {
        if (!set_max_dynamic_smem(reinterpret_cast<const void*>(kern), kPlSmem)) return false;
        const int pairs = std::min(p.tiles, resident_pairs(reinterpret_cast<const void*>(kern), kPlSmem, kPlThreads));
        return pairs > 0 && launch_dep(kern, 2 * pairs, kPlThreads, kPlSmem, st, ma, mw, p);
    };
    const bool ok = p.segs > 1 ? (g.diag ? run(gemm_tc_planes_kernel<true, true>) : run(gemm_tc_planes_kernel<false, true>))
                               : (g.diag ? run(gemm_tc_planes_kernel<true, false>) : run(gemm_tc_planes_kernel<false, false>));
    return ok ? SSM_OK : SSM_ERR_CUDA;
}

}  // namespace ssm
