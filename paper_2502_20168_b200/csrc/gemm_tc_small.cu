// Tensor-core projections for problems of few tiles: training batches of a few thousand rows, single steps, and
// the layers of a stack.
//
// The kernels of gemm_tc.cu walk 128 x 256 or 256 x 256 accumulator tiles, which is what a machine full of tiles
// wants; 1024 rows x 512 columns are 16 such tiles, so 132 of 148 SMs idled and the time was the serial chain of
// one tile's k-blocks (15 - 25 us with the six plane products of fp32 operands).  Here
//  * a tile is 128 rows x 64, 128 or 256 columns, and a cluster of 1, 2 or 4 CTAs shares one tile, each taking a
//    part of the contraction; the parts are added through distributed shared memory in the order of the ranks, so
//    results repeat bit for bit and no partial sum goes through memory;
//  * or two CTAs take a tile of 256 rows together (cta_group::2), each with half of the weight tile in its shared
//    memory: a third less to bring in per k-block where there are enough rows (4096 x 1024 x 1024, two products of
//    planes: 17.8 -> 16.1 us back to back);
//  * a k-block brings every plane of both operands into shared memory once and all products of the schedule are
//    issued from it (the other kernels load a pair of planes per product: 12 tiles instead of 6);
//  * an fp32 A operand needs no planes in memory: the warps that later run the epilogue read it, split it into its
//    three bf16 planes and write them to the operand stages themselves;
//  * the accumulator tile is staged in shared memory (over the operand stages, which are free by then) and read
//    back by rows, so that the epilogue's operands and results are plain coalesced accesses in any type.
#include <algorithm>

#include "kernels.h"
#include "small_tile.cuh"

namespace ssm {
namespace tc {

// Epilogue warps: 8, or 16 for tiles of 256 columns, whose CTAs are never shared (a CTA of 18 warps takes about
// 1 us longer to start than one of 10, which small tiles would notice).
__host__ __device__ constexpr int sm_epi_warps(int bn) { return bn == 256 ? 16 : 8; }
__host__ __device__ constexpr int sm_threads(int bn) { return 64 + 32 * sm_epi_warps(bn); }
constexpr int kSmMaxStages = 6;
constexpr size_t kSmSmemMax = 218 * 1024;        // of the 227 KB a CTA can have (the rest: static shared memory)

struct SmallTnArgs {
    int M, N;                  // rows; output columns
    int n_tiles, cluster;      // tiles along N; CTAs per tile
    int k_blocks;              // per product
    int stages, stage_bytes;
    int planes_a, planes_w, n_prod;
    uint32_t prod_a, prod_w;   // product j: plane (prod_a >> 4 j) & 15 of A, (prod_w >> 4 j) & 15 of W
    int a_plane, w_plane_cols, w_plane_rows, w_stacked;   // where the planes lie (w_stacked: hi / lo blocks of 128 rows)
    const float* a_f32;        // A as fp32 [M, K] (planes made here), or NULL: bf16 planes by TMA
    __nv_bfloat16* a_planes;   // or NULL: the planes made here also go to memory (by the CTAs of the first column tile)
    int K;
    // epilogue
    void* out;
    const float* diag;
    const void* skip;
    const void* dot;
    const float* add;
    float* dot_part;
    __nv_bfloat16* gate_out;
    bool out_bf16, skip_bf16, dot_bf16;
    WsHeader* hdr;
};

// Epilogues: fp32 result; out = acc + diag * skip (+ add) with, if asked for, the column sums of skip * dot over the
// rows of this CTA; fp32 result and out2 = skip * sigmoid(acc) in bf16.
enum SmallEpi { kSmStore, kSmDiag, kSmGate };

struct SmallBars {
    uint64_t full[kSmMaxStages], empty[kSmMaxStages], done;
    uint32_t tmem;
    int abort_flag;
};

template <int kBN, int kEpi, bool kSplitA, bool kBf16, bool kPair>
__global__ void __launch_bounds__(sm_threads(kBN), 1)
gemm_tc_tn_small_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmW, SmallTnArgs p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ SmallBars bars;
    uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    constexpr int kSmEpiWarps = sm_epi_warps(kBN);
    constexpr int kWRows = kPair ? kBN / 2 : kBN;   // weight rows this CTA loads
    constexpr int kWTile = kWRows * BK * 2;
    constexpr int kPitch = kBN + 4;   // staging: floats per row; 16 bytes of padding keep both directions free of bank conflicts
    volatile int* abort_flag = &bars.abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int crank = (int)cluster_ctarank(), rank = kPair ? 0 : crank, tile = (int)blockIdx.x / (kPair ? 2 : p.cluster);
    const int m_tile = kPair ? 2 * (tile / p.n_tiles) + crank : tile / p.n_tiles;
    const int m0 = m_tile * BM, n0 = (tile % p.n_tiles) * kBN;
    if (threadIdx.x == 0) {
        for (int i = 0; i < p.stages; ++i) {
            mbar_init(smem_u32(&bars.full[i]), kSplitA ? 1 + kSmEpiWarps : 1);
            mbar_init(smem_u32(&bars.empty[i]), 1);
        }
        mbar_init(smem_u32(&bars.done), 1);
        bars.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();
    // Several products: the last one (hi hi) has an accumulator of its own, the small ones share a second, and the two
    // are added once.  (In one accumulator every small term would be rounded at the magnitude of the sum: measured 2 - 3 x
    // the error on the gradients of small fp32 layers.)
    const uint32_t tmem_cols = p.n_prod > 1 ? 2 * kBN : kBN;
    if (warp == 1) {
        if (kPair) tmem_alloc_pair(smem_u32(&bars.tmem), tmem_cols);
        else tmem_alloc(smem_u32(&bars.tmem), tmem_cols);
    }
    tc_fence_before();
    if (kPair) cluster_sync_all();   // the other CTA's barriers are set up
    else __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = bars.tmem;
    grid_dep_wait();   // the set-up above ran beside the end of the kernel before this one
    grid_dep_launch();
    const int kb0 = p.k_blocks * rank / p.cluster, kb1 = p.k_blocks * (rank + 1) / p.cluster;
    const uint32_t a_bytes = (uint32_t)p.planes_a * kSmATile;

    if (warp == 0) {
        if (elect_one()) {
            if (!kSplitA) prefetch_tmap(&tmA);
            prefetch_tmap(&tmW);
        }
        const uint32_t bytes = (uint32_t)p.planes_w * kWTile + (kSplitA ? 0u : a_bytes);
        const int wn = n0 + (kPair ? crank * kWRows : 0), wrow = p.w_stacked ? (wn / 128) * 256 + wn % 128 : wn;
        int stage = 0;
        uint32_t phase = 0;
        for (int kb = kb0; kb < kb1; ++kb) {
            if (!mbar_wait_warp(smem_u32(&bars.empty[stage]), phase ^ 1u, abort_flag)) break;
            // (a pair counts both CTAs' loads on the barrier of CTA 0, which issues the MMAs)
            const uint32_t full = kPair ? map_to_cta(smem_u32(&bars.full[stage]), 0) : smem_u32(&bars.full[stage]);
            if (elect_one()) {
                const uint32_t dst = smem_u32(tiles) + (uint32_t)stage * (uint32_t)p.stage_bytes;
                if (!kPair || crank == 0) mbar_expect_tx(smem_u32(&bars.full[stage]), kPair ? 2 * bytes : bytes);
                auto load = [&](uint32_t to, const CUtensorMap* map, int c0, int c1) {
                    if (kPair) tma_load_2d_pair(to, map, full, c0, c1);
                    else tma_load_2d(to, map, full, c0, c1);
                };
                if (!kSplitA)
                    for (int a = 0; a < p.planes_a; ++a) load(dst + a * kSmATile, &tmA, a * p.a_plane + kb * BK, m0);
                for (int w = 0; w < p.planes_w; ++w)
                    load(dst + a_bytes + w * kWTile, &tmW, w * p.w_plane_cols + kb * BK, wrow + w * p.w_plane_rows);
            }
            if (++stage == p.stages) {
                stage = 0;
                phase ^= 1u;
            }
        }
    } else if (warp == 1) {
        if (!kPair || crank == 0) {
            constexpr uint32_t idesc = instr_desc(kPair ? 2 * BM : BM, kBN, 0, 0);
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int kb = kb0; kb < kb1; ++kb) {
                if (!(ok = mbar_wait_warp(smem_u32(&bars.full[stage]), phase, abort_flag))) break;
                tc_fence_after();
                const uint32_t base = smem_u32(tiles) + (uint32_t)stage * (uint32_t)p.stage_bytes;
                if (elect_one()) {
                    for (int j = 0; j < p.n_prod; ++j) {
                        const bool small = j < p.n_prod - 1;
                        const uint32_t d_tmem = tmem_base + (small ? (uint32_t)kBN : 0u);
                        const bool first = kb == kb0 && (j == 0 || !small);
                        const uint64_t ad = smem_desc_kmajor(base + ((p.prod_a >> (4 * j)) & 15u) * kSmATile);
                        const uint64_t wd = smem_desc_kmajor(base + a_bytes + ((p.prod_w >> (4 * j)) & 15u) * kWTile);
#pragma unroll
                        for (int k = 0; k < BK / UK; ++k) {
                            if (kPair) umma_bf16_pair(d_tmem, ad + (uint64_t)(2 * k), wd + (uint64_t)(2 * k), idesc, (uint32_t)!(first && k == 0));
                            else umma_bf16(d_tmem, ad + (uint64_t)(2 * k), wd + (uint64_t)(2 * k), idesc, (uint32_t)!(first && k == 0));
                        }
                    }
                    if (kPair) umma_commit_pair(smem_u32(&bars.empty[stage]));
                    else umma_commit(smem_u32(&bars.empty[stage]));
                }
                if (++stage == p.stages) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
            if (ok && elect_one()) {
                if (kPair) umma_commit_pair(smem_u32(&bars.done));
                else umma_commit(smem_u32(&bars.done));
            }
        }
    } else {
        if (kSplitA) {
            const int te = threadIdx.x - 64;
            SplitA<32 * kSmEpiWarps> sp;   // the next k-block's values are on their way while this one is split and stored
            if (kb0 < kb1) sp.fetch(p.a_f32, p.K, p.M, m0, kb0, te);
            int stage = 0;
            uint32_t phase = 0;
            for (int kb = kb0; kb < kb1; ++kb) {
                if (!mbar_wait(smem_u32(&bars.empty[stage]), phase ^ 1u, abort_flag)) break;
                sp.store(tiles + (size_t)stage * p.stage_bytes, p.M, m0, te, n0 == 0 ? p.a_planes : nullptr, p.K, kb);
                if (kb + 1 < kb1) sp.fetch(p.a_f32, p.K, p.M, m0, kb + 1, te);
                fence_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bars.full[stage]));
                if (++stage == p.stages) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
        }
    }

    // Epilogue: CTA `rank` finishes rows [rank, rank + 1) * 128 / cluster of the tile; a thread keeps its 4 columns and
    // takes every kRowGroups-th row, kU rows at a time.
    constexpr int kC4 = kBN / 4, kRowGroups = 32 * kSmEpiWarps / kC4, kU = kBN == 256 && !kBf16 ? 4 : 8;
    const int te = (int)threadIdx.x - 64, c4 = te % kC4, rg = te / kC4;
    const int parts = kPair ? 1 : p.cluster;   // CTAs whose parts of a row are added
    const int rows = BM / parts, row_base = rank * rows;
    const int n = n0 + 4 * c4;
    Raw4<kBf16> sk[kU], dt[kU];
    // the epilogue's operands come from far: the first rows are asked for while the MMAs run
    auto fetch_operands = [&](int r0) {
#pragma unroll
        for (int i = 0; i < kU; ++i) {
            const int r = r0 + i * kRowGroups, m = m0 + row_base + r;
            if (kEpi != kSmStore && r < rows && m < p.M && n < p.N) {
                const size_t e = (size_t)m * p.N + n;
                sk[i].load(p.skip, p.skip_bf16, e);
                if (kEpi == kSmDiag && p.dot) dt[i].load(p.dot, p.dot_bf16, e);
            }
        }
    };
    if (warp >= 2) {
        fetch_operands(rg);
        if (mbar_wait(smem_u32(&bars.done), 0, abort_flag)) {
            // this CTA's part of the tile -> shared memory (every operand stage has been read: the MMAs are done)
            tc_fence_after();
            const int q = warp & 3, grp = (warp - 2) >> 2;   // TMEM lane quarter; every fourth slab of 32 columns
            float* row = reinterpret_cast<float*>(tiles) + (size_t)(q * 32 + lane) * kPitch;
            const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16);
#pragma unroll 1
            for (int c = grp * 32; c < kBN; c += 32 * (kSmEpiWarps / 4)) {
                uint32_t r[32];
                tmem_ld32(t_row + (uint32_t)c, r);
                if (p.n_prod > 1) {
                    uint32_t r2[32];
                    tmem_ld32(t_row + (uint32_t)(kBN + c), r2);
                    tmem_ld_wait();
#pragma unroll
                    for (int j = 0; j < 32; ++j) r[j] = __float_as_uint(__uint_as_float(r[j]) + __uint_as_float(r2[j]));
                } else {
                    tmem_ld_wait();
                }
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    *reinterpret_cast<float4*>(row + c + 4 * j) =
                        make_float4(__uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1]), __uint_as_float(r[4 * j + 2]),
                                    __uint_as_float(r[4 * j + 3]));
            }
            tc_fence_before();
        }
    }
    __syncwarp();
    if (parts > 1) cluster_sync_all();   // the parts of all CTAs of the cluster are in place
    else __syncthreads();
    if (warp >= 2 && !*abort_flag) {
        const bool n_ok = n < p.N;
        float4 dg = make_float4(0.f, 0.f, 0.f, 0.f), dsum = dg;
        if (kEpi == kSmDiag && n_ok) dg = *reinterpret_cast<const float4*>(p.diag + n);
        for (int r0 = rg; r0 < rows; r0 += kU * kRowGroups) {
            if (r0 != rg) fetch_operands(r0);
#pragma unroll
            for (int i0 = 0; i0 < kU; i0 += 4) {
                const int r1 = r0 + i0 * kRowGroups;
                if (r1 >= rows) break;
                const float* own = reinterpret_cast<const float*>(tiles) + (size_t)(row_base + r1) * kPitch + 4 * c4;
                float4 v[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int r = r1 + i * kRowGroups, m = m0 + row_base + r;
                    v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (kEpi == kSmDiag && p.add && r < rows && m < p.M && n_ok)
                        v[i] = *reinterpret_cast<const float4*>(p.add + (size_t)m * p.N + n);
                }
                for (int q = 0; q < parts; ++q) {
                    const uint32_t a = map_to_cta(smem_u32(own), (uint32_t)q);
                    float4 t[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (r1 + i * kRowGroups < rows)
                            t[i] = parts == 1 ? *reinterpret_cast<const float4*>(own + (size_t)i * kRowGroups * kPitch)
                                                  : ld_cluster_f4(a + (uint32_t)i * (kRowGroups * kPitch * 4u));
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (r1 + i * kRowGroups < rows) v[i].x += t[i].x, v[i].y += t[i].y, v[i].z += t[i].z, v[i].w += t[i].w;
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int r = r1 + i * kRowGroups, m = m0 + row_base + r;
                    if (r >= rows || m >= p.M || !n_ok) continue;
                    const size_t e = (size_t)m * p.N + n;
                    if (kEpi == kSmStore) {
                        *reinterpret_cast<float4*>(reinterpret_cast<float*>(p.out) + e) = v[i];
                    } else if (kEpi == kSmDiag) {
                        const float4 s4 = sk[i0 + i].get(p.skip_bf16);
                        v[i].x = fmaf(dg.x, s4.x, v[i].x);
                        v[i].y = fmaf(dg.y, s4.y, v[i].y);
                        v[i].z = fmaf(dg.z, s4.z, v[i].z);
                        v[i].w = fmaf(dg.w, s4.w, v[i].w);
                        store4_io(p.out, p.out_bf16, e, v[i]);
                        if (p.dot) {
                            const float4 d4 = dt[i0 + i].get(p.dot_bf16);
                            dsum.x = fmaf(s4.x, d4.x, dsum.x);
                            dsum.y = fmaf(s4.y, d4.y, dsum.y);
                            dsum.z = fmaf(s4.z, d4.z, dsum.z);
                            dsum.w = fmaf(s4.w, d4.w, dsum.w);
                        }
                    } else {
                        const float4 s4 = sk[i0 + i].get(true);
                        *reinterpret_cast<float4*>(reinterpret_cast<float*>(p.out) + e) = v[i];
                        *reinterpret_cast<uint2*>(p.gate_out + e) =
                            pack4_bf16(make_float4(s4.x * sigmoid_f<__nv_bfloat16>(v[i].x), s4.y * sigmoid_f<__nv_bfloat16>(v[i].y), s4.z * sigmoid_f<__nv_bfloat16>(v[i].z), s4.w * sigmoid_f<__nv_bfloat16>(v[i].w)));
                    }
                }
            }
        }
        if (kEpi == kSmDiag && p.dot) {
            // column sums over this CTA's rows: the row groups added in a fixed order, one row of dot_part per CTA
            __shared__ float4 red[32 * kSmEpiWarps];
            red[te] = dsum;
            asm volatile("bar.sync 1, %0;" ::"n"(32 * kSmEpiWarps) : "memory");
            if (rg == 0 && n_ok) {
                float4 t = red[c4];
#pragma unroll
                for (int g = 1; g < kRowGroups; ++g) {
                    const float4 u = red[g * kC4 + c4];
                    t.x += u.x, t.y += u.y, t.z += u.z, t.w += u.w;
                }
                *reinterpret_cast<float4*>(p.dot_part + (size_t)(m_tile * parts + rank) * p.N + n) = t;
            }
        }
    }
    // nobody leaves (or frees tensor memory) while another CTA may still read its part
    tc_fence_before();
    __syncwarp();
    if (kPair || p.cluster > 1) cluster_sync_all();
    else __syncthreads();
    tc_fence_after();
    if (warp == 1) {
        if (kPair) tmem_dealloc_pair(tmem_base, tmem_cols);
        else tmem_dealloc(tmem_base, tmem_cols);
    }
    if (threadIdx.x == 0 && *abort_flag && p.hdr) p.hdr->status = SSM_ERR_TIMEOUT;
}

// ---------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------
namespace {

struct SmallShape {
    int bn, cluster, stages;
    bool pair;
};

size_t stage_bytes_of(int bn, int planes_a, int planes_w, bool pair) {
    return (size_t)planes_a * kSmATile + (size_t)planes_w * (pair ? bn / 2 : bn) * BK * 2;
}

// Tile width and cluster size, or a CTA pair: the choice with the shortest estimated time.  The estimate for single CTAs and
// clusters is a fit, in microseconds, to timings of all of them on twenty shapes from 16 x 256 x 256 to 4096 x 1024 x 1024,
// back to back (within 10 % of the measured time, and the one it picks within 8 % of the fastest): a wave of CTAs takes a
// fixed part that grows with the tile (start, first loads, epilogue), its k-blocks at 48 bytes of operands per cycle and SM
// (L2), 0.95 us where fp32 operands are split on the way, and the exchange between the CTAs of a cluster.  Pairs go through
// the same formula with their own operand bytes; it was not fitted to them, only checked on whole passes, with pairs / with
// single CTAs and clusters: gate of 4096 x 1024 102.4 / 108.2 us, of 4096 x 512 47.9 / 49.7, layer 64 x 100 (256, 128)
// 55.4 / 57.4, 32 x 128 (512, 256) 63.5 / 63.5, 32 x 128 (1024, 512) 114.6 / 114.2.
SmallShape pick_small(int M, int N, int k_blocks, int planes_a, int planes_w, bool split_a, bool w_stacked) {
    SmallShape best{0, 0, 0, false};
    double best_t = 0.0;
    const int m_tiles = (M + BM - 1) / BM, sms = device_sm_count();
    auto consider = [&](int bn, int c, bool pair) {
        const size_t sb = stage_bytes_of(bn, planes_a, planes_w, pair);
        const int stages = std::min<int>(kSmMaxStages, (int)((kSmSmemMax - 1024) / sb));
        if (stages < 2) return;
        const int ctas = (pair ? (m_tiles + 1) / 2 * 2 : m_tiles * c) * ((N + bn - 1) / bn);
        const int slots = pair || c == 2 ? sms - 4 : (c == 1 ? sms : sms - 16);   // clusters must fit a GPC
        const int waves = (ctas + slots - 1) / slots;
        const double per_kb = std::max((double)sb / 91000.0, split_a ? 0.95 : 0.0);
        const double exchange = c == 1 ? 0.0 : bn * c / 256.0;
        const double t = waves * (4.6 + bn * 0.0115 + exchange + ((k_blocks + c - 1) / c) * per_kb);
        if (best.bn == 0 || t < best_t) {
            best_t = t;
            best = {bn, c, stages, pair};
        }
    };
    for (int bn = 64; bn <= (w_stacked ? 128 : 256); bn *= 2)
        for (int c = 1; c <= 4 && c <= k_blocks; c *= 2) consider(bn, c, false);
    if (!split_a)
        for (int bn = 128; bn <= 256; bn *= 2) consider(bn, 1, true);
    return best;
}

template <int kBN, int kEpi, bool kSplitA, bool kBf16, bool kPair>
int launch_small(const CUtensorMap& ma, const CUtensorMap& mw, const SmallTnArgs& p, int grid, size_t smem, cudaStream_t st) {
    auto kern = gemm_tc_tn_small_kernel<kBN, kEpi, kSplitA, kBf16, kPair>;
    if (!set_max_dynamic_smem(reinterpret_cast<const void*>(kern), kSmSmemMax)) return SSM_ERR_CUDA;
    count_launch();
    return launch_dep_cluster(kern, kPair ? 2u : (unsigned)p.cluster, grid, sm_threads(kBN), smem, st, ma, mw, p) ? SSM_OK : SSM_ERR_CUDA;
}

}  // namespace
}  // namespace tc

int launch_gemm_tc_tn_small(const GemmTcTN& g, cudaStream_t st) {
    using namespace tc;
    const int epi = g.gate_out ? kSmGate : (g.store_f32 && !g.diag ? kSmStore : kSmDiag);
    if (g.K % BK != 0 || g.N_out % 64 != 0 || g.n_products > 8) return SSM_ERR_SHAPE;
    if (epi == kSmDiag && (!g.diag || !g.skip)) return SSM_ERR_SHAPE;
    if (epi == kSmGate && (!g.skip || !g.skip_bf16)) return SSM_ERR_SHAPE;
    SmallTnArgs p{};
    p.M = g.M;
    p.N = g.N_out;
    p.K = g.K;
    p.k_blocks = g.K / BK;
    if (g.split_w) {          // hi / lo blocks of 128 weight rows; lo product first
        p.planes_a = 1, p.planes_w = 2, p.n_prod = 2;
        p.prod_a = 0x00u, p.prod_w = 0x01u;
        p.w_plane_rows = 128, p.w_stacked = 1;
    } else if (g.n_products > 0) {
        p.planes_a = g.planes_a, p.planes_w = g.planes_w, p.n_prod = g.n_products;
        p.prod_a = g.prod_a, p.prod_w = g.prod_w;
        p.w_plane_cols = g.K;
    } else {
        p.planes_a = p.planes_w = p.n_prod = 1;
    }
    p.a_plane = g.K;
    p.a_f32 = g.a_f32 ? reinterpret_cast<const float*>(g.A) : nullptr;
    p.a_planes = reinterpret_cast<__nv_bfloat16*>(g.a_planes_out);
    if (g.a_f32 && p.planes_a != 3) return SSM_ERR_SHAPE;
    p.out = g.out, p.diag = g.diag, p.skip = g.skip, p.dot = g.dot, p.add = g.add;
    p.dot_part = g.dot_part, p.gate_out = reinterpret_cast<__nv_bfloat16*>(g.gate_out);
    p.out_bf16 = !g.store_f32, p.skip_bf16 = g.skip_bf16, p.dot_bf16 = g.dot_bf16;
    p.hdr = g.hdr;
    const SmallShape s = pick_small(g.M, g.N_out, p.k_blocks, p.planes_a, p.planes_w, g.a_f32, p.w_stacked != 0);
    if (s.bn == 0) return SSM_ERR_SHAPE;
    p.cluster = s.cluster;
    p.stages = s.stages;
    p.stage_bytes = (int)stage_bytes_of(s.bn, p.planes_a, p.planes_w, s.pair);
    p.n_tiles = (g.N_out + s.bn - 1) / s.bn;
    const size_t smem = std::max((size_t)p.stages * p.stage_bytes, (size_t)BM * (s.bn + 4) * 4) + 1024;
    const int m_tiles = (g.M + BM - 1) / BM, grid = (s.pair ? (m_tiles + 1) / 2 * 2 : m_tiles * p.cluster) * p.n_tiles;
    if (g.dot_rows) *g.dot_rows = s.pair ? (m_tiles + 1) / 2 * 2 : m_tiles * p.cluster;
    CUtensorMap ma, mw;
    const uint64_t w_rows = (uint64_t)g.N_out * (p.w_stacked ? p.planes_w : 1);
    const uint64_t w_cols = (uint64_t)g.K * (p.w_stacked ? 1 : p.planes_w);
    if (!make_map(&mw, g.W, w_rows, w_cols, BK, (uint32_t)(s.pair ? s.bn / 2 : s.bn))) return SSM_ERR_CUDA;
    ma = mw;   // unused when A is split here
    if (!g.a_f32 && !make_map(&ma, g.A, (uint64_t)g.M, (uint64_t)g.K * p.planes_a, BK, BM)) return SSM_ERR_CUDA;
    const bool io_bf16 = g.skip_bf16 && (!g.dot || g.dot_bf16);
#define SSM_SMALL(EPI, SPLIT, BF)                                                             \
    do {                                                                                      \
        if constexpr (!SPLIT) {   /* (an fp32 operand is split by single CTAs) */                             \
            if (s.pair && s.bn == 128) return launch_small<128, EPI, false, BF, true>(ma, mw, p, grid, smem, st); \
            if (s.pair) return launch_small<256, EPI, false, BF, true>(ma, mw, p, grid, smem, st);                \
        }                                                                                                     \
        if (s.bn == 64) return launch_small<64, EPI, SPLIT, BF, false>(ma, mw, p, grid, smem, st);            \
        if (s.bn == 128) return launch_small<128, EPI, SPLIT, BF, false>(ma, mw, p, grid, smem, st);          \
        return launch_small<256, EPI, SPLIT, BF, false>(ma, mw, p, grid, smem, st);                           \
    } while (0)
    if (epi == kSmGate) SSM_SMALL(kSmGate, false, true);
    if (epi == kSmStore && g.a_f32) SSM_SMALL(kSmStore, true, true);
    if (epi == kSmStore) SSM_SMALL(kSmStore, false, true);
    if (g.a_f32) SSM_SMALL(kSmDiag, true, false);
    if (io_bf16) SSM_SMALL(kSmDiag, false, true);
    return SSM_ERR_SHAPE;   // planes of A with fp32 skip or dot: left to gemm_tc_planes.cu
#undef SSM_SMALL
}

// One partial row of column sums per CTA along M.
int tc_tn_small_max_dot_rows(int M) { return 4 * ((M + tc::BM - 1) / tc::BM); }

}  // namespace ssm
