// Weight gradients of fp32 layers: the products of a backward pass (gBbar = s^T u and dC = gy^T conj(x)) as sums of
// products of bf16 planes, both of a layer, or all of a stack's layers, in one launch.
//   part[s, i, j] = sum over the rows m of slice s of A[m, i] B[m, j],  A [K, I], B [K, J] as bf16 planes
// Both operands are contiguous in the output index (MN-major tiles of [64 rows][64 columns]).  One CTA per 128 x 128
// tile, slice of the rows and product: a k-block brings every plane of both operands in once (96 KB) and all six
// products are issued from it; the kernel this replaces loaded a pair of planes per product (288 KB for a tile of
// twice the size) and took one launch per product.  The last product (hi hi) has an accumulator of its own (see
// gemm_tc_small.cu).  The tensor core truncates at every addition, so the error of a sum grows with the length of its
// chain: after kNpSegment k-blocks the epilogue warps take the tile out of tensor memory and add it to their registers
// while the next segment runs in the other half of tensor memory (64000 rows: dB 1.6e-5 off without).
// kPair: a CTA pair takes a tile of 256 x 128, each CTA 128 columns of A and 64 of B (72 KB a k-block).  A 128 x 128 x 16
// MMA takes 97 cycles because its operands come out of shared memory at 8 KB per 64 tensor-core cycles, a pair's 256 x
// 128 x 16 takes 70: both products of 64000 x 512 x 512 350 / 286 us.  Where I leaves half of a pair's last tile empty and there
// are few tiles (I = 128, 384), one CTA per tile is at least as fast.
#include <algorithm>

#include "kernels.h"
#include "tcgen05.cuh"

namespace ssm {
namespace tc {

constexpr int kNpTile = 128 * BK * 2;    // one plane of an operand tile of a k-block
constexpr int kNpMaxStages = 4;
constexpr int kNpSegment = 4;            // k-blocks per segment: 256 rows, 16 chained additions
constexpr int kNpThreads = 64 + 256;     // producer, MMA, eight epilogue warps
constexpr size_t kNpSmemMax = 220 * 1024;

struct NtPlanesArgs {
    int K, I, J, j_tiles, blocks_per_split;
    int stages, stage_bytes;
    WsHeader* hdr;
    struct Product {
        int planes_a, planes_b, n_prod;
        uint32_t pa, pb;
        float* part;
    } product[2 * kLayerBatch];
};
template <int kN>
struct NtPlanesMaps {   // (a single layer does not carry a batch's 8 KB of tensor maps through its launch)
    CUtensorMap a[kN], b[kN];
};

struct NtPlanesBars {
    uint64_t full[kNpMaxStages], empty[kNpMaxStages], done[2], free[2];
    uint32_t tmem;
    int abort_flag;
};

template <int kN, bool kPair>
__global__ void __launch_bounds__(kNpThreads, 1)
gemm_tc_nt_planes_kernel(const __grid_constant__ NtPlanesMaps<kN> maps, const __grid_constant__ NtPlanesArgs p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ NtPlanesBars bars;
    uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    volatile int* abort_flag = &bars.abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const NtPlanesArgs::Product& pr = p.product[blockIdx.z];
    const CUtensorMap *ta = &maps.a[blockIdx.z], *tb = &maps.b[blockIdx.z];
    constexpr int kBTile = kPair ? kNpTile / 2 : kNpTile;   // one plane of this CTA's columns of B
    const int rank = kPair ? (int)cluster_ctarank() : 0, tile = kPair ? (int)blockIdx.x >> 1 : (int)blockIdx.x;
    const int i0 = (tile / p.j_tiles) * (kPair ? 256 : 128) + 128 * rank, j0 = (tile % p.j_tiles) * 128;
    const int total = (p.K + BK - 1) / BK;
    const int kb0 = (int)blockIdx.y * p.blocks_per_split, kb1 = min(total, kb0 + p.blocks_per_split);
    const int planes_a = pr.planes_a, planes_b = pr.planes_b;
    if (threadIdx.x == 0) {
        for (int i = 0; i < p.stages; ++i) {
            mbar_init(smem_u32(&bars.full[i]), 1);
            mbar_init(smem_u32(&bars.empty[i]), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&bars.done[i]), 1);
            mbar_init(smem_u32(&bars.free[i]), kPair ? 16 : 8);
        }
        bars.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        prefetch_tmap(ta);
        prefetch_tmap(tb);
    }
    __syncwarp();
    if (warp == 1) {
        if (kPair) tmem_alloc_pair(smem_u32(&bars.tmem), 512);
        else tmem_alloc(smem_u32(&bars.tmem), 512);
    }
    tc_fence_before();
    if (kPair) cluster_sync_all();   // the other CTA's barriers are set up
    else __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = bars.tmem;
    grid_dep_wait();
    grid_dep_launch();

    if (warp == 0) {
        const uint32_t bytes = (uint32_t)planes_a * kNpTile + (uint32_t)planes_b * kBTile;
        int stage = 0;
        uint32_t phase = 0;
        for (int kb = kb0; kb < kb1; ++kb) {
            if (!mbar_wait_warp(smem_u32(&bars.empty[stage]), phase ^ 1u, abort_flag)) break;
            // (a pair counts both CTAs' loads on the barrier of CTA 0, which issues the MMAs)
            const uint32_t full = kPair ? map_to_cta(smem_u32(&bars.full[stage]), 0) : smem_u32(&bars.full[stage]);
            uint32_t dst = smem_u32(tiles) + (uint32_t)stage * (uint32_t)p.stage_bytes;
            if (elect_one()) {
                if (rank == 0) mbar_expect_tx(smem_u32(&bars.full[stage]), kPair ? 2 * bytes : bytes);
                auto load = [&](uint32_t to, const CUtensorMap* map, int c0) {
                    if (kPair) tma_load_2d_pair(to, map, full, c0, kb * BK);
                    else tma_load_2d(to, map, full, c0, kb * BK);
                };
                for (int q = 0; q < planes_a; ++q, dst += kNpTile) {
                    load(dst, ta, q * p.I + i0);
                    load(dst + kNpTile / 2, ta, q * p.I + i0 + 64);
                }
                for (int q = 0; q < planes_b; ++q, dst += kBTile) {
                    load(dst, tb, q * p.J + j0 + 64 * rank);
                    if (!kPair) load(dst + kNpTile / 2, tb, q * p.J + j0 + 64);
                }
            }
            if (++stage == p.stages) {
                stage = 0;
                phase ^= 1u;
            }
        }
    } else if (warp == 1) {
        if (kb0 < kb1 && rank == 0) {
            constexpr uint32_t idesc = instr_desc(kPair ? 256 : 128, 128, 1, 1);
            const int n_prod = pr.n_prod;
            const uint32_t pa = pr.pa, pb = pr.pb;
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int kb = kb0; kb < kb1; ++kb) {
                const int seg = (kb - kb0) / kNpSegment, buf = seg & 1;
                const bool seg_first = (kb - kb0) % kNpSegment == 0;
                if (seg_first && seg >= 2) {   // the epilogue has taken segment seg - 2 out of this half of tensor memory
                    if (!(ok = mbar_wait_warp(smem_u32(&bars.free[buf]), (uint32_t)((seg >> 1) - 1) & 1u, abort_flag))) break;
                    tc_fence_after();
                }
                if (!(ok = mbar_wait_warp(smem_u32(&bars.full[stage]), phase, abort_flag))) break;
                tc_fence_after();
                const uint32_t base = smem_u32(tiles) + (uint32_t)stage * (uint32_t)p.stage_bytes;
                if (elect_one()) {
                    for (int j = 0; j < n_prod; ++j) {
                        const bool small = j < n_prod - 1;
                        const uint32_t d_tmem = tmem_base + 256u * (uint32_t)buf + (small ? 128u : 0u);
                        const bool first = seg_first && (j == 0 || !small);
                        const uint64_t ad = smem_desc_mnmajor(base + ((pa >> (4 * j)) & 15u) * kNpTile);
                        const uint64_t bd = smem_desc_mnmajor(base + (uint32_t)planes_a * kNpTile + ((pb >> (4 * j)) & 15u) * kBTile);
#pragma unroll
                        for (int k = 0; k < BK / UK; ++k) {   // 16 rows of 128 bytes further: +128 in the address field
                            if (kPair) umma_bf16_pair(d_tmem, ad + (uint64_t)(128 * k), bd + (uint64_t)(128 * k), idesc, (uint32_t)!(first && k == 0));
                            else umma_bf16(d_tmem, ad + (uint64_t)(128 * k), bd + (uint64_t)(128 * k), idesc, (uint32_t)!(first && k == 0));
                        }
                    }
                    auto commit = [&](uint64_t* bar) {
                        if (kPair) umma_commit_pair(smem_u32(bar));
                        else umma_commit(smem_u32(bar));
                    };
                    commit(&bars.empty[stage]);
                    if (kb + 1 == kb1 || (kb + 1 - kb0) % kNpSegment == 0) commit(&bars.done[buf]);
                }
                if (++stage == p.stages) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
        }
    } else {
        const int q = warp & 3, half = (warp - 2) >> 2;
        const int row = i0 + q * 32 + lane;
        float* dst = pr.part + ((size_t)blockIdx.y * p.I + row) * p.J + j0 + 64 * half;
        const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16) + 64u * (uint32_t)half;
        float sum[64];
#pragma unroll
        for (int j = 0; j < 64; ++j) sum[j] = 0.f;
        const int segs = (max(0, kb1 - kb0) + kNpSegment - 1) / kNpSegment;
        bool ok = true;
        for (int seg = 0; seg < segs; ++seg) {
            const int buf = seg & 1;
            if (!(ok = mbar_wait(smem_u32(&bars.done[buf]), (uint32_t)(seg >> 1) & 1u, abort_flag))) break;
            tc_fence_after();
#pragma unroll
            for (int c = 0; c < 64; c += 32) {
                uint32_t v[32], w[32];
                tmem_ld32(t_row + 256u * (uint32_t)buf + (uint32_t)c, v);
                tmem_ld32(t_row + 256u * (uint32_t)buf + 128u + (uint32_t)c, w);
                tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 32; ++j) sum[c + j] += __uint_as_float(v[j]) + __uint_as_float(w[j]);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if (kPair) mbar_arrive_cluster(map_to_cta(smem_u32(&bars.free[buf]), 0));
                else mbar_arrive(smem_u32(&bars.free[buf]));
            }
        }
        if (ok && row < p.I)
#pragma unroll
            for (int j = 0; j < 16; ++j)
                *reinterpret_cast<float4*>(dst + 4 * j) = make_float4(sum[4 * j], sum[4 * j + 1], sum[4 * j + 2], sum[4 * j + 3]);
    }
    // nobody leaves (or frees tensor memory) while the other CTA may still signal or compute
    tc_fence_before();
    __syncwarp();
    if (kPair) cluster_sync_all();
    else __syncthreads();
    tc_fence_after();
    if (warp == 1) {
        if (kPair) tmem_dealloc_pair(tmem_base, 512);
        else tmem_dealloc(tmem_base, 512);
    }
    if (threadIdx.x == 0 && *abort_flag && p.hdr) p.hdr->status = SSM_ERR_TIMEOUT;
}

}  // namespace tc

// Pairs: where I fills their tiles, and a slice is long enough to pay for the pair's set-up (1024 rows of 256 x 256, one
// k-block per slice: a pass of that layer takes 64.1 us with single CTAs, 64.9 with pairs; stack of four layers of
// 1024 rows, 512 x 512, 16 k-blocks per slice: 338.5 and 335.0).
static bool nt_planes_pairs(int I, int blocks_per_slice) { return blocks_per_slice >= 4 && (I % 256 == 0 || I >= 640); }

// Slices of the rows: the shortest estimated time, rounds of CTAs (pairs: on all but the few SMs that clusters of two cannot
// use) times the k-blocks of a slice and what a CTA costs besides, about six k-blocks.  Up to 4096 rows that is one round;
// with 16 pair tiles of 64000 rows 4 slices would leave 8 of 72 pairs without work, 9 take two full rounds: a pass
// of the 64 x 1000 layer (512, 256) 1408 / 1395 us.
int tc_nt_planes_splits(int K, int I, int J, int n_products) {
    const int blocks = (K + tc::BK - 1) / tc::BK, most = std::min(blocks, 64);
    auto slices = [&](int i_tiles, int slots) {
        const int units = std::max(n_products * i_tiles * (J / 128), 1);
        int best = 1;
        long best_t = 0;
        for (int s = 1; s <= most && (s == 1 || (long)units * s <= 3L * slots); ++s) {
            const long t = (long)((units * s + slots - 1) / slots) * ((blocks + s - 1) / s + 6);
            if (s == 1 || t < best_t) best = s, best_t = t;
        }
        return best;
    };
    const int single = slices(I / 128, device_sm_count());
    return nt_planes_pairs(I, blocks / single) ? slices((I + 255) / 256, (device_sm_count() - 4) / 2) : single;
}

template <int kN, bool kPair>
static int launch_nt_planes(int K, int I, int J, int splits, int n, const GemmTcNtPlanes* products, WsHeader* hdr, cudaStream_t st) {
    using namespace tc;
    auto kern = gemm_tc_nt_planes_kernel<kN, kPair>;
    if (!set_max_dynamic_smem(reinterpret_cast<const void*>(kern), kNpSmemMax)) return SSM_ERR_CUDA;
    const int blocks = (K + BK - 1) / BK;
    NtPlanesArgs p{};
    NtPlanesMaps<kN> maps{};
    p.K = K, p.I = I, p.J = J, p.j_tiles = J / 128, p.hdr = hdr;
    p.blocks_per_split = (blocks + splits - 1) / splits;
    int stage_bytes = 0;
    for (int z = 0; z < n; ++z) {
        const GemmTcNtPlanes& q = products[z];
        if (q.n_products < 2 || q.n_products > 8) return SSM_ERR_SHAPE;
        p.product[z] = {q.planes_a, q.planes_b, q.n_products, q.prod_a, q.prod_b, q.part};
        stage_bytes = std::max(stage_bytes, q.planes_a * kNpTile + q.planes_b * (kPair ? kNpTile / 2 : kNpTile));
        if (!make_map(&maps.a[z], q.A, (uint64_t)K, (uint64_t)I * q.planes_a, 64, BK)) return SSM_ERR_CUDA;
        if (!make_map(&maps.b[z], q.B, (uint64_t)K, (uint64_t)J * q.planes_b, 64, BK)) return SSM_ERR_CUDA;
    }
    p.stage_bytes = stage_bytes;
    p.stages = std::min<int>(kNpMaxStages, (int)((kNpSmemMax - 1024) / p.stage_bytes));
    if (p.stages < 2) return SSM_ERR_SHAPE;
    count_launch();
    const dim3 grid((unsigned)((kPair ? 2 * ((I + 255) / 256) : I / 128) * p.j_tiles), (unsigned)splits, (unsigned)n);
    return launch_dep_cluster(kern, kPair ? 2u : 1u, grid, kNpThreads, (size_t)p.stages * p.stage_bytes + 1024, st, maps, p) ? SSM_OK : SSM_ERR_CUDA;
}

int launch_gemm_tc_nt_planes(int K, int I, int J, int splits, int n_products, const GemmTcNtPlanes* products, WsHeader* hdr,
                             cudaStream_t st) {
    if (I % 128 != 0 || J % 128 != 0) return SSM_ERR_SHAPE;
    for (int first = 0; first < n_products; first += 2 * kLayerBatch) {
        const int n = std::min(2 * kLayerBatch, n_products - first);
        auto run = [&](auto launch) { return launch(K, I, J, splits, n, products + first, hdr, st); };
        const int rc = nt_planes_pairs(I, (K + tc::BK - 1) / tc::BK / splits) ? (n <= 2 ? run(launch_nt_planes<2, true>) : run(launch_nt_planes<2 * kLayerBatch, true>))
                                          : (n <= 2 ? run(launch_nt_planes<2, false>) : run(launch_nt_planes<2 * kLayerBatch, false>));
        if (rc) return rc;
    }
    return SSM_OK;
}

}  // namespace ssm
