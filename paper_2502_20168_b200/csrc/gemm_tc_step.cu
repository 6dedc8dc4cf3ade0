// Single-step mode in one kernel: Bu = Bbar u, x_next = keep Abar x_prev + Bu, y = Re(C x_next) + D u for B trajectories.
//
// As three kernels (projection, recurrence, projection) a step of 4096 trajectories at H = 512, P = 256 took 25 us,
// most of it launches, pipeline fills and the trip of Bu and x through memory.  Here a cluster of CTAs owns 128
// trajectories.  In the first phase its CTAs compute tiles of kBN columns of Bu (K = H) and apply the recurrence in
// the epilogue: x_next leaves in fp32, and for bf16 I/O as the bf16 operand of the second phase.  One cluster barrier
// later every CTA computes tiles of kBN columns of y (K = 2P) from the whole rows of x, which are in L2.  The weights
// of the first k-blocks of the second phase are loaded while the first phase's epilogue still runs.
// Bound by operand delivery from L2 (per CTA 384 + 256 KB at that size) and by the latency of the chain
// load - MMA - epilogue - barrier - load - MMA - epilogue.
//
// bf16 I/O: weights of the first phase as hi + lo bf16 (two products), one bf16 product in the second, as in the
// layer.  fp32 I/O: both phases as six products of bf16 planes, the fp32 operand split on its way to shared memory.
// With several products the last one (hi hi) has an accumulator of its own (see gemm_tc_small.cu).
#include <algorithm>

#include "kernels.h"
#include "small_tile.cuh"

namespace ssm {
namespace tc {

constexpr int kStEpiWarps = 8, kStEpiThreads = 32 * kStEpiWarps, kStThreads = 64 + kStEpiThreads;
constexpr int kStMaxStages = 6;
constexpr size_t kStSmemMax = 222 * 1024;

struct StepArgs {
    int M, H, P;
    int cluster;               // CTAs per 128 trajectories
    int n_tiles[2], k_blocks[2];   // tiles of kBN columns, k-blocks of a product, per phase
    int stages, stage_bytes;
    const void* u;             // [M, H] io
    const uint8_t* done;       // [M] or NULL
    const float4* x_prev;      // [M, P / 2] pairs of states
    float4* x_next;
    __nv_bfloat16* x_bf16;     // bf16 I/O: [M, 2P], operand of the second phase
    const float4 *Abar, *Alo;
    const float* D;
    void* y;                   // [M, H] io
    WsHeader* hdr;
};

// Products of a phase: first operand planes, second operand planes, and the schedule (see GemmTcTN).
template <bool kF32, int kPhase> struct StepProducts;
template <int kPhase> struct StepProducts<true, kPhase> {
    static constexpr int planes_a = 3, planes_w = 3, n = 6;
    static constexpr uint32_t a = 0x001102u, w = 0x010120u;
};
template <> struct StepProducts<false, 0> {
    static constexpr int planes_a = 1, planes_w = 2, n = 2;
    static constexpr uint32_t a = 0x00u, w = 0x01u;
};
template <> struct StepProducts<false, 1> {
    static constexpr int planes_a = 1, planes_w = 1, n = 1;
    static constexpr uint32_t a = 0x0u, w = 0x0u;
};

struct StepBars {
    uint64_t full[kStMaxStages], empty[kStMaxStages], done, free;
    uint32_t tmem;
    int abort_flag;   // a wait of the load or MMA warp gave up
    int epi_abort;    // a wait of an epilogue warp did: written before their barrier, read after it, so that they agree
};

struct Ring {   // position in the ring of operand stages
    int stage = 0;
    uint32_t phase = 0;
    __device__ __forceinline__ void next(int stages) {
        if (++stage == stages) {
            stage = 0;
            phase ^= 1u;
        }
    }
};

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// Orders generic-proxy accesses to global memory with the TMA unit's.
__device__ __forceinline__ void fence_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }

template <int kBN, bool kF32>
__global__ void __launch_bounds__(kStThreads, 1)
step_kernel(const __grid_constant__ CUtensorMap tmU, const __grid_constant__ CUtensorMap tmX,
            const __grid_constant__ CUtensorMap tmWb, const __grid_constant__ CUtensorMap tmWc, StepArgs p) {
    using P0 = StepProducts<kF32, 0>;
    using P1 = StepProducts<kF32, 1>;
    extern __shared__ uint8_t smem_raw[];
    __shared__ StepBars bars;
    uint8_t* tiles = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* staging = tiles + (size_t)p.stages * p.stage_bytes;
    constexpr int kWTile = kBN * BK * 2, kPitch = kBN + 4;
    constexpr uint32_t kTmem = 2 * kBN;   // accumulators: hi hi, and the small products
    constexpr uint32_t a_bytes = (kF32 ? 3u : 1u) * kSmATile;
    volatile int* abort_flag = &bars.abort_flag;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)cluster_ctarank(), m0 = ((int)blockIdx.x / p.cluster) * BM;
    if (threadIdx.x == 0) {
        for (int i = 0; i < p.stages; ++i) {
            mbar_init(smem_u32(&bars.full[i]), kF32 ? 1 + kStEpiWarps : 1);
            mbar_init(smem_u32(&bars.empty[i]), 1);
        }
        mbar_init(smem_u32(&bars.done), 1);
        mbar_init(smem_u32(&bars.free), kStEpiWarps);
        bars.abort_flag = bars.epi_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        prefetch_tmap(&tmWb);
        prefetch_tmap(&tmWc);
        if (!kF32) {
            prefetch_tmap(&tmU);
            prefetch_tmap(&tmX);
        }
    }
    __syncwarp();
    if (warp == 1) tmem_alloc(smem_u32(&bars.tmem), kTmem);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = bars.tmem;
    grid_dep_wait();
    grid_dep_launch();

    if (warp == 0) {
        Ring r;
        // W tiles of k-block kb of column tile t
        auto load_w = [&](int ph, int t, int kb, int stage, uint32_t full) {
            const uint32_t dst = smem_u32(tiles) + (uint32_t)stage * (uint32_t)p.stage_bytes + a_bytes;
            const int n0 = t * kBN;
            if (kF32) {   // planes side by side along K
                const CUtensorMap* tm = ph ? &tmWc : &tmWb;
                const int K = ph ? 2 * p.P : p.H;
#pragma unroll
                for (int w = 0; w < 3; ++w) tma_load_2d(dst + w * kWTile, tm, full, w * K + kb * BK, n0);
            } else if (ph == 0) {   // hi / lo blocks of 128 rows
                const int row = (n0 / 128) * 256 + n0 % 128;
                tma_load_2d(dst, &tmWb, full, kb * BK, row);
                tma_load_2d(dst + kWTile, &tmWb, full, kb * BK, row + 128);
            } else {
                tma_load_2d(dst, &tmWc, full, kb * BK, n0);
            }
        };
        auto load_a = [&](int ph, int kb, int stage, uint32_t full) {
            if (!kF32) tma_load_2d(smem_u32(tiles) + (uint32_t)stage * (uint32_t)p.stage_bytes, ph ? &tmX : &tmU, full, kb * BK, m0);
        };
        constexpr uint32_t bytes0 = P0::planes_w * kWTile + (kF32 ? 0u : a_bytes);
        constexpr uint32_t bytes1 = P1::planes_w * kWTile + (kF32 ? 0u : a_bytes);
        bool ok = true;
        for (int t = rank; t < p.n_tiles[0] && ok; t += p.cluster)
            for (int kb = 0; kb < p.k_blocks[0]; ++kb, r.next(p.stages)) {
                if (!(ok = mbar_wait_warp(smem_u32(&bars.empty[r.stage]), r.phase ^ 1u, abort_flag))) break;
                if (elect_one()) {
                    const uint32_t full = smem_u32(&bars.full[r.stage]);
                    mbar_expect_tx(full, bytes0);
                    load_a(0, kb, r.stage, full);
                    load_w(0, t, kb, r.stage, full);
                }
            }
        __syncwarp();
        cluster_arrive();
        // the weights of the first k-blocks of the second phase do not wait for the states
        Ring r1 = r;
        int pre = 0;
        const bool any = rank < p.n_tiles[1];
        if (ok && any)
            for (; pre < p.stages && pre < p.k_blocks[1]; ++pre, r.next(p.stages)) {
                if (!(ok = mbar_wait_warp(smem_u32(&bars.empty[r.stage]), r.phase ^ 1u, abort_flag))) break;
                if (elect_one()) {
                    const uint32_t full = smem_u32(&bars.full[r.stage]);
                    mbar_expect_tx(full, bytes1);
                    load_w(1, rank, pre, r.stage, full);
                }
            }
        __syncwarp();
        cluster_wait();
        if (!kF32 && elect_one()) {
            fence_async_global();
            for (int kb = 0; kb < pre; ++kb, r1.next(p.stages)) load_a(1, kb, r1.stage, smem_u32(&bars.full[r1.stage]));
        }
        for (int t = rank; t < p.n_tiles[1] && ok; t += p.cluster)
            for (int kb = t == rank ? pre : 0; kb < p.k_blocks[1]; ++kb, r.next(p.stages)) {
                if (!(ok = mbar_wait_warp(smem_u32(&bars.empty[r.stage]), r.phase ^ 1u, abort_flag))) break;
                if (elect_one()) {
                    const uint32_t full = smem_u32(&bars.full[r.stage]);
                    mbar_expect_tx(full, bytes1);
                    load_a(1, kb, r.stage, full);
                    load_w(1, t, kb, r.stage, full);
                }
            }
        __syncwarp();
    } else if (warp == 1) {
        Ring r;
        uint32_t free_phase = 0;
        bool ok = true, used = false;
        auto run_phase = [&](int ph, int n_prod, uint32_t pa, uint32_t pw) {
            constexpr uint32_t idesc = instr_desc(BM, kBN, 0, 0);
            for (int t = rank; t < p.n_tiles[ph] && ok; t += p.cluster) {
                if (used) {   // the epilogue has taken the previous tile out of tensor memory
                    if (!(ok = mbar_wait_warp(smem_u32(&bars.free), free_phase, abort_flag))) break;
                    free_phase ^= 1u;
                    tc_fence_after();
                }
                used = true;
                for (int kb = 0; kb < p.k_blocks[ph]; ++kb, r.next(p.stages)) {
                    if (!(ok = mbar_wait_warp(smem_u32(&bars.full[r.stage]), r.phase, abort_flag))) break;
                    tc_fence_after();
                    const uint32_t base = smem_u32(tiles) + (uint32_t)r.stage * (uint32_t)p.stage_bytes;
                    if (elect_one()) {
                        for (int j = 0; j < n_prod; ++j) {
                            const bool small = j < n_prod - 1;
                            const uint32_t d_tmem = tmem_base + (small ? (uint32_t)kBN : 0u);
                            const bool first = kb == 0 && (j == 0 || !small);
                            const uint64_t ad = smem_desc_kmajor(base + ((pa >> (4 * j)) & 15u) * kSmATile);
                            const uint64_t wd = smem_desc_kmajor(base + a_bytes + ((pw >> (4 * j)) & 15u) * kWTile);
#pragma unroll
                            for (int k = 0; k < BK / UK; ++k)
                                umma_bf16(d_tmem, ad + (uint64_t)(2 * k), wd + (uint64_t)(2 * k), idesc, (uint32_t)!(first && k == 0));
                        }
                        umma_commit(smem_u32(&bars.empty[r.stage]));
                    }
                }
                if (ok && elect_one()) umma_commit(smem_u32(&bars.done));
            }
        };
        run_phase(0, P0::n, P0::a, P0::w);
        __syncwarp();
        cluster_arrive();
        cluster_wait();
        run_phase(1, P1::n, P1::a, P1::w);
        __syncwarp();
    } else {
        constexpr int kC4 = kBN / 4, kRowGroups = kStEpiThreads / kC4, kRows = BM / kRowGroups;
        constexpr int kU = kRows < 8 ? kRows : 8;   // rows whose operands are in flight per thread
        const int te = (int)threadIdx.x - 64, c4 = te % kC4, rg = te / kC4;
        Ring r;
        uint32_t done_phase = 0;
        SplitA<kStEpiThreads> sp;
        volatile int* epi_abort = &bars.epi_abort;
        auto epi_sync = [] { asm volatile("bar.sync 1, %0;" ::"n"(kStEpiThreads) : "memory"); };
        auto feed = [&](const float* a, int K, int kbs) {   // fp32: this tile's A operand
            sp.fetch(a, K, p.M, m0, 0, te);
            for (int kb = 0; kb < kbs; ++kb, r.next(p.stages)) {
                if (!mbar_wait_warp(smem_u32(&bars.empty[r.stage]), r.phase ^ 1u, epi_abort)) break;
                sp.store(tiles + (size_t)r.stage * p.stage_bytes, p.M, m0, te);
                if (kb + 1 < kbs) sp.fetch(a, K, p.M, m0, kb + 1, te);
                fence_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bars.full[r.stage]));
            }
        };
        auto drain = [&](bool two) {   // accumulators -> staging rows; false when aborting
            const bool ok = mbar_wait_warp(smem_u32(&bars.done), done_phase, epi_abort);
            done_phase ^= 1u;
            tc_fence_after();
            const int q = warp & 3, grp = (warp - 2) >> 2;
            if (ok) {
                float* row = reinterpret_cast<float*>(staging) + (size_t)(q * 32 + lane) * kPitch;
                const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16);
#pragma unroll 1
                for (int c = grp * 32; c < kBN; c += 64) {
                    uint32_t v[32], w[32];
                    tmem_ld32(t_row + (uint32_t)c, v);
                    if (two) tmem_ld32(t_row + (uint32_t)(kBN + c), w);
                    tmem_ld_wait();
                    if (two)
#pragma unroll
                        for (int j = 0; j < 32; ++j) v[j] = __float_as_uint(__uint_as_float(v[j]) + __uint_as_float(w[j]));
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        *reinterpret_cast<float4*>(row + c + 4 * j) =
                            make_float4(__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]),
                                        __uint_as_float(v[4 * j + 2]), __uint_as_float(v[4 * j + 3]));
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bars.free));
            epi_sync();
            return !*epi_abort;
        };
        const float* own = reinterpret_cast<const float*>(staging) + 4 * c4;

        // ---- first phase: Bu tiles, the recurrence in the epilogue
        const int P2 = p.P / 2;
        for (int t = rank; t < p.n_tiles[0]; t += p.cluster) {
            const int pp = t * (kBN / 4) + c4;   // this thread's pair of states
            const bool n_ok = pp < P2;
            float4 xp[kU], a = make_float4(0.f, 0.f, 0.f, 0.f), al = a;
            bool keep[kU];
            auto fetch = [&](int i0) {
#pragma unroll
                for (int i = 0; i < kU; ++i) {
                    const int m = m0 + rg + (i0 + i) * kRowGroups;
                    keep[i] = false;
                    if (m < p.M && n_ok) {
                        xp[i] = p.x_prev[(size_t)m * P2 + pp];
                        keep[i] = !(p.done && p.done[m] != 0);
                    }
                }
            };
            if (n_ok) {
                a = p.Abar[pp];
                al = p.Alo[pp];
            }
            fetch(0);
            if (kF32) feed(reinterpret_cast<const float*>(p.u), p.H, p.k_blocks[0]);
            if (!drain(true)) break;
#pragma unroll 1
            for (int i0 = 0; i0 < kRows; i0 += kU) {
                if (i0) fetch(i0);
#pragma unroll
                for (int i = 0; i < kU; ++i) {
                    const int row = rg + (i0 + i) * kRowGroups, m = m0 + row;
                    if (m >= p.M || !n_ok) continue;
                    float4 v = *reinterpret_cast<const float4*>(own + (size_t)row * kPitch);
                    if (keep[i]) {   // Abar as an fp32 pair, the small products first
                        v.x = fmaf(a.x, xp[i].x, fmaf(-a.y, xp[i].y, fmaf(al.x, xp[i].x, fmaf(-al.y, xp[i].y, v.x))));
                        v.y = fmaf(a.x, xp[i].y, fmaf(a.y, xp[i].x, fmaf(al.x, xp[i].y, fmaf(al.y, xp[i].x, v.y))));
                        v.z = fmaf(a.z, xp[i].z, fmaf(-a.w, xp[i].w, fmaf(al.z, xp[i].z, fmaf(-al.w, xp[i].w, v.z))));
                        v.w = fmaf(a.z, xp[i].w, fmaf(a.w, xp[i].z, fmaf(al.z, xp[i].w, fmaf(al.w, xp[i].z, v.w))));
                    }
                    p.x_next[(size_t)m * P2 + pp] = v;
                    if (!kF32) *reinterpret_cast<uint2*>(p.x_bf16 + (size_t)m * 2 * p.P + 4 * pp) = pack4_bf16(v);
                }
            }
            epi_sync();   // staging free
        }
        if (!kF32) {   // the other CTAs' TMA units read what was just written
            __threadfence();
            fence_async_global();
        }
        cluster_arrive();
        cluster_wait();

        // ---- second phase: y tiles
        for (int t = rank; t < p.n_tiles[1]; t += p.cluster) {
            const int n = t * kBN + 4 * c4;
            const bool n_ok = n < p.H;
            Raw4<!kF32> sk[kU];
            auto fetch = [&](int i0) {
#pragma unroll
                for (int i = 0; i < kU; ++i) {
                    const int m = m0 + rg + (i0 + i) * kRowGroups;
                    if (m < p.M && n_ok) sk[i].load(p.u, !kF32, (size_t)m * p.H + n);
                }
            };
            fetch(0);
            const float4 dg = n_ok ? *reinterpret_cast<const float4*>(p.D + n) : make_float4(0.f, 0.f, 0.f, 0.f);
            if (kF32) feed(reinterpret_cast<const float*>(p.x_next), 2 * p.P, p.k_blocks[1]);
            if (!drain(P1::n > 1)) break;
#pragma unroll 1
            for (int i0 = 0; i0 < kRows; i0 += kU) {
                if (i0) fetch(i0);
#pragma unroll
                for (int i = 0; i < kU; ++i) {
                    const int row = rg + (i0 + i) * kRowGroups, m = m0 + row;
                    if (m >= p.M || !n_ok) continue;
                    float4 v = *reinterpret_cast<const float4*>(own + (size_t)row * kPitch);
                    const float4 s4 = sk[i].get(!kF32);
                    v.x = fmaf(dg.x, s4.x, v.x);
                    v.y = fmaf(dg.y, s4.y, v.y);
                    v.z = fmaf(dg.z, s4.z, v.z);
                    v.w = fmaf(dg.w, s4.w, v.w);
                    store4_io(p.y, !kF32, (size_t)m * p.H + n, v);
                }
            }
            epi_sync();
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem_base, kTmem);
    if (threadIdx.x == 0 && (*abort_flag || *reinterpret_cast<volatile int*>(&bars.epi_abort)) && p.hdr) p.hdr->status = SSM_ERR_TIMEOUT;
}

// ---------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------
namespace {

struct StepShape {
    int bn, cluster, stages, stage_bytes;
};

// Tile width and cluster size by an estimate in microseconds built like that of the few-tile projections (fixed cost of a
// tile, k-blocks at the slower of L2 and tensor core, both phases).  Its constants are taken over from there, not fitted
// to this kernel.
StepShape pick_step(int M, int H, int P, bool f32) {
    StepShape best{0, 0, 0, 0};
    double best_t = 0.0;
    const int m_tiles = (M + BM - 1) / BM, sms = device_sm_count();
    for (int bn = 32; bn <= (f32 ? 64 : 128); bn *= 2) {
        const int w0 = (f32 ? 3 : 2) * bn * BK * 2, w1 = (f32 ? 3 : 1) * bn * BK * 2, a = (f32 ? 3 : 1) * kSmATile;
        const int sb = a + w0;
        const int stages = std::min<int>(kStMaxStages, (int)((kStSmemMax - 2048 - (size_t)BM * (bn + 4) * 4) / sb));
        if (stages < 2) continue;
        for (int c = 1; c <= 8; c *= 2) {
            const int slots = c == 1 ? sms : (c == 2 ? sms - 4 : (c == 4 ? sms - 16 : sms - 36));   // clusters must fit a GPC
            const int waves = (m_tiles * c + slots - 1) / slots;
            const int i0 = ((2 * P + bn - 1) / bn + c - 1) / c, i1 = ((H + bn - 1) / bn + c - 1) / c;
            const double mma = 4.0 * std::max(bn / 2.0, (128 + bn) / 4.0) / 1900.0;   // of one product and k-block
            const double kb0 = std::max((f32 ? w0 + 32768 : sb) / 91000.0, (f32 ? 6 : 2) * mma);
            const double kb1 = std::max((f32 ? w1 + 32768 : a + w1) / 91000.0, (f32 ? 6 : 1) * mma);
            const double t = waves * (3.0 + i0 * (1.5 + 0.012 * bn + (H / BK) * kb0) + i1 * (1.5 + 0.012 * bn + (2 * P / BK) * kb1));
            if (best.bn == 0 || t < best_t) {
                best_t = t;
                best = {bn, c, stages, sb};
            }
        }
    }
    return best;
}

template <int kBN, bool kF32>
int launch_step_t(const CUtensorMap& mu, const CUtensorMap& mx, const CUtensorMap& mb, const CUtensorMap& mc, const StepArgs& p,
                  cudaStream_t st) {
    auto kern = step_kernel<kBN, kF32>;
    const size_t smem = (size_t)p.stages * p.stage_bytes + (size_t)BM * (kBN + 4) * 4 + 1024;
    if (!set_max_dynamic_smem(reinterpret_cast<const void*>(kern), kStSmemMax)) return SSM_ERR_CUDA;
    count_launch();
    const unsigned grid = (unsigned)((p.M + BM - 1) / BM * p.cluster);
    return launch_dep_cluster(kern, (unsigned)p.cluster, grid, kStThreads, smem, st, mu, mx, mb, mc, p) ? SSM_OK : SSM_ERR_CUDA;
}

}  // namespace
}  // namespace tc

// fp32 I/O above 256 columns is left to the projections of gemm_tc_small.cu: every CTA here splits the whole rows of
// its operands again for its few columns (H = 512: 24.5 us at 256 - 1024 trajectories against 19.5 - 24.9 as three
// kernels, 47 against 38 at 4096; H = 256: 14.8 against 15.8, 16.3 against 22.5).
bool use_step_kernel(int H, int P, bool f32) { return !f32 || std::max(H, 2 * P) <= 256; }

int launch_step(const StepCall& g, cudaStream_t st) {
    using namespace tc;
    if (g.H % BK != 0 || g.P % (BK / 2) != 0) return SSM_ERR_SHAPE;
    const StepShape s = pick_step(g.B, g.H, g.P, g.f32);
    if (s.bn == 0) return SSM_ERR_SHAPE;
    StepArgs p{};
    p.M = g.B, p.H = g.H, p.P = g.P, p.cluster = s.cluster, p.stages = s.stages, p.stage_bytes = s.stage_bytes;
    p.n_tiles[0] = (2 * g.P + s.bn - 1) / s.bn, p.n_tiles[1] = (g.H + s.bn - 1) / s.bn;
    p.k_blocks[0] = g.H / BK, p.k_blocks[1] = 2 * g.P / BK;
    p.u = g.u, p.done = g.done, p.D = g.D, p.y = g.y, p.hdr = g.hdr;
    p.x_prev = reinterpret_cast<const float4*>(g.x_prev), p.x_next = reinterpret_cast<float4*>(g.x_next);
    p.x_bf16 = reinterpret_cast<__nv_bfloat16*>(g.x_bf16);
    p.Abar = reinterpret_cast<const float4*>(g.Abar), p.Alo = reinterpret_cast<const float4*>(g.Alo);
    const uint64_t H = (uint64_t)g.H, P2 = 2 * (uint64_t)g.P, M = (uint64_t)g.B;
    CUtensorMap mu, mx, mb, mc;
    bool ok = g.f32 ? make_map(&mb, g.Wb, P2, 3 * H, BK, (uint32_t)s.bn) && make_map(&mc, g.Wc, H, 3 * P2, BK, (uint32_t)s.bn)
                    : make_map(&mb, g.Wb, 2 * P2, H, BK, (uint32_t)s.bn) && make_map(&mc, g.Wc, H, P2, BK, (uint32_t)s.bn);
    mu = mx = mb;   // unused with fp32 I/O
    if (!g.f32) ok = ok && make_map(&mu, g.u, M, H, BK, BM) && make_map(&mx, g.x_bf16, M, P2, BK, BM);
    if (!ok) return SSM_ERR_CUDA;
    if (g.f32) return s.bn == 32 ? launch_step_t<32, true>(mu, mx, mb, mc, p, st) : launch_step_t<64, true>(mu, mx, mb, mc, p, st);
    if (s.bn == 32) return launch_step_t<32, false>(mu, mx, mb, mc, p, st);
    if (s.bn == 64) return launch_step_t<64, false>(mu, mx, mb, mc, p, st);
    return launch_step_t<128, false>(mu, mx, mb, mc, p, st);
}

}  // namespace ssm
