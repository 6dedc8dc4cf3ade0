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
#include "scan_math.cuh"
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
    TileScan scan;
    int tile_rows, seqs;       // rows of a tile: BM, or seqs whole sequences
    WsHeader* hdr;
};

// Epilogues: fp32 result; out = acc + diag * skip (+ add) with, if asked for, the column sums of skip * dot over the
// rows of this CTA; fp32 result and out2 = skip * sigmoid(acc) in bf16; the scan of the result's rows (columns 2 p, 2 p + 1 are
// state p), which leaves in its place, forward or backward.
//
// The scans: a tile then holds whole sequences, and CTA `rank` finishes all rows of its share of the tile's columns.  A
// thread has one state and kRows rows; the groups of rows are joined in order through shared memory, as in the streaming
// kernels.  As kernels of their own the scans of 1024 rows took 4 (forward) and 6 us (backward) of a pass, all latency: forward and
// backward of 16 x 64 steps at H, P = 256, 128 62.9 -> 55.3 us, a stack of four layers of 512, 256 319 -> 287.
enum SmallEpi { kSmStore, kSmDiag, kSmGate, kSmScanFwd, kSmScanBwd };
__host__ __device__ constexpr bool sm_scans(int epi) { return epi >= kSmScanFwd; }

struct SmallBars {
    uint64_t full[kSmMaxStages], empty[kSmMaxStages], done;
    uint32_t tmem;
    int abort_flag;
};

// What a scanning thread reads from afar, asked for while the MMAs run; kRows rows of one state.
template <int kEpi, int kRows>
struct ScanThread {
    int b, t0, len, row0, groups, g;   // sequence, first step, steps, row in the tile; groups of a sequence, the thread's
    int p;                             // state
    bool mine;
    uint32_t flags;
    float2 a, al, first, before[kEpi == kSmScanBwd ? kRows : 1];
    __device__ __forceinline__ void fetch(const SmallTnArgs& k, int m_tile, int col0, int te) {
        constexpr int kStates = 2 * kRows;
        const TileScan& s = k.scan;
        groups = (s.T + kRows - 1) / kRows;
        const int slot = te / kStates, seq = slot / groups;
        g = slot - seq * groups;
        b = m_tile * k.seqs + seq;
        t0 = g * kRows;
        len = min(kRows, s.T - t0);
        row0 = seq * s.T + t0;
        p = col0 / 2 + te % kStates;
        mine = seq < k.seqs && b < s.B;
        flags = 0;
        a = al = first = make_float2(0.f, 0.f);
        if (!mine) return;
        a = s.Abar[p], al = s.Alo[p];
        const size_t m = (size_t)b * s.T + t0, P = (size_t)k.N / 2;
        if (s.done)
#pragma unroll
            for (int i = 0; i < kRows; ++i)
                if (i < len && s.done[m + i] != 0) flags |= 1u << i;
        if (kEpi == kSmScanFwd) {
            if (g == 0 && s.x0) first = s.x0[(size_t)b * P + p];
        } else {
            if (g == groups - 1 && s.gxT) first = s.gxT[(size_t)b * P + p];
#pragma unroll
            for (int i = 0; i < kRows; ++i) {
                before[i] = make_float2(0.f, 0.f);
                if (i < len && t0 + i > 0) before[i] = s.x[(m + i - 1) * P + p];
                else if (i < len && s.x0) before[i] = s.x0[(size_t)b * P + p];
            }
        }
    }
};

template <int kBN, int kEpi, bool kSplitA, bool kBf16, bool kPair, int kScanRows = 0>
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
    const int m0 = m_tile * (sm_scans(kEpi) ? p.tile_rows : BM), n0 = (tile % p.n_tiles) * kBN;
    const int m_end = sm_scans(kEpi) ? min(p.M, m0 + p.tile_rows) : p.M;
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
            if (kb0 < kb1) sp.fetch(p.a_f32, p.K, m_end, m0, kb0, te);
            int stage = 0;
            uint32_t phase = 0;
            for (int kb = kb0; kb < kb1; ++kb) {
                if (!mbar_wait(smem_u32(&bars.empty[stage]), phase ^ 1u, abort_flag)) break;
                sp.store(tiles + (size_t)stage * p.stage_bytes, m_end, m0, te, n0 == 0 ? p.a_planes : nullptr, p.K, kb);
                if (kb + 1 < kb1) sp.fetch(p.a_f32, p.K, m_end, m0, kb + 1, te);
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
            if ((kEpi == kSmDiag || kEpi == kSmGate) && r < rows && m < p.M && n < p.N) {
                const size_t e = (size_t)m * p.N + n;
                sk[i].load(p.skip, p.skip_bf16, e);
                if (kEpi == kSmDiag && p.dot) dt[i].load(p.dot, p.dot_bf16, e);
            }
        }
    };
    ScanThread<kEpi, kScanRows ? kScanRows : 1> sc;
    if (warp >= 2) {
        if (sm_scans(kEpi)) sc.fetch(p, m_tile, n0 + rank * (kBN / parts), te);
        else fetch_operands(rg);
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
    if (sm_scans(kEpi) && warp >= 2) {
        constexpr bool kBwd = kEpi == kSmScanBwd;
        constexpr int kR = kScanRows ? kScanRows : 1, kStates = 2 * kR;
        __shared__ float4 agg[32 * kSmEpiWarps];
        auto epi_sync = [] { asm volatile("bar.sync 1, %0;" ::"n"(32 * kSmEpiWarps) : "memory"); };
        const float2 zero = make_float2(0.f, 0.f);
        const size_t P = (size_t)p.N / 2;
        float2 v[kR], a = sc.a, al = sc.al, aR, aRl;
        cpow2_pair<kR>(a, al, aR, aRl);
        if (kBwd) a = cconj(a), al = cconj(al), aR = cconj(aR), aRl = cconj(aRl);
        // this thread's rows: the sum of the parts of all CTAs
        const float* own = reinterpret_cast<const float*>(tiles) + (size_t)sc.row0 * kPitch + rank * (kBN / parts) + 2 * (te % kStates);
#pragma unroll
        for (int i = 0; i < kR; ++i) v[i] = zero;
        if (sc.mine)
            for (int q = 0; q < parts; ++q) {
                const uint32_t from = map_to_cta(smem_u32(own), (uint32_t)q);
                float2 t[kR];
#pragma unroll
                for (int i = 0; i < kR; ++i)
                    if (i < sc.len) t[i] = ld_cluster_f2(from + (uint32_t)i * (kPitch * 4u));
#pragma unroll
                for (int i = 0; i < kR; ++i)
                    if (i < sc.len) v[i] = cadd(v[i], t[i]);
            }
        // a group's own contribution; the first one that is folded starts from what enters the sequence
        float2 e = sc.first;
        const bool cut = sc.flags != 0u || (kBwd ? sc.g == sc.groups - 1 : sc.g == 0);
#pragma unroll
        for (int j = 0; j < kR; ++j) {
            const int i = kBwd ? kR - 1 - j : j;
            if (i >= sc.len) continue;
            if (!kBwd) e = cfma2(a, al, (sc.flags >> i) & 1u ? zero : e, v[i]);
            else if (i == sc.len - 1) e = cadd(v[i], e);   // (the state's gradient s; what it hands on, conj(Abar) s, is rounded once, below)
            else e = cfma2(a, al, (sc.flags >> (i + 1)) & 1u ? zero : e, v[i]);
        }
        if (kBwd) e = (sc.flags & 1u) ? zero : cfma2(a, al, e, zero);
        agg[te] = make_float4(e.x, e.y, cut ? 1.f : 0.f, 0.f);
        epi_sync();
        float2 c = sc.first, gA = zero;
        if (sc.mine && !*abort_flag) {
            const int ahead = kBwd ? sc.groups - 1 - sc.g : sc.g;
#pragma unroll 4
            for (int j = ahead; j > 0; --j) {   // the groups before this one, the furthest first
                const float4 o = agg[te + (kBwd ? j : -j) * kStates];
                c = o.z != 0.f ? make_float2(o.x, o.y) : cfma2(aR, aRl, c, make_float2(o.x, o.y));
            }
            float2* dst = reinterpret_cast<float2*>(p.out) + ((size_t)sc.b * p.scan.T + sc.t0) * P + sc.p;
#pragma unroll
            for (int j = 0; j < kR; ++j) {
                const int i = kBwd ? kR - 1 - j : j;
                if (i >= sc.len) continue;
                const bool flag = (sc.flags >> i) & 1u;
                if (!kBwd) c = cfma2(a, al, flag ? zero : c, v[i]);
                else if (i == sc.len - 1) c = cadd(v[i], c);
                else c = cfma2(a, al, (sc.flags >> (i + 1)) & 1u ? zero : c, v[i]);
                dst[(size_t)i * P] = c;
                if (kBwd && !flag) gA = cfma(c, cconj(sc.before[kBwd ? i : 0]), gA);
            }
            if (kBwd) c = (sc.flags & 1u) ? zero : cfma2(a, al, c, zero);
            float2* end = kBwd ? p.scan.gx0 : p.scan.xT;
            if (end && (kBwd ? sc.g == 0 : sc.g == sc.groups - 1)) end[(size_t)sc.b * P + sc.p] = c;
        }
        if (kBwd) {   // sum of the groups of a sequence, in order
            epi_sync();
            agg[te] = make_float4(gA.x, gA.y, 0.f, 0.f);
            epi_sync();
            if (sc.mine && sc.g == 0 && !*abort_flag) {
                double re = (double)gA.x, im = (double)gA.y;   // (dDelta takes differences of these sums)
#pragma unroll 4
                for (int j = 1; j < sc.groups; ++j) re += (double)agg[te + j * kStates].x, im += (double)agg[te + j * kStates].y;
                p.scan.gA_part[(size_t)sc.b * P + sc.p] = make_float2((float)re, (float)im);
            }
        }
    }
    if (!sm_scans(kEpi) && warp >= 2 && !*abort_flag) {
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

// Rows of a scanning thread for a cluster size: kBN / cluster columns of the tile are 2 kRows states.
constexpr int scan_rows(int cluster) { return 64 / (4 * cluster); }
// Whole sequences of a tile, so that their groups of rows find a slot of the 256 scanning threads each.
int scan_seqs(int T, int cluster) {
    const int r = scan_rows(cluster), slots = 256 / (2 * r), groups = (T + r - 1) / r;
    return std::min(BM / T, slots / groups);
}

// Tile width and cluster size, or a CTA pair: the choice with the shortest estimated time.  The estimate for single CTAs and
// clusters is a fit, in microseconds, to timings of all of them on twenty shapes from 16 x 256 x 256 to 4096 x 1024 x 1024,
// back to back (within 10 % of the measured time, and the one it picks within 8 % of the fastest): a wave of CTAs takes a
// fixed part that grows with the tile (start, first loads, epilogue), its k-blocks at 48 bytes of operands per cycle and SM
// (L2), 0.95 us where fp32 operands are split on the way, and the exchange between the CTAs of a cluster.  Pairs go through
// the same formula with their own operand bytes; it was not fitted to them, only checked on whole passes, with pairs / with
// single CTAs and clusters: gate of 4096 x 1024 102.4 / 108.2 us, of 4096 x 512 47.9 / 49.7, layer 64 x 100 (256, 128)
// 55.4 / 57.4, 32 x 128 (512, 256) 63.5 / 63.5, 32 x 128 (1024, 512) 114.6 / 114.2.
SmallShape pick_small(int M, int N, int k_blocks, int planes_a, int planes_w, bool split_a, bool w_stacked,
                      const TileScan* scan = nullptr, double* us = nullptr) {
    SmallShape best{0, 0, 0, false};
    double best_t = 0.0;
    const int sms = device_sm_count();
    auto consider = [&](int bn, int c, bool pair) {
        const int seqs = scan ? scan_seqs(scan->T, c) : 0;
        if (scan && seqs == 0) return;
        const int m_tiles = scan ? (scan->B + seqs - 1) / seqs : (M + BM - 1) / BM;
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
    if (scan) {   // (the scans are built for 64 columns and clusters of 2 and 4)
        for (int c = 2; c <= 4 && c <= k_blocks; c *= 2) consider(64, c, false);
        if (us) *us = best_t;
        return best;
    }
    for (int bn = 64; bn <= (w_stacked ? 128 : 256); bn *= 2)
        for (int c = 1; c <= 4 && c <= k_blocks; c *= 2) consider(bn, c, false);
    if (!split_a)
        for (int bn = 128; bn <= 256; bn *= 2) consider(bn, 1, true);
    if (us) *us = best_t;
    return best;
}

template <int kBN, int kEpi, bool kSplitA, bool kBf16, bool kPair, int kScanRows = 0>
int launch_small(const CUtensorMap& ma, const CUtensorMap& mw, const SmallTnArgs& p, int grid, size_t smem, cudaStream_t st) {
    auto kern = gemm_tc_tn_small_kernel<kBN, kEpi, kSplitA, kBf16, kPair, kScanRows>;
    if (!set_max_dynamic_smem(reinterpret_cast<const void*>(kern), kSmSmemMax)) return SSM_ERR_CUDA;
    count_launch();
    return launch_dep_cluster(kern, kPair ? 2u : (unsigned)p.cluster, grid, sm_threads(kBN), smem, st, ma, mw, p) ? SSM_OK : SSM_ERR_CUDA;
}

}  // namespace
}  // namespace tc

int launch_gemm_tc_tn_small(const GemmTcTN& g, cudaStream_t st) {
    using namespace tc;
    const int epi = g.scan ? (g.scan->gA_part ? kSmScanBwd : kSmScanFwd) : g.gate_out ? kSmGate : (g.store_f32 && !g.diag ? kSmStore : kSmDiag);
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
    const SmallShape s = pick_small(g.M, g.N_out, p.k_blocks, p.planes_a, p.planes_w, g.a_f32, p.w_stacked != 0, g.scan);
    if (s.bn == 0) return SSM_ERR_SHAPE;
    if (g.scan) p.scan = *g.scan, p.seqs = scan_seqs(g.scan->T, s.cluster), p.tile_rows = p.seqs * g.scan->T;
    p.cluster = s.cluster;
    p.stages = s.stages;
    p.stage_bytes = (int)stage_bytes_of(s.bn, p.planes_a, p.planes_w, s.pair);
    p.n_tiles = (g.N_out + s.bn - 1) / s.bn;
    const size_t smem = std::max((size_t)p.stages * p.stage_bytes, (size_t)BM * (s.bn + 4) * 4) + 1024;
    const int m_tiles = g.scan ? (g.scan->B + p.seqs - 1) / p.seqs : (g.M + BM - 1) / BM, grid = (s.pair ? (m_tiles + 1) / 2 * 2 : m_tiles * p.cluster) * p.n_tiles;
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
    if (epi == kSmScanBwd) {   // (the gradient is fp32 there)
        if (!g.a_f32) return SSM_ERR_DTYPE;
        return s.cluster == 4 ? launch_small<64, kSmScanBwd, true, true, false, scan_rows(4)>(ma, mw, p, grid, smem, st)
                              : launch_small<64, kSmScanBwd, true, true, false, scan_rows(2)>(ma, mw, p, grid, smem, st);
    }
    if (epi == kSmScanFwd && g.a_f32)
        return s.cluster == 4 ? launch_small<64, kSmScanFwd, true, true, false, scan_rows(4)>(ma, mw, p, grid, smem, st)
                              : launch_small<64, kSmScanFwd, true, true, false, scan_rows(2)>(ma, mw, p, grid, smem, st);
    if (epi == kSmScanFwd)
        return s.cluster == 4 ? launch_small<64, kSmScanFwd, false, true, false, scan_rows(4)>(ma, mw, p, grid, smem, st)
                              : launch_small<64, kSmScanFwd, false, true, false, scan_rows(2)>(ma, mw, p, grid, smem, st);
    if (epi == kSmGate) SSM_SMALL(kSmGate, false, true);
    if (epi == kSmStore && g.a_f32) SSM_SMALL(kSmStore, true, true);
    if (epi == kSmStore) SSM_SMALL(kSmStore, false, true);
    if (g.a_f32) SSM_SMALL(kSmDiag, true, false);
    if (io_bf16) SSM_SMALL(kSmDiag, false, true);
    return SSM_ERR_SHAPE;   // planes of A with fp32 skip or dot: left to gemm_tc_planes.cu
#undef SSM_SMALL
}

// The estimate of the projection on whole sequences (64 columns, clusters) may be 3 us above the best without: what a scan of
// its own costs in the cheaper direction, the forward pass.  us per forward and backward pass in a graph, apart -> together: 8 x 50 (256, 128) 57.3 -> 49.3, 16 x 100
// 67.5 -> 57.6, 64 x 16 (256, 256) 66.9 -> 59.5, 8 x 128 (512, 256) 82.1 -> 73.9; at 10 x 100 (512, 256), 20 x 70 (256, 128) and
// 16 x 64 (1024, 512), where the tiles would need another round, they stay apart.
bool tc_tile_scan_supported(int B, int T, int H, int P, bool a_bf16) {
    using namespace tc;
    if (T < 8 || T > BM || H % BK != 0 || (2 * P) % 64 != 0 || tc_planes_many_tiles(B * T, 2 * P)) return false;
    TileScan scan{};
    scan.B = B, scan.T = T;
    double with = 0.0, without = 0.0;
    const SmallShape s = pick_small(B * T, 2 * P, H / BK, a_bf16 ? 1 : 3, 3, !a_bf16, false, &scan, &with);
    pick_small(B * T, 2 * P, H / BK, a_bf16 ? 1 : 3, 3, !a_bf16, false, nullptr, &without);
    return s.bn != 0 && with <= without + 3.0;
}

// One partial row of column sums per CTA along M.
int tc_tn_small_max_dot_rows(int M) { return 4 * ((M + tc::BM - 1) / tc::BM); }

}  // namespace ssm
