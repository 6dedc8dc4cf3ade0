// Single-step mode for a few trajectories: one kernel on the CUDA cores, Bu with the recurrence, then y.
//
// A tensor-core tile has 128 rows; with 16 trajectories it is idle work, and the chain of loads, MMAs and epilogues
// behind it (12 us per step at B = 16, H = 256, P = 128, fp32) is all latency.  The sums themselves are small
// (33 M multiply-adds per projection at 32 x 1024 x 1024: 1 us of the machine's FMA rate), so here a cluster of CTAs
// takes 8 trajectories and a warp 4 output columns x 8 rows at a time: its lanes split the contraction (4 neighbouring
// indices per lane and step, so that every load is a coalesced 256 or 512 bytes), and the 32 partial sums of a lane are
// added over the warp by a halving exchange that leaves one result per lane.  fp32 sums.  The new states go to the
// shared memory of every CTA of the cluster, from where its warps project them after one cluster barrier; the weights of
// a warp's first columns there are on their way meanwhile.
// Bound by latency: a launch, two trips to L2 and the barrier.  Measured per step: see halves_shorter.
#include <algorithm>
#include <type_traits>

#include "kernels.h"
#include "tcgen05.cuh"

namespace ssm {

constexpr int kSsCols = 4, kSsRows = 8, kSsWarps = 8;

struct StepSmallArgs {
    int M, H, P2, cluster;     // trajectories, features, state components (2P), CTAs per 8 trajectories
    const void* u;             // [M, H] io
    const __nv_bfloat16 *Wb, *Wc;
    size_t b_pitch, b_plane, c_pitch, c_plane;   // elements between rows of a weight matrix and between its planes
    const uint8_t* done;
    const float2 *Abar, *Alo;
    const float* x_prev;
    float* x_next;             // may be x_prev: a component is read and written by the same thread
    const float* D;
    void* y;                   // [M, H] io
};

__device__ __forceinline__ float4 bf16x4(uint2 r) {
    return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xffff0000u), __uint_as_float(r.y << 16),
                       __uint_as_float(r.y & 0xffff0000u));
}

// Four neighbouring rows of a weight matrix whose kPlanes bf16 planes (hi, lo, or hi, mid, lo) are added; kStacked: hi / lo
// in blocks of 128 rows (which four columns never cross).
template <int kPlanes, bool kStacked>
struct WeightCols {
    const __nv_bfloat16* row;
    size_t pitch, plane;
    __device__ __forceinline__ WeightCols(const __nv_bfloat16* W, int n0, size_t pitch_, size_t plane_)
        : row(W + (size_t)(kStacked ? (n0 / 128) * 256 + n0 % 128 : n0) * pitch_), pitch(pitch_), plane(plane_) {}
    struct Raw {
        uint2 r[kPlanes][kSsCols];
        __device__ __forceinline__ float4 get(int c) const {
            float4 w = bf16x4(r[0][c]);
#pragma unroll
            for (int q = 1; q < kPlanes; ++q) {
                const float4 t = bf16x4(r[q][c]);
                w.x += t.x, w.y += t.y, w.z += t.z, w.w += t.w;
            }
            return w;
        }
    };
    __device__ __forceinline__ void load(Raw& o, int k) const {
#pragma unroll
        for (int q = 0; q < kPlanes; ++q)
#pragma unroll
            for (int c = 0; c < kSsCols; ++c) o.r[q][c] = *reinterpret_cast<const uint2*>(row + c * pitch + q * plane + k);
    }
};

template <typename Raw, typename Rows>
__device__ __forceinline__ void add_products(float (&acc)[kSsRows * kSsCols], const Raw& w, const Rows& a) {
    float4 wv[kSsCols];
#pragma unroll
    for (int c = 0; c < kSsCols; ++c) wv[c] = w.get(c);
#pragma unroll
    for (int r = 0; r < kSsRows; ++r) {
        const float4 x = a.get(r);
#pragma unroll
        for (int c = 0; c < kSsCols; ++c) {
            float& s = acc[r * kSsCols + c];
            s = fmaf(x.x, wv[c].x, fmaf(x.y, wv[c].y, fmaf(x.z, wv[c].z, fmaf(x.w, wv[c].w, s))));
        }
    }
}

// The warp's sums of value l = 4 row + column: lane l returns it.
__device__ __forceinline__ float warp_exchange(float (&acc)[kSsRows * kSsCols], int lane) {
#pragma unroll
    for (int h = 16; h >= 1; h >>= 1) {
        const bool upper = (lane & h) != 0;
#pragma unroll
        for (int j = 0; j < h; ++j) {
            const float send = upper ? acc[j] : acc[j + h];
            const float keep = upper ? acc[j + h] : acc[j];
            acc[j] = keep + __shfl_xor_sync(0xffffffffu, send, h);
        }
    }
    return acc[0];
}

// Rows of u as loaded, 4 neighbouring values of each; rows of the new states in shared memory.
template <bool kF32>
struct RowsU {
    typename std::conditional<kF32, float4, uint2>::type r[kSsRows];
    __device__ __forceinline__ void load(const void* u, int m0, int M, int H, int k) {
#pragma unroll
        for (int i = 0; i < kSsRows; ++i) {
            const size_t e = (size_t)min(m0 + i, M - 1) * H + k;
            if constexpr (kF32) r[i] = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(u) + e);
            else r[i] = *reinterpret_cast<const uint2*>(reinterpret_cast<const __nv_bfloat16*>(u) + e);
        }
    }
    __device__ __forceinline__ float4 get(int i) const {
        if constexpr (kF32) return r[i];
        else return bf16x4(r[i]);
    }
};
struct RowsX {
    const float4* x;
    int pitch;   // in float4
    __device__ __forceinline__ float4 get(int i) const { return x[i * pitch]; }
};

// Column n = 2 p + c of the new state: real or imaginary part of state p; the other part sits in the neighbouring lane.
__device__ __forceinline__ float recurrence(int n, float xp, bool keep, float2 a, float2 al, float v) {
    const float xq = __shfl_xor_sync(0xffffffffu, xp, 1), s = (n & 1) ? 1.f : -1.f;
    return keep ? fmaf(a.x, xp, fmaf(s * a.y, xq, fmaf(al.x, xp, fmaf(s * al.y, xq, v)))) : v;
}
template <bool kF32>
__device__ __forceinline__ float load_u(const StepSmallArgs& p, size_t e) {
    return kF32 ? reinterpret_cast<const float*>(p.u)[e] : __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(p.u)[e]);
}
template <bool kF32>
__device__ __forceinline__ void store_y(const StepSmallArgs& p, size_t e, float v, float d, float u) {
    v = fmaf(d, u, v);
    if (kF32) reinterpret_cast<float*>(p.y)[e] = v;
    else reinterpret_cast<__nv_bfloat16*>(p.y)[e] = __float2bfloat16_rn(v);
}

template <bool kF32>
__global__ void __launch_bounds__(32 * kSsWarps)
step_small_kernel(const __grid_constant__ StepSmallArgs p) {
    constexpr int kAhead = 2;   // steps of 128 whose loads are in flight together (registers; 4 with bf16 I/O: 5 % slower)
    extern __shared__ float4 x_s[];   // [8 rows][2P]: the new states
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int rank = (int)tc::cluster_ctarank(), m0 = ((int)blockIdx.x / p.cluster) * kSsRows;
    const int n0 = (rank * kSsWarps + w) * kSsCols, n = n0 + lane % kSsCols, m = m0 + lane / kSsCols;
    const bool ok = m < p.M;
    asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");   // (every CTA runs before its shared memory is written)
    grid_dep_wait();
    grid_dep_launch();
    // ---- Bu and the recurrence
    if (n0 < p.P2) {
        using W = WeightCols<kF32 ? 3 : 2, !kF32>;
        const W wb(p.Wb, n0, p.b_pitch, p.b_plane);
        float acc[kSsRows * kSsCols] = {};
        float2 a, al;
        float xp = 0.f;
        bool keep = false;
#pragma unroll 1
        for (int k = 4 * lane; k < p.H; k += 128 * kAhead) {
            typename W::Raw wr[kAhead];
            RowsU<kF32> ur[kAhead];
#pragma unroll
            for (int i = 0; i < kAhead; ++i)
                if (k + 128 * i < p.H) {
                    wb.load(wr[i], k + 128 * i);
                    ur[i].load(p.u, m0, p.M, p.H, k + 128 * i);
                }
            if (k < 128) {
                a = p.Abar[n >> 1], al = p.Alo[n >> 1];
                if (ok) xp = p.x_prev[(size_t)m * p.P2 + n];
                keep = ok && !(p.done && p.done[m] != 0);
            }
#pragma unroll
            for (int i = 0; i < kAhead; ++i)
                if (k + 128 * i < p.H) add_products(acc, wr[i], ur[i]);
        }
        float v = warp_exchange(acc, lane);
        v = recurrence(n, xp, keep, a, al, v);
        if (ok) p.x_next[(size_t)m * p.P2 + n] = v;
        // a row's four components as one store; lane l % 4 serves every fourth CTA of the cluster
        float4 v4;
        v4.x = __shfl_sync(0xffffffffu, v, lane & ~3);
        v4.y = __shfl_sync(0xffffffffu, v, (lane & ~3) + 1);
        v4.z = __shfl_sync(0xffffffffu, v, (lane & ~3) + 2);
        v4.w = __shfl_sync(0xffffffffu, v, (lane & ~3) + 3);
        asm volatile("barrier.cluster.wait;" ::: "memory");
        const uint32_t to = tma::smem_u32(x_s + ((lane / kSsCols) * p.P2 + n0) / 4);
        for (int q = lane % kSsCols; q < p.cluster; q += kSsCols) tc::st_cluster_f4(tc::map_to_cta(to, (uint32_t)q), v4);
    } else {
        asm volatile("barrier.cluster.wait;" ::: "memory");
    }
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    // ---- y from the states of this cluster's rows; the first weights are on their way before these are complete
    if (n0 >= p.H) {
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
        return;
    }
    using W = WeightCols<kF32 ? 3 : 1, false>;
    const W wc(p.Wc, n0, p.c_pitch, p.c_plane);
    const size_t e = (size_t)m * p.H + n;
    float acc[kSsRows * kSsCols] = {};
    const float d = p.D[n];
    const float u = ok ? load_u<kF32>(p, e) : 0.f;
    typename W::Raw wr[kAhead];
#pragma unroll
    for (int i = 0; i < kAhead; ++i)
        if (4 * lane + 128 * i < p.P2) wc.load(wr[i], 4 * lane + 128 * i);
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
#pragma unroll 1
    for (int k = 4 * lane; k < p.P2; k += 128 * kAhead) {
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
            const int ki = k + 128 * i;
            if (ki >= p.P2) break;
            add_products(acc, wr[i], RowsX{x_s + ki / 4, p.P2 / 4});
            if (ki + 128 * kAhead < p.P2) wc.load(wr[i], ki + 128 * kAhead);
        }
    }
    const float v = warp_exchange(acc, lane);
    if (ok) store_y<kF32>(p, e, v, d, u);
}

// The two halves as kernels of their own, on as many SMs as there are.  (They keep their own sums, exchange and epilogue: on the functions
// above, 8 rows of the input loaded together, 16 x (1024, 512) takes 10.8 us instead of 9.6 in bf16 and 1 x (640, 192) 7.1 instead of 6.5 in
// fp32; with only the exchange and the epilogue shared still 0.1 us more.)
struct StepHalfArgs {
    int M, N, K;               // rows, output columns, contraction
    const void* a;             // first phase: u [M, K] io;  second: x_next [M, K] fp32
    const __nv_bfloat16* W;
    size_t w_pitch, w_plane;   // elements between rows of W and between its planes
    const uint8_t* done;       // first phase
    const float2 *Abar, *Alo;
    const float* x_prev;
    float* x_next;
    const float* D;            // second phase
    const void* u;
    void* y;
};

// kPlanes: bf16 planes of a weight (hi, lo, or hi, mid, lo) that are added.  kStacked: hi / lo in blocks of 128 rows.
template <bool kFirst, bool kAf32, bool kIoF32, int kPlanes, bool kStacked>
__global__ void __launch_bounds__(256)
step_half_kernel(StepHalfArgs p) {
    grid_dep_wait();
    grid_dep_launch();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int n0 = (blockIdx.x * (blockDim.x >> 5) + w) * kSsCols, m0 = blockIdx.y * kSsRows;
    if (n0 >= p.N) return;   // (N is a multiple of 4)
    const __nv_bfloat16* wrow[kSsCols];
#pragma unroll
    for (int c = 0; c < kSsCols; ++c) {
        const int n = n0 + c;
        wrow[c] = p.W + (size_t)(kStacked ? (n / 128) * 256 + n % 128 : n) * p.w_pitch;
    }
    float acc[kSsRows * kSsCols];
#pragma unroll
    for (int i = 0; i < kSsRows * kSsCols; ++i) acc[i] = 0.f;
#pragma unroll 2
    for (int k = 4 * lane; k < p.K; k += 128) {
        float4 wv[kSsCols];
#pragma unroll
        for (int c = 0; c < kSsCols; ++c) {
            wv[c] = bf16x4(*reinterpret_cast<const uint2*>(wrow[c] + k));
#pragma unroll
            for (int q = 1; q < kPlanes; ++q) {
                const float4 t = bf16x4(*reinterpret_cast<const uint2*>(wrow[c] + q * p.w_plane + k));
                wv[c].x += t.x, wv[c].y += t.y, wv[c].z += t.z, wv[c].w += t.w;
            }
        }
#pragma unroll
        for (int r = 0; r < kSsRows; ++r) {
            const size_t e = (size_t)min(m0 + r, p.M - 1) * p.K + k;
            const float4 a = kAf32 ? *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(p.a) + e)
                                   : bf16x4(*reinterpret_cast<const uint2*>(reinterpret_cast<const __nv_bfloat16*>(p.a) + e));
#pragma unroll
            for (int c = 0; c < kSsCols; ++c) {
                float& s = acc[r * kSsCols + c];
                s = fmaf(a.x, wv[c].x, fmaf(a.y, wv[c].y, fmaf(a.z, wv[c].z, fmaf(a.w, wv[c].w, s))));
            }
        }
    }
    // lane l ends with the sum of value l = 4 row + column over the warp
#pragma unroll
    for (int h = 16; h >= 1; h >>= 1) {
        const bool upper = (lane & h) != 0;
#pragma unroll
        for (int j = 0; j < h; ++j) {
            const float send = upper ? acc[j] : acc[j + h];
            const float keep = upper ? acc[j + h] : acc[j];
            acc[j] = keep + __shfl_xor_sync(0xffffffffu, send, h);
        }
    }
    const int m = m0 + lane / kSsCols, n = n0 + lane % kSsCols;
    const bool ok = m < p.M;
    float v = acc[0];
    if (kFirst) {   // column n = 2 p + c: real or imaginary part of state p; the other part sits in the neighbouring lane
        const float2 a = p.Abar[n >> 1], al = p.Alo[n >> 1];
        const float xp = ok ? p.x_prev[(size_t)m * p.N + n] : 0.f;
        const float xq = __shfl_xor_sync(0xffffffffu, xp, 1);
        const float s = (n & 1) ? 1.f : -1.f;
        if (ok) {
            if (!(p.done && p.done[m] != 0)) v = fmaf(a.x, xp, fmaf(s * a.y, xq, fmaf(al.x, xp, fmaf(s * al.y, xq, v))));
            p.x_next[(size_t)m * p.N + n] = v;
        }
    } else if (ok) {
        const size_t e = (size_t)m * p.N + n;
        const float u = kIoF32 ? reinterpret_cast<const float*>(p.u)[e] : __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(p.u)[e]);
        v = fmaf(p.D[n], u, v);
        if (kIoF32) reinterpret_cast<float*>(p.y)[e] = v;
        else reinterpret_cast<__nv_bfloat16*>(p.y)[e] = __float2bfloat16_rn(v);
    }
}

// Against the cluster kernel of gemm_tc_step.cu, us per step, the two halves / that one:
//   bf16 I/O: B = 64, H = 512: 9.6 / 11.1, B = 96: 12.5 / 11.6;  H = 1024: B = 32: 15.2 / 17.7, B = 48: 19.3 / 17.9;
//   fp32 I/O: H = 512: B = 64: 11.6 / 21.9;  H = 1024: B = 32: 18.3 (three kernels: 21.4), B = 48: 26.1 (21.9).
bool use_step_small(int B, int H, int P) { return (long long)B * std::max(H, 2 * P) <= 32768; }

static auto step_cluster_kernel(bool f32) { return f32 ? step_small_kernel<true> : step_small_kernel<false>; }
// The halves take less time on the device than the one kernel where its clusters are small or hold few rows, and more host time nearly
// everywhere (two launches: 7.3 us).  us per step in a graph, halves / one kernel (B, H, P):
//   fp32, clusters of 16: 1, 512, 256 6.9 / 7.7, 4 7.7 / 7.7, 8 9.7 / 7.7;  1, 384, 192 5.5 / 6.5, 4 6.1 / 6.5, 5 6.9 / 6.5;  16, 512, 256 9.9 / 7.7;
//         4, 384, 64 4.6 / 5.4, 16 5.0 / 5.5, 16, 512, 64 6.0 / 6.0;  of 8: 1, 256, 128 4.7 / 4.6, 16 6.2 / 4.7, 96 6.6 / 4.9;  2, 256, 64 4.0 / 4.2, 8 4.5 / 4.2;
//         of 4: 8, 128, 64 3.5 / 3.7, 112 3.8 / 3.9, 224 4.7 / 3.9;
//   bf16, clusters of 8: 1, 256, 128 4.2 / 4.2, 16 4.6 / 4.4;  1, 256, 64 3.6 / 4.0, 8 3.9 / 4.0, 32 4.1 / 4.1;  of 4: 8, 128, 64 3.4 / 3.6, 224 4.6 / 3.8.
// Eager: 16, 256, 128 7.3 / 5.0, 16, 512, 256 10.5 / 8.3;  1, 512, 256 7.5 / 8.2, 3 8.0 / 8.3;  1, 384, 256 7.3 / 7.6, 2 7.5 / 7.6.  The results are the same bits.
static bool halves_shorter(const StepCall& g, int cluster, cudaStream_t st) {
    const int P2 = 2 * g.P;
    const int products = g.H * P2;   // (at most 512 x 512)
    const bool in_graph = g.B <= (cluster == 4 ? 112 : cluster == 8 ? (std::min(g.H, P2) == 128 ? 2 : 0) : (P2 == 128 ? 16 : products < 512 * 512 ? 4 : 3));
    const bool eager = cluster == 16 && g.B <= 3 && products >= (g.B == 1 ? 384 : 512) * 512;
    return in_graph == eager ? eager : (capturing(st) ? in_graph : eager);
}

// CTAs of a cluster that takes a step's columns in one round, or 0: the halves apart.  The clusters have to run in one round (us in a graph,
// halves / one kernel: 128, 256, 128, 16 clusters of 8, fp32 7.4 / 8.7, bf16 6.6 / 8.1;  64, 512, 256 in fp32, 8 of 16, 11.0 / 14.4), on a device that
// holds fewer than a B200 as well.  Wider ones, with several rounds of columns a warp, are slower throughout (8, 1024, 512 in fp32 16.8 / 40), as are
// clusters of 16 with bf16 I/O (16, 512, 256 6.2 / 6.7).
static int step_small_cluster(const StepCall& g, cudaStream_t st) {
    const int width = std::max(g.H, 2 * g.P), row_groups = (g.B + kSsRows - 1) / kSsRows;
    if (std::min(g.H, 2 * g.P) < 128) return 0;   // (every lane has a share of both contractions)
    int c = 4;
    while (c * kSsWarps * kSsCols < width) c *= 2;
    const int most = c <= 8 ? 112 : (c == 16 && g.f32 ? 64 : 0);   // CTAs
    if (row_groups * c > most || halves_shorter(g, c, st)) return 0;
    const size_t smem = kSsRows * kSsWarps * kSsCols * 16 * sizeof(float);   // (of the widest)
    return resident_clusters(reinterpret_cast<const void*>(step_cluster_kernel(g.f32)), c, smem, 32 * kSsWarps) >= row_groups ? c : 0;
}

static int launch_step_cluster(const StepCall& g, int cluster, cudaStream_t st) {
    const size_t H = (size_t)g.H, P2 = 2 * (size_t)g.P;
    StepSmallArgs p{};
    p.M = g.B, p.H = g.H, p.P2 = 2 * g.P, p.cluster = cluster;
    p.u = g.u, p.done = g.done, p.Abar = g.Abar, p.Alo = g.Alo, p.D = g.D, p.y = g.y;
    p.Wb = (const __nv_bfloat16*)g.Wb, p.Wc = (const __nv_bfloat16*)g.Wc;
    p.x_prev = reinterpret_cast<const float*>(g.x_prev), p.x_next = reinterpret_cast<float*>(g.x_next);
    if (g.f32) p.b_pitch = 3 * H, p.b_plane = H, p.c_pitch = 3 * P2, p.c_plane = P2;
    else p.b_pitch = H, p.b_plane = 128 * H, p.c_pitch = P2;
    count_launch();
    const unsigned grid = (unsigned)((g.B + kSsRows - 1) / kSsRows * cluster);
    return launch_dep_cluster(step_cluster_kernel(g.f32), (unsigned)cluster, grid, 32 * kSsWarps, kSsRows * P2 * sizeof(float), st, p) ? SSM_OK : SSM_ERR_CUDA;
}

int launch_step_small(const StepCall& g, cudaStream_t st) {
    if (const int cluster = step_small_cluster(g, st)) return launch_step_cluster(g, cluster, st);
    StepHalfArgs p{};
    p.M = g.B;
    p.done = g.done, p.Abar = g.Abar, p.Alo = g.Alo;
    p.x_prev = reinterpret_cast<const float*>(g.x_prev), p.x_next = reinterpret_cast<float*>(g.x_next);
    p.D = g.D, p.u = g.u, p.y = g.y;
    StepHalfArgs q = p;
    p.a = g.u, p.N = 2 * g.P, p.K = g.H, p.W = (const __nv_bfloat16*)g.Wb;
    q.a = g.x_next, q.N = g.H, q.K = 2 * g.P, q.W = (const __nv_bfloat16*)g.Wc;
    auto grid = [&](int N, int warps) { return dim3((unsigned)((N / kSsCols + warps - 1) / warps), (unsigned)((g.B + kSsRows - 1) / kSsRows)); };
    // warps per CTA: as many as still leave a CTA per SM
    auto warps_of = [&](int N) {
        int w = 8;
        while (w > 1 && (N / kSsCols / w) * ((g.B + kSsRows - 1) / kSsRows) < device_sm_count()) w /= 2;
        return w;
    };
    const int w0 = warps_of(p.N), w1 = warps_of(q.N);
    bool ok;
    count_launch(2);
    if (g.f32) {
        p.w_pitch = 3 * (size_t)p.K, p.w_plane = (size_t)p.K;
        q.w_pitch = 3 * (size_t)q.K, q.w_plane = (size_t)q.K;
        ok = launch_dep(step_half_kernel<true, true, true, 3, false>, grid(p.N, w0), 32 * w0, 0, st, p) &&
             launch_dep(step_half_kernel<false, true, true, 3, false>, grid(q.N, w1), 32 * w1, 0, st, q);
    } else {
        p.w_pitch = (size_t)p.K, p.w_plane = 128 * (size_t)p.K;
        q.w_pitch = (size_t)q.K;
        ok = launch_dep(step_half_kernel<true, false, false, 2, true>, grid(p.N, w0), 32 * w0, 0, st, p) &&
             launch_dep(step_half_kernel<false, true, false, 1, false>, grid(q.N, w1), 32 * w1, 0, st, q);
    }
    return ok ? SSM_OK : SSM_ERR_CUDA;
}

}  // namespace ssm
