// Single-step mode for a few trajectories: two kernels on the CUDA cores, Bu with the recurrence, then y.
//
// A tensor-core tile has 128 rows; with 16 trajectories it is idle work, and the chain of loads, MMAs and epilogues
// behind it (12 us per step at B = 16, H = 256, P = 128, fp32) is all latency.  The sums themselves are small
// (33 M multiply-adds per projection at 32 x 1024 x 1024: 1 us of the machine's FMA rate), so here a warp owns 4
// output columns x 8 rows: its lanes split the contraction (4 neighbouring indices per lane and step, so that every
// load is a coalesced 256 or 512 bytes), the 32 partial sums of a lane are added over the warp by a halving
// exchange that leaves one result per lane, and the eight warps of a CTA share its 8 rows through L1.  fp32 sums.
// Bound by launch latency and by reading the weights from L2.  Measured per step (B, H, P): see use_step_small.
#include <algorithm>

#include "kernels.h"

namespace ssm {

constexpr int kSsCols = 4, kSsRows = 8;

struct StepSmallArgs {
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

__device__ __forceinline__ float4 bf16x4(uint2 r) {
    return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xffff0000u), __uint_as_float(r.y << 16),
                       __uint_as_float(r.y & 0xffff0000u));
}

// kPlanes: bf16 planes of a weight (hi, lo, or hi, mid, lo) that are added.  kStacked: hi / lo in blocks of 128 rows.
template <bool kFirst, bool kAf32, bool kIoF32, int kPlanes, bool kStacked>
__global__ void __launch_bounds__(256)
step_small_kernel(StepSmallArgs p) {
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

// Where these kernels win: us per step back to back, this pair of kernels / the cluster kernel of gemm_tc_step.cu,
//   bf16 I/O: B = 64, H = 512: 9.6 / 11.1, B = 96: 12.5 / 11.6;  H = 1024: B = 32: 15.2 / 17.7, B = 48: 19.3 / 17.9;
//             H = 256: 6.9 - 7.7 / 7.1 - 7.6 up to B = 128;
//   fp32 I/O: H = 256: B = 16: 6.5 / 12.1, B = 128: 7.5 / 14.5;  H = 512: B = 64: 11.6 / 21.9;
//             H = 1024: B = 32: 18.3 (three kernels: 21.4), B = 48: 26.1 (21.9).
bool use_step_small(int B, int H, int P) { return (long long)B * std::max(H, 2 * P) <= 32768; }

int launch_step_small(const StepCall& g, cudaStream_t st) {
    StepSmallArgs p{};
    p.M = g.B;
    p.done = g.done, p.Abar = g.Abar, p.Alo = g.Alo;
    p.x_prev = reinterpret_cast<const float*>(g.x_prev), p.x_next = reinterpret_cast<float*>(g.x_next);
    p.D = g.D, p.u = g.u, p.y = g.y;
    StepSmallArgs q = p;
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
        ok = launch_dep(step_small_kernel<true, true, true, 3, false>, grid(p.N, w0), 32 * w0, 0, st, p) &&
             launch_dep(step_small_kernel<false, true, true, 3, false>, grid(q.N, w1), 32 * w1, 0, st, q);
    } else {
        p.w_pitch = (size_t)p.K, p.w_plane = 128 * (size_t)p.K;
        q.w_pitch = (size_t)q.K;
        ok = launch_dep(step_small_kernel<true, false, false, 2, true>, grid(p.N, w0), 32 * w0, 0, st, p) &&
             launch_dep(step_small_kernel<false, true, false, 1, false>, grid(q.N, w1), 32 * w1, 0, st, q);
    }
    return ok ? SSM_OK : SSM_ERR_CUDA;
}

}  // namespace ssm
