// A layer's forward and backward pass in one kernel each, for small layers of widths that the tensor cores do not take.
//
// As ten dependent launches a layer of 64 steps, 32 features and 16 states took 31 us (eager 36.5), 3 us each, of which the sums are
// a fraction.  Here a cluster of CTAs takes one sequence through the whole pass.  Each CTA owns a part of the states: it
// projects onto them, scans them (groups of rows per state, joined in order, as in the streaming kernels) and forms
// their weight gradients; the scanned states go to the shared memory of all CTAs of the cluster, each of which
// projects them onto its part of the features.  The weights are used as the caller stores them: gamma, the factor of
// the discretisation, multiplies the projected inputs and, conjugated, the gradients of the states, so that its
// double-precision evaluation (its four functions on different warps) runs while the inputs arrive.  What of that could leave the
// range of fp32 where gamma B does not is computed in its order (an overflowed B u) or scaled exactly (gradients where |gamma| > 1).
// fp32 throughout; Abar as an fp32 pair, its power over a group's rows and the adjoint of the discretisation
// evaluated in double.  A single sequence finishes its parameter gradients itself; several leave them as slices for
// launch_layer_tail, or s for the products of the separate kernels where the slices would need more room than those.
// Bound by latency: one trip to memory, the exponentials, six barriers and the fetch of the instructions, which each launch runs once.  Of
// the cycles between two instructions of a warp at 1 x 64 (32, 16), barriers are 39 % forward and 28 % backward, missing instructions 29 %
// backward; no unit is above 19 % at 14 sequences.  Measured: see ls_cluster.
#include <type_traits>

#include "kernels.h"
#include "scan_math.cuh"
#include "tcgen05.cuh"
#include "zoh.cuh"

namespace ssm {
namespace {

constexpr int kLsThreads = 256, kLsWarps = kLsThreads / 32;
constexpr size_t kLsSmemMax = 200 * 1024;
constexpr int kLsDotGroups = 8;   // row groups of dD's sums
constexpr int kLsChain = 8;       // rows that are summed before they are added to the rest (in one chain of 500: dB 2.5 x further off)

// Rows of a scanning thread: the kLsThreads / states groups along time share the sequence; not fewer than 4.
__host__ __device__ inline int ls_group_rows(int T, int states) {
    const int groups = kLsThreads / states, r = (T + groups - 1) / groups;
    return r < 4 ? 4 : r;
}

struct LsSmem {   // offsets in floats; every row starts on a 16-byte boundary
    int hp, xp, fp, wp, cp;    // pitches: u and gy; own states; all states; weights of the own states; of the own features
    int u, gy, x, s, full, wstate, wfeat, parts, zoh, apow, agg, sums, gq, flags, total;
    __host__ __device__ LsSmem(int T, int H, int P, int cluster, bool bwd) {
        const int pc = P / cluster, hc = H / cluster;
        hp = H + 4, fp = 2 * P + 4, xp = 2 * pc + 4;
        wp = bwd ? 2 * pc + 4 : 2 * H + 4;   // C[h][own p], or B[own p][h]
        cp = bwd ? 2 * hc + 4 : 2 * P + 4;   // B[p][own h], or C[own h][p]
        xp = (xp + 3) / 4 * 4, wp = (wp + 3) / 4 * 4, cp = (cp + 3) / 4 * 4;
        int o = 0;
        auto take = [&o](int n) {
            const int at = o;
            o += (n + 3) / 4 * 4;
            return at;
        };
        u = take(T * hp);
        gy = take(bwd ? T * hp : 0);
        x = take(bwd ? T * xp : 0);
        s = take(T * xp);
        full = take(T * fp);
        wstate = take((bwd ? H : pc) * wp);
        wfeat = take((bwd ? P : hc) * cp);
        parts = take(P * 10);          // doubles: sin, cos; sin of half; expm1; exp
        zoh = take(P * (int)(sizeof(ZohTerms) / 4));
        apow = take(4 * pc);
        agg = take(2 * kLsThreads);    // a group's own contribution, or sums
        sums = take(kLsDotGroups * hc > 256 ? kLsDotGroups * hc : 256);   // (kLsThreads)
        gq = take(2 * pc * ((H + 31) / 32));
        flags = take((T + 3) / 4);
        total = o;
    }
};

struct LsArgs {
    int T, H, P, cluster;
    const float2* Lambda; const float* Delta; const float2 *Bc, *Cc;
    const float* D;
    const void* u;
    const uint8_t* done;
    const float2 *x0, *gxT;
    const void* gy;
    float2* x;        // [B, T, P]: kept for the backward pass
    void* out;        // y or du
    float2 *xT, *gx0;
    float2 *part_b, *part_c;  // [B, H, P], or with s
    float2* s;                // [B, T, P]: the weight gradients are left to others
    float2* gA_part;          // [B, P]
    float* dD_part;           // [B, H]; a single sequence: dD itself
    float2 *dLambda, *dB, *dC;   // a single sequence
    float* dDelta;
    WsHeader* hdr;
    bool single;
};

template <int kBytes>
__device__ __forceinline__ void copy_async(float* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(tma::smem_u32(dst)), "l"(src), "n"(kBytes) : "memory");
}
// `rows` rows of n_float2 pairs, `src_pitch` pairs apart.
__device__ __forceinline__ void copy_pairs(float* dst, int pitch, const float2* src, int src_pitch, int rows, int n_pairs) {
    for (int i = threadIdx.x; i < rows * n_pairs; i += kLsThreads) {
        const int r = i / n_pairs, c = i - r * n_pairs;
        copy_async<8>(dst + r * pitch + 2 * c, src + (size_t)r * src_pitch + c);
    }
}
// [rows][cols] of IO (contiguous, cols % 8 == 0) -> fp32 rows of `pitch`.
template <typename IO>
__device__ __forceinline__ void load_rows(float* dst, int pitch, const IO* src, int rows, int cols) {
    const int q = cols / 4;
#pragma unroll 4
    for (int i = threadIdx.x; i < rows * q; i += kLsThreads) {
        const int r = i / q, c = 4 * (i - r * q);
        if constexpr (sizeof(IO) == 4) {
            copy_async<16>(dst + r * pitch + c, src + 4 * (size_t)i);
        } else {
            const uint2 t = ld_stream(reinterpret_cast<const uint2*>(src) + i);
            *reinterpret_cast<float4*>(dst + r * pitch + c) =
                make_float4(__uint_as_float(t.x << 16), __uint_as_float(t.x & 0xffff0000u), __uint_as_float(t.y << 16),
                            __uint_as_float(t.y & 0xffff0000u));
        }
    }
}

// Rows (kR per thread) x columns: out(row, column, sum) after step(accumulator[kR], row pointers, column, k) over k in
// fours, which go to two accumulators in turn (half the chain, and closer to the exact sum); kR = 1 where that many threads
// are there.
__device__ __forceinline__ float add(float a, float b) { return a + b; }
__device__ __forceinline__ float2 add(float2 a, float2 b) { return cadd(a, b); }
template <int kR, typename Acc, typename Step, typename Out>
__device__ __forceinline__ void product_rows(const float* a, int pa, int M, int N, int K, Step step, Out out) {
    for (int i = threadIdx.x; i < (M + kR - 1) / kR * N; i += kLsThreads) {
        const int m0 = i / N * kR, n = i - i / N * N;
        const float* ar[kR];
        Acc acc[kR] = {}, acc2[kR] = {};
#pragma unroll
        for (int r = 0; r < kR; ++r) ar[r] = a + min(m0 + r, M - 1) * pa;
        for (int k = 0; k < K; k += 8) {   // (K is a multiple of 8)
            step(acc, ar, n, k);
            step(acc2, ar, n, k + 4);
        }
#pragma unroll
        for (int r = 0; r < kR; ++r)
            if (m0 + r < M) out(m0 + r, n, add(acc[r], acc2[r]));
    }
}

__device__ __forceinline__ float4 f4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float2 f2(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ bool finite(float2 v) { return isfinite(v.x + v.y); }
__device__ __forceinline__ void cluster_arrive_release() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait_acquire() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

template <typename IO, bool kBwd>
__global__ void __launch_bounds__(kLsThreads)
layer_small_kernel(const __grid_constant__ LsArgs p) {
    extern __shared__ float4 ls_raw[];
    float* sm = reinterpret_cast<float*>(ls_raw);
    const int T = p.T, H = p.H, P = p.P, C = p.cluster, tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const int rank = (int)tc::cluster_ctarank(), b = (int)blockIdx.x / C;
    const int pc = P / C, hc = H / C, p0 = rank * pc, h0 = rank * hc;
    const LsSmem o(T, H, P, C, kBwd);
    float *u = sm + o.u, *gy = sm + o.gy, *x = sm + o.x, *s = sm + o.s, *full = sm + o.full, *wstate = sm + o.wstate, *wfeat = sm + o.wfeat;
    double* parts = reinterpret_cast<double*>(sm + o.parts);
    ZohTerms* zoh = reinterpret_cast<ZohTerms*>(sm + o.zoh);
    float4* apow = reinterpret_cast<float4*>(sm + o.apow);
    float2 *agg = reinterpret_cast<float2*>(sm + o.agg), *gq = reinterpret_cast<float2*>(sm + o.gq);
    float* sums = sm + o.sums;
    uint8_t* flags = reinterpret_cast<uint8_t*>(sm + o.flags);
    float* scale = sm + o.parts + 10 * pc;   // backward: what the states' gradients are divided by, in the room of the other CTAs' parts
    const float2 zero = make_float2(0.f, 0.f);
    if (kBwd && tid < P) scale[tid] = 1.f;
    if (kBwd && tid == 0) scale[P] = 1.f;   // (P <= kLsThreads)
    cluster_arrive_release();   // (every CTA runs before its shared memory is written)
    grid_dep_wait();
    grid_dep_launch();
    if (tid == 0 && blockIdx.x == 0 && !kBwd) p.hdr->status = 0;

    // ---- inputs and parameters are on their way while the functions of the discretisation are evaluated
    load_rows<IO>(u, o.hp, reinterpret_cast<const IO*>(p.u) + (size_t)b * T * H, T, H);
    if (kBwd) {
        load_rows<IO>(gy, o.hp, reinterpret_cast<const IO*>(p.gy) + (size_t)b * T * H, T, H);
        copy_pairs(wstate, o.wp, p.Cc + p0, P, H, pc);
        copy_pairs(x, o.xp, p.x + (size_t)b * T * P + p0, P, T, pc);
        copy_pairs(wfeat, o.cp, p.Bc + h0, H, P, hc);
    } else {
        copy_pairs(wstate, o.wp, p.Bc + (size_t)p0 * H, H, pc, H);
        copy_pairs(wfeat, o.cp, p.Cc + (size_t)h0 * P, P, hc, P);
    }
    for (int i = tid; i < T; i += kLsThreads) flags[i] = p.done ? p.done[(size_t)b * T + i] != 0 : 0;
    for (int q = p0 + (w >> 2) * 32 + lane; q < p0 + pc; q += 32 * (kLsWarps / 4)) {
        const double lr = p.Lambda[q].x, li = p.Lambda[q].y, d = p.Delta[q];
        double* z = parts + 5 * (q - p0);
        if ((w & 3) == 0) sincos(li * d, z, z + 1);
        else if ((w & 3) == 1) z[2] = sin(0.5 * (li * d));
        else if ((w & 3) == 2) z[3] = expm1(lr * d);
        else z[4] = exp(lr * d);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();

    // ---- own states: B u, or g_x = gy conj(C)
    {
        auto out = [&](int t, int q, float2 v) { *reinterpret_cast<float2*>(s + t * o.xp + 2 * q) = v; };
        auto run = [&](auto rows_per_thread) {
            constexpr int kR = decltype(rows_per_thread)::value;
            product_rows<kR, float2>(kBwd ? gy : u, o.hp, T, pc, H, [&](float2(&acc)[kR], const float* (&ar)[kR], int q, int k) {
                float2 wv[4];
                if (kBwd) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) wv[i] = f2(wstate + (k + i) * o.wp + 2 * q), wv[i].y = -wv[i].y;
                } else {
                    const float4 t0 = f4(wstate + q * o.wp + 2 * k), t1 = f4(wstate + q * o.wp + 2 * k + 4);
                    wv[0] = make_float2(t0.x, t0.y), wv[1] = make_float2(t0.z, t0.w);
                    wv[2] = make_float2(t1.x, t1.y), wv[3] = make_float2(t1.z, t1.w);
                }
#pragma unroll
                for (int r = 0; r < kR; ++r) {
                    const float4 v = f4(ar[r] + k);
                    acc[r].x = fmaf(v.w, wv[3].x, fmaf(v.z, wv[2].x, fmaf(v.y, wv[1].x, fmaf(v.x, wv[0].x, acc[r].x))));
                    acc[r].y = fmaf(v.w, wv[3].y, fmaf(v.z, wv[2].y, fmaf(v.y, wv[1].y, fmaf(v.x, wv[0].y, acc[r].y))));
                }
            }, out);
        };
        if (T * pc <= kLsThreads) run(std::integral_constant<int, 1>());
        else run(std::integral_constant<int, 4>());
    }
    const int rows = ls_group_rows(T, pc);
    for (int q = tid; q < pc; q += kLsThreads) {
        const double lr = p.Lambda[p0 + q].x, li = p.Lambda[p0 + q].y, *z = parts + 5 * q, n = lr * lr + li * li;
        ZohTerms t;
        const double er = z[3] * z[1] - 2.0 * z[2] * z[2], ei = z[4] * z[0];
        t.ar = er + 1.0, t.ai = ei;
        t.gr = (er * lr + ei * li) / n, t.gi = (ei * lr - er * li) / n;
        zoh[q] = t;
        double re = 1.0, im = 0.0, br = t.ar, bi = t.ai;   // Abar^rows
        for (int e = rows; e > 0; e >>= 1) {
            if (e & 1) {
                const double r2 = re * br - im * bi;
                im = re * bi + im * br;
                re = r2;
            }
            const double r2 = br * br - bi * bi;
            bi = 2.0 * br * bi;
            br = r2;
        }
        const float hr = (float)re, hi = (float)im;
        apow[q] = make_float4(hr, hi, (float)(re - (double)hr), (float)(im - (double)hi));
    }
    __syncthreads();

    // ---- the recurrence: thread (own state q, group g) has rows [t0, t1)
    const int q = tid % pc, g = tid / pc, t0 = g * rows, t1 = min(T, t0 + rows), n_groups = (T + rows - 1) / rows;
    const bool mine = tid < kLsThreads / pc * pc && t0 < T, last = g == n_groups - 1;
    float2 a = zero, al = zero, aR = zero, aRl = zero, gamma = zero, gammal = zero, first = zero;
    float own_scale = 1.f;
    bool cut = kBwd ? last : g == 0;   // nothing is added to what the first group to be folded ends with
    float* vq = s + 2 * q;
    if (mine) {
        const ZohTerms z = zoh[q];
        a = make_float2((float)z.ar, (float)z.ai);
        al = make_float2((float)(z.ar - (double)a.x), (float)(z.ai - (double)a.y));
        gamma = make_float2((float)z.gr, (float)z.gi);
        gammal = make_float2((float)(z.gr - (double)gamma.x), (float)(z.gi - (double)gamma.y));
        aR = make_float2(apow[q].x, apow[q].y), aRl = make_float2(apow[q].z, apow[q].w);
        if (kBwd) a = cconj(a), al = cconj(al), aR = cconj(aR), aRl = cconj(aRl), gamma = cconj(gamma), gammal = cconj(gammal);
        if (kBwd && fabsf(gamma.x) + fabsf(gamma.y) > 1.f) {   // conj(gamma) s may leave the range of s: B takes a power of two of gamma
            const float by = fminf(2.f * __uint_as_float(__float_as_uint(fabsf(gamma.x) + fabsf(gamma.y)) & 0x7f800000u), 0x1p127f), div = 1.f / by;
            gamma = make_float2(div * gamma.x, div * gamma.y), gammal = make_float2(div * gammal.x, div * gammal.y);
            own_scale = by;
        }
        const float2* from = kBwd ? p.gxT : p.x0;
        if (cut && from) first = from[(size_t)b * P + p0 + q];
        float2 e = first;
        if (!kBwd) {
            float2 dropped = zero;
            for (int t = t0; t < t1; ++t) {
                const float2 v = cfma2(gamma, gammal, f2(vq + t * o.xp), zero);
                *reinterpret_cast<float2*>(vq + t * o.xp) = v;
                if (flags[t]) dropped = cadd(dropped, e), e = zero, cut = true;
                e = cfma2(a, al, e, v);
            }
            if (!finite(cadd(dropped, e))) {   // B u may have left the range of fp32, which gamma B u need not have done
                e = first;
#pragma unroll 1
                for (int t = t0; t < t1; ++t) {
                    float2 v = f2(vq + t * o.xp);
                    if (!finite(v)) {
                        v = zero;
#pragma unroll 1
                        for (int h = 0; h < H; ++h) {
                            const float2 bg = cfma2(gamma, gammal, f2(wstate + q * o.wp + 2 * h), zero);
                            v.x = fmaf(u[t * o.hp + h], bg.x, v.x);
                            v.y = fmaf(u[t * o.hp + h], bg.y, v.y);
                        }
                        *reinterpret_cast<float2*>(vq + t * o.xp) = v;
                    }
                    e = cfma2(a, al, flags[t] ? zero : e, v);
                }
            }
        } else {
            e = cadd(f2(vq + (t1 - 1) * o.xp), e);   // (the state's gradient s; conj(Abar) s, which it hands on, is rounded once, at the end)
            cut = cut || flags[t1 - 1];
            for (int t = t1 - 2; t >= t0; --t) {
                e = cfma2(a, al, flags[t + 1] ? zero : e, f2(vq + t * o.xp));
                cut = cut || flags[t];
            }
            e = flags[t0] ? zero : cfma2(a, al, e, zero);
        }
        agg[tid] = e;
        sums[tid] = cut ? 1.f : 0.f;
    }
    __syncthreads();
    cluster_wait_acquire();
    float2 gA = zero;
    if (mine) {
        float2 c = first;
        auto join = [&](int j) {
            const float2 e = agg[j * pc + q];
            c = sums[j * pc + q] != 0.f ? e : cfma2(aR, aRl, c, e);
        };
        if (!kBwd) {
#pragma unroll 4
            for (int j = 0; j < g; ++j) join(j);
        } else {
#pragma unroll 4
            for (int j = n_groups - 1; j > g; --j) join(j);
        }
        const uint32_t to = tma::smem_u32(full) + 8u * (uint32_t)(p0 + q);
        auto share = [&](int t, float2 v) {
            for (int r = 0; r < C; ++r)
                asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(tc::map_to_cta(to + 4u * (uint32_t)(t * o.fp), (uint32_t)r)),
                             "f"(v.x), "f"(v.y) : "memory");
        };
        if (!kBwd) {
            for (int t = t0; t < t1; ++t) {
                if (flags[t]) c = zero;
                c = cfma2(a, al, c, f2(vq + t * o.xp));
                share(t, c);
                p.x[((size_t)b * T + t) * P + p0 + q] = c;
            }
            if (t1 == T && p.xT) p.xT[(size_t)b * P + p0 + q] = c;
        } else {
            const float* xq = x + 2 * q;
            for (int t = t1 - 1; t >= t0; --t) {
                const float2 v = f2(vq + t * o.xp);
                c = t == t1 - 1 ? cadd(v, c) : cfma2(a, al, flags[t + 1] ? zero : c, v);
                *reinterpret_cast<float2*>(vq + t * o.xp) = c;
                share(t, cfma2(gamma, gammal, c, zero));
                if (p.s) p.s[((size_t)b * T + t) * P + p0 + q] = c;
                if (!flags[t]) {
                    const float2 before = t > 0 ? f2(xq + (t - 1) * o.xp) : (p.x0 ? p.x0[(size_t)b * P + p0 + q] : zero);
                    gA = cfma(c, cconj(before), gA);
                }
            }
            c = flags[t0] ? zero : cfma2(a, al, c, zero);
            if (t0 == 0 && p.gx0) p.gx0[(size_t)b * P + p0 + q] = c;
            if (t0 == 0 && own_scale != 1.f)
                for (int r = 0; r < C; ++r)
                    for (const int i : {p0 + q, P})   // (entry P: there are any)
                        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(tc::map_to_cta(tma::smem_u32(scale + i), (uint32_t)r)), "f"(own_scale)
                                     : "memory");
        }
    }
    cluster_arrive_release();

    if (kBwd) {
        // ---- of the own states, while the others finish: gBbar = s^T u, dC = gy^T conj(x), and the sums of gAbar
        __syncthreads();
        if (mine) agg[tid] = gA;
        const int chunks = (H + 31) / 32;
        for (int i = w; i < (p.s ? 0 : 2 * pc * chunks); i += kLsWarps) {   // a warp: one state, 32 features
            const bool is_c = i >= pc * chunks;
            const int j = is_c ? i - pc * chunks : i, st = j / chunks, h = (j - st * chunks) * 32 + lane;
            const float *av = (is_c ? gy : u) + min(h, H - 1), *bv = (is_c ? x : s) + 2 * st;
            float2 acc = zero;
            auto row = [&](int t, float2& to) {
                const float v = av[t * o.hp];
                const float2 z = f2(bv + t * o.xp);
                to.x = fmaf(v, z.x, to.x);
                to.y = fmaf(v, z.y, to.y);
            };
            int t = 0;
#pragma unroll 2
            for (; t + kLsChain <= T; t += kLsChain) {
                float2 part = zero;
#pragma unroll
                for (int i = 0; i < kLsChain; ++i) row(t + i, part);
                acc = cadd(acc, part);
            }
            for (; t < T; ++t) row(t, acc);
            const size_t e_c = (size_t)h * P + p0 + st;
            if (!p.single) {
                if (h < H) ((is_c ? p.part_c : p.part_b) + (size_t)b * H * P)[e_c] = acc;
            } else if (is_c) {
                if (h < H) p.dC[e_c] = cconj(acc);
            } else {
                float2 gg = zero;
                if (h < H) {
                    const size_t e = (size_t)(p0 + st) * H + h;
                    p.dB[e] = cmul(make_float2((float)zoh[st].gr, -(float)zoh[st].gi), acc);
                    gg = cmul(cconj(p.Bc[e]), acc);
                }
#pragma unroll
                for (int m = 16; m > 0; m >>= 1) {
                    gg.x += __shfl_xor_sync(0xffffffffu, gg.x, m);
                    gg.y += __shfl_xor_sync(0xffffffffu, gg.y, m);
                }
                if (lane == 0) gq[j] = gg;
            }
        }
        // dD of the own features
        for (int i = tid; i < hc * kLsDotGroups; i += kLsThreads) {
            const int grp = i / hc, h = h0 + i - grp * hc;
            float d = 0.f;
            int t = grp;
            for (; t + kLsDotGroups * (kLsChain - 1) < T; t += kLsDotGroups * kLsChain) {
                float part = 0.f;
#pragma unroll
                for (int j = 0; j < kLsChain; ++j) part = fmaf(gy[(t + kLsDotGroups * j) * o.hp + h], u[(t + kLsDotGroups * j) * o.hp + h], part);
                d += part;
            }
            for (; t < T; t += kLsDotGroups) d = fmaf(gy[t * o.hp + h], u[t * o.hp + h], d);
            sums[i] = d;
        }
        __syncthreads();
        if (tid < hc) {
            float d = 0.f;
#pragma unroll
            for (int i = 0; i < kLsDotGroups; ++i) d += sums[i * hc + tid];
            p.dD_part[(size_t)b * H + h0 + tid] = d;
        }
        const int st = kLsThreads - 1 - tid;   // (other warps than dD's)
        if (st < pc) {
            double ar = 0.0, ai = 0.0, gr = 0.0, gi = 0.0;
#pragma unroll 4
            for (int j = 0; j < n_groups; ++j) ar += (double)agg[j * pc + st].x, ai += (double)agg[j * pc + st].y;
            if (p.single) {
                for (int j = 0; j < chunks; ++j) gr += (double)gq[st * chunks + j].x, gi += (double)gq[st * chunks + j].y;
                zoh_adjoint(zoh[st], p.Lambda[p0 + st], p.Delta[p0 + st], ar, ai, gr, gi, p.dLambda[p0 + st], p.dDelta[p0 + st]);
            } else {
                p.gA_part[(size_t)b * P + p0 + st] = make_float2((float)ar, (float)ai);
            }
        }
    }
    // ---- own features: y = Re(C x) + D u, or du = Re(conj(B) conj(gamma) s) + D gy
    cluster_wait_acquire();
    if (kBwd && scale[P] != 1.f) {
        for (int i = tid; i < P * hc; i += kLsThreads) {
            float2* w2 = reinterpret_cast<float2*>(wfeat + i / hc * o.cp) + i % hc;
            *w2 = make_float2(scale[i / hc] * w2->x, scale[i / hc] * w2->y);
        }
        __syncthreads();
    }
    {
        const float* skip = kBwd ? gy : u;
        auto out = [&](int t, int h, float v) {
            reinterpret_cast<IO*>(p.out)[((size_t)b * T + t) * H + h0 + h] = from_f32<IO>(fmaf(p.D[h0 + h], skip[t * o.hp + h0 + h], v));
        };
        auto run = [&](auto rows_per_thread) {
            constexpr int kR = decltype(rows_per_thread)::value;
            product_rows<kR, float>(full, o.fp, T, hc, 2 * P, [&](float(&acc)[kR], const float* (&ar)[kR], int h, int k) {
                float4 wv;
                if (kBwd) {
                    const float2 t0 = f2(wfeat + (k / 2) * o.cp + 2 * h), t1 = f2(wfeat + (k / 2 + 1) * o.cp + 2 * h);
                    wv = make_float4(t0.x, t0.y, t1.x, t1.y);
                } else {
                    wv = f4(wfeat + h * o.cp + k);
                    wv.y = -wv.y, wv.w = -wv.w;
                }
#pragma unroll
                for (int r = 0; r < kR; ++r) {
                    const float4 v = f4(ar[r] + k);
                    acc[r] = fmaf(v.w, wv.w, fmaf(v.z, wv.z, fmaf(v.y, wv.y, fmaf(v.x, wv.x, acc[r]))));
                }
            }, out);
        };
        if (T * hc <= kLsThreads) run(std::integral_constant<int, 1>());
        else run(std::integral_constant<int, 4>());
    }
}

// us per forward and backward pass in a graph (forward alone), ten launches -> this (B x T, H, P): 1 x 64, 32, 16 30.9 -> 15.5 (eager
// 36.5 -> 15.9), 1 x 1, 16, 8 17.2 -> 11.2 (6.2 -> 4.7), 1 x 512, 16, 16 41.2 -> 34.9, 14 x 64, 72, 104 62.5 -> 47.6 (25.0 -> 13.9), 4 x 128, 96, 40 47.3 -> 45.3
// (123 K multiply-adds a projection and CTA: the limit is 131 K);  clusters of 4: 32 x 64, 40, 40 44.8 -> 45.7 (15.4 -> 9.7), 20 x 128, 32, 64
// 55.4 -> 45.2, 32 x 261, 24, 8 107 -> 38.5 (51.4 -> 10.4);  with the weight gradients as products: 32 x 10, 184, 128 73.9 -> 47.7 (32.5 -> 14.9),
// 14 x 16, 192, 128 71.7 -> 41.1 (31.2 -> 11.6), 4 x 2, 208, 256 92.5 -> 29.8 (43.1 -> 9.9), 15 x 13, 24, 24 in bf16 34.5 -> 24.6 (12.9 -> 6.1).  Of 135 shapes
// none is slower by more than 2 %, and the forward pass alone never.  Where the clusters do not run in one round: 16 x 128, 64, 64 (clusters of 8) 53.9 -> 73.2, 36 x 64, 64, 64 (of 4) 55.7 -> 58.6.  One CTA per sequence, 148 x 64, 32, 16: 59.6 -> 76.0.
int ls_cluster(int B, int T, int H, int P) {
    if (P > kLsThreads || T > 512 || H > 256 || B > 32) return 0;
    const int c = B <= 14 ? 8 : 4;
    return (long long)T * H * 2 * P <= (long long)c << 17 && (size_t)LsSmem(T, H, P, c, true).total * 4 <= kLsSmemMax ? c : 0;
}

// Whether the device runs that many clusters at the same time (of the backward pass, which takes more shared memory and registers;
// asked for in steps of 40 KB; no device: a B200 is planned for).
template <typename IO>
bool ls_resident(int cluster, int B, int T, int H, int P) {
    const void* kern = reinterpret_cast<const void*>(layer_small_kernel<IO, true>);
    constexpr size_t kStep = 40 * 1024;
    static_assert(kLsSmemMax % kStep == 0, "steps of shared memory");
    const size_t smem = ((size_t)LsSmem(T, H, P, cluster, true).total * 4 + kStep - 1) / kStep * kStep;
    const int n = resident_clusters(kern, cluster, smem, kLsThreads);
    return n < 0 || n >= B;
}

template <typename IO, bool kBwd>
int launch_ls(LsArgs p, int B, cudaStream_t st) {
    auto kern = layer_small_kernel<IO, kBwd>;
    if (!set_max_dynamic_smem(reinterpret_cast<const void*>(kern), kLsSmemMax)) return SSM_ERR_CUDA;
    p.cluster = ls_cluster(B, p.T, p.H, p.P);
    p.single = B == 1;
    count_launch();
    const size_t smem = (size_t)LsSmem(p.T, p.H, p.P, p.cluster, kBwd).total * 4;
    return launch_dep_cluster(kern, (unsigned)p.cluster, (unsigned)(B * p.cluster), kLsThreads, smem, st, p) ? SSM_OK : SSM_ERR_CUDA;
}

}  // namespace

int layer_small_cluster(int B, int T, int H, int P, bool bf16) {
    const int c = ls_cluster(B, T, H, P);
    return c && (bf16 ? ls_resident<__nv_bfloat16>(c, B, T, H, P) : ls_resident<float>(c, B, T, H, P)) ? c : 0;
}

int launch_layer_small_fwd(const LayerSmall& g, cudaStream_t st) {
    LsArgs p{};
    p.T = g.T, p.H = g.H, p.P = g.P, p.Lambda = g.Lambda, p.Delta = g.Delta, p.Bc = g.Bc, p.Cc = g.Cc, p.D = g.D, p.u = g.u;
    p.done = g.done, p.x0 = g.x0, p.x = g.x, p.out = g.out, p.xT = g.xT, p.hdr = g.hdr;
    return g.bf16 ? launch_ls<__nv_bfloat16, false>(p, g.B, st) : launch_ls<float, false>(p, g.B, st);
}

int launch_layer_small_bwd(const LayerSmall& g, const GradTail& tail, float2* s, float2* gA_part, float* dD_part, cudaStream_t st) {
    LsArgs p{};
    p.T = g.T, p.H = g.H, p.P = g.P, p.Lambda = g.Lambda, p.Delta = g.Delta, p.Bc = g.Bc, p.Cc = g.Cc, p.D = g.D, p.u = g.u;
    p.done = g.done, p.x0 = g.x0, p.gxT = g.gxT, p.gy = g.gy, p.x = g.x, p.out = g.out, p.gx0 = g.gx0;
    p.part_b = (float2*)tail.part_b, p.part_c = (float2*)tail.part_c, p.s = s, p.gA_part = gA_part;
    p.dD_part = g.B == 1 ? tail.sum_out[0] : dD_part;
    p.dLambda = tail.dLambda, p.dDelta = tail.dDelta, p.dB = tail.dB, p.dC = tail.dC;
    return g.bf16 ? launch_ls<__nv_bfloat16, true>(p, g.B, st) : launch_ls<float, true>(p, g.B, st);
}

}  // namespace ssm
