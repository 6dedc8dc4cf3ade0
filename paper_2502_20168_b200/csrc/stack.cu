// Wrapper of the stacked sequence model: out = LayerNorm(u + GELU(v)) * w + b with v = SSM(u),
// forward and backward.  A warp per row of up to 1024 features, a CTA per wider row; arithmetic in fp32.  Only the stack's own
// input, output and their gradients are in the I/O type; what passes between the layers (v, the
// layer inputs, the gradients handed down) is fp32, hence the separate element types below.
#include "kernels.h"

namespace ssm {

constexpr int kRowThreads = 128;
constexpr float kLnEps = 1e-5f;

__device__ __forceinline__ float gelu_f(float v) { return 0.5f * v * (1.f + erff(v * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float v) {
    return 0.5f * (1.f + erff(v * 0.70710678118654752f)) + v * 0.3989422804014327f * expf(-0.5f * v * v);
}

// Sum over the CTA; every thread gets the result.
__device__ __forceinline__ float block_sum(float v, float* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < kRowThreads / 32; ++w) t += red[w];
    return t;
}

// TI: type of the layer input u; TO: type of out.
template <typename TI, typename TO>
__global__ void __launch_bounds__(kRowThreads)
stack_fwd_kernel(int H, const TI* u, const float* v, const float* w,
                 const float* b, TO* out, float* mu_out,
                 float* rstd_out) {
    grid_dep_wait();
    grid_dep_launch();
    __shared__ float red[kRowThreads / 32];
    const size_t row = blockIdx.x;
    const TI* ur = u + row * H;
    const float* vr = v + row * H;
    float sum = 0.f;
    for (int h = threadIdx.x; h < H; h += kRowThreads) sum += to_f32<TI>(ur[h]) + gelu_f(vr[h]);
    const float mu = block_sum(sum, red) / (float)H;
    float sq = 0.f;
    for (int h = threadIdx.x; h < H; h += kRowThreads) {
        const float z = to_f32<TI>(ur[h]) + gelu_f(vr[h]) - mu;
        sq = fmaf(z, z, sq);
    }
    const float rstd = rsqrtf(block_sum(sq, red) / (float)H + kLnEps);
    for (int h = threadIdx.x; h < H; h += kRowThreads) {
        const float z = to_f32<TI>(ur[h]) + gelu_f(vr[h]);
        out[row * H + h] = from_f32<TO>(fmaf((z - mu) * rstd, w[h], b[h]));
    }
    if (threadIdx.x == 0) {
        mu_out[row] = mu;
        rstd_out[row] = rstd;
    }
}

// gz = LayerNorm'(g) (the gradient of the residual branch);  gv = gz * GELU'(v) (what the SSM
// backward takes).  TG: type of the incoming gradient g; TI: type of the layer input u.
template <typename TG, typename TI>
__global__ void __launch_bounds__(kRowThreads)
stack_bwd_kernel(int H, const TG* g, const TI* u, const float* v,
                 const float* w, const float* mu_in, const float* rstd_in,
                 float* gz_out, float* gv) {
    grid_dep_wait();
    grid_dep_launch();
    __shared__ float red[kRowThreads / 32];
    const size_t row = blockIdx.x;
    const TG* gr = g + row * H;
    const TI* ur = u + row * H;
    const float* vr = v + row * H;
    const float mu = mu_in[row], rstd = rstd_in[row];
    float s1 = 0.f, s2 = 0.f;
    for (int h = threadIdx.x; h < H; h += kRowThreads) {
        const float zhat = (to_f32<TI>(ur[h]) + gelu_f(vr[h]) - mu) * rstd;
        const float gh = to_f32<TG>(gr[h]) * w[h];
        s1 += gh;
        s2 = fmaf(gh, zhat, s2);
    }
    const float m1 = block_sum(s1, red) / (float)H;
    const float m2 = block_sum(s2, red) / (float)H;
    for (int h = threadIdx.x; h < H; h += kRowThreads) {
        const float vv = vr[h];
        const float zhat = (to_f32<TI>(ur[h]) + gelu_f(vv) - mu) * rstd;
        const float gz = rstd * (to_f32<TG>(gr[h]) * w[h] - m1 - zhat * m2);
        gz_out[row * H + h] = gz;
        gv[row * H + h] = gz * gelu_grad_f(vv);
    }
}

// part_w[grp, h] = sum over the group's rows of g * zhat;  part_b[grp, h] = sum of g.
constexpr int kLnGradRows = 64;
template <typename TG, typename TI>
__global__ void __launch_bounds__(256)
ln_param_grad_kernel(int M, int H, const TG* g, const TI* u, const float* v,
                     const float* mu_in, const float* rstd_in,
                     float* part_w, float* part_b) {
    grid_dep_wait();
    grid_dep_launch();
    __shared__ float sw[8][33], sb[8][33];
    const int h = blockIdx.y * 32 + threadIdx.x;
    const int r0 = blockIdx.x * kLnGradRows, r1 = min(M, r0 + kLnGradRows);   // row groups along x (no 65535 limit)
    float aw = 0.f, ab = 0.f;
    if (h < H)
        for (int r = r0 + threadIdx.y; r < r1; r += 8) {
            const size_t i = (size_t)r * H + h;
            const float zhat = (to_f32<TI>(u[i]) + gelu_f(v[i]) - mu_in[r]) * rstd_in[r];
            const float gg = to_f32<TG>(g[i]);
            aw = fmaf(gg, zhat, aw);
            ab += gg;
        }
    sw[threadIdx.y][threadIdx.x] = aw;
    sb[threadIdx.y][threadIdx.x] = ab;
    __syncthreads();
    if (threadIdx.y == 0 && h < H) {
        float tw = 0.f, tb = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            tw += sw[i][threadIdx.x];
            tb += sb[i][threadIdx.x];
        }
        part_w[(size_t)blockIdx.x * H + h] = tw;
        part_b[(size_t)blockIdx.x * H + h] = tb;
    }
}

// ---- rows of up to 1024 features: one warp per row ------------------------------------------------
// The row stays in registers (a lane owns the groups of 4 features lane, lane + 32, ...), so u, v and g are read once
// and GELU is evaluated once, where the kernels above read the row two or three times.  The backward kernel also keeps
// the sums for dw and db of its features over the rows a warp takes and leaves one row of partial sums per CTA, which
// used to be a second pass over g, u and v and two column sums.  1024 rows x 512: forward 4.8 -> 3.0 us, backward with
// the parameter sums 15.6 (four launches) -> 4.6 (one).  Latency-bound at such sizes, HBM-bound from 10^5 rows on.
constexpr int kLnWarps = 8;
template <typename T>
__device__ __forceinline__ float4 ln_load4(const T* p);
template <>
__device__ __forceinline__ float4 ln_load4<float>(const float* p) { return *reinterpret_cast<const float4*>(p); }
template <>
__device__ __forceinline__ float4 ln_load4<__nv_bfloat16>(const __nv_bfloat16* p) {
    const uint2 r = *reinterpret_cast<const uint2*>(p);
    return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xffff0000u), __uint_as_float(r.y << 16),
                       __uint_as_float(r.y & 0xffff0000u));
}
__device__ __forceinline__ void ln_store4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void ln_store4(__nv_bfloat16* p, float4 v) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
    *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <int NI, typename TI, typename TO>
__global__ void __launch_bounds__(32 * kLnWarps)
stack_fwd_row_kernel(int M, int H, const TI* u, const float* v, const float* w, const float* b, TO* out, float* mu_out,
                     float* rstd_out) {
    grid_dep_wait();
    grid_dep_launch();
    const int lane = threadIdx.x & 31;
    const float inv = 1.f / (float)H;
    for (int row = blockIdx.x * kLnWarps + (threadIdx.x >> 5); row < M; row += gridDim.x * kLnWarps) {
        float4 z[NI];
        float sum = 0.f;
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const int h = 4 * (lane + 32 * i);
            z[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (h < H) {
                const float4 a = ln_load4<TI>(u + (size_t)row * H + h), x = ln_load4<float>(v + (size_t)row * H + h);
                z[i] = make_float4(a.x + gelu_f(x.x), a.y + gelu_f(x.y), a.z + gelu_f(x.z), a.w + gelu_f(x.w));
                sum += (z[i].x + z[i].y) + (z[i].z + z[i].w);
            }
        }
        const float mu = warp_sum(sum) * inv;
        float sq = 0.f;
#pragma unroll
        for (int i = 0; i < NI; ++i)
            if (4 * (lane + 32 * i) < H) {
                z[i].x -= mu, z[i].y -= mu, z[i].z -= mu, z[i].w -= mu;
                sq = fmaf(z[i].x, z[i].x, fmaf(z[i].y, z[i].y, fmaf(z[i].z, z[i].z, fmaf(z[i].w, z[i].w, sq))));
            }
        const float rstd = rsqrtf(warp_sum(sq) * inv + kLnEps);
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const int h = 4 * (lane + 32 * i);
            if (h < H) {
                const float4 ww = ln_load4<float>(w + h), bb = ln_load4<float>(b + h);
                ln_store4(out + (size_t)row * H + h, make_float4(fmaf(z[i].x * rstd, ww.x, bb.x), fmaf(z[i].y * rstd, ww.y, bb.y),
                                                                 fmaf(z[i].z * rstd, ww.z, bb.z), fmaf(z[i].w * rstd, ww.w, bb.w)));
            }
        }
        if (lane == 0) {
            mu_out[row] = mu;
            rstd_out[row] = rstd;
        }
    }
}

template <int NI, typename TG, typename TI>
__global__ void __launch_bounds__(32 * kLnWarps)
stack_bwd_row_kernel(int M, int H, const TG* g, const TI* u, const float* v, const float* w, const float* mu_in,
                     const float* rstd_in, float* gz_out, float* gv, float* part_w, float* part_b) {
    __shared__ float4 red[kLnWarps][32];
    grid_dep_wait();
    grid_dep_launch();
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const float inv = 1.f / (float)H;
    float4 dw[NI], db[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) dw[i] = db[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int row = blockIdx.x * kLnWarps + wp; row < M; row += gridDim.x * kLnWarps) {
        const float mu = mu_in[row], rstd = rstd_in[row];
        float4 zh[NI], gh[NI], gd[NI];   // normalised row, g w, GELU'(v)
        float s1 = 0.f, s2 = 0.f;
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const int h = 4 * (lane + 32 * i);
            zh[i] = gh[i] = gd[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (h < H) {
                const float4 a = ln_load4<TI>(u + (size_t)row * H + h), x = ln_load4<float>(v + (size_t)row * H + h);
                const float4 gg = ln_load4<TG>(g + (size_t)row * H + h), ww = ln_load4<float>(w + h);
                zh[i] = make_float4((a.x + gelu_f(x.x) - mu) * rstd, (a.y + gelu_f(x.y) - mu) * rstd,
                                    (a.z + gelu_f(x.z) - mu) * rstd, (a.w + gelu_f(x.w) - mu) * rstd);
                gd[i] = make_float4(gelu_grad_f(x.x), gelu_grad_f(x.y), gelu_grad_f(x.z), gelu_grad_f(x.w));
                gh[i] = make_float4(gg.x * ww.x, gg.y * ww.y, gg.z * ww.z, gg.w * ww.w);
                dw[i].x = fmaf(gg.x, zh[i].x, dw[i].x), dw[i].y = fmaf(gg.y, zh[i].y, dw[i].y);
                dw[i].z = fmaf(gg.z, zh[i].z, dw[i].z), dw[i].w = fmaf(gg.w, zh[i].w, dw[i].w);
                db[i].x += gg.x, db[i].y += gg.y, db[i].z += gg.z, db[i].w += gg.w;
                s1 += (gh[i].x + gh[i].y) + (gh[i].z + gh[i].w);
                s2 = fmaf(gh[i].x, zh[i].x, fmaf(gh[i].y, zh[i].y, fmaf(gh[i].z, zh[i].z, fmaf(gh[i].w, zh[i].w, s2))));
            }
        }
        const float m1 = warp_sum(s1) * inv, m2 = warp_sum(s2) * inv;
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const int h = 4 * (lane + 32 * i);
            if (h < H) {
                const float4 gz = make_float4(rstd * (gh[i].x - m1 - zh[i].x * m2), rstd * (gh[i].y - m1 - zh[i].y * m2),
                                              rstd * (gh[i].z - m1 - zh[i].z * m2), rstd * (gh[i].w - m1 - zh[i].w * m2));
                ln_store4(gz_out + (size_t)row * H + h, gz);
                ln_store4(gv + (size_t)row * H + h, make_float4(gz.x * gd[i].x, gz.y * gd[i].y, gz.z * gd[i].z, gz.w * gd[i].w));
            }
        }
    }
    // the CTA's warps added in a fixed order: one row of partial sums per CTA
#pragma unroll
    for (int i = 0; i < 2 * NI; ++i) {
        __syncthreads();
        red[wp][lane] = i < NI ? dw[i % NI] : db[i % NI];
        __syncthreads();
        const int h = 4 * (lane + 32 * (i % NI));
        if (wp == 0 && h < H) {
            float4 t = red[0][lane];
#pragma unroll
            for (int q = 1; q < kLnWarps; ++q) {
                const float4 x = red[q][lane];
                t.x += x.x, t.y += x.y, t.z += x.z, t.w += x.w;
            }
            ln_store4((i < NI ? part_w : part_b) + (size_t)blockIdx.x * H + h, t);
        }
    }
}

// CTAs of the row kernels: enough to give every warp a row, at most two per SM; in the backward pass as many such rounds
// as it takes to leave a warp no more than kLnRows rows, since its sums for dw and db are chains of fp32 additions
// (1048576 x 128 in one round, 443 rows a warp: dw 4.2e-7 off, 1.5e-7 with 16; 591 / 516 us; 64000 x 512 134 / 142).
constexpr int kLnRows = 16;
static int ln_row_blocks(int M, bool bwd) {
    const int need = (M + kLnWarps - 1) / kLnWarps, round = 2 * device_sm_count();
    if (need <= round) return need;
    const int least = bwd ? (M + kLnWarps * kLnRows - 1) / (kLnWarps * kLnRows) : 1;
    return (least + round - 1) / round * round;
}
static bool ln_by_rows(int H) { return H <= 1024; }

static inline int ln_groups(int M) { return (M + kLnGradRows - 1) / kLnGradRows; }

// Rows of partial sums of dw and db (each) that launch_stack_bwd leaves, and the floats they and its scratch take.
static int stack_part_rows(int M, int H) { return ln_by_rows(H) ? ln_row_blocks(M, true) : ln_groups(M); }
size_t stack_tmp_floats(int M, int H) {
    const int g = stack_part_rows(M, H);
    return 2 * ((size_t)g * H + colsum_tmp_floats(g, H));
}

template <typename TI, typename TO>
static void stack_fwd_launch(int M, int H, const void* u, const float* v, const float* w, const float* b, void* out, float* mu,
                             float* rstd, cudaStream_t st) {
    const int blocks = ln_row_blocks(M, false), threads = 32 * kLnWarps;
    const TI* uu = (const TI*)u;
    TO* oo = (TO*)out;
    if (H <= 256) launch_dep(stack_fwd_row_kernel<2, TI, TO>, blocks, threads, 0, st, M, H, uu, v, w, b, oo, mu, rstd);
    else if (H <= 512) launch_dep(stack_fwd_row_kernel<4, TI, TO>, blocks, threads, 0, st, M, H, uu, v, w, b, oo, mu, rstd);
    else if (ln_by_rows(H)) launch_dep(stack_fwd_row_kernel<8, TI, TO>, blocks, threads, 0, st, M, H, uu, v, w, b, oo, mu, rstd);
    else launch_dep(stack_fwd_kernel<TI, TO>, M, kRowThreads, 0, st, H, uu, v, w, b, oo, mu, rstd);
}

void launch_stack_fwd(bool u_bf16, bool out_bf16, int M, int H, const void* u, const float* v, const float* w,
                      const float* b, void* out, float* mu, float* rstd, cudaStream_t st) {
    using bf = __nv_bfloat16;
    count_launch();
    if (u_bf16 && out_bf16) stack_fwd_launch<bf, bf>(M, H, u, v, w, b, out, mu, rstd, st);
    else if (u_bf16) stack_fwd_launch<bf, float>(M, H, u, v, w, b, out, mu, rstd, st);
    else if (out_bf16) stack_fwd_launch<float, bf>(M, H, u, v, w, b, out, mu, rstd, st);
    else stack_fwd_launch<float, float>(M, H, u, v, w, b, out, mu, rstd, st);
}

template <typename TG, typename TI>
static void stack_bwd_launch(int M, int H, const void* g, const void* u, const float* v, const float* w, const float* mu,
                             const float* rstd, float* gz, float* gv, float* part_w, float* part_b, cudaStream_t st) {
    const TG* gg = (const TG*)g;
    const TI* uu = (const TI*)u;
    const int blocks = ln_row_blocks(M, true), threads = 32 * kLnWarps;
    count_launch(ln_by_rows(H) ? 1 : 2);
    if (H <= 256) launch_dep(stack_bwd_row_kernel<2, TG, TI>, blocks, threads, 0, st, M, H, gg, uu, v, w, mu, rstd, gz, gv, part_w, part_b);
    else if (H <= 512) launch_dep(stack_bwd_row_kernel<4, TG, TI>, blocks, threads, 0, st, M, H, gg, uu, v, w, mu, rstd, gz, gv, part_w, part_b);
    else if (ln_by_rows(H)) launch_dep(stack_bwd_row_kernel<8, TG, TI>, blocks, threads, 0, st, M, H, gg, uu, v, w, mu, rstd, gz, gv, part_w, part_b);
    else {
        dim3 blk(32, 8), grid(ln_groups(M), (H + 31) / 32);
        launch_dep(stack_bwd_kernel<TG, TI>, M, kRowThreads, 0, st, H, gg, uu, v, w, mu, rstd, gz, gv);
        launch_dep(ln_param_grad_kernel<TG, TI>, grid, blk, 0, st, M, H, gg, uu, v, mu, rstd, part_w, part_b);
    }
}

void launch_stack_bwd(bool g_bf16, bool u_bf16, int M, int H, const void* g, const void* u, const float* v,
                      const float* w, const float* mu, const float* rstd, float* gz, float* gv, float* tmp,
                      const float** dw_part, const float** db_part, int* part_rows, cudaStream_t st) {
    using bf = __nv_bfloat16;
    const int rows = stack_part_rows(M, H);
    const size_t half = stack_tmp_floats(M, H) / 2;
    float *part_w = tmp, *part_b = tmp + half;
    if (g_bf16 && u_bf16) stack_bwd_launch<bf, bf>(M, H, g, u, v, w, mu, rstd, gz, gv, part_w, part_b, st);
    else if (g_bf16) stack_bwd_launch<bf, float>(M, H, g, u, v, w, mu, rstd, gz, gv, part_w, part_b, st);
    else if (u_bf16) stack_bwd_launch<float, bf>(M, H, g, u, v, w, mu, rstd, gz, gv, part_w, part_b, st);
    else stack_bwd_launch<float, float>(M, H, g, u, v, w, mu, rstd, gz, gv, part_w, part_b, st);
    *dw_part = launch_reduce_rows(part_w, rows, H, part_w + (size_t)rows * H, kMaxPartialRows, part_rows, st);
    *db_part = launch_reduce_rows(part_b, rows, H, part_b + (size_t)rows * H, kMaxPartialRows, part_rows, st);
}

}  // namespace ssm
