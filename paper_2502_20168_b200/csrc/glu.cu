// Half-GLU gate of the S5 sequence layer (Appendix "S5 Sequence Layer"):
//   x1 = GELU(v),  z = W^T x1 (row by row: z[m, j] = sum_i x1[m, i] W[i, j]),  out = v * sigmoid(z)
// and its backward.  The two H x H contractions per direction and the weight gradient run on the
// projection GEMMs of this library; this file holds what surrounds them: operand packing and
// the elementwise passes (each streams [B*T, H] arrays once: HBM-bound).
#include "kernels.h"

namespace ssm {
namespace {

__device__ __forceinline__ float gelu_f(float v) { return 0.5f * v * (1.f + erff(v * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float v) {
    return 0.5f * (1.f + erff(v * 0.70710678118654752f)) + v * 0.3989422804014327f * expf(-0.5f * v * v);
}

constexpr int kThreads = 256;
inline int blocks_for(size_t n) {
    const size_t b = (n + kThreads - 1) / kThreads;
    return (int)(b < 148 * 32 ? b : 148 * 32);
}

// The elementwise passes work on groups of 8 consecutive elements (H is a multiple of 8): 16- or
// 32-byte accesses per array and thread.
struct F8 {
    float x[8];
};
template <typename T> __device__ __forceinline__ F8 load8(const T* p);
template <> __device__ __forceinline__ F8 load8<float>(const float* p) {
    const float4 a = ld_stream(reinterpret_cast<const float4*>(p)), b = ld_stream(reinterpret_cast<const float4*>(p) + 1);
    return F8{{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}};
}
template <> __device__ __forceinline__ F8 load8<__nv_bfloat16>(const __nv_bfloat16* p) {
    const uint4 r = ld_stream(reinterpret_cast<const uint4*>(p));
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&r);
    F8 o;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 f = __bfloat1622float2(h[i]);
        o.x[2 * i] = f.x;
        o.x[2 * i + 1] = f.y;
    }
    return o;
}
template <typename T> __device__ __forceinline__ void store8(T* p, const F8& v);
template <> __device__ __forceinline__ void store8<float>(float* p, const F8& v) {
    reinterpret_cast<float4*>(p)[0] = make_float4(v.x[0], v.x[1], v.x[2], v.x[3]);
    reinterpret_cast<float4*>(p)[1] = make_float4(v.x[4], v.x[5], v.x[6], v.x[7]);
}
template <> __device__ __forceinline__ void store8<__nv_bfloat16>(__nv_bfloat16* p, const F8& v) {
    uint4 r;
    __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&r);
#pragma unroll
    for (int i = 0; i < 4; ++i) h[i] = __floats2bfloat162_rn(v.x[2 * i], v.x[2 * i + 1]);
    *reinterpret_cast<uint4*>(p) = r;
}
// hi = bf16(v), lo = bf16(v - hi) into two planes `plane` elements apart
__device__ __forceinline__ void store8_planes(__nv_bfloat16* p, size_t plane, const F8& v) {
    F8 hi_f, lo;
    uint4 r;
    __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&r);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        h[i] = __floats2bfloat162_rn(v.x[2 * i], v.x[2 * i + 1]);
        const float2 f = __bfloat1622float2(h[i]);
        hi_f.x[2 * i] = f.x;
        hi_f.x[2 * i + 1] = f.y;
    }
    *reinterpret_cast<uint4*>(p) = r;
#pragma unroll
    for (int i = 0; i < 8; ++i) lo.x[i] = v.x[i] - hi_f.x[i];
    store8<__nv_bfloat16>(p + plane, lo);
}

// Weight operands.  tc: bf16 planes hi, lo = bf16(w - hi) side by side along the reduction index:
//   Wz [H, 2H]: row j (output column of z = x1 W), reduction index i: W[i, j], i.e. W transposed;
//   Wn [H, 2H]: row i (output column of g_x1 = gz W^T), reduction index j: W[i, j].
// Wt_f32 (CUDA-core path): W transposed.  A block turns a 32 x 32 tile round in shared memory, so that both directions
// move 64 to 128 contiguous bytes per warp (H = 1024: 38 -> 6 us against one thread per element with strided stores).
// Also clears the status word of the workspace header.
__device__ __forceinline__ void pack_weights(int tile, int H, const float* W, __nv_bfloat16* Wz, __nv_bfloat16* Wn, float* Wt_f32, WsHeader* hdr) {
    __shared__ float t[32][33];
    const int n = (H + 31) / 32, lane = threadIdx.x & 31, w = threadIdx.x >> 5, i0 = tile / n * 32, j0 = tile % n * 32;
    if (threadIdx.x == 0 && tile == 0) hdr->status = 0;
    auto put = [&](__nv_bfloat16* base, int row, int k, float v) {
        const __nv_bfloat16 hi = __float2bfloat16_rn(v);
        base[(size_t)row * 2 * H + k] = hi;
        base[(size_t)row * 2 * H + H + k] = __float2bfloat16_rn(v - __bfloat162float(hi));
    };
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int i = i0 + w + 8 * q, j = j0 + lane;
        if (i < H && j < H) {
            const float v = W[(size_t)i * H + j];
            t[w + 8 * q][lane] = v;
            if (Wn) put(Wn, i, j, v);
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int j = j0 + w + 8 * q, i = i0 + lane;
        if (i < H && j < H) {
            const float v = t[lane][w + 8 * q];
            if (Wz) put(Wz, j, i, v);
            if (Wt_f32) Wt_f32[(size_t)j * H + i] = v;
        }
    }
}

// What the gate's GEMM reads, in one launch (two are a few us longer: both are short and neither fills the machine): the
// first blocks lay the weights out, the others compute
// x1 = GELU(v): fp32 [M, H], or bf16 [M, 2H] with the high halves in columns [0, H) and the low
// halves (bf16(x1 - hi)) in [H, 2H): one operand for the gate's GEMM with both planes along K, two
// column blocks for the weight-gradient products.  A single bf16 rounding of x1 is not enough there.
template <typename IO, bool kPlanes>
__global__ void __launch_bounds__(kThreads)
glu_pre_kernel(int pack_blocks, size_t n, int H, const IO* v, void* x1, const float* W, __nv_bfloat16* Wz, __nv_bfloat16* Wn, float* Wt_f32,
               WsHeader* hdr) {
    grid_dep_wait();
    grid_dep_launch();
    if ((int)blockIdx.x < pack_blocks) {
        pack_weights((int)blockIdx.x, H, W, Wz, Wn, Wt_f32, hdr);
        return;
    }
    const size_t step = (size_t)(gridDim.x - pack_blocks) * kThreads * 8;
    for (size_t e = ((size_t)(blockIdx.x - pack_blocks) * kThreads + threadIdx.x) * 8; e < n; e += step) {
        F8 a = load8<IO>(v + e);
#pragma unroll
        for (int i = 0; i < 8; ++i) a.x[i] = gelu_f(a.x[i]);
        if (kPlanes) {
            const size_t m = e / H, h = e % H;   // a group of 8 stays inside one row (H % 8 == 0)
            store8_planes(reinterpret_cast<__nv_bfloat16*>(x1) + m * 2 * H + h, (size_t)H, a);
        } else {
            store8<float>(reinterpret_cast<float*>(x1) + e, a);
        }
    }
}

template <typename IO>
__global__ void glu_out_kernel(size_t n, const IO* v, const float* z, IO* out) {
    grid_dep_wait();
    grid_dep_launch();
    for (size_t e = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) * 8; e < n; e += (size_t)gridDim.x * blockDim.x * 8) {
        const F8 a = load8<IO>(v + e), zz = load8<float>(z + e);
        F8 o;
#pragma unroll
        for (int i = 0; i < 8; ++i) o.x[i] = a.x[i] * sigmoid_f<IO>(zz.x[i]);
        store8<IO>(out + e, o);
    }
}

// gz = gout * v * s (1 - s), s = sigmoid(z): fp32, or two bf16 planes hi / lo `plane` elements apart
template <typename IO, bool kPlanes>
__global__ void glu_gz_kernel(size_t n, const IO* v, const IO* gout,
                              const float* z, void* gz, size_t plane) {
    grid_dep_wait();
    grid_dep_launch();
    for (size_t e = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) * 8; e < n; e += (size_t)gridDim.x * blockDim.x * 8) {
        const F8 a = load8<IO>(v + e), g = load8<IO>(gout + e), zz = load8<float>(z + e);
        F8 o;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float s = sigmoid_f<IO>(zz.x[i]);
            o.x[i] = g.x[i] * a.x[i] * s * (1.f - s);
        }
        if (kPlanes) store8_planes(reinterpret_cast<__nv_bfloat16*>(gz) + e, plane, o);
        else store8<float>(reinterpret_cast<float*>(gz) + e, o);
    }
}

// The last launch of the backward pass: the first blocks add the slices of dW, the others compute
// gv = gout * sigmoid(z) + g_x1 * GELU'(v)
template <typename IO>
__global__ void __launch_bounds__(kThreads)
glu_post_kernel(int reduce_blocks, const float* part, int splits, size_t n_w, float* dW, size_t n, const IO* v, const IO* gout,
                const float* z, const float* gx1, IO* gv) {
    grid_dep_wait();
    grid_dep_launch();
    if ((int)blockIdx.x < reduce_blocks) {
        const size_t quads = n_w / 4, step = (size_t)reduce_blocks * kThreads;
        for (size_t e = (size_t)blockIdx.x * kThreads + threadIdx.x; e < quads; e += step) {
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
            for (int s = 0; s < splits; ++s) {
                const float4 t = ld_stream(reinterpret_cast<const float4*>(part + (size_t)s * n_w) + e);
                acc.x += t.x, acc.y += t.y, acc.z += t.z, acc.w += t.w;
            }
            reinterpret_cast<float4*>(dW)[e] = acc;
        }
        return;
    }
    const size_t step = (size_t)(gridDim.x - reduce_blocks) * kThreads * 8;
    for (size_t e = ((size_t)(blockIdx.x - reduce_blocks) * kThreads + threadIdx.x) * 8; e < n; e += step) {
        const F8 a = load8<IO>(v + e), g = load8<IO>(gout + e), zz = load8<float>(z + e), x = load8<float>(gx1 + e);
        F8 o;
#pragma unroll
        for (int i = 0; i < 8; ++i) o.x[i] = g.x[i] * sigmoid_f<IO>(zz.x[i]) + x.x[i] * gelu_grad_f(a.x[i]);
        store8<IO>(gv + e, o);
    }
}

}  // namespace

void launch_glu_pre(bool io_bf16, bool planes, size_t n, int H, const void* v, void* x1, const float* W, void* Wz, void* Wn,
                    float* Wt_f32, WsHeader* hdr, cudaStream_t st) {
    count_launch();
    const int tiles = ((H + 31) / 32) * ((H + 31) / 32), b = tiles + blocks_for(n / 8);
    auto wz = (__nv_bfloat16*)Wz, wn = (__nv_bfloat16*)Wn;
    if (io_bf16 && planes)
        launch_dep(glu_pre_kernel<__nv_bfloat16, true>, b, kThreads, 0, st, tiles, n, H, (const __nv_bfloat16*)v, x1, W, wz, wn, Wt_f32, hdr);
    else if (io_bf16)
        launch_dep(glu_pre_kernel<__nv_bfloat16, false>, b, kThreads, 0, st, tiles, n, H, (const __nv_bfloat16*)v, x1, W, wz, wn, Wt_f32, hdr);
    else
        launch_dep(glu_pre_kernel<float, false>, b, kThreads, 0, st, tiles, n, H, (const float*)v, x1, W, wz, wn, Wt_f32, hdr);
}

void launch_glu_out(bool io_bf16, size_t n, const void* v, const float* z, void* out, cudaStream_t st) {
    count_launch();
    const int b = blocks_for(n / 8);
    if (io_bf16) launch_dep(glu_out_kernel<__nv_bfloat16>, b, kThreads, 0, st, n, (const __nv_bfloat16*)v, z, (__nv_bfloat16*)out);
    else launch_dep(glu_out_kernel<float>, b, kThreads, 0, st, n, (const float*)v, z, (float*)out);
}

void launch_glu_gz(bool io_bf16, bool planes, size_t n, const void* v, const void* gout, const float* z, void* gz,
                   cudaStream_t st) {
    count_launch();
    const int b = blocks_for(n / 8);
    if (io_bf16 && planes)
        launch_dep(glu_gz_kernel<__nv_bfloat16, true>, b, kThreads, 0, st, n, (const __nv_bfloat16*)v, (const __nv_bfloat16*)gout, z, gz, n);
    else if (io_bf16)
        launch_dep(glu_gz_kernel<__nv_bfloat16, false>, b, kThreads, 0, st, n, (const __nv_bfloat16*)v, (const __nv_bfloat16*)gout, z, gz, n);
    else
        launch_dep(glu_gz_kernel<float, false>, b, kThreads, 0, st, n, (const float*)v, (const float*)gout, z, gz, n);
}

void launch_glu_post(bool io_bf16, const float* part, int splits, size_t n_w, float* dW, size_t n, const void* v, const void* gout,
                     const float* z, const float* gx1, void* gv, cudaStream_t st) {
    count_launch();
    const int rb = blocks_for(n_w / 4), b = rb + blocks_for(n / 8);
    if (io_bf16)
        launch_dep(glu_post_kernel<__nv_bfloat16>, b, kThreads, 0, st, rb, part, splits, n_w, dW, n, (const __nv_bfloat16*)v,
                   (const __nv_bfloat16*)gout, z, gx1, (__nv_bfloat16*)gv);
    else
        launch_dep(glu_post_kernel<float>, b, kThreads, 0, st, rb, part, splits, n_w, dW, n, (const float*)v, (const float*)gout, z, gx1,
                   (float*)gv);
}

}  // namespace ssm
