// fp32 tensors as bf16 planes, for fp32-accurate projections on the bf16 tensor cores.
//
// A value v is carried as three bf16 numbers, hi = bf16(v), mid = bf16(v - hi), lo = bf16(v - hi - mid):
// 3 x 8 mantissa bits, so hi + mid + lo = v exactly (up to underflow).  A matrix [M, K] becomes
// [M, 3K] with the planes side by side along K; the product of two such matrices is the sum of the
// six plane products whose terms are not below 2^-24 of the result (hi hi, hi mid, mid hi, mid mid,
// hi lo, lo hi), which the GEMM kernels accumulate (see GemmTcTN).
#include <algorithm>

#include "kernels.h"

namespace ssm {

__device__ __forceinline__ void split3(float v, __nv_bfloat16& hi, __nv_bfloat16& mid, __nv_bfloat16& lo) {
    hi = __float2bfloat16_rn(v);
    const float r1 = v - __bfloat162float(hi);
    mid = __float2bfloat16_rn(r1);
    lo = __float2bfloat16_rn(r1 - __bfloat162float(mid));
}

// in [M, K] fp32 -> out [M, 3K] bf16 (planes side by side).  One thread per 4 neighbouring elements.  HBM-bound:
// 64000 x 512 (328 MB) 52 us, 6.3 TB/s.
// The loads of four quads are issued before the first store (89 us with one at a time).
__global__ void __launch_bounds__(256)
split_planes_kernel(const float* in, size_t M, int K, __nv_bfloat16* out) {
    grid_dep_wait();
    grid_dep_launch();
    constexpr int kU = 4;
    const size_t quads = M * (size_t)(K / 4), step = (size_t)gridDim.x * blockDim.x;
    for (size_t q0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q0 < quads; q0 += kU * step) {
        float4 v[kU];
#pragma unroll
        for (int i = 0; i < kU; ++i)
            if (q0 + i * step < quads) v[i] = ld_stream(reinterpret_cast<const float4*>(in) + q0 + i * step);
#pragma unroll
        for (int i = 0; i < kU; ++i) {
            const size_t q = q0 + i * step;
            if (q >= quads) break;
            const size_t m = q / (K / 4);
            const int k = (int)(q - m * (K / 4)) * 4;
            const float vv[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
            __nv_bfloat16 h[4], d[4], l[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) split3(vv[j], h[j], d[j], l[j]);
            __nv_bfloat16* row = out + m * 3 * (size_t)K + k;
            *reinterpret_cast<uint2*>(row) = *reinterpret_cast<const uint2*>(h);
            *reinterpret_cast<uint2*>(row + K) = *reinterpret_cast<const uint2*>(d);
            *reinterpret_cast<uint2*>(row + 2 * (size_t)K) = *reinterpret_cast<const uint2*>(l);
        }
    }
}

void launch_split_planes(const float* in, size_t M, int K, void* out, cudaStream_t st) {
    const size_t quads = M * (size_t)(K / 4);
    const int blocks = (int)std::min<size_t>((quads + 255) / 256, 148 * 8);
    count_launch();
    launch_dep(split_planes_kernel, blocks, 256, 0, st, in, M, K, (__nv_bfloat16*)out);
}

}  // namespace ssm
