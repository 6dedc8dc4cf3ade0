// Pieces shared by the kernels on 128-row tiles whose epilogue runs from shared memory (gemm_tc_small.cu,
// gemm_tc_step.cu): typed 4-element accesses and the split of fp32 operands into bf16 planes.
#pragma once

#include "tcgen05.cuh"

namespace ssm {
namespace tc {

constexpr int kSmATile = BM * BK * 2;   // one plane of the A tile of a k-block

// Four neighbouring values of an epilogue operand as loaded; decoded when they are used, so that many can be in
// flight.  kBf16: the operands are known to be bf16 (half the registers), else the flag says.
template <bool kBf16> struct Raw4;
template <> struct Raw4<true> {
    uint2 r;
    __device__ __forceinline__ void load(const void* p, bool, size_t i) {
        r = *reinterpret_cast<const uint2*>(reinterpret_cast<const __nv_bfloat16*>(p) + i);
    }
    __device__ __forceinline__ float4 get(bool) const {
        return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xffff0000u), __uint_as_float(r.y << 16),
                           __uint_as_float(r.y & 0xffff0000u));
    }
};
template <> struct Raw4<false> {
    uint4 r;
    __device__ __forceinline__ void load(const void* p, bool bf16, size_t i) {
        if (bf16) {
            const uint2 t = *reinterpret_cast<const uint2*>(reinterpret_cast<const __nv_bfloat16*>(p) + i);
            r.x = t.x, r.y = t.y;
        } else {
            r = *reinterpret_cast<const uint4*>(reinterpret_cast<const float*>(p) + i);
        }
    }
    __device__ __forceinline__ float4 get(bool bf16) const {
        if (bf16) return Raw4<true>{make_uint2(r.x, r.y)}.get(true);
        return make_float4(__uint_as_float(r.x), __uint_as_float(r.y), __uint_as_float(r.z), __uint_as_float(r.w));
    }
};
__device__ __forceinline__ uint2 pack4_bf16(float4 v) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
    return make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
}
__device__ __forceinline__ void store4_io(void* p, bool bf16, size_t i, float4 v) {
    if (!bf16) *reinterpret_cast<float4*>(reinterpret_cast<float*>(p) + i) = v;
    else *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(p) + i) = pack4_bf16(v);
}

// Eight fp32 values -> the 16-byte chunks of their three bf16 planes (hi + mid + lo = value).
__device__ __forceinline__ void split8(const float4 a, const float4 b, uint4& hi, uint4& mid, uint4& lo) {
    const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    uint32_t* h = &hi.x;
    uint32_t* m = &mid.x;
    uint32_t* l = &lo.x;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __nv_bfloat162 p = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
        const float2 pf = __bfloat1622float2(p);
        const float r0 = v[2 * i] - pf.x, r1 = v[2 * i + 1] - pf.y;
        const __nv_bfloat162 q = __floats2bfloat162_rn(r0, r1);
        const float2 qf = __bfloat1622float2(q);
        const __nv_bfloat162 t = __floats2bfloat162_rn(r0 - qf.x, r1 - qf.y);
        h[i] = *reinterpret_cast<const uint32_t*>(&p);
        m[i] = *reinterpret_cast<const uint32_t*>(&q);
        l[i] = *reinterpret_cast<const uint32_t*>(&t);
    }
}

// fp32 rows of A -> the three planes of a K-major operand tile, by `kThreads` threads: 128 rows x 8 chunks of 8 values
// per k-block, so that 8 threads read a row's 256 bytes.  fetch() asks for a k-block's values, store() splits and
// writes them; rows past M are left alone (what they hold only reaches result rows past M).
template <int kThreads>
struct SplitA {
    static constexpr int kC = 1024 / kThreads, kStep = kThreads / 8;   // chunks per thread, rows between them
    float4 va[kC], vb[kC];
    __device__ __forceinline__ void fetch(const float* a, int K, int M, int m0, int kb, int te) {
#pragma unroll
        for (int i = 0; i < kC; ++i) {
            const int m = m0 + (te >> 3) + kStep * i;
            if (m < M) {
                const float4* src = reinterpret_cast<const float4*>(a + (size_t)m * K + kb * BK + 8 * (te & 7));
                va[i] = src[0];
                vb[i] = src[1];
            }
        }
    }
    // `planes` (may be NULL): the three planes also go to [M, 3K] in global memory.
    __device__ __forceinline__ void store(uint8_t* dst, int M, int m0, int te, __nv_bfloat16* planes = nullptr, int K = 0,
                                          int kb = 0) const {
#pragma unroll
        for (int i = 0; i < kC; ++i) {
            const int r = (te >> 3) + kStep * i;
            if (m0 + r >= M) continue;
            uint4 hi, mid, lo;
            split8(va[i], vb[i], hi, mid, lo);
            uint8_t* q = dst + r * 128 + (((te & 7) ^ (r & 7)) << 4);   // the 128-byte swizzle of a K-major tile
            *reinterpret_cast<uint4*>(q) = hi;
            *reinterpret_cast<uint4*>(q + kSmATile) = mid;
            *reinterpret_cast<uint4*>(q + 2 * kSmATile) = lo;
            if (planes) {
                __nv_bfloat16* g = planes + (size_t)(m0 + r) * 3 * K + kb * BK + 8 * (te & 7);
                *reinterpret_cast<uint4*>(g) = hi;
                *reinterpret_cast<uint4*>(g + K) = mid;
                *reinterpret_cast<uint4*>(g + 2 * (size_t)K) = lo;
            }
        }
    }
};

}  // namespace tc
}  // namespace ssm
