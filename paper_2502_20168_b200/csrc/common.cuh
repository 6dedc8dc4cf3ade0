// Shared device/host helpers of the S5 SSM library (sm_100a only).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

#include "../../include/ssm.h"

namespace ssm {

// ---- complex arithmetic on float2 ---------------------------------------------------
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a * x + b
__device__ __forceinline__ float2 cfma(float2 a, float2 x, float2 b) {
    return make_float2(fmaf(a.x, x.x, fmaf(-a.y, x.y, b.x)), fmaf(a.x, x.y, fmaf(a.y, x.x, b.y)));
}
__device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }

// ---- programmatic dependent launch -------------------------------------------------------
// Every kernel of the library is launched so that its blocks may start while the kernel before it on the stream
// still drains, and calls grid_dep_wait before it touches global memory: the wait ends when that kernel has completed
// and its writes are visible.  Since every kernel waits, completion is transitive along the stream.
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next kernel's blocks start where there is room for them.
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Streaming loads (no reuse expected), volatile so that they stay behind grid_dep_wait.
__device__ __forceinline__ float ld_stream(const float* p) {
    float v;
    asm volatile("ld.global.cs.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float2 ld_stream(const float2* p) {
    float2 v;
    asm volatile("ld.global.cs.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ float4 ld_stream(const float4* p) {
    float4 v;
    asm volatile("ld.global.cs.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t ld_stream(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.global.cs.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint2 ld_stream(const uint2* p) {
    uint2 v;
    asm volatile("ld.global.cs.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ uint4 ld_stream(const uint4* p) {
    uint4 v;
    asm volatile("ld.global.cs.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

// ---- io element access ----------------------------------------------------------------
template <typename T> __device__ __forceinline__ float to_f32(T v);
template <> __device__ __forceinline__ float to_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f32(float v);
template <> __device__ __forceinline__ float from_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// 1 / (1 + exp(-z)).  With t = exp(-|z|) <= 1 the divisor lies in [1, 2], where the approximate reciprocal is good to 2 ulp of
// fp32 (of 1 / (1 + exp(-z)) it makes 0 for z < -87.3).  A result in IO = float gets a Newton step, after which the
// reciprocal is at most a unit in the last place off; bf16 results come out the same without it (share of outputs that differ
// from the rounded exact ones 2.3e-4 either way, 2.4e-4 with exact quotients; a projection of 4096 x 1024 with the gate
// 32.7 us, with exact quotients 33.5).
template <typename IO>
__device__ __forceinline__ float sigmoid_f(float z) {
    const float t = expf(-fabsf(z)), d = 1.f + t;
    float r = __fdividef(1.f, d);
    if (sizeof(IO) == 4) r = fmaf(r, fmaf(-d, r, 1.f), r);
    return z < 0.f ? t * r : r;
}

// ---- workspace header -------------------------------------------------------------------
// First 256 bytes of every workspace.  `status` is written by kernels whose bounded waits
// give up.
struct WsHeader {
    int status;
    int pad[63];
};
static_assert(sizeof(WsHeader) == 256, "header is one 256-byte line group");

inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

inline int check_shape(const ssm_shape* s) {
    if (!s) return SSM_ERR_NULL;
    if (s->B < 1 || s->T < 1 || s->H < 8 || s->P < 8 || (s->H % 8) || (s->P % 8)) return SSM_ERR_SHAPE;
    if ((int64_t)s->B * s->T >= (int64_t)1 << 31) return SSM_ERR_SHAPE;
    if (s->io_dtype != SSM_F32 && s->io_dtype != SSM_BF16) return SSM_ERR_DTYPE;
    if (s->reserved != 0) return SSM_ERR_SHAPE;
    return SSM_OK;
}
inline bool misaligned(const void* p, size_t a = 16) { return (reinterpret_cast<uintptr_t>(p) % a) != 0; }

// Measurement hooks (profile.cu): launch counter and optional per-stage event timing.
void count_launch(int n = 1);
// Number of SMs of the current device, cached per device ordinal (148 where no device answers).
int device_sm_count();
// Raises a kernel's dynamic shared-memory limit, once per (kernel, device) (device_setup.cu).
bool set_max_dynamic_smem(const void* kernel, size_t bytes);
// Clusters of `cluster` CTAs of a kernel that the current device runs at the same time, cached per (kernel, cluster, shared memory,
// device); 0: it cannot launch them; -1: no device answers.  Lets the kernel be launched with that much shared memory and in clusters of 16.
int resident_clusters(const void* kernel, int cluster, size_t smem_bytes, int threads);
// Whether what is launched on a stream goes into a graph.
inline bool capturing(cudaStream_t st) {
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &status) == cudaSuccess) return status == cudaStreamCaptureStatusActive;
    (void)cudaGetLastError();
    return false;
}
// Launches a kernel of the library: programmatic dependent launch (see grid_dep_wait), optionally in clusters.
// Between two kernels of a few microseconds the start of the second used to stand idle for about 2 us; its blocks now
// set up while the first drains (projection of 4096 x 512 x 512 back to back: 12.3 -> 9.4 us).
template <typename... KArgs, typename... Args>
inline bool launch_dep_cluster(void (*kernel)(KArgs...), unsigned cluster, dim3 grid, dim3 block, size_t smem,
                               cudaStream_t st, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...) == cudaSuccess;
}
template <typename... KArgs, typename... Args>
inline bool launch_dep(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
    return launch_dep_cluster(kernel, 1, grid, block, smem, st, std::forward<Args>(args)...);
}

// The same launch without the overlap: the grid is placed when the kernel before it has ended, one block per SM first.
template <typename... KArgs, typename... Args>
inline bool launch_after(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...) == cudaSuccess;
}

class StageTimer {
  public:
    StageTimer(const char* name, cudaStream_t st);
    ~StageTimer();
  private:
    cudaStream_t st_;
    int idx_;
};

#define SSM_RETURN_IF_CUDA_ERROR()                              \
    do {                                                        \
        if (cudaPeekAtLastError() != cudaSuccess) {             \
            (void)cudaGetLastError();                           \
            return SSM_ERR_CUDA;                                \
        }                                                       \
    } while (0)

}  // namespace ssm
