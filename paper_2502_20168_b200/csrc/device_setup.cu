// Per-device, per-kernel set-up that launchers would otherwise repeat on every call.
#include <map>
#include <mutex>
#include <tuple>
#include <utility>

#include "common.cuh"

namespace ssm {

// The dynamic shared-memory limit is an attribute of the function in one device's context:
// set it the first time a kernel is launched on a device, remember that it was.
bool set_max_dynamic_smem(const void* kernel, size_t bytes) {
    static std::mutex mu;
    static std::map<std::pair<const void*, int>, size_t> done;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    std::lock_guard<std::mutex> lock(mu);
    auto it = done.find({kernel, dev});
    if (it != done.end() && it->second >= bytes) return true;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    done[{kernel, dev}] = bytes;
    return true;
}

// What the device holds depends on the kernel's registers and shared memory and on how its SMs are grouped: asked once.
int resident_clusters(const void* kernel, int cluster, size_t smem_bytes, int threads) {
    using Key = std::tuple<const void*, int, size_t, int>;
    static std::mutex mu;
    static std::map<Key, int> cache;
    static thread_local Key last_key;   // (a loop of steps asks the same again and again: 0.1 us less of its host time)
    static thread_local int last = 0;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        (void)cudaGetLastError();
        return -1;
    }
    const Key key(kernel, cluster, smem_bytes, dev);
    if (key == last_key) return last;
    std::lock_guard<std::mutex> lock(mu);
    last_key = key;
    const auto it = cache.find(key);
    if (it != cache.end()) return last = it->second;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(cluster * device_sm_count()), 1, 1);
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = smem_bytes;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if ((smem_bytes > 48 * 1024 && !set_max_dynamic_smem(kernel, smem_bytes)) ||
        (cluster > 8 && cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) ||
        cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        n = 0;
    }
    return last = cache[key] = n;
}

// Workspace layouts, operand packing order and kernel choices depend on the SM count, so it is
// looked up for the device that is current, once per ordinal.
int device_sm_count() {
    constexpr int kMaxDevices = 64;
    static std::mutex mu;
    static int cache[kMaxDevices] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        (void)cudaGetLastError();
        return 148;
    }
    std::lock_guard<std::mutex> lock(mu);
    if (!cache[dev]) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
            (void)cudaGetLastError();
            return 148;
        }
        cache[dev] = n;
    }
    return cache[dev];
}

}  // namespace ssm
