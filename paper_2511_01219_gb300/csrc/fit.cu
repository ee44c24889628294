// What the launches need to know of a kernel before every launch, asked of the
// driver once: how many CTAs of a shape an SM holds, and that the kernel may
// use that much dynamic shared memory.  The answers depend on the device, the
// kernel and the shape alone, so they are kept for the process (at most
// kMaxFits of them), under a mutex: any context, stream or thread may ask (a
// limit set once held in a second driver context of the device and after
// cudaDeviceReset and cuDevicePrimaryCtxReset: the runtime keeps it).  A
// batch asked the driver some 20 times, 10 to 15 us of host time that a small
// call waits for.
#include <cuda_runtime.h>
#include <stdint.h>

#include <functional>
#include <mutex>
#include <unordered_map>

#include "relo_internal.h"

namespace relo {

namespace {

struct FitKey {
    const void *kernel;
    int device, threads;
    size_t smem;
    bool operator==(const FitKey &o) const {
        return kernel == o.kernel && device == o.device && threads == o.threads && smem == o.smem;
    }
};
struct FitHash {
    size_t operator()(const FitKey &k) const {
        size_t h = std::hash<const void *>()(k.kernel);
        for (size_t v : {(size_t)k.device, (size_t)k.threads, k.smem}) h = h * 1000003u ^ v;
        return h;
    }
};

constexpr size_t kMaxFits = 4096;
std::mutex g_mu;
std::unordered_map<FitKey, int, FitHash> g_fits;       // resident CTAs per SM
std::unordered_map<FitKey, size_t, FitHash> g_limits;  // (kernel, device): the dynamic shared memory it may use

// g_mu held: raises the kernel's limit to smem (never lowers it: another thread may be about to launch with more)
cudaError_t raise_limit(const void *kernel, int device, size_t smem) {
    size_t &limit = g_limits[FitKey{kernel, device, 0, 0}];
    if (smem <= limit) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) limit = smem;
    return e;
}

}  // namespace

cudaError_t allow_smem(const void *kernel, size_t smem) {
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(g_mu);
    return raise_limit(kernel, dev, smem);
}

cudaError_t resident_ctas(const void *kernel, int threads, size_t smem, int *ctas) {
    int dev = 0;
    *ctas = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const FitKey key{kernel, dev, threads, smem};
    std::lock_guard<std::mutex> lk(g_mu);
    const auto it = g_fits.find(key);
    if (it != g_fits.end()) {
        *ctas = it->second;
        return cudaSuccess;
    }
    if ((e = raise_limit(kernel, dev, smem)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas, kernel, threads, smem)) != cudaSuccess) return e;
    if (g_fits.size() >= kMaxFits) g_fits.clear();
    g_fits.emplace(key, *ctas);
    return cudaSuccess;
}

}  // namespace relo
