// relo_edt_noalloc: the exact squared EDT of a grid, for callers that cannot
// allocate device memory.
//
// Some callers may not call cudaMalloc at all once they are running: a
// robot's real-time localisation loop that only allocates at start-up
// (a device allocation can block inside the driver for an unbounded time),
// or a host framework that owns every byte of device memory through its own
// pool and forbids raw allocations by the libraries it loads.  This entry
// point lets them compute the EDT lookup table with memory they already own:
// the caller passes the grid and the output, and the only scratch, the
// occupancy words, the column-segment summaries and the bands' flags, lives in
// file-scope __device__ arrays of a fixed maximum size.  The passes are those of
// the map precompute (edt_band.cuh); with column distances in memory and one
// thread per cell scanning a row they took 38 us on 1000 x 777, now 24.5.
//
// Consequences, stated for the user:
//   - Maps up to kNoAllocMaxSide x kNoAllocMaxSide cells (1024 x 1024) are
//     accepted; larger ones are rejected with RELO_E_INVALID_ARG.
//   - Every GPU that loads the library holds the scratch (0.7 MiB) until the
//     process exits.
//   - The first call on a device looks up the scratch's device address with
//     that device current; make that first call before any stream capture.
//     The address is kept for the life of the process: after cudaDeviceReset
//     (or any reset of the device's primary context) the module, and with it
//     the scratch, is gone, so do not call this entry point on that device
//     again in the same process.
//   - A CUDA error already pending in the calling thread (left by earlier
//     work) is reported as RELO_E_CUDA before anything is launched, and is
//     left in place for its owner; the launches are checked, and a
//     failed first launch stops the call.
//   - All calls on one device share the scratch: calls whose work overlaps on
//     the GPU (for example on two streams at once) race and give wrong
//     results.  Each call overwrites every scratch element it reads, so
//     nothing has to start at zero and no clearing is needed.
//   - No cudaMalloc, cudaFree or allocating library routine is called.
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "../../include/relo.h"
#include "edt_band.cuh"

namespace {

constexpr int kNoAllocMaxSide = 1024;
constexpr int kNoAllocMaxTiles = kNoAllocMaxSide / 8;
constexpr int kMaxDevices = 64;

struct NoAllocScratch {
    uint64_t words[kNoAllocMaxTiles * kNoAllocMaxTiles];
    short2 summ[kNoAllocMaxTiles / kSegTiles * kNoAllocMaxSide];
    short2 span[kNoAllocMaxTiles * kNoAllocMaxSide];
    int far[kNoAllocMaxTiles + 1];
};
static __device__ __align__(256) NoAllocScratch g_scratch;

std::mutex g_mu;
NoAllocScratch *g_scratch_addr[kMaxDevices] = {nullptr};
int g_n_sm[kMaxDevices] = {0};

__global__ void __launch_bounds__(256) k_na_tiles(const int8_t *__restrict__ grid, EdtTiles t, bool vec) {
    edt_tiles(grid, t, vec, nullptr, [](uint64_t, int, int) {});
}

// device address of the scratch and number of SMs of the current device (looked up once per device)
cudaError_t scratch_for_current_device(NoAllocScratch **scratch, int *n_sm) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_scratch_addr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_scratch);
        if (e != cudaSuccess) return e;
        e = cudaDeviceGetAttribute(&g_n_sm[dev], cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        g_scratch_addr[dev] = static_cast<NoAllocScratch *>(p);
    }
    *scratch = g_scratch_addr[dev];
    *n_sm = g_n_sm[dev];
    return cudaSuccess;
}

}  // namespace

extern "C" int relo_edt_noalloc(const int8_t *grid_dev, int32_t w, int32_t h, int32_t *d2_dev, void *stream) {
    if (!grid_dev || !d2_dev || w < 1 || h < 1) return RELO_E_INVALID_ARG;
    if (w > kNoAllocMaxSide || h > kNoAllocMaxSide) return RELO_E_INVALID_ARG;
    NoAllocScratch *sc = nullptr;
    int n_sm = 0;
    if (scratch_for_current_device(&sc, &n_sm) != cudaSuccess) return RELO_E_CUDA;
    // an error left by the caller's own earlier work: report it, launch nothing, leave it pending
    if (cudaPeekAtLastError() != cudaSuccess) return RELO_E_CUDA;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const EdtTiles t{sc->words, sc->summ, sc->span, sc->far, nullptr, w, h, (w + 7) / 8, (h + 7) / 8};
    const bool vec = (w & 7) == 0 && (reinterpret_cast<uintptr_t>(grid_dev) & 7) == 0;
    k_na_tiles<<<dim3((t.TW + 31) / 32, edt_summary_rows(h)), dim3(32, 8), 0, s>>>(grid_dev, t, vec);
    if (cudaGetLastError() != cudaSuccess) return RELO_E_CUDA;
    if (launch_edt_bands(t, EdtOut{d2_dev, nullptr, nullptr, 0, 0, 0}, n_sm, s) != cudaSuccess) return RELO_E_CUDA;
    return RELO_OK;
}
