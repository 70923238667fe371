// What the launchers ask the CUDA runtime about a kernel, remembered per kernel and device: the
// answers do not change while the process runs, and asking on every launch took a
// tenth of the host's time of a short call (phi_64 of perf/cases.py: 232 -> 216 us a pass).
// Bounded: one entry per kernel, device, block size and shared memory size in use; guarded by
// a mutex, so any thread may launch.
#include <map>
#include <mutex>
#include <tuple>

#include "common.cuh"

namespace pdgb {

static std::mutex g_mu;

cudaError_t launch_smem(const void* kernel, size_t bytes) {
    static std::map<std::pair<const void*, int>, size_t> largest;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e) return e;
    std::lock_guard<std::mutex> lock(g_mu);
    size_t& had = largest[{kernel, dev}];
    if (bytes <= had) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (!e) had = bytes;
    return e;
}

cudaError_t launch_occupancy(const void* kernel, int threads, size_t smem, int* per_sm) {
    static std::map<std::tuple<const void*, int, int, size_t>, int> known;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e) return e;
    std::lock_guard<std::mutex> lock(g_mu);
    const auto key = std::make_tuple(kernel, dev, threads, smem);
    const auto it = known.find(key);
    if (it != known.end()) {
        *per_sm = it->second;
        return cudaSuccess;
    }
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, kernel, threads, smem);
    if (!e && known.size() < 4096) known[key] = *per_sm;
    return e;
}

}  // namespace pdgb
