// sg_launch.cuh -- launch helpers of the pass launchers: shared-memory opt-ins
// and occupancies cached per kernel, launches with programmatic stream
// serialization, NVTX ranges.
#pragma once
#include <cuda_runtime.h>

#include <map>
#include <mutex>
#include <tuple>
#include <utility>

#include <nvtx3/nvToolsExt.h>

namespace sg {

// Dynamic shared memory above the 48 KB default needs an opt-in; carveout
// asks for the largest shared-memory split of L1 (several blocks of a
// shared-memory-heavy kernel per SM).  Done once per kernel, device and
// size: later launches (for example while a stream is being captured) make
// no attribute calls.
struct LaunchCache {
    std::mutex mu;
    std::map<std::tuple<const void*, int, int, size_t>, int> occ;  // (kernel, device, threads, smem) -> blocks/SM
    std::map<std::tuple<const void*, int>, size_t> smem;            // (kernel, device) -> opted-in bytes
};
static LaunchCache& launch_cache()
{
    static LaunchCache c;
    return c;
}
static int current_device()
{
    int d = 0;
    if (cudaGetDevice(&d) != cudaSuccess) {
        cudaGetLastError();
        d = 0;
    }
    return d;
}

template <typename K>
static cudaError_t set_smem(K kernel, size_t smem, bool carveout = false)
{
    LaunchCache& c = launch_cache();
    const auto key = std::make_tuple((const void*)kernel, current_device());
    std::lock_guard<std::mutex> lock(c.mu);
    auto it = c.smem.find(key);
    if (it != c.smem.end() && it->second >= smem) return cudaSuccess;
    cudaError_t e = cudaSuccess;
    if (smem > 48 * 1024) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess && carveout)
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e == cudaSuccess) c.smem[key] = it != c.smem.end() && it->second > smem ? it->second : smem;
    return e;
}

// NVTX range around the enqueue of one pass (visible in Nsight timelines;
// near-free when no tool is attached)
struct PassRange {
    explicit PassRange(const char* name) { nvtxRangePushA(name); }
    ~PassRange() { nvtxRangePop(); }
};

// Launch with programmatic stream serialization: the kernel may start while
// the previous one on the stream finishes; it waits (sg_grid_dep_wait)
// before it reads that kernel's results.
template <typename... KArgs, typename... Args>
static cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, int block, size_t smem, cudaStream_t st,
                              Args&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// Blocks of a kernel resident on the GPU at once (occupancy x SMs), cached
// per kernel, device and launch shape.
template <typename K>
static int resident_blocks(K kernel, int threads, size_t smem, int sms)
{
    LaunchCache& c = launch_cache();
    const auto key = std::make_tuple((const void*)kernel, current_device(), threads, smem);
    int occ = 0;
    {
        std::lock_guard<std::mutex> lock(c.mu);
        auto it = c.occ.find(key);
        if (it != c.occ.end()) occ = it->second;
    }
    if (occ == 0) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, threads, smem) != cudaSuccess || occ < 1) {
            cudaGetLastError();
            occ = 1;
        }
        std::lock_guard<std::mutex> lock(c.mu);
        c.occ[key] = occ;
    }
    return occ * (sms > 0 ? sms : 1);
}

}  // namespace sg
