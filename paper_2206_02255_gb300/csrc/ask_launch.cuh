// ask_launch.cuh -- launches of the ASK chain's kernels.
//
// The kernels of a chain after its first (init, plainly launched; then levels
// and leaves) are launched as programmatic dependents of the kernel before
// them on the stream: each says at its start that its own dependent may be
// launched (chain_start), and waits there for the kernels before it to finish
// before it touches memory.  So a kernel's launch and the set-up of its CTAs
// overlap the end of the one before; what it reads and writes is ordered as in
// plain stream order, since the wait covers the whole earlier grid and its
// memory operations, and that grid has itself waited for the one before it.
// A call in a row of calls, every kernel plain -> this way: n = 256 50.6 -> 47.3
// us, n = 1024 61.8 -> 54.8, n = 1999 without allocation 199.4 -> 190.7, n = 3001
// 376 -> 369, n = 16384 1636 -> 1626; a captured graph is the same either way.
//
// The init kernel depends on whatever the stream held before: a CDP2 render of
// the same scratch, say, whose grids launch the rest of their work from the
// device.  The wait is defined for the grid before, not for the grids that it
// has launched in its turn, so init takes plain stream order, which covers
// those (45.4 us at n = 256, 53.2 at n = 1024 with init a dependent too).
//
// The deep-zoom kernels are launched plainly: their grids leave room on an SM,
// and CTAs placed while the kernel before still holds a part of the SMs end
// up unevenly spread (float-float, n = 3000: 7.67 ms against 7.28).
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <utility>

namespace ask {

__device__ __forceinline__ void chain_start()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <typename... KArgs, typename... Args>
cudaError_t launch_chained(void (*kernel)(KArgs...), int grid, int threads, size_t smem, cudaStream_t s,
                           Args &&...args)
{
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
    if (e != cudaSuccess)
        cudaGetLastError();  // reported here, not by the process's next check
    return e;
}

// Answers of resident_ctas, by device (0: not asked yet).
constexpr int kKnownDevices = 64;
struct PerDevice {
    std::atomic<int> ctas[kKnownDevices] = {};
};

// CTAs of a kernel that fit an SM of the current device at once (at least 1).
// `known` keeps the answer; a query that failed counts as 1 this once.
template <typename K>
int resident_ctas(K kernel, int threads, size_t smem, PerDevice *known = nullptr)
{
    int dev = -1, per_sm = 0;
    if (known && cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < kKnownDevices &&
        (per_sm = known->ctas[dev].load(std::memory_order_relaxed)) > 0)
        return per_sm;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem) != cudaSuccess ||
        per_sm < 1) {
        cudaGetLastError();  // not the launch's error
        return 1;
    }
    if (known && dev >= 0 && dev < kKnownDevices)
        known->ctas[dev].store(per_sm, std::memory_order_relaxed);
    return per_sm;
}

}  // namespace ask
