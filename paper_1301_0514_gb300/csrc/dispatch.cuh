// Runtime grid size -> compile-time template argument.
#pragma once

#include <map>
#include <mutex>
#include <type_traits>
#include <utility>

#include <cuda_runtime.h>

namespace scint {

template <typename F>
cudaError_t dispatch_n(int n, F&& f) {
    switch (n) {
        case 16: return f(std::integral_constant<int, 16>{});
        case 32: return f(std::integral_constant<int, 32>{});
        case 64: return f(std::integral_constant<int, 64>{});
        case 128: return f(std::integral_constant<int, 128>{});
        case 256: return f(std::integral_constant<int, 256>{});
        case 512: return f(std::integral_constant<int, 512>{});
        case 1024: return f(std::integral_constant<int, 1024>{});
        case 2048: return f(std::integral_constant<int, 2048>{});
        case 4096: return f(std::integral_constant<int, 4096>{});
        case 8192: return f(std::integral_constant<int, 8192>{});
        case 16384: return f(std::integral_constant<int, 16384>{});
        default: return cudaErrorInvalidValue;
    }
}

// Opt a kernel into more than 48 KB of dynamic shared memory, once per kernel
// and device (later calls, e.g. inside a stream capture, make no CUDA call).
template <typename K>
inline cudaError_t set_smem(K kernel, size_t bytes) {
    if (bytes <= 48 * 1024) return cudaSuccess;
    static std::mutex mu;
    static std::map<std::pair<int, const void*>, size_t> done;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const auto key = std::make_pair(dev, reinterpret_cast<const void*>(kernel));
    std::lock_guard<std::mutex> lk(mu);
    auto it = done.find(key);
    if (it != done.end() && it->second >= bytes) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) done[key] = bytes;
    return e;
}

// Clusters of cs blocks of a kernel that are resident on the device at once (the
// grid of a persistent kernel), queried once per kernel and device; call after set_smem.
template <typename K>
inline cudaError_t active_clusters(K kernel, int cs, int threads, size_t smem, int* out) {
    static std::mutex mu;
    static std::map<std::pair<int, const void*>, int> seen;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const auto key = std::make_pair(dev, reinterpret_cast<const void*>(kernel));
    std::lock_guard<std::mutex> lk(mu);
    auto it = seen.find(key);
    if (it != seen.end()) {
        *out = it->second;
        return cudaSuccess;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cs * 1024);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int nc = 0;
    e = cudaOccupancyMaxActiveClusters(&nc, kernel, &cfg);
    if (e != cudaSuccess) return e;
    if (nc < 1) return cudaErrorInvalidConfiguration;
    seen[key] = nc;
    *out = nc;
    return cudaSuccess;
}

// Blocks of a kernel that are resident on the device at once, queried once per kernel and
// device; call after set_smem.
template <typename K>
inline cudaError_t resident_blocks(K kernel, int threads, size_t smem, int* out) {
    static std::mutex mu;
    static std::map<std::pair<int, const void*>, int> seen;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const auto key = std::make_pair(dev, reinterpret_cast<const void*>(kernel));
    std::lock_guard<std::mutex> lk(mu);
    auto it = seen.find(key);
    if (it != seen.end()) {
        *out = it->second;
        return cudaSuccess;
    }
    int sms = 0, per_sm = 0;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem)) != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    *out = seen[key] = sms * per_sm;
    return cudaSuccess;
}

// Start of a kernel launched by launch_next: wait for the kernel before (all of it, and its memory)
// before touching anything, then let the next one of the stream be set up.  In this order one kernel at
// most waits on the chip; the other way round a whole chain of them piles up beside the one that works
// (256^2 in 64-bit, 20 passes as a graph: 59 us a pass in this order, 165 in the other).
// What the kernel before wrote is read by plain loads (or __ldcg, or TMA): the read-only path (__ldg) is for
// memory that stands still from the reading kernel's start, which here lies before the wait.  What an
// earlier kernel of the stream wrote stands still by then: the one before has waited for it.
__device__ __forceinline__ void begin_after_previous() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// Launch a kernel that begins with begin_after_previous: it is set up while the kernel before it ends
// (programmatic dependent launch).  Between the short kernels of a small call the gaps had been a third of
// its time (1024^2 at one wavelength with one curve 34.8 -> 24.6 us, 256^2 in 64-bit 65.6 -> 59.4).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_next(void (*k)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, std::forward<Args>(args)...);
}
// Passes that are launched so (the synthesis' above 512^2 are not, synth.cu): grids of at most 65536 threads, a fifth of what the chip holds (N lines of
// N / 16 threads: to 1024^2), and at most eight times as many thread-wavelengths.  A longer pass hides its
// own launch, and its waiting blocks take room from the one that works, this stream's or another's: with
// every pass let in, 4096^2 at one wavelength went from 668 to 677 us, and with 1024^2 at 32 wavelengths
// let in the batched workload of eight streams from 106.5 to 107.2 ms.  An early grid waits for the whole
// of the one before in any case, so the order of memory is that of plain launches.
constexpr int kEarlyThreads = 65536, kEarlyWork = 8 * kEarlyThreads;
template <int N>
__device__ __forceinline__ void begin_pass() {
    if constexpr (N <= 1024) begin_after_previous();
}
template <int N, typename... KArgs, typename... Args>
inline cudaError_t launch_pass(int count, void (*k)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                               Args&&... args) {
    if constexpr (N <= 1024) {
        const size_t threads = (size_t)grid.x * block.x;
        if (threads <= kEarlyThreads && threads * count <= kEarlyWork)
            return launch_next(k, grid, block, smem, s, std::forward<Args>(args)...);
    }
    k<<<grid, block, smem, s>>>(std::forward<Args>(args)...);
    return cudaGetLastError();
}

// Launch k with clusters of cs blocks along x (cs == 1: ordinary launch).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_k(void (*k)(KArgs...), int cs, dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                            Args&&... args) {
    if (cs == 1) {
        k<<<grid, block, smem, s>>>(std::forward<Args>(args)...);
        return cudaGetLastError();
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, std::forward<Args>(args)...);
}

}  // namespace scint
