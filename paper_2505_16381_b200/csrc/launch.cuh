// Kernel launches of the library.  Kernels that follow one another in a call are launched with programmatic stream
// serialization: a kernel's CTAs may start, and set up their barriers and tensor memory, while the last CTAs of the kernel
// before it still run.  The rules that make that safe:
//  * Every kernel launched here calls grid_wait() in every thread before its first access to global memory, and before any
//    return: it comes back once the kernel before it has completed and that kernel's writes are visible.
//  * grid_launch() comes after grid_wait().  The next kernel can then start only when everything before this kernel is
//    complete; the wait alone covers only the kernel directly in front (with the release placed first, a decoding step read
//    stale cache lines that the step before had written, two kernels back).  It also keeps a whole chain of kernels from
//    crowding onto the SMs early (float32 forward of 2 x 256 x 64: 35 instead of 20 us per call).
//  * A kernel that allocates tensor memory calls grid_launch() only after it has: otherwise a CTA of the next kernel on the same
//    SM could take the columns that a CTA of this one still needs, and then wait for it.
// Gained, with the memsets in front of the first kernels gone as well: training step of 2 x 256 x 64 196 -> 159 us, gated 16 x
// 3001 x 64 480 -> 447 us, decoding step of 128 x 700 x 64 19 -> 16 us.
#pragma once
#include <atomic>
#include <cuda_runtime.h>

namespace path {

__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

constexpr int kMaxCachedDevices = 64;

// SMs of the current device.
inline cudaError_t sm_count(int& sms) {
    static std::atomic<int> known[kMaxCachedDevices];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool cached = dev < kMaxCachedDevices;
    if (cached && (sms = known[dev].load(std::memory_order_relaxed)) > 0) return cudaSuccess;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess && cached) known[dev].store(sms, std::memory_order_relaxed);
    return e;
}

// Launches KERN.  More than 48 KB of dynamic shared memory has to be asked for once per kernel and device.
template <auto KERN, class... Args>
cudaError_t launch(dim3 grid, unsigned block, size_t smem, cudaStream_t st, const Args&... args) {
    if (smem > 48 * 1024) {
        static std::atomic<unsigned> allowed[kMaxCachedDevices];
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev >= kMaxCachedDevices || allowed[dev].load(std::memory_order_relaxed) < smem) {
            e = cudaFuncSetAttribute(KERN, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
            if (dev < kMaxCachedDevices) allowed[dev].store((unsigned)smem, std::memory_order_relaxed);
        }
    }
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, KERN, args...);
    if (e != cudaSuccess) (void)cudaGetLastError();   // reported by the return code; the host's next CUDA call must not find it
    return e;
}

}  // namespace path
