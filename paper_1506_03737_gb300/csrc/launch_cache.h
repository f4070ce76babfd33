// Host-side launch helpers of the persistent FFT kernels: the dynamic shared-memory attribute
// and the persistent grid size (resident CTAs per SM x SMs), cached per device.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <mutex>

namespace colapm {

template <typename K>
static cudaError_t set_smem(K kernel, size_t bytes) {
    if (bytes <= 48 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// Persistent grid: resident CTAs per SM x SMs.
template <typename K>
static int persistent_grid(K kernel, int threads, size_t smem) {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, smem);
    if (per < 1) per = 1;
    return per * sms;
}

// Launch configuration of one kernel on each device: its dynamic shared-memory attribute (set
// once per device, raised when a larger size is asked for) and the persistent grid for that size.
// A mutex guards it, so launchers may run from several host threads and on several devices.
constexpr int kMaxDevices = 64;
struct GridCache {
    std::mutex mu;
    int grid[kMaxDevices] = {};
    size_t smem[kMaxDevices] = {};
};

template <typename K>
static cudaError_t cached_grid(GridCache& c, K kernel, int threads, size_t smem, int* grid) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(c.mu);
    if (!c.grid[dev] || smem > c.smem[dev]) {
        e = set_smem(kernel, smem);
        if (e != cudaSuccess) return e;
        if (smem > c.smem[dev]) c.smem[dev] = smem;
        c.grid[dev] = persistent_grid(kernel, threads, c.smem[dev]);
    }
    *grid = c.grid[dev];
    return cudaSuccess;
}

// Launches that may overlap the end of the kernel before them (programmatic stream serialization): the CTAs of
// the next kernel are placed as soon as every CTA of this one has started and there is room, load their
// constant tables and wait in pdl_wait() until the kernel before has completed and its writes are visible.
// Every kernel launched by launch_dep calls pdl_wait() before it touches anything but constant tables (written
// before the stream's work began); kernels whose predecessors did the same are then ordered as without it.
// What that kernel may still be writing is read through plain pointers (or __ldcg, __ldcs): `const T* __restrict__` and
// __ldg promise that the memory does not change while the kernel runs, which leaves the compiler free to load it on
// the path that is not coherent, or before the wait.
// A step on a 64^3 or 128^3 mesh is a chain of 3-12 us kernels, of which the start and the table loads
// were 1-2 us each: a step at 64^3 went from 89 to 76 us, ten at 128^3 with P(k) from 908 to 817 us.
// `overlap` is for such short kernels only (overlap_mesh): kernels that follow one another without a gap
// share one split of an SM's memory into L1 and shared memory, which cost the 512^3 step 3% (the gather lives
// off L1) and a batch with meshes up to 384^3 on two streams 11% (waiting CTAs hold room the other
// stream's kernels could use).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;"); }

constexpr bool overlap_mesh(int side) { return side <= 128; }

template <typename... P, typename... A>
static cudaError_t launch_dep(bool overlap, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = overlap ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace colapm
