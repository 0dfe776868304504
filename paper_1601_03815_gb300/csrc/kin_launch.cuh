// Launches whose start overlaps the end of the kernel before them.
//
// A step of a small box lasts a few microseconds, most of them the gap between
// one grid's last block and the next grid's first.  launch_next gives the grid
// the programmatic-serialization attribute: its blocks may become resident as
// soon as every block of the kernel before it on the stream has called
// grid_begin (or ended), and grid_begin itself returns only when that kernel is
// complete and its writes are visible.  A kernel launched this way therefore
//   * calls grid_begin before it reads or writes any global memory, and
//   * reads what the kernels before it wrote with load_l2 or plain loads, never
//     through the read-only path, which may hold lines from before they ended.
// After anything but such a kernel (a copy, another library's kernel) the
// launch is an ordinary one.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <utility>

namespace kin {

__device__ __forceinline__ void grid_begin() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Allow KERNEL bytes of dynamic shared memory on the current device; set once per
// device that this process launches on.
template <auto KERNEL>
cudaError_t allow_smem(size_t bytes) {
    static std::atomic<unsigned long long> configured{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
    if (bit && (configured.load() & bit)) return cudaSuccess;
    e = cudaFuncSetAttribute(KERNEL, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) configured.fetch_or(bit);
    return e;
}

template <typename... P, typename... A>
cudaError_t launch_next(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(std::forward<A>(args))...);
}

}  // namespace kin
