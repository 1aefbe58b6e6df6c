// Launches that overlap their start with the end of the kernel before them in the stream (programmatic
// dependent launch). A kernel launched with launch_pdl() may begin once every block of its predecessor has called
// pdl_trigger() or ended: it calls pdl_wait() before it touches anything another kernel writes or reads, and reads
// what others wrote with plain loads only (a read-only load may be moved above the wait). In the small
// grids a launch's own latency (about 2 us) is a large part of its time.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace adr {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Only grids of at most a quarter of the SMs start early: blocks that wait hold room that kernels of other streams could
// use. Three runs at a time, early against plain: 16 blocks 1.23x to 1.5x (32^2, 8 x 9 FP64), 36 blocks 1.18x (48^2
// FP64); 63 blocks 0.89x (400 x 40 FP32), 120 blocks 0.86x (20 x 24 x 16 FP64).
inline bool starts_early(long long blocks) {
    static const int sms = [] {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        return v;
    }();
    return blocks <= sms / 4;
}

template <typename... P, typename... A>
cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s, A&&... args) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(unsigned(threads));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = starts_early((long long)grid.x * grid.y * grid.z) ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, P(std::forward<A>(args))...);
}

}  // namespace adr
