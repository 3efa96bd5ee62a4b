// overlap.cuh -- kernels of one stream that follow one another closely: a
// kernel may be launched while its predecessor drains (programmatic dependent
// launch), does what needs no memory, and waits for the predecessor's end
// before it touches any.
//
// Every kernel launched by launch_overlapped calls await_previous, in every
// thread, before its first access to global memory: it then returns only
// after all earlier work of the stream, since each kernel before it did the
// same.  Work of other kinds (copies, event waits, kernels launched otherwise)
// is ordered as ever.
//
// A clear, a fold and a render of a small raster are mostly the gaps between
// them.  Measured, us per pass without and with (every kernel waiting): 1856 x
// 2208, four members out and four in with a histogram, 37.0 and 29.5 to 33.6 by
// the run; 1501 x 1103 x 100 53.2 and 45.8; 1856 x 2208 x 64 depths 172.4 and
// 165.6; 1024^2 x 16 streamed 104.3 and 99.2; 4096^2 x 1024 2367 and 2359.
#pragma once

#include <utility>

#include <cuda_runtime.h>

namespace cpt {

__device__ __forceinline__ void await_previous() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the next kernel may be launched
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <typename... Params, typename... Args>
cudaError_t launch_overlapped(void (*kernel)(Params...), dim3 grid, unsigned threads, size_t smem, cudaStream_t s,
                              Args &&...args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

}  // namespace cpt
