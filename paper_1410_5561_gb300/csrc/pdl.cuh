// Programmatic dependent launch: the kernel of one step is set up while the step before it still
// runs, and waits for its results on the device instead of at a kernel boundary. For steps that
// take microseconds (64^3: see launch_plain) the boundary is most of the time.
#pragma once
#include <cuda_runtime.h>

namespace stg {

// First statement of a kernel launched with launch_dependent: lets the next such kernel of the
// stream be set up, then waits until everything before this one has completed and is visible.
__device__ __forceinline__ void dependent_begin() {
    asm volatile("griddepcontrol.launch_dependents;\n\tgriddepcontrol.wait;\n" ::: "memory");
}

// Launches a kernel that begins with dependent_begin(); early = false: at the kernel boundary as usual.
template <typename... P, typename... A>
cudaError_t launch_dependent(bool early, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                             A... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

}  // namespace stg
