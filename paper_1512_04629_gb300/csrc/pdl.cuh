// pdl.cuh -- programmatic dependent launch of the solve-path kernels.
#pragma once
#include <cuda_runtime.h>

#include <cstdlib>
#include <utility>

#include "common.cuh"

namespace amg {

// Programmatic dependent launch: the solve-path kernels go out with the
// stream-serialisation attribute, so the next kernel's blocks are scheduled
// while the current one runs (its launch latency is hidden), and every such
// kernel begins with pdl_begin(): it lets its own dependent launch, then
// waits until the kernel before it has completed and its writes are visible.
// Without the attribute (or with AMG_PDL=0) both instructions do nothing.
__device__ __forceinline__ void pdl_begin() {
    asm volatile("griddepcontrol.launch_dependents;\n\tgriddepcontrol.wait;" ::: "memory");
}
// The two halves, for kernels that load what no earlier kernel of the solve
// writes -- the operator, its layout, its diagonal -- in between, so that
// these loads overlap the kernel before.  Everything a solve kernel reads that
// way is complete before its first launch: setup and re-sparsification end
// with a stream synchronisation, and so does each layout built for a timed
// trial.
__device__ __forceinline__ void pdl_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// vectors written by the kernel before: coherent loads that stay behind the
// dependency wait (a read-only load may be moved above it by the compiler)
__device__ __forceinline__ double ld_dyn(const double *p) {
    double v;
    asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float ld_dyn(const float *p) {
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}

inline bool pdl_enabled() {
    static const bool on = [] {
        const char *e = std::getenv("AMG_PDL");
        return !(e && e[0] == '0');
    }();
    return on;
}

template <typename... KArgs, typename... Args>
void pdl_launch(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args &&...args) {
    if (!pdl_enabled()) {
        kern<<<grid, block, smem, s>>>(std::forward<Args>(args)...);
        return;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    AMG_CUDA(cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...));
}

}  // namespace amg
