// Programmatic dependent launch of the kernels of a chain.
#pragma once

#include <cuda_runtime.h>

#include "kernels.h"
#include "nm_internal.h"

namespace nm {

// Wait for the predecessor's results, then let the successor start: only two
// kernels of a chain are ever in flight together. What is loaded before this
// point is matrix data, which no kernel in flight writes: the host waits for the
// kernels that make it, at assembly and on first use (to_f32, ensure_df,
// build_clusters). Blocks are read after it, by plain (not read-only path)
// loads.
__device__ __forceinline__ void dep_sync() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Launch of a kernel that calls dep_sync: it may start while its predecessor
// on the stream drains.
template <typename... P, typename... A>
int launch_dependent(void (*k)(P...), dim3 grid, unsigned threads, cudaStream_t s, const A&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    NM_CUDA(cudaLaunchKernelEx(&cfg, k, args...));
    count_launch();
    return NM_OK;
}

}  // namespace nm
