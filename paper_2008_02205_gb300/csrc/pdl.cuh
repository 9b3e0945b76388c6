// Programmatic dependent launch of the FP32 L-apply: the kernel may start while its
// predecessor in the stream drains, sets up its barriers, fetches its first operator
// records (written when the operators are formed, which ends with a stream
// synchronisation) and then waits for it.
//
// Every kernel launched with launch_pdl calls pdl_wait() in all threads before it touches
// anything that an earlier kernel writes or reads, and before it ends: so a kernel that
// has completed implies that all its predecessors have.  pdl_trigger() lets a successor
// launched this way start; it fires when every block has called it or has ended, so all
// blocks of this kernel are running by then.
//
// Applies back to back at 32^2 S4: 4.0 -> 3.0 us.  Tried on every kernel of the Krylov loops
// and not kept there: blocks that wait hold registers and shared memory that the
// running kernel's successors need (eight batched problems 37.5 -> 40.5 ms, 32^2 S4 FP64
// step 20.5 -> 24.3).
#pragma once

#include <cuda_runtime.h>

namespace mlpg {

__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;\n"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
// a pointer whose loads stay behind pdl_wait(), also where the compiler knows them read-only
template <typename T>
__device__ __forceinline__ T *after_wait(T *p) {
    asm volatile("" : "+l"(p));
    return p;
}

template <typename... KA, typename... A>
inline cudaError_t launch_pdl(void (*kernel)(KA...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KA>(args)...);
}

}  // namespace mlpg
