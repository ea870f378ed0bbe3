// launch.cuh -- programmatic dependent launch: a call's kernels (spline build, fold, summation) follow one
// another on a stream, and each may be put on the chip while the one before it still runs; it does
// what needs none of that one's results (barriers, tensor memory, harmonics), then waits for its
// completion.  Every kernel launched by launch_pdl executes pdl_wait() in every block, and before it reads
// or writes anything that an earlier kernel may use, with these exceptions:
//   k_rb_pack_a, k_rb64_pack_a  write the packed coefficients (scratch at the address of an earlier call's)
//                               and read the caller's coefficients before it;
//   k_direct_ring, k_mode_select  read the caller's arrays before it;
//   k_build                     reads jobs and factors, which the host has waited for, before it.
// The first four are right only because the kernel just before each is launched plainly (<<<>>>: it starts
// when everything queued ahead has ended) and uses none of that memory otherwise.  That launch is
// checked before the dependent one is queued: without it the dependent one would overlap whatever came before.
//
// What the kernels before it write is read by ordinary loads: not by __ldg, nor through a const
// __restrict__ pointer.  Those may take the read-only path, which is specified only for data that does
// not change while the kernel runs (its blocks are there before that data is), and the compiler may
// move them up across the wait.
#pragma once

#include <cuda_runtime.h>

namespace fewsum {

// Waits until the kernels this one depends on have completed and their writes are visible.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Lets the next kernel's blocks be scheduled once every block of this one has got here.
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... P, typename... A>
inline cudaError_t launch_pdl(void (*kernel)(P...), unsigned grid, unsigned threads, size_t smem,
                              cudaStream_t st, A &&...args)
{
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

}  // namespace fewsum
