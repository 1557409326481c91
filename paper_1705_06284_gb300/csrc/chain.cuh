// Transform stages launched ahead of their turn.  Every stage needs all of the
// one before it, so a plain launch leaves the GPU idle from the last block of
// one to the first of the next.  With programmatic stream serialisation the
// next kernel's blocks are set up while this one runs and wait on the device.
// chain_begin is the first statement of such a kernel, for all its threads: it
// allows the next launch and then waits until the kernel before has completed
// with its writes visible.  Since every block waits before it does anything
// else, completion is transitive along the chain and buffers may be reused as
// in an ordinary stream.  `chained` is the kernel's last argument, whether it
// belongs to such a chain (the forward z pass, which begins one, is launched the
// ordinary way and only allows the next launch: its wait returns at once).
// Other launches skip both: the x stage's tens of thousands of blocks that find
// nothing to do paid for the wait (0.47 -> 0.57 ms at 512^3).
#pragma once

#include <cuda_runtime.h>

#include "fbs_internal.h"

namespace fbs {

__device__ __forceinline__ void chain_begin(int chained) {
    if (!chained) return;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Chaining pays where the gaps between launches count and costs where the
// blocks waiting for their turn displace running ones.  Measured with every
// launch of an evaluation chained: 32^3, 6 bins 62.5 -> 55 us, but 192^3, 48
// bins (levels of 60 M and 104 M shell-field values) 1,337 -> 1,435 us.  With
// the stages alone 62.5 -> 54.3 us, 64^3, 12 bins 74.5 -> 66.0 us, 108^3, 10 bins
// with quadruplets (12.6 M values) 303 -> 297 us;
// a chained reduction or contraction, which wait beside long kernels, gave
// nothing or cost 8 us: they are launched the ordinary way.
constexpr long long kChainValues = 1LL << 24;  // at most this many values written by the stage

// k<<<grid, threads, smem, stream>>>(args..., chained), chained to the kernel
// before it when `chained`.
template <class... P, class... A>
void launch_chained(bool chained, void (*k)(P...), dim3 grid, int threads, size_t smem, cudaStream_t stream, A... args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = stream;
    c.attrs = &at;
    c.numAttrs = chained ? 1 : 0;
    FBS_CUDA(cudaLaunchKernelEx(&c, k, args..., (int)chained));
}

}  // namespace fbs
