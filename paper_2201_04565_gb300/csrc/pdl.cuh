// pdl.cuh -- programmatic dependent launch for the time-step chain.
//
// A time step of a small specimen takes less time than the gap between two
// dependent launches (drain, launch latency, table loads). The kernels of the
// chain are therefore launched with programmatic stream serialization: the
// next kernel's blocks become resident while the current one still runs, load
// what no time step writes (tables, topology), and wait on the device until
// the kernels before it have completed and their writes are visible.
//
// Rules that every kernel of the chain keeps:
//   - pdl_begin() comes before the first read or write of anything that a
//     kernel of the chain writes; only constants of the context are read
//     before it;
//   - what an earlier kernel of the chain wrote is not read through const
//     __restrict__ parameters (such loads count as invariant and may be moved
//     above the wait);
//   - the next kernel is released only after the wait, so that at most two
//     kernels of the chain are in flight.
// Launched without the attribute, pdl_begin() does nothing.
#pragma once

#include <cuda_runtime.h>

namespace lsm {

__device__ __forceinline__ void pdl_begin()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... P, typename... Q>
cudaError_t launch_pdl(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Q &&...args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

}  // namespace lsm
