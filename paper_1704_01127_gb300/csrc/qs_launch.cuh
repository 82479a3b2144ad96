// Launches whose start may overlap the end of the kernel before them on the
// state's stream.  Inside qs_run_circuit consecutive sweeps are chained
// (qs_state::chain): the next sweep's blocks start once every block of the
// present one has started, set up what does not depend on the state (operands
// to shared memory, tensor memory, tables) and wait for the present sweep to
// finish before they touch an amplitude.  Every kernel launched this way calls
// chain_start() first and chain_wait() before its first access to the state;
// without a chain both do nothing.  20 qubits complex64, 16 sweeps: 149 -> 95 us a
// circuit; 83 gates on 16 qubits: 401 -> 323 us (a sweep of a small state is
// launch, set-up and one tile); large states gain the ramp between sweeps
// (28 qubits complex64 1.5%).
#pragma once

#include <cuda_runtime.h>

#include "qs_internal.h"

namespace {

__device__ __forceinline__ void chain_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// chain: s->chain, or false for a kernel that must not start early.  The blocks that do
// start go to the SMs that are free first, as many as fit there, and stay: a kernel
// with a fixed number of blocks for the whole GPU is spread evenly only if no SM can
// hold more than its share of them (the tensor-core sweeps' shared memory, the phase
// sweep's registers), or if it has no work to speak of.
template <typename... P, typename... A>
cudaError_t launch_sweep(const qs_state *s, bool chain, void (*kernel)(P...), int grid, int block, size_t smem, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = (cudaStream_t)s->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = chain ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace
