// Launches whose prologue overlaps the kernel before them (programmatic
// dependent launch), for the kernels of one evaluation.
//
// A kernel launched by launch_chained may start while its predecessor on the
// stream still runs (once every CTA of that one has called chain_release, or
// has ended) and calls chain_wait before it touches anything another kernel
// writes or reads: the wait ends when the predecessor has ended and its writes
// are visible. Every kernel of the chain waits, so the order is transitive. A
// kernel that does not call chain_wait must not be launched this way.
//
// What it saves is the launch latency and the prologue (barrier and
// tensor-memory set-up, tables) of each of the five to seven kernels of an
// evaluation. `chain` off is an ordinary launch: a plan chains (chain_call in
// mfbd_api.cu) where that was faster.
#pragma once

#include <cuda_runtime.h>

namespace mfbd_dev {

__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... Params, class... Args>
cudaError_t launch_chained(bool chain, void (*kern)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                           const Args&... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = chain ? 1 : 0;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, Params(args)...);
    if (e != cudaSuccess) cudaGetLastError();
    return e;
}

}  // namespace mfbd_dev
