// Chained launches.  Most of the library's work is chains of short kernels, each
// reading what the one before it wrote.  launch() marks a kernel so that it may
// be set up on the device while the one before it in the stream ends; every
// kernel launched so calls chain_enter() before its first access to memory that
// another kernel writes or reads, which waits for the kernels before it, their
// memory operations included.
// A kernel's end is what lets the next one be placed.  Letting it be placed
// earlier (griddepcontrol.launch_dependents after the wait) made the n = 4096 LU
// 2.5 ms slower: blocks placed while the tensor-core GEMM holds most SMs crowd on
// the few that are free.
// What such a kernel reads is loaded by plain loads, never as read-only data: a
// read-only load could be moved above the wait or served from a line cached
// before it.
// ozlu_gemm by FP8, DD 32 x 32 x 32 (4 kernels): 20.6 us with plain launches, 13.3
// with these; QD 96 x 96 x 96: 32.8 and 22.3; QD n = 1000 LU: 8.03 and 7.48 ms.
#pragma once

#include <cuda_runtime.h>

namespace ozlu {

__device__ __forceinline__ void chain_enter() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// kernel<<<grid, block, smem, s>>>(args...), as above
template <typename... P, typename... A>
cudaError_t launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, const A&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace ozlu
