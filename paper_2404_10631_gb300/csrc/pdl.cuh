// Programmatic dependent launch: the kernels of one call follow each other in
// a stream, most of them a few microseconds long, so the launch of the next
// one is made while the one before is still running. A kernel launched so may
// start before its predecessor has finished: pdl_wait() is its first
// statement that touches memory (it returns when every kernel before it has
// completed and its writes are visible; at once after an ordinary launch).
// pdl_next() lets the successor's CTAs be placed from now on. Only kernels of
// a few microseconds give that leave, after their own wait, and those that may
// have more to do only once they know that they have not: CTAs that wait
// hold their place, which other streams' kernels may need. (The second KNN
// pass gave it at once: a 48 x 48 frame on another stream beside a 1024 x 1024
// map of noise, lambda 0.1, took 39 ms, now 0.09 ms; the filter alone on 416 x
// 512 23.0 -> 23.4 us.) Measured, calls of
// one context back to back: a 48 x 48 x 125 snapshot classified (9 kernels) 88
// -> 68 us, the PCA of 416 x 512 x 128 107 -> 91 us, the filter alone (2
// kernels) 28.7 -> 23.3 us; four pushbroom frames in flight 301 -> 309 us, all
// of 303 - 323 us from run to run.
#pragma once

#include <cuda_runtime.h>

namespace hsc {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_next()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// kern<<<grid, block, smem, st>>>(args...), allowed to start before the
// stream's previous kernel has finished.
template <typename... P, typename... A>
inline cudaError_t launch_pdl(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                              A... args)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, P(args)...);
}

}  // namespace hsc
