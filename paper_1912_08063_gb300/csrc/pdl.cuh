// Programmatic dependent launch of the step kernels.  A step reads what the step before it
// wrote, so on a stream its launch would wait for that kernel to end, and the launch and the
// CTAs' set-up would lie bare between steps.  Launched with the programmatic attribute, a
// kernel's CTAs start as those of the kernel before it run out, do the work that depends on
// no other kernel (barriers, tensor memory, loads of W and the sponge, which are complete
// when a call starts) and then wait for the kernel before to end.  Measured on GB300, whole
// calls: 2-D 517 x 900 at 16th order 3.09 -> 2.09 ms (500 steps), 96^3 16th-order gradient
// 23.9 -> 20.4 ms, serving mix 39 -> 34 ms, 64-shot FWI iteration 95.9 -> 93.4 ms, 1024^3
// forward 379 -> 349 ms.  (Which streaming steps are launched so: k_step3d.cu.)
#pragma once

#include <cuda_runtime.h>

namespace fwi {

// The next kernel of the stream may start its CTAs as this kernel's run out.
__device__ __forceinline__ void pdl_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Returns when the kernels this one follows have ended and their writes are visible.  Every
// thread calls it before it touches anything that work on the stream may write.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... P, class... A>
cudaError_t launch_pdl(void (*fn)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, const A &...args)
{
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fn, args...);
}

}  // namespace fwi
