// Programmatic dependent launch of the step kernels.  A step reads what the step before it
// wrote, so on a stream its launch would wait for that kernel to end, and the launch and the
// CTAs' set-up would lie bare between steps.  Launched with the programmatic attribute, a
// kernel's CTAs start as those of the kernel before it run out, do the work that depends on
// no other kernel (barriers, tensor memory, loads of W and the sponge, which are complete
// when a call starts) and then wait for the kernel before to end.  Measured on GB300, whole
// calls: 2-D 517 x 900 at 16th order 3.09 -> 2.09 ms (500 steps), 96^3 16th-order gradient
// 23.9 -> 20.4 ms, serving mix 39 -> 34 ms, 64-shot FWI iteration 95.9 -> 93.4 ms, 1024^3
// forward 379 -> 349 ms.  (Which streaming steps are launched so: k_step3d.cu.)
//
// Such a kernel runs while the one before it still writes, so what that one or an earlier
// programmatic kernel may write (states, gradient sums, codes, scales, maxima, traces) is not
// read-only for its lifetime: it is read after the wait, with plain or volatile loads, through
// pointers without __restrict__.  The non-coherent path (__ldg, or what the compiler makes of
// const and __restrict__) asks for memory that nobody writes while the kernel runs, and lets a
// load move above the wait.  It stays for what is complete before a call's first step: W, the
// sponge, the receiver map and the tap tables.
#pragma once

#include <cuda_runtime.h>

namespace fwi {

// The next kernel of the stream may start its CTAs as this kernel's run out.
__device__ __forceinline__ void pdl_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Returns when the kernels this one follows have ended and their writes are visible.  Every
// thread calls it before it touches anything that work on the stream may write.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// 16 and 8 bytes of such data past L1, for values that a kernel reads once.  (__ldcg and its like
// are no volatile loads: the compiler may move them above the wait.)
__device__ __forceinline__ uint4 load_cg(const uint4 *p)
{
    uint4 v;
    asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

__device__ __forceinline__ uint2 load_cg(const uint2 *p)
{
    uint2 v;
    asm volatile("ld.global.cg.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}

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
