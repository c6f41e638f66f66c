// Programmatic stream serialisation of kernels that follow one another in a stream.
#pragma once

#include <cuda_runtime.h>

namespace cmlbm {

// Launch with programmatic stream serialisation: the grid is set up while the preceding kernel of
// the stream still runs, and its blocks wait (pdl_wait()) until that kernel has completed and its writes are
// visible.  Back-to-back step kernels otherwise start about 2.4 us apart (dependent launches resolve in 2 us
// ticks): 16^3 FP32 4.1 -> 2.5 us per step, 64^3 13.3 -> 10.9 us.  Without a preceding kernel it is a plain
// launch.  The next grid is not triggered early: its waiting blocks then held slots of the running one
// (32^3: 2.6 -> 4.5 us).
//
// Rules for the kernels launched here:
//  * pdl_wait() comes before the first access to memory that another kernel reads or writes.  Only set-up of
//    the block's own (barriers, tensor memory, prefetched descriptors) may stand before it.
//  * The kernel's life begins before the wait, while the preceding kernel may still be writing.  So memory that
//    a kernel of the stream writes is not read-only for that life: it is read through plain pointers, never
//    through __ldg or a `const T* __restrict__` parameter.  Those allow the load to move above the wait, and
//    its non-coherent form is undefined for such data; a plain pointer is held behind the wait by its "memory"
//    clobber.  `__restrict__` stays right for what is only written, and `const __restrict__` for memory that
//    only the host writes.
template <typename... P, typename... A>
inline cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = st;
    c.attrs = at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}

// Waits until the kernel before this one in its stream has completed and its writes are visible
// (returns at once in a kernel launched without programmatic serialisation, see launch_pdl).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

}  // namespace cmlbm
