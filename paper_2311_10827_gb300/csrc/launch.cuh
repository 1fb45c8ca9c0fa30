// Launching the kernels of a step loop back to back.  Internal header.
//
// A step's kernel depends on the whole of the one before it, so an ordinary
// launch leaves the GPU idle between them: the last CTAs drain, their stores
// are flushed, then the next grid is set up and scheduled.  These kernels are
// launched with programmatic stream serialization: the next grid is set up and
// scheduled once every CTA of the one before has exited, and waits in pdl_wait
// until that grid's stores are visible.  Every read or write of device memory
// follows pdl_wait, so the order of the stream is kept; a kernel launched
// without the attribute is serialized as usual.  Launches can be captured into
// graphs, which keep the dependency kind.
//
// Measured (whole runs, ordinary launches -> these): 301 x 203 FP32 with
// diagnostics every 25 steps 1917 -> 1485 us per 200 steps, the adjoint of 400
// steps at 512 x 512 25.4 -> 22.0 ms, 128 x 128 FP32 in graphs 1787 -> 1680 us per
// 400 steps, 100 x 75 x 130 BF16 offsets 7.84 -> 7.59 ms.  Scheduling the next
// grid earlier (griddepcontrol.launch_dependents at the start of a kernel) was
// worse: 1024 x 1024 3446 -> 3574 us per 100 steps against 3424 this way, its
// waiting CTAs taking the slots of SMs that still work.
#pragma once

#include <cuda_runtime.h>

namespace wblbm {

// Waits until the grid before this one has completed and its stores are
// visible, and passes on an index.  The kernels read what that grid
// wrote through the read-only path, and the compiler takes such loads for
// loads of constants, which a memory clobber does not hold back: only an address
// formed from a value that the wait itself defines orders them.  So a kernel
// takes an index along x, of its block or its thread, from here, and every
// address of such a load contains it; a load whose address contains neither
// takes its pointer through after_wait.
__device__ __forceinline__ int pdl_wait(unsigned index)
{
    asm volatile("griddepcontrol.wait;" : "+r"(index)::"memory");
    return (int)index;
}
// p, not before a pdl_wait above (volatile statements keep their order).
template <class T>
__device__ __forceinline__ T *after_wait(T *p)
{
    asm volatile("" : "+l"(p));
    return p;
}

template <class... P, class... A>
cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                       A... args)
{
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace wblbm
