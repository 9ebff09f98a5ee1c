// Programmatic dependent launch: a kernel launched with pdl_launch may be set
// up, and its blocks placed, while the kernel before it in the stream drains.
// Each kernel so launched waits at pdl_wait() until that kernel (and with it
// all earlier ones, since each of them waits too) has finished and its
// writes are visible, and must not touch global memory that another kernel
// writes before.  pdl_trigger() lets the next kernel start its own set-up.
// Pointers to what other kernels write are not __restrict__ parameters of a
// kernel so launched: that would promise that nothing, the wait included,
// changes what they point to while the kernel runs, and allow their loads
// before the wait or through the non-coherent path, whose lines an earlier
// kernel's blocks may have fetched before the data were there.  (Tables laid
// out at set-up may be.)  The kernels load a point's values before they store.
// A kernel that allocates tensor memory triggers only once its block holds its
// columns: the allocation waits for columns without a limit, and blocks of
// several launches and contexts share an SM's 512.  A dependent's block is
// placed when every block before it has triggered, so whoever holds columns
// while it waits, waits for blocks that hold theirs, and no cycle can form.
// (Triggered earlier, a dependent could take the columns that its own
// predecessor was still to get.)
// The loops of a small-grid minimisation are chains of kernels of a few
// microseconds, where the gap between dependent kernels (about 1.5 us) counts.
// Measured (GB300, one evaluation in a captured loop, plain -> dependent):
// VT84F 32^3 73.4 -> 63.6 us, 48^3 92.3 -> 85.4, 128^3 572 -> 566; ftTF 60^3
// 92.7 -> 87.2, 32^3 unchanged.
#pragma once

#include <cuda_runtime.h>

namespace ofdft {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_enter()
{
    pdl_wait();
    pdl_trigger();
}

template <typename... P, typename... A>
void pdl_launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args)
{
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &at;
    c.numAttrs = 1;
    cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}

}  // namespace ofdft
