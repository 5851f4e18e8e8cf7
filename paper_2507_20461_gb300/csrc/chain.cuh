/*
 * Chained launches (programmatic dependent launch, CUDA programming guide).
 *
 * The kernels of a step depend on each other in a row, and a small grid's
 * step is mostly the time between them.  A kernel launched with launch_chained
 * may be brought onto the SMs while the one before it in the stream still
 * drains; its first statement, after_previous, waits until that kernel has
 * ended and its writes are visible, and lets the next one be brought up.  So
 * no kernel reads or writes memory before everything earlier in the stream is
 * complete (each waits for its predecessor, which waited for its own), and the
 * order is that of ordinary launches.
 * GB300, a pass, plain / chained: 4 steps of 64^2 mixed 245 / 178 us, 20 steps of
 * 400 cells 1055 / 964 us, 2 steps of 2048^2 3.97 / 3.92 ms, 256^3 equal.
 */
#pragma once
#include <cuda_runtime.h>

namespace gks {

/* First statement of a kernel that launch_chained starts, before any access to
 * memory.  The kernel is on the SMs while its predecessors, and theirs, still
 * write.  The wait orders what the compiler must take as touched by it: the
 * target of a __restrict__ parameter is not, and a load through a const one may
 * even become non-coherent.  So the pointers of such a kernel carry no
 * __restrict__, but for what no kernel of the chain writes (a batch's
 * descriptors and tile lists, uploaded before its first launch), and nothing is
 * read by __ldg, whose target may not change while the kernel is resident.
 * Without either a load does not move past a store before it, so the updates
 * read everything before they store. */
__device__ __forceinline__ void after_previous()
{
#ifdef __CUDA_ARCH__
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
#endif
}

/* Blocks from the last to the first (rev) or in order: the kernels of a step
 * alternate, so each begins with what the one before it wrote last, which L2
 * still holds (99 x 64 x 50 viscous 1246 to 1218 us a pass, 256^3 24.57 to 24.51 ms). */
__device__ __forceinline__ unsigned block_in_order(bool rev) { return rev ? gridDim.x - 1 - blockIdx.x : blockIdx.x; }

#ifdef __CUDACC__
template <typename... K, typename... A>
cudaError_t launch_chained(void (*kernel)(K...), dim3 blocks, unsigned threads, cudaStream_t stream, A... args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = blocks;
    cfg.blockDim = dim3(threads);
    cfg.stream = stream;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<K>(args)...);
}
#endif

} // namespace gks
