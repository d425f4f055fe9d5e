// Dependent launches: the kernels of a run follow one another on one stream,
// and on small maps the gaps between them (the next grid is set up only once
// the last block has left) are a good part of its time.
//
// A kernel launched with launch_next may be set up while the kernel before it
// on the stream still runs: its blocks take places that are free and stop in
// grid_wait() until that kernel has completed and its writes are visible.
// Every thread of such a kernel calls grid_wait() before it touches memory,
// so a kernel's end implies the end of all before it, and a later kernel's
// wait for its predecessor covers the whole chain.  grid_release() lets the
// next such launch be set up; the last kernel of a call does not call it, and
// the first kernel of a run is a plain launch, so that neither a caller's own
// work nor the run starts early.  Both are no-ops between plain launches, and a
// launch that follows anything but a kernel is a plain one.
// Measured against plain launches: a replayed run of a 128x128 plane 29.7 to
// 28.8 us, of a 200x200x150 map with its network passes 383 to 370 us, of a
// 160x160x120 map 110.7 to 109.8 us; not replayed, 72 to 63 us, 427 to 399 us
// and 151 to 138 us.  A batch of eight planes and eight volumes: no change.
#pragma once
#include <cuda_runtime.h>

namespace gk {

__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... K, class... A>
inline cudaError_t launch_next(void (*kernel)(K...), dim3 grid, unsigned threads, size_t smem, cudaStream_t s,
                               A&&... args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<K>(args)...);
}

}  // namespace gk
