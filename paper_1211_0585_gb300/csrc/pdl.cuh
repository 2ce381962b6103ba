// Programmatic dependent launch: a kernel of an iteration is launched while the
// one before it still runs, and waits on the device for that one's end and
// memory before it reads anything of the iteration. The launch, the block
// scheduling and the reads of tables that no kernel of an iteration writes then
// overlap the tail of the kernel before: 6 % of the cooled solve at Nside 16 (four
// kernels of 4 to 12 us an iteration), 1 to 2 % at Nside 256. Every kernel launched this way calls
// pdl_wait() in every thread before any return, so that "the one before has
// ended" also covers the ones before that.
#pragma once

#include <cuda_runtime.h>

namespace wfk {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// the next kernel of the stream may be scheduled once every CTA of this one has come here (after pdl_wait: before it,
// whole graphs of small kernels sat on the SMs waiting for one another)
__device__ __forceinline__ void pdl_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Up to a CTA an SM: a larger grid's first CTAs (the longest, where a launch orders them so) would pile up on the SMs
// that the kernel before left first instead of spreading, and the cooled solve at Nside 512 took 507 ms instead of
// 455.
constexpr unsigned kPdlCtas = 152;

template <class... P, class... A>
void launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, const A &...args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = grid.x * grid.y * grid.z <= kPdlCtas;
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = s;
  c.attrs = &at;
  c.numAttrs = 1;
  cudaLaunchKernelEx(&c, kernel, P(args)...);
}

}  // namespace wfk
