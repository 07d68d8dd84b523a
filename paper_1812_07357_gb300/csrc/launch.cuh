// Order of a launch against the launch before it in the stream, and the
// device side of it (programmatic dependent launch).
//
//   kOrdinary  starts when everything before it has finished.
//   kChained   starts while the launch before it drains: its blocks read the
//              plan's constant tables, then wait for that launch to finish
//              (grid_order).  For a launch whose predecessor is a single
//              launch of the same call, so that its end is the end of all work
//              before it.
//   kLeads     ordinary, and the launches after it run beside it: the first launch
//              of a pass over boxes of several plane shapes or z lengths.
//   kBeside    starts while the launch before it drains and computes beside it:
//              the later launches of such a pass.  Its grid has one block (or
//              cluster) more than it has work, which only waits for that launch
//              to finish (grid_join), so the end of each launch of the pass
//              implies the end of the one before it.  The launch after the pass is
//              kOrdinary again.  That wait is what orders the pass in a CUDA graph, whose
//              only full edge into the next pass comes from the pass's last
//              launch (a stream would wait for all of them).  It always ends: a
//              launch starts beside another only when every block of that one
//              has started.
//
// Every kernel here lets its successor start as soon as all its own blocks have
// (grid_release), so a successor's blocks only take the room that the last
// wave leaves.
//
// The register kernels have instantiations of their own for kLeads and kBeside
// (MANY): the release alone changed the code of every launch that has no
// successor beside it.  Steps replayed from graphs, without it / with it / with a
// join tested behind the loads of the job: 8 boxes of 48^3 rho form 60.3 / 61.7 /
// 61.9 us, 128 boxes of 96^3 2.832 / 2.836 / 2.839 ms.  The join is a block of its own
// because a wait of block 0 at the end of every kernel took 2.909.
//
// Chained are the line kernels (any_lines.cuh, any_z.cuh, the exchange) of calls
// that launch directly: a PIC cycle of a 64^3 box 71 -> 62 us, forward + inverse
// FFT of 240 x 200 x 180 187 -> 177 us.  Not the register kernels: a z block that
// starts on an SM still set up for the plane kernels' shared memory keeps
// their small L1 (128 boxes of 96^3: 2.90 -> 3.22 ms per step).  Not captured
// steps: 32^3 FP64 45 -> 56 us per step.  Beside: the register kernels of a batch
// of many box shapes, 60 launches a step whose tails overlap (40 uneven boxes
// 1.51 -> 1.28 ms per step).
#pragma once

#include <cuda_runtime.h>

#include "psatd_internal.h"

namespace psatd {

__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;"); }
__device__ __forceinline__ void grid_order(int order) {
  grid_release();
  if (order == kChained) asm volatile("griddepcontrol.wait;" ::: "memory");
}
// Whether this block of a kBeside launch is one of the last `n`, which only
// wait (grid_join).
__device__ __forceinline__ bool grid_extra(int order, unsigned n = 1) {
  return order == kBeside && blockIdx.x + n >= gridDim.x;
}
__device__ __forceinline__ void grid_join() {
  grid_release();
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
// The grid of a launch of `blocks` blocks per y index, and the extra ones when kBeside.
inline bool order_of_many(int order) { return order == kLeads || order == kBeside; }
inline dim3 ordered_grid(int order, unsigned blocks, unsigned y, unsigned n = 1) {
  return dim3(blocks + (order == kBeside ? n : 0u), y);
}

template <typename... P, typename... A>
cudaError_t launch_ordered(int order, void (*kernel)(P...), dim3 grid, int threads, int smem, cudaStream_t st,
                           A... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = dim3((unsigned)threads);
  c.dynamicSmemBytes = (size_t)smem;
  c.stream = st;
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &attr;
  c.numAttrs = order == kChained || order == kBeside ? 1 : 0;
  return cudaLaunchKernelEx(&c, kernel, P(args)...);
}

}  // namespace psatd
