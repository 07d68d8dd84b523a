// Launchers of the generic kernels for one precision and radix class; each is
// instantiated in a translation unit of its own (any_part_<k>.cu).
#pragma once

#include "fft_codelets.cuh"
#include "psatd_internal.h"

namespace psatd {

template <typename T, int CLS>
struct AnyPart {
  static void fwd_x(dim3 grid, const DevPlan& P, const FieldPtrs& f, void* spec, int64_t sstride, const RowJob* jobs,
                    const LineCfg& c, const GatherGrid* ggrid, int ngather, cudaStream_t st);
  static void col(dim3 grid, int dir, int axis, const DevPlan& P, void* spec, int64_t sstride, const ColJob* jobs,
                  const LineCfg& c, cudaStream_t st);
  static void inv_x(dim3 grid, const DevPlan& P, const FieldPtrs& f, void* spec, int64_t sstride, const RowJob* jobs,
                    const LineCfg& c, int interior_only, cudaStream_t st);
  static void z_update(dim3 grid, int form, const DevPlan& P, void* spec, int64_t sstride, const ColJob* jobs,
                       const LineCfg& c, int nft, cudaStream_t st);
  static cudaError_t configure(int smem);   // raise the dynamic shared memory limit
};

}  // namespace psatd
