#pragma once

#include "any_lines.cuh"
#include "any_part.h"
#include "any_z.cuh"
#include "launch.cuh"

namespace psatd {

template <typename T, int CLS>
void AnyPart<T, CLS>::fwd_x(dim3 grid, const DevPlan& P, const FieldPtrs& f, void* spec, int64_t sstride,
                            const RowJob* jobs, const LineCfg& c, const GatherGrid* ggrid, int ngather,
                            cudaStream_t st) {
  cx<T>* s = static_cast<cx<T>*>(spec);
  if (ggrid)
    launch_ordered(P.order, k_fwd_x<T, CLS, true>, grid, c.threads, c.smem, st, P, f, s, sstride, jobs, ggrid, ngather, c.lg);
  else
    launch_ordered(P.order, k_fwd_x<T, CLS, false>, grid, c.threads, c.smem, st, P, f, s, sstride, jobs, ggrid, ngather, c.lg);
}

template <typename T, int CLS>
void AnyPart<T, CLS>::col(dim3 grid, int dir, int axis, const DevPlan& P, void* spec, int64_t sstride,
                          const ColJob* jobs, const LineCfg& c, cudaStream_t st) {
  cx<T>* s = static_cast<cx<T>*>(spec);
  if (dir < 0)
    launch_ordered(P.order, k_col<T, -1, CLS>, grid, c.threads, c.smem, st, P, s, sstride, axis, jobs, c.lg);
  else
    launch_ordered(P.order, k_col<T, 1, CLS>, grid, c.threads, c.smem, st, P, s, sstride, axis, jobs, c.lg);
}

template <typename T, int CLS>
void AnyPart<T, CLS>::inv_x(dim3 grid, const DevPlan& P, const FieldPtrs& f, void* spec, int64_t sstride,
                            const RowJob* jobs, const LineCfg& c, int interior_only, cudaStream_t st) {
  launch_ordered(P.order, k_inv_x<T, CLS>, grid, c.threads, c.smem, st, P, f, static_cast<const cx<T>*>(spec), sstride, jobs,
                                                   interior_only, c.lg);
}

template <typename T, int CLS>
void AnyPart<T, CLS>::z_update(dim3 grid, int form, const DevPlan& P, void* spec, int64_t sstride, const ColJob* jobs,
                               const LineCfg& c, int nft, cudaStream_t st) {
  cx<T>* s = static_cast<cx<T>*>(spec);
  const int NT = c.threads;
  switch (form) {
    case kVacuum: launch_ordered(P.order, k_z_update<T, kVacuum, CLS>, grid, NT, c.smem, st, P, s, sstride, jobs, nft, c.lg); break;
    case kJForm: launch_ordered(P.order, k_z_update<T, kJForm, CLS>, grid, NT, c.smem, st, P, s, sstride, jobs, nft, c.lg); break;
    case kPml: launch_ordered(P.order, k_z_update<T, kPml, CLS>, grid, NT, c.smem, st, P, s, sstride, jobs, nft, c.lg); break;
    default: launch_ordered(P.order, k_z_update<T, kRhoForm, CLS>, grid, NT, c.smem, st, P, s, sstride, jobs, nft, c.lg); break;
  }
}

template <typename T, int CLS>
cudaError_t AnyPart<T, CLS>::configure(int smem) {
  cudaError_t e = cudaSuccess;
  for (const void* k : {(const void*)k_fwd_x<T, CLS, false>, (const void*)k_fwd_x<T, CLS, true>,
                        (const void*)k_inv_x<T, CLS>, (const void*)k_col<T, -1, CLS>, (const void*)k_col<T, 1, CLS>,
                        (const void*)k_z_update<T, kVacuum, CLS>, (const void*)k_z_update<T, kJForm, CLS>,
                        (const void*)k_z_update<T, kRhoForm, CLS>, (const void*)k_z_update<T, kPml, CLS>}) {
    // the opt-in maximum less the kernel's static shared memory
    cudaFuncAttributes fa{};
    cudaError_t r = cudaFuncGetAttributes(&fa, k);
    if (r == cudaSuccess)
      r = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem - (int)fa.sharedSizeBytes);
    if (r != cudaSuccess) e = r;
  }
  return e;
}

}  // namespace psatd
