// Host side of the generic kernels (any_lines.cuh, any_z.cuh): dispatch by
// precision and radix class, and the launch sizes that a list of lines needs.
#include <cuda_runtime.h>

#include <cstdint>

#include "any_fft.cuh"
#include "any_part.h"
#include "psatd_internal.h"

namespace psatd {

extern template struct AnyPart<float, 0>;
extern template struct AnyPart<float, 1>;
extern template struct AnyPart<double, 0>;
extern template struct AnyPart<double, 1>;

namespace {

constexpr int64_t kMaxGridX = 2147483647LL;

// f(AnyPart) of the precision and class, then the launch status
template <typename F>
cudaError_t dispatch(int prec, const LineCfg& c, int64_t njobs, int nf, F&& f) {
  if (njobs <= 0 || nf <= 0) return cudaSuccess;
  if (njobs > kMaxGridX) return cudaErrorInvalidConfiguration;
  const dim3 grid((unsigned)njobs, nf);
  if (prec == 32) {
    if (c.cls)
      f(AnyPart<float, 1>{}, grid);
    else
      f(AnyPart<float, 0>{}, grid);
  } else {
    if (c.cls)
      f(AnyPart<double, 1>{}, grid);
    else
      f(AnyPart<double, 0>{}, grid);
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_fwd_x(int prec, const DevPlan& P, const FieldPtrs& f, int nf, void* spec, int64_t sstride,
                         const RowJob* jobs, int64_t njobs, const LineCfg& c, const GatherGrid* ggrid, int ngather,
                         cudaStream_t st) {
  return dispatch(prec, c, njobs, nf,
                  [&](auto p, dim3 g) { p.fwd_x(g, P, f, spec, sstride, jobs, c, ggrid, ngather, st); });
}

cudaError_t launch_col(int prec, int dir, int axis, const DevPlan& P, void* spec, int64_t sstride, int nf,
                       const ColJob* jobs, int64_t njobs, const LineCfg& c, cudaStream_t st) {
  return dispatch(prec, c, njobs, nf, [&](auto p, dim3 g) { p.col(g, dir, axis, P, spec, sstride, jobs, c, st); });
}

cudaError_t launch_inv_x(int prec, const DevPlan& P, const FieldPtrs& f, int nf, void* spec, int64_t sstride,
                         const RowJob* jobs, int64_t njobs, const LineCfg& c, int interior_only, cudaStream_t st) {
  return dispatch(prec, c, njobs, nf,
                  [&](auto p, dim3 g) { p.inv_x(g, P, f, spec, sstride, jobs, c, interior_only, st); });
}

cudaError_t launch_z_update(int prec, int form, const DevPlan& P, void* spec, int64_t sstride, const ColJob* jobs,
                            int64_t njobs, const LineCfg& c, int nft, cudaStream_t st) {
  return dispatch(prec, c, njobs, 1,
                  [&](auto p, dim3 g) { p.z_update(g, form, P, spec, sstride, jobs, c, nft, st); });
}

cudaError_t configure_kernels(int prec, int smem) {
  const cudaError_t a = prec == 32 ? AnyPart<float, 0>::configure(smem) : AnyPart<double, 0>::configure(smem);
  const cudaError_t b = prec == 32 ? AnyPart<float, 1>::configure(smem) : AnyPart<double, 1>::configure(smem);
  return a != cudaSuccess ? a : b;
}

int line_tile_width(int prec) { return prec == 32 ? line_tile<float>() : line_tile<double>(); }

// Shared memory, threads and class that lines of length n need, on top of
// what c already covers (rows: x lines, else columns).
void line_cover(LineCfg& c, int prec, const AxisPlan& a, bool rows) {
  const int w = line_tile_width(prec), csz = prec == 32 ? 8 : 16;
  const int len = !rows ? a.n : prec == 32 ? row_line_pitch(a) : (a.n + 1) | 1;
  const int r = a.r1 > a.r2 ? a.r1 : a.r2;
  c.smem = c.smem > w * len * csz ? c.smem : w * len * csz;
  const int t = (w * r + 31) / 32 * 32;
  c.threads = c.threads > t ? c.threads : t;
  if (r > 16) c.cls = 1;
}

// Columns per z tile (a power of two, its logarithm in c.lg) and the shared
// memory of the longest line n2_max: the widest tile of at most 128-byte rows
// that leaves room for the blocks an SM can hold (FP32 two of 256 threads: two
// boxes of 384 x 256 x 256 2.90 ms per step with 8 columns, 98 KB, against 3.26
// with 4; FP64 three of 128: 128^3 rho form 2.62 ms either way, 64 x 64 x 256
// 0.93 against 0.98 with two wider ones) and gives the `columns` columns of the
// launch a tile per SM (64^3, 10 slots: 264 tiles of 8 columns run at once, 528
// of 4 columns took two waves, 16.5 us against 12); `widest` > 0: no wider than
// that.
void z_cover(LineCfg& c, int prec, int form, int n2_max, int64_t columns, int widest, int sms, int optin) {
  const int csz = prec == 32 ? 8 : 16, ns = spec_slots(form);
  const int lo = prec == 32 ? 2 : 1, hi = prec == 32 ? 4 : 3;   // log2 of the narrowest and widest tile
  const int budget = (prec == 32 ? 112 : 75) * 1024;
  auto bytes = [&](int lg) { return ns * z_slot_pitch(csz, n2_max, 1 << lg) * csz; };
  int lg = hi;
  while (lg > lo && (bytes(lg) > budget || (columns >> lg) < sms)) --lg;
  while (lg > lo - 1 && (bytes(lg) > optin || (widest > 0 && (1 << lg) > widest))) --lg;
  c.lg = lg;
  c.smem = bytes(lg);
}

}  // namespace psatd
