// Host side of the generic kernels (any_lines.cuh, any_z.cuh): dispatch by
// precision and radix class, and the launch sizes that a list of lines needs.
#include <cuda_runtime.h>

#include <cstdint>
#include <utility>
#include <vector>

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

cudaError_t configure_kernels(int prec, int smem, int classes) {
  cudaError_t e = cudaSuccess;
  if (classes & 1) e = prec == 32 ? AnyPart<float, 0>::configure(smem) : AnyPart<double, 0>::configure(smem);
  if (e == cudaSuccess && (classes & 2))
    e = prec == 32 ? AnyPart<float, 1>::configure(smem) : AnyPart<double, 1>::configure(smem);
  return e;
}

// Shared memory, threads and class that lines of length n need in tiles of
// 1 << c.lg, on top of what c already covers (rows: x lines, else columns).
void line_cover(LineCfg& c, int prec, const AxisPlan& a, bool rows) {
  const int w = 1 << c.lg, csz = prec == 32 ? 8 : 16;
  const int len = !rows ? a.n : prec == 32 ? row_line_pitch(a) : (a.n + 1) | 1;
  const int r = a.r1 > a.r2 ? a.r1 : a.r2;
  c.smem = c.smem > w * len * csz ? c.smem : w * len * csz;
  // columns of radices above 16 (112 registers): two sub-transforms per thread, so
  // that two or three blocks fit an SM (forward + inverse FFT of 240 x 200 x 180,
  // 200 = 10 * 20: 173 -> 153 us)
  int items = !rows && r > 16 ? (r + 1) / 2 : r;
  // FP64 rows of radices above 16 (252 registers): 128 threads where they hold pass
  // 2, a thread per sub-transform of the smaller radix (line_plan puts it first),
  // so that two blocks fit an SM and one computes while the other loads; pass 1
  // loops.  250^3 vacuum 27.6 -> 23.2 ms per step, 324 x 96 x 96 rho form 4.75 ->
  // 4.23, 500 x 96 x 96 7.25 -> 6.69.  Above 128 one block fits either way and
  // needs its warps: 1000 x 64 x 64 6.01 ms with 224 threads, 6.44 with 160.
  if (rows && prec == 64 && r > 16 && w * a.r1 <= 128) items = 128 / w;
  const int t = (w * items + 31) / 32 * 32;
  c.threads = c.threads > t ? c.threads : t;
  if (r > 16) c.cls = 1;
}

namespace {
// warp instructions (in lane operations) of `items` threads of `ops` operations each in blocks of nt
double lane_ops(int items, double ops, int nt) { return (items + nt - 1) / nt * nt * ops; }
double radix_total(int r) { return r * radix_ops(r); }
}  // namespace

// Tile of the x or y passes over `lines` (length, number of lines): FP32 16, FP64
// the one of 8 and 16 that wastes fewer lanes in the last warp of a pass, 8
// while 16 would leave SMs without work (`sms` x 4 tiles of six slots) and for
// radices above 16 (registers).  90 = 9 * 10: 72 and 80 threads of 96 in tiles
// of 8, 144 and 160 of 160 in tiles of 16.
int line_lg(int prec, const std::vector<std::pair<AxisPlan, int64_t>>& lines, int sms) {
  if (prec == 32) return 4;
  double cost[2] = {0, 0};
  int64_t total = 0;
  for (const auto& l : lines) {
    const AxisPlan& a = l.first;
    if (a.r1 > 16 || a.r2 > 16) return 3;
    for (int k = 0; k < 2; ++k) {
      const int w = 8 << k;
      cost[k] += (double)l.second / w *
                 (lane_ops(w * a.r2, radix_total(a.r1), 32) + lane_ops(w * a.r1, radix_total(a.r2), 32));
    }
    total += l.second;
  }
  return total * 6 / 16 >= 4 * sms && cost[1] < 0.97 * cost[0] ? 4 : 3;
}

// Threads of a z block: FP32 256; FP64 128, or 96 where that wastes fewer lanes over
// the passes and the update (some 190 operations per mode) of the lines of
// `axes` and the launch fills the SMs (`tiles`; a small one needs every warp: 32^3
// 46 us per step with 128, 48 with 64).  J form, z length 72: 128 threads run
// 77 % full, 96 threads 95 %; with the tiles of line_lg, 8 boxes of 100 x 90 x 72
// 6.33 -> 5.70 ms.
void z_threads_for(LineCfg& c, int prec, int form, int nft, const std::vector<AxisPlan>& axes, int64_t tiles,
                   int sms) {
  c.threads = prec == 32 ? 256 : 128;
  if (prec == 32 || tiles < 3 * sms) return;
  const int tx = 1 << c.lg, fout = fields_out(form);
  auto cost = [&](int nt) {
    double v = 0;
    for (const AxisPlan& a : axes)
      v += (lane_ops(nft * a.r2 * tx, radix_total(a.r1), nt) + lane_ops(nft * a.r1 * tx, radix_total(a.r2), nt) +
            lane_ops(a.n * tx, 190, nt) + lane_ops(fout * a.r1 * tx, radix_total(a.r2), nt) +
            lane_ops(fout * a.r2 * tx, radix_total(a.r1), nt)) /
           ((double)a.n * tx);
    return v;
  };
  if (cost(96) < 0.97 * cost(128)) c.threads = 96;
}

// Whether the z pass may start while the y pass drains (kChained).  Its early
// blocks go wherever room is, so with more than one tile per SM but fewer than
// the blocks an SM holds (registers: 3, 2 with radices above 16; shared memory)
// they stack on the SMs that drain first and leave others idle, which the FP64
// pipe does not hide: one step of a 64^3 box, vacuum (264 tiles) 292 us chained, 248
// not; 48^3 132, 118; 32 x 32 x 256 314, 257.  With fewer or more tiles it gains: 16^3 33.1
// against 34.9, 64^3 rho form (528) 329, 332.  FP32 is the same either way.
int z_chains(int prec, const LineCfg& c, int64_t tiles, int sms) {
  if (prec == 32 || tiles <= sms) return 1;
  const int hold = c.cls ? 2 : 3, fit = 227 * 1024 / (c.smem + 1024);
  return (tiles + sms - 1) / sms >= (hold < fit ? hold : fit);
}

// Columns per z tile (a power of two, its logarithm in c.lg) and the shared
// memory of the longest line n2_max: the widest tile of at most 128-byte rows
// that leaves room for the blocks an SM can hold (FP32 two of 256 threads: two
// boxes of 384 x 256 x 256 2.90 ms per step with 8 columns, 98 KB, against 3.26
// with 4; FP64 three of 128: 128^3 rho form 2.62 ms either way, 64 x 64 x 256
// 0.93 against 0.98 with two wider ones) and gives the `columns` columns of the
// launch a tile per SM (64^3, 10 slots: 264 tiles of 8 columns run at once, 528
// of 4 columns took two waves, 16.5 us against 12); `widest` > 0: no wider than
// the power of two from there up.
void z_cover(LineCfg& c, int prec, int form, int n2_max, int64_t columns, int widest, int sms, int optin) {
  const int csz = prec == 32 ? 8 : 16, ns = spec_slots(form);
  const int lo = prec == 32 ? 2 : 1, hi = prec == 32 ? 4 : 3;   // log2 of the narrowest and widest tile
  const int budget = (prec == 32 ? 112 : 75) * 1024;
  auto bytes = [&](int lg) { return ns * z_slot_pitch(csz, n2_max, 1 << lg) * csz; };
  int lg = hi;
  while (lg > lo && (bytes(lg) > budget || (columns >> lg) < sms)) --lg;
  while (lg > lo - 1 && (bytes(lg) > optin || (widest > 0 && (1 << lg) >= 2 * widest))) --lg;
  c.lg = lg;
  c.smem = bytes(lg);
}

}  // namespace psatd
