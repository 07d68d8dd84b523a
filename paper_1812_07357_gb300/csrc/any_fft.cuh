// FFT lines of any 5-smooth length up to 512, the building block of the
// generic kernels (any_lines.cuh, any_z.cuh): every length is done in two
// register passes over run-time radices,
//
//   N = r1 * r2:  pass 1, one thread per (line, n2): a DFT of the r1 samples
//                 (a_in n2 + r2 n1) mod N, n1 < r1;
//                 pass 2, one thread per (line, k1): a DFT of the r2 results,
//                 giving the outputs (a_out k1 + s_out k2) mod N, k2 < r2,
//
// with the prime-factor mapping where r1 and r2 are coprime (no twiddles:
// a_in = r1, a_out = r2 (r2^-1 mod r1), s_out = r1 (r1^-1 mod r2)), else
// decimation in time (a_in = 1, a_out = 1, s_out = r1, twiddles w_N^(n2 k1)).
// The radices are chosen per length by the host (line_plan): fewest
// operations per point, then balanced passes.
//
// Why two large radices: the data pass through shared memory once per pass, so
// two passes are the fewest that a length above the register file allows, and
// the operation count is what bounds FP64 (two FP64 lanes per SM).  Why
// run-time radices: the lengths are about 70 per axis, and a kernel per
// length and form would be hundreds of kernels; the switch is uniform over the
// block and costs one branch per pass.  Lanes run over the lines of a tile
// (128 bytes of columns, or as many rows), so every radix and every index map
// reads shared memory without bank conflicts.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "fft_codelets.cuh"
#include "psatd_internal.h"

namespace psatd {
namespace {

// Lines of a tile (adjacent complex columns, or rows), a power of two 1 << lg:
// FP32 16, 128 bytes of columns; FP64 8 or 16, whichever wastes fewer lanes
// (line_lg: an FP64 instruction costs a warp the same however few lanes it has).
constexpr int kMaxLines = 16;
template <typename T>
__device__ __forceinline__ int line_lg(int lg) {
  return sizeof(T) == 4 ? 4 : lg;
}

// Row pitch of the FP32 x kernels in shared memory: sub-transform k1 at
// k1 * (r2 | 1), so that lanes along n2 and lanes along k1 both read it without
// bank conflicts; the natural-order row needs r1 * r2 of it.
__host__ __device__ __forceinline__ int row_line_pitch(const AxisPlan& a) { return a.r1 * (a.r2 | 1); }

// complex elements between two slots of a z tile: n2 * tx and a pad that puts
// each slot one row (tx columns) further within a 128-byte line, so that lanes
// over (column, slot) read different banks whatever the tile's width
__host__ __device__ constexpr int z_slot_pitch(int csz, int n2, int tx) {
  const int line = 128 / csz, p = n2 * tx;
  return p + (tx % line + line - p % line) % line;
}

// Threads of a block at most: a tile times the largest radix of the class
// (class 0: radices up to 16, class 1: up to 32; FP64 class 1 in tiles of 8).
template <typename T, int CLS>
constexpr int line_threads() {
  return sizeof(T) == 8 && CLS ? 8 * 32 : kMaxLines * (CLS ? 32 : 16);
}

// Call f(std::integral_constant<int, r>) for a run-time radix r.
template <int CLS, typename F>
__device__ __forceinline__ void with_radix(int r, F&& f) {
  switch (r) {
#define PSATD_ARM(R)                          \
  case R:                                     \
    f(std::integral_constant<int, R>{});      \
    break;
    PSATD_ARM(1) PSATD_ARM(2) PSATD_ARM(3) PSATD_ARM(4) PSATD_ARM(5) PSATD_ARM(6) PSATD_ARM(8) PSATD_ARM(9)
    PSATD_ARM(10) PSATD_ARM(12) PSATD_ARM(15) PSATD_ARM(16)
    default:
      if constexpr (CLS) {
        switch (r) {
          PSATD_ARM(18) PSATD_ARM(20) PSATD_ARM(24) PSATD_ARM(25) PSATD_ARM(27) PSATD_ARM(30) PSATD_ARM(32)
        }
      }
      break;
#undef PSATD_ARM
  }
}

// Exact e / d for 0 <= e, d < 2^16 with m = floor((2^32 - 1) / d) + 1 (for
// d = 1 that constant wraps to 0 and the quotient is e itself).
__device__ __forceinline__ unsigned line_magic(int d) { return 0xFFFFFFFFu / (unsigned)d + 1u; }
__device__ __forceinline__ int line_div(int e, unsigned m) { return m ? (int)__umulhi((unsigned)e, m) : e; }

// asynchronous global -> shared copy of one complex element
__device__ __forceinline__ void cp_async(float2* s, const float2* g) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(s);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_async(double2* s, const double2* g) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(s);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

// The radices of one length in registers.
struct Line {
  int n, r1, r2, a_in, a_out, s_out;
  bool wrap;
  __device__ __forceinline__ explicit Line(const AxisPlan& a)
      : n(a.n), r1(a.r1), r2(a.r2), a_in(a.a_in), a_out(a.a_out), s_out(a.s_out), wrap(a.wrap != 0) {}
  // i + step modulo n, both below n
  __device__ __forceinline__ int next(int i, int step) const {
    i += step;
    return i >= n ? i - n : i;
  }
  // first output of sub-transform k1
  __device__ __forceinline__ int out0(int k1) const {
    const int i = a_out * k1;
    return wrap ? i % n : i;
  }
  // output index held at (k1, k2)
  __device__ __forceinline__ int freq(int k1, int k2) const { return (a_out * k1 + s_out * k2) % n; }
};

// Pass 1 of sub-transform n2: load(i) gives sample i, store(k1, i, v) takes
// result k1, whose place in an in-place transform is sample index i.
// WRAP = false: a length planned without prime-factor maps.
template <typename T, int R, int DIR, bool WRAP, typename Load, typename Store>
__device__ __forceinline__ void line_pass1(const Line& l, int n2, const cx<T>* __restrict__ tw, Load&& load,
                                           Store&& store) {
  cx<T> v[R];
  const int i0 = WRAP ? l.a_in * n2 : n2;
  int i = i0;
#pragma unroll
  for (int j = 0; j < R; ++j) {
    v[j] = load(i);
    i = WRAP ? l.next(i, l.r2) : i + l.r2;
  }
  Dft<T, R, DIR>::run(v);
  if (!(WRAP && l.wrap) && n2) {
#pragma unroll
    for (int k = 1; k < R; ++k) v[k] = twmul<DIR>(v[k], tw[n2 * k]);
  }
  i = i0;
#pragma unroll
  for (int k = 0; k < R; ++k) {
    store(k, i, v[k]);
    i = WRAP ? l.next(i, l.r2) : i + l.r2;
  }
}

}  // namespace
}  // namespace psatd
