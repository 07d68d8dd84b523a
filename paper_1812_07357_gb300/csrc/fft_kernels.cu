// Generic FFT passes of the PSATD push: boxes of any even 5-smooth size, both
// precisions, every form (the absorbing layers too), the stand-alone
// transforms and the ranks of a distributed group.  The fused z pass is in
// any_z.cu.
//
// Spectral layout of one box and one field slot (the "half spectrum"):
//   element (mx, my, mz), mx in [0, n0/2], at mx + hx*(my + n1*mz), hx = n0/2+1.
//
// Passes of one step (S1..S3 of the PSATD push):
//   fwd_x      real rows -> packed complex FFT of length n0/2 -> R2C split
//   col (y)    complex FFT along y of a tile of columns
//   z_update   (any_z.cu) complex FFT along z, the per-mode update, inverse along z
//   col (y)    inverse along y (only z planes that hold interior cells)
//   inv_x      C2R merge -> inverse packed FFT -> real rows (interior only)
//
// The lines run through two register passes of any_fft.cuh.  A tile is 128
// bytes of columns: k_col loads its samples straight from HBM into the
// registers of pass 1 and stores the outputs of pass 2 straight back, one trip
// through shared memory and one barrier between; columns are numbered through
// the planes of a box (the z columns of a box are one contiguous run), so only
// a box's last tile is partial.
//
// What bounds them: FP64 the two FP64 lanes of an SM (operation count), FP32
// memory latency.  Measured against radix-8 Stockham passes in shared memory
// (two barriers per pass, run-time modulo per butterfly, one tile of 4096
// points per block), GB300: absorbing layers, 8 boxes of 96^3 FP32 4.19 ->
// 0.79 ms per step; FP64 J form, 8 boxes of 100 x 90 x 72 8.53 -> 6.40 ms;
// forward + inverse FFT of 240 x 200 x 180 FP32 858 -> 190 us; 32^3 FP64 157
// -> 46 us per step (tiles of 128 bytes instead of 4096 points fill the chip).
#include <cuda_runtime.h>

#include <cstdint>

#include "any_fft.cuh"
#include "fft_codelets.cuh"
#include "psatd_internal.h"
#include "psatd_update.cuh"

namespace psatd {

namespace {

// Pass 2 along rows in shared memory: every thread holds one sub-transform
// (lane = row) and stores its outputs in natural order behind a barrier.
template <typename T, int DIR, int CLS>
__device__ __forceinline__ void rows_pass2(cx<T>* row, const Line& l, int k1, bool live) {
  with_radix<CLS>(l.r2, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    cx<T> v[R];
    live = live && k1 < l.r1;
    if (live) {
      int i = l.r2 * k1;
#pragma unroll
      for (int j = 0; j < R; ++j) {
        v[j] = row[i];
        i = l.next(i, l.a_in);
      }
      Dft<T, R, DIR>::run(v);
    }
    __syncthreads();
    if (live) {
      int k = l.out0(k1);
#pragma unroll
      for (int j = 0; j < R; ++j) {
        row[k] = v[j];
        k = l.next(k, l.s_out);
      }
    }
  });
  __syncthreads();
}

// Pass 1 along rows, in place.
template <typename T, int DIR, int CLS>
__device__ __forceinline__ void rows_pass1(cx<T>* row, const Line& l, int n2, bool live,
                                           const cx<T>* __restrict__ tw) {
  if (live && n2 < l.r2)
    with_radix<CLS>(l.r1, [&](auto rc) {
      line_pass1<T, decltype(rc)::value, DIR>(
          l, n2, tw, [&](int i) { return row[i]; }, [&](int, int i, cx<T> v) { row[i] = v; });
    });
  __syncthreads();
}

}  // namespace

// ---------------------------------------------------------------------------
// S1, x axis: real rows -> half spectrum (R2C via a packed complex FFT)
// z[m] = x[2m] + i x[2m+1];  Z = FFT_L(z);  with A = (Z[k] + conj Z[L-k])/2,
// B = (Z[k] - conj Z[L-k])/(2i) and w = exp(-2 pi i/n0):
// X[k] = A + w^k B,  X[L-k] = conj(A - w^k B)   (w^(L-k) = -conj w^k)
// ---------------------------------------------------------------------------
template <typename T, int CLS>
__global__ void __launch_bounds__(line_threads<T, CLS>()) k_fwd_x(DevPlan P, FieldPtrs F, cx<T>* spec,
                                                                  int64_t sstride, const RowJob* __restrict__ jobs) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<T>* sm = reinterpret_cast<cx<T>*>(smem_raw);
  constexpr int W = line_tile<T>();
  const RowJob J = jobs[blockIdx.x];
  const int f = blockIdx.y;
  const BoxDev& bx = P.boxes[J.box];
  const ShapeDev& sh = P.shapes[bx.shape];
  const Line l(sh.ax);
  const int L = l.n, hx = L + 1, PX = L | 1;   // odd row pitch
  const int64_t soff = bx.soff;
  const cx<T>* in = reinterpret_cast<const cx<T>*>(reinterpret_cast<const T*>(F.p[f]) + bx.foff) + (int64_t)J.r0 * L;
  const unsigned mL = line_magic(L);
  for (int e = threadIdx.x; e < J.nr * L; e += blockDim.x) cp_async(sm + e + line_div(e, mL) * (PX - L), in + e);
  cp_async_wait();
  __syncthreads();
  const int c = threadIdx.x % W, g = threadIdx.x / W;
  const bool live = c < J.nr;
  rows_pass1<T, -1, CLS>(sm + c * PX, l, g, live, cpool<T>(P) + sh.ax.tw);
  rows_pass2<T, -1, CLS>(sm + c * PX, l, g, live);
  const cx<T>* post = cpool<T>(P) + sh.post;
  cx<T>* out = spec + f * sstride + soff + (int64_t)J.r0 * hx;
  const int H = L / 2 + 1;
  const unsigned mH = line_magic(H);
  for (int e = threadIdx.x; e < J.nr * H; e += blockDim.x) {
    const int r = line_div(e, mH), k = e - r * H;
    const cx<T> a = sm[r * PX + k], b = sm[r * PX + (k == 0 ? 0 : L - k)];
    cx<T>* o = out + (int64_t)r * hx;
    if (k == 0) {
      o[0] = mk<T>(a.x + a.y, T(0));
      o[L] = mk<T>(a.x - a.y, T(0));
      continue;
    }
    const cx<T> w = post[k];
    const cx<T> A = mk<T>(a.x + b.x, a.y - b.y);
    const cx<T> t = cmul(rmul(T(0.5), w), mk<T>(a.y + b.y, b.x - a.x));
    o[k] = mk<T>(T(0.5) * A.x + t.x, T(0.5) * A.y + t.y);
    if (2 * k != L) o[L - k] = mk<T>(T(0.5) * A.x - t.x, t.y - T(0.5) * A.y);
  }
}

// ---------------------------------------------------------------------------
// Column FFT along y (axis 1) or z (axis 2) of J.nm columns from column J.m0
// of plane J.plane on, running on through the planes that follow.
// ---------------------------------------------------------------------------
template <typename T, int DIR, int CLS>
__global__ void __launch_bounds__(line_threads<T, CLS>()) k_col(DevPlan P, cx<T>* spec, int64_t sstride, int axis,
                                                                const ColJob* __restrict__ jobs) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int W = line_tile<T>();
  const ColJob J = jobs[blockIdx.x];
  const BoxDev& bx = P.boxes[J.box];
  const ShapeDev& sh = P.shapes[bx.shape];
  const int hx = sh.hx, n1 = bx.n[1];
  const Line l(axis == 1 ? sh.ay : sh.az);
  const cx<T>* tw = cpool<T>(P) + (axis == 1 ? sh.ay.tw : sh.az.tw);
  const int c = threadIdx.x % W, g0 = threadIdx.x / W, gs = blockDim.x / W;
  const bool live = c < J.nm;
  // first element of this lane's column, and the step between its samples
  int m = J.m0 + c, pl = J.plane;
  int stride = n1 * hx;
  if (axis == 1) {
    while (m >= hx) {
      m -= hx;
      ++pl;
    }
    stride = hx;
  }
  cx<T>* g = spec + blockIdx.y * sstride + bx.soff + (int64_t)pl * (axis == 1 ? n1 * hx : hx) + m;
  cx<T>* col = reinterpret_cast<cx<T>*>(smem_raw) + c;   // place p of the column at col[p * W]
  if (live)
    with_radix<CLS>(l.r1, [&](auto rc) {
      for (int n2 = g0; n2 < l.r2; n2 += gs)
        line_pass1<T, decltype(rc)::value, DIR>(
            l, n2, tw, [&](int i) { return g[(int64_t)i * stride]; },
            [&](int k, int, cx<T> v) { col[(k * l.r2 + n2) * W] = v; });
    });
  __syncthreads();
  if (live)
    with_radix<CLS>(l.r2, [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      for (int k1 = g0; k1 < l.r1; k1 += gs) {
        cx<T> v[R];
#pragma unroll
        for (int j = 0; j < R; ++j) v[j] = col[(k1 * R + j) * W];
        Dft<T, R, DIR>::run(v);
        int k = l.out0(k1);
#pragma unroll
        for (int j = 0; j < R; ++j) {
          g[(int64_t)k * stride] = v[j];
          k = l.next(k, l.s_out);
        }
      }
    });
}

// ---------------------------------------------------------------------------
// S3, x axis: half spectrum -> real rows (C2R), with 1/(n0 n1 n2).
// With s = X[k] + conj X[L-k], u = (X[k] - conj X[L-k]) w^-k, w = exp(-2 pi i/n0):
// Z'[k] = s + i u,  Z'[L-k] = conj s + i conj u,  k <= L/2;
// z = IFFT_L(Z') (unnormalised);  x[2m] = Re z[m], x[2m+1] = Im z[m].
// ---------------------------------------------------------------------------
template <typename T, int CLS>
__global__ void __launch_bounds__(line_threads<T, CLS>()) k_inv_x(DevPlan P, FieldPtrs F, const cx<T>* spec,
                                                                  int64_t sstride, const RowJob* __restrict__ jobs,
                                                                  int interior_only) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<T>* sm = reinterpret_cast<cx<T>*>(smem_raw);
  constexpr int W = line_tile<T>();
  const RowJob J = jobs[blockIdx.x];
  const int f = blockIdx.y;
  const BoxDev& bx = P.boxes[J.box];
  const ShapeDev& sh = P.shapes[bx.shape];
  const Line l(sh.ax);
  const int L = l.n, hx = L + 1, n0 = 2 * L, PX = hx | 1;
  const T scale = T(1.0 / ((double)n0 * bx.n[1] * bx.n[2]));
  T* out = reinterpret_cast<T*>(F.p[f]) + bx.foff + (int64_t)J.r0 * n0;
  const int xlo = interior_only ? bx.ng_lo[0] : 0;
  const int nxi = (interior_only ? n0 - bx.ng_hi[0] : n0) - xlo;
  const cx<T>* in = spec + f * sstride + bx.soff + (int64_t)J.r0 * hx;
  const unsigned mh = line_magic(hx);
  for (int e = threadIdx.x; e < J.nr * hx; e += blockDim.x) cp_async(sm + e + line_div(e, mh) * (PX - hx), in + e);
  cp_async_wait();
  __syncthreads();
  const cx<T>* post = cpool<T>(P) + sh.post;
  const int H = L / 2 + 1;
  const unsigned mH = line_magic(H);
  for (int e = threadIdx.x; e < J.nr * H; e += blockDim.x) {
    const int r = line_div(e, mH), k = e - r * H;
    cx<T>* row = sm + r * PX;
    const cx<T> a = row[k], b = conjg(row[L - k]);
    const cx<T> s = a + b, u = cmulc(a - b, post[k]);
    row[k] = rmul(scale, mk<T>(s.x - u.y, s.y + u.x));
    if (k != 0 && 2 * k != L) row[L - k] = rmul(scale, mk<T>(s.x + u.y, u.x - s.y));
  }
  __syncthreads();
  const int c = threadIdx.x % W, g = threadIdx.x / W;
  const bool live = c < J.nr;
  rows_pass1<T, 1, CLS>(sm + c * PX, l, g, live, cpool<T>(P) + sh.ax.tw);
  rows_pass2<T, 1, CLS>(sm + c * PX, l, g, live);
  if (((xlo | nxi) & 1) == 0) {   // whole pairs of cells
    const int np = nxi / 2;
    const unsigned mp = line_magic(np);
    for (int e = threadIdx.x; e < J.nr * np; e += blockDim.x) {
      const int r = line_div(e, mp), m = xlo / 2 + e - r * np;
      reinterpret_cast<cx<T>*>(out)[(int64_t)r * L + m] = sm[r * PX + m];
    }
  } else {
    const unsigned mx = line_magic(nxi);
    for (int e = threadIdx.x; e < J.nr * nxi; e += blockDim.x) {
      const int r = line_div(e, mx), x = xlo + e - r * nxi;
      const cx<T> z = sm[r * PX + (x >> 1)];
      out[(int64_t)r * n0 + x] = (x & 1) ? z.y : z.x;
    }
  }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
namespace {
constexpr int64_t kMaxGridX = 2147483647LL;
}  // namespace

cudaError_t launch_fwd_x(int prec, const DevPlan& P, const FieldPtrs& f, int nf, void* spec, int64_t sstride,
                         const RowJob* jobs, int64_t njobs, const LineCfg& c, cudaStream_t st) {
  if (njobs <= 0 || nf <= 0) return cudaSuccess;
  if (njobs > kMaxGridX) return cudaErrorInvalidConfiguration;
  dim3 grid((unsigned)njobs, nf);
#define PSATD_GO(T, C2, CLS) \
  k_fwd_x<T, CLS><<<grid, c.threads, c.smem, st>>>(P, f, (C2*)spec, sstride, jobs)
  if (prec == 32) {
    if (c.cls) PSATD_GO(float, float2, 1); else PSATD_GO(float, float2, 0);
  } else {
    if (c.cls) PSATD_GO(double, double2, 1); else PSATD_GO(double, double2, 0);
  }
#undef PSATD_GO
  return cudaGetLastError();
}

cudaError_t launch_col(int prec, int dir, int axis, const DevPlan& P, void* spec, int64_t sstride, int nf,
                       const ColJob* jobs, int64_t njobs, const LineCfg& c, cudaStream_t st) {
  if (njobs <= 0 || nf <= 0) return cudaSuccess;
  if (njobs > kMaxGridX) return cudaErrorInvalidConfiguration;
  dim3 grid((unsigned)njobs, nf);
#define PSATD_GO(T, C2, DIR, CLS) \
  k_col<T, DIR, CLS><<<grid, c.threads, c.smem, st>>>(P, (C2*)spec, sstride, axis, jobs)
  if (prec == 32) {
    if (dir < 0) {
      if (c.cls) PSATD_GO(float, float2, -1, 1); else PSATD_GO(float, float2, -1, 0);
    } else {
      if (c.cls) PSATD_GO(float, float2, 1, 1); else PSATD_GO(float, float2, 1, 0);
    }
  } else {
    if (dir < 0) {
      if (c.cls) PSATD_GO(double, double2, -1, 1); else PSATD_GO(double, double2, -1, 0);
    } else {
      if (c.cls) PSATD_GO(double, double2, 1, 1); else PSATD_GO(double, double2, 1, 0);
    }
  }
#undef PSATD_GO
  return cudaGetLastError();
}

cudaError_t launch_inv_x(int prec, const DevPlan& P, const FieldPtrs& f, int nf, void* spec, int64_t sstride,
                         const RowJob* jobs, int64_t njobs, const LineCfg& c, int interior_only, cudaStream_t st) {
  if (njobs <= 0 || nf <= 0) return cudaSuccess;
  if (njobs > kMaxGridX) return cudaErrorInvalidConfiguration;
  dim3 grid((unsigned)njobs, nf);
#define PSATD_GO(T, C2, CLS) \
  k_inv_x<T, CLS><<<grid, c.threads, c.smem, st>>>(P, f, (const C2*)spec, sstride, jobs, interior_only)
  if (prec == 32) {
    if (c.cls) PSATD_GO(float, float2, 1); else PSATD_GO(float, float2, 0);
  } else {
    if (c.cls) PSATD_GO(double, double2, 1); else PSATD_GO(double, double2, 0);
  }
#undef PSATD_GO
  return cudaGetLastError();
}

template <typename T, int CLS>
static cudaError_t configure_t(int smem) {
  cudaError_t e = cudaSuccess;
  for (const void* k : {(const void*)k_fwd_x<T, CLS>, (const void*)k_inv_x<T, CLS>, (const void*)k_col<T, -1, CLS>,
                        (const void*)k_col<T, 1, CLS>}) {
    const cudaError_t r = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (r != cudaSuccess) e = r;
  }
  return e;
}

cudaError_t configure_kernels(int prec, int smem) {
  cudaError_t e = configure_any_z(prec, smem);
  for (const cudaError_t r : {prec == 32 ? configure_t<float, 0>(smem) : configure_t<double, 0>(smem),
                              prec == 32 ? configure_t<float, 1>(smem) : configure_t<double, 1>(smem)})
    if (r != cudaSuccess) e = r;
  return e;
}

int line_tile_width(int prec) { return prec == 32 ? line_tile<float>() : line_tile<double>(); }

// Shared memory, threads and class that lines of length n need, on top of
// what c already covers (kind 0: columns, 1: rows of n complex elements, 2:
// rows of n + 1).
void line_cover(LineCfg& c, int prec, const AxisPlan& a, int kind) {
  const int w = line_tile_width(prec), csz = prec == 32 ? 8 : 16;
  const int len = kind == 0 ? a.n : kind == 1 ? (a.n | 1) : ((a.n + 1) | 1);
  const int r = a.r1 > a.r2 ? a.r1 : a.r2;
  c.smem = c.smem > w * len * csz ? c.smem : w * len * csz;
  const int t = (w * r + 31) / 32 * 32;
  c.threads = c.threads > t ? c.threads : t;
  if (r > 16) c.cls = 1;
}

}  // namespace psatd
