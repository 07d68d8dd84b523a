// Generic FFT passes of the PSATD push: boxes of any even 5-smooth size, both
// precisions, every form (the absorbing layers too), the stand-alone
// transforms and the ranks of a distributed group.  The fused z pass is in
// any_z.cuh.
//
// Spectral layout of one box and one field slot (the "half spectrum"):
//   element (mx, my, mz), mx in [0, n0/2], at mx + hx*(my + n1*mz), hx = n0/2+1.
//
// Passes of one step (S1..S3 of the PSATD push):
//   fwd_x      real rows -> packed complex FFT of length n0/2 -> R2C split
//   col (y)    complex FFT along y of a tile of columns
//   z_update   (any_z.cuh) complex FFT along z, the per-mode update, inverse along z
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
// FP32 x rows take no prime-factor maps, so their lanes run along the row: the
// forward kernel loads its samples (gathered from the cells that own them with
// the deferred exchange) and the inverse kernel merges pairs and stores its
// outputs straight between HBM and registers.  FP64 rows are staged in shared
// memory with lanes across the rows, which any map reads without conflicts:
// there the operation count decides, and coprime radices save the twiddles.
//
// What bounds them: FP64 the two FP64 lanes of an SM (84 % busy), FP32 memory
// latency and instruction issue.  Measured on GB300 against radix-8 Stockham
// passes in shared memory (two barriers per pass, run-time modulo per butterfly,
// 4096 points per block): a 100 x 90 x 80 box with absorbing layers FP32 726 ->
// 119 us per step; FP64 J form, 8 boxes of 100 x 90 x 72 8.52 -> 5.70 ms; forward +
// inverse FFT of 240 x 200 x 180 FP32 with a filter between 856 -> 152 us; 32^3 FP64
// 157 -> 46 us per step.  Against a kernel per length with whole tiles staged in
// shared memory: two FP32 boxes of 384 x 256 x 256 3.74 -> 2.92 ms per step, 256^3
// FP32 1.33 -> 1.05, 128^3 FP64 rho form 3.03 -> 2.61.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "any_fft.cuh"
#include "fft_codelets.cuh"
#include "launch.cuh"
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

// Pass 1 along rows, in place: sub-transforms n2, n2 + gs, ... (class 0: a thread
// for each).
template <typename T, int DIR, int CLS>
__device__ __forceinline__ void rows_pass1(cx<T>* row, const Line& l, int n2, int gs, bool live,
                                           const cx<T>* __restrict__ tw) {
  if (live && n2 < l.r2)
    with_radix<CLS>(l.r1, [&](auto rc) {
      do {
        line_pass1<T, decltype(rc)::value, DIR, true>(
            l, n2, tw, [&](int i) { return row[i]; }, [&](int, int i, cx<T> v) { row[i] = v; });
        n2 += gs;
      } while (CLS && n2 < l.r2);
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
template <typename T>
__device__ __forceinline__ void split_rows(const cx<T>* sm, int pitch, int nr, int L, const cx<T>* __restrict__ post,
                                           cx<T>* out) {
  const int H = L / 2 + 1;
  const unsigned mH = line_magic(H);
  for (int e = threadIdx.x; e < nr * H; e += blockDim.x) {
    const int r = line_div(e, mH), k = e - r * H;
    const cx<T> a = sm[r * pitch + k], b = sm[r * pitch + (k == 0 ? 0 : L - k)];
    cx<T>* o = out + r * (L + 1);
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

// GATHER (deferred exchange): the samples of a row come from the cells that own
// them, up to three bands of columns per row from the plane's gather grid.
template <typename T>
struct RowBands {
  int64_t src[kMaxLines][3];   // element x of band i is src[.][i] + x
  int x[kMaxLines][2];         // the bands' first columns (past the first band)
  __device__ __forceinline__ int64_t at(int r, int col) const {
    return src[r][(col >= x[r][0]) + (col >= x[r][1])] + col;
  }
};

template <typename T, int CLS, bool GATHER>
__global__ void __launch_bounds__(line_threads<T, CLS>())
    k_fwd_x(DevPlan P, FieldPtrs F, cx<T>* spec, int64_t sstride, const RowJob* __restrict__ jobs,
            const GatherGrid* __restrict__ ggrid, int ngather, int lg) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<T>* sm = reinterpret_cast<cx<T>*>(smem_raw);
  const int lw = line_lg<T>(lg), W = 1 << lw;
  const RowJob J = jobs[blockIdx.x];
  const int f = blockIdx.y;
  const BoxDev& bx = P.boxes[J.box];
  const ShapeDev& sh = P.shapes[bx.shape];
  const Line l(sh.ax);
  const int L = l.n;
  const cx<T>* tw = cpool<T>(P) + sh.ax.tw;
  const cx<T>* in = reinterpret_cast<const cx<T>*>(reinterpret_cast<const T*>(F.p[f]) + bx.foff) + (int64_t)J.r0 * L;
  cx<T>* out = spec + f * sstride + bx.soff + (int64_t)J.r0 * (L + 1);
  __shared__ RowBands<T> bands;
  const T* fb = reinterpret_cast<const T*>(F.p[f]);
  const bool gather = GATHER && f < ngather;
  grid_order(P.order);
  if (gather) {
    if (threadIdx.x < J.nr) {
      const int t = threadIdx.x, r = J.r0 + t, n1 = bx.n[1], z = r / n1, y = r - z * n1;
      const GatherGrid& G = ggrid[bx.gplane + z];
      const int iy = (y >= G.y1) + (y >= G.y2);
      const int dy = y - (iy == 0 ? 0 : iy == 1 ? G.y1 : G.y2);
      bands.src[t][0] = G.base[3 * iy] + (int64_t)dy * G.pitch[3 * iy];
      bands.src[t][1] = G.base[3 * iy + 1] + (int64_t)dy * G.pitch[3 * iy + 1] - G.x1;
      bands.src[t][2] = G.base[3 * iy + 2] + (int64_t)dy * G.pitch[3 * iy + 2] - G.x2;
      bands.x[t][0] = G.x1;
      bands.x[t][1] = G.x2;
    }
    __syncthreads();
  }
  // complex sample i of row r of the tile
  auto sample = [&](int r, int i) -> const cx<T>* {
    return gather ? reinterpret_cast<const cx<T>*>(fb + bands.at(r, 2 * i)) : in + r * L + i;
  };
  if constexpr (sizeof(T) == 4) {
    // lanes along the row: samples straight from HBM, n2 adjacent
    const int pitch = row_line_pitch(sh.ax), p2 = l.r2 | 1;
    {
      const int r = line_div(threadIdx.x, line_magic(l.r2)), n2 = threadIdx.x - r * l.r2;
      if (r < J.nr)
        with_radix<CLS>(l.r1, [&](auto rc) {
          line_pass1<T, decltype(rc)::value, -1, false>(
              l, n2, tw, [&](int i) { return *sample(r, i); },
              [&](int k, int, cx<T> v) { sm[r * pitch + k * p2 + n2] = v; });
        });
    }
    __syncthreads();
    with_radix<CLS>(l.r2, [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      const int r = line_div(threadIdx.x, line_magic(l.r1)), k1 = threadIdx.x - r * l.r1;
      cx<T> v[R];
      if (r < J.nr) {
#pragma unroll
        for (int j = 0; j < R; ++j) v[j] = sm[r * pitch + k1 * p2 + j];
        Dft<T, R, -1>::run(v);
      }
      __syncthreads();
      if (r < J.nr) {
#pragma unroll
        for (int j = 0; j < R; ++j) sm[r * pitch + k1 + l.r1 * j] = v[j];
      }
    });
    __syncthreads();
    split_rows<T>(sm, pitch, J.nr, L, cpool<T>(P) + sh.post, out);
  } else {
    // lanes across the rows (any index map free of bank conflicts), the rows staged in shared memory
    const int PX = L | 1;   // odd row pitch
    const unsigned mL = line_magic(L);
    for (int e = threadIdx.x; e < J.nr * L; e += blockDim.x) {
      const int r = line_div(e, mL);
      cp_async(sm + e + r * (PX - L), sample(r, e - r * L));
    }
    cp_async_wait();
    __syncthreads();
    const int c = threadIdx.x & (W - 1), g = threadIdx.x >> lw;
    const bool live = c < J.nr;
    rows_pass1<T, -1, CLS>(sm + c * PX, l, g, blockDim.x >> lw, live, tw);
    rows_pass2<T, -1, CLS>(sm + c * PX, l, g, live);
    split_rows<T>(sm, PX, J.nr, L, cpool<T>(P) + sh.post, out);
  }
}

// ---------------------------------------------------------------------------
// Column FFT along y (axis 1) or z (axis 2) of J.nm columns from column J.m0
// of plane J.plane on, running on through the planes that follow.
// ---------------------------------------------------------------------------
template <typename T, int DIR, int CLS>
__global__ void __launch_bounds__(line_threads<T, CLS>()) k_col(DevPlan P, cx<T>* spec, int64_t sstride, int axis,
                                                                const ColJob* __restrict__ jobs, int lg) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lw = line_lg<T>(lg), W = 1 << lw;
  const ColJob J = jobs[blockIdx.x];
  const BoxDev& bx = P.boxes[J.box];
  const ShapeDev& sh = P.shapes[bx.shape];
  const int hx = sh.hx, n1 = bx.n[1];
  const Line l(axis == 1 ? sh.ay : sh.az);
  const cx<T>* tw = cpool<T>(P) + (axis == 1 ? sh.ay.tw : sh.az.tw);
  const int c = threadIdx.x & (W - 1), g0 = threadIdx.x >> lw, gs = blockDim.x >> lw;
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
  cx<T>* col = reinterpret_cast<cx<T>*>(smem_raw) + c;   // place p of the column at col[p << lw]
  grid_order(P.order);
  if (live)
    with_radix<CLS>(l.r1, [&](auto rc) {
      for (int n2 = g0; n2 < l.r2; n2 += gs)
        line_pass1<T, decltype(rc)::value, DIR, true>(
            l, n2, tw, [&](int i) { return g[(int64_t)i * stride]; },
            [&](int k, int, cx<T> v) { col[(k * l.r2 + n2) << lw] = v; });
    });
  __syncthreads();
  if (live)
    with_radix<CLS>(l.r2, [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      for (int k1 = g0; k1 < l.r1; k1 += gs) {
        cx<T> v[R];
#pragma unroll
        for (int j = 0; j < R; ++j) v[j] = col[(k1 * R + j) << lw];
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
__global__ void __launch_bounds__(line_threads<T, CLS>(), sizeof(T) == 4 && !CLS ? 3 : 1) k_inv_x(DevPlan P, FieldPtrs F, const cx<T>* spec,
                                                                  int64_t sstride, const RowJob* __restrict__ jobs,
                                                                  int interior_only, int lg) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<T>* sm = reinterpret_cast<cx<T>*>(smem_raw);
  const int lw = line_lg<T>(lg), W = 1 << lw;
  const RowJob J = jobs[blockIdx.x];
  const int f = blockIdx.y;
  const BoxDev& bx = P.boxes[J.box];
  const ShapeDev& sh = P.shapes[bx.shape];
  const Line l(sh.ax);
  const int L = l.n, hx = L + 1, n0 = 2 * L;
  const cx<T>* tw = cpool<T>(P) + sh.ax.tw;
  const cx<T>* post = cpool<T>(P) + sh.post;
  T* out = reinterpret_cast<T*>(F.p[f]) + bx.foff + (int64_t)J.r0 * n0;
  const int xlo = interior_only ? bx.ng_lo[0] : 0;
  const int nxi = (interior_only ? n0 - bx.ng_hi[0] : n0) - xlo;
  const bool pairs = ((xlo | nxi) & 1) == 0;   // whole pairs of cells
  const cx<T>* in = spec + f * sstride + bx.soff + (int64_t)J.r0 * hx;
  grid_order(P.order);
  if constexpr (sizeof(T) == 4) {
    // lanes along the row: every thread merges its own samples from HBM (both
    // ends of a pair, the other end from L1) and stores its outputs to HBM
    const T scale = sh.scale32;
    const int pitch = row_line_pitch(sh.ax), p2 = l.r2 | 1;
    {
      const int r = line_div(threadIdx.x, line_magic(l.r2)), n2 = threadIdx.x - r * l.r2;
      if (r < J.nr)
        with_radix<CLS>(l.r1, [&](auto rc) {
          line_pass1<T, decltype(rc)::value, 1, false>(
              l, n2, tw,
              [&](int i) {
                const cx<T> a = in[r * hx + i], b = conjg(in[r * hx + L - i]);
                const cx<T> s = a + b, u = cmulc(a - b, post[i]);
                return rmul(scale, mk<T>(s.x - u.y, s.y + u.x));
              },
              [&](int k, int, cx<T> v) { sm[r * pitch + k * p2 + n2] = v; });
        });
    }
    __syncthreads();
    const int r = line_div(threadIdx.x, line_magic(l.r1)), k1 = threadIdx.x - r * l.r1;
    if (r < J.nr)
      with_radix<CLS>(l.r2, [&](auto rc) {
        constexpr int R = decltype(rc)::value;
        cx<T> v[R];
#pragma unroll
        for (int j = 0; j < R; ++j) v[j] = sm[r * pitch + k1 * p2 + j];
        Dft<T, R, 1>::run(v);
        T* o = out + r * n0;
        if (pairs) {
#pragma unroll
          for (int j = 0; j < R; ++j) {
            const int x = 2 * (k1 + l.r1 * j);
            if ((unsigned)(x - xlo) < (unsigned)nxi) *reinterpret_cast<cx<T>*>(o + x) = v[j];
          }
        } else {
#pragma unroll
          for (int j = 0; j < R; ++j) {
            const int x = 2 * (k1 + l.r1 * j);
            if ((unsigned)(x - xlo) < (unsigned)nxi) o[x] = v[j].x;
            if ((unsigned)(x + 1 - xlo) < (unsigned)nxi) o[x + 1] = v[j].y;
          }
        }
      });
  } else {
    const T scale = sh.scale64;
    const int PX = hx | 1;
    const unsigned mh = line_magic(hx);
    for (int e = threadIdx.x; e < J.nr * hx; e += blockDim.x) cp_async(sm + e + line_div(e, mh) * (PX - hx), in + e);
    cp_async_wait();
    __syncthreads();
    const int H = L / 2 + 1;
    const unsigned mH = line_magic(H);
    for (int e = threadIdx.x; e < J.nr * H; e += blockDim.x) {
      const int r = line_div(e, mH), k = e - r * H;
      cx<T>* row = sm + r * PX;
      const cx<T> a = row[k], b = conjg(row[L - k]);
      const cx<T> s = rmul(scale, a + b), u = cmulc(a - b, rmul(scale, post[k]));
      row[k] = mk<T>(s.x - u.y, s.y + u.x);
      if (k != 0 && 2 * k != L) row[L - k] = mk<T>(s.x + u.y, u.x - s.y);
    }
    __syncthreads();
    const int c = threadIdx.x & (W - 1), g = threadIdx.x >> lw;
    const bool live = c < J.nr;
    rows_pass1<T, 1, CLS>(sm + c * PX, l, g, blockDim.x >> lw, live, tw);
    rows_pass2<T, 1, CLS>(sm + c * PX, l, g, live);
    if (pairs) {
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
}

}  // namespace psatd
