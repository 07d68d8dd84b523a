// The generic fused z pass (S1 z, S2, S3 z): boxes of any even 5-smooth z
// length, both precisions, every form, absorbing layers included.
//
//   k_z_update  a tile of TX adjacent z columns (of the box's contiguous run of
//               n1 * hx columns), every field slot: z FFT, per-mode update,
//               inverse z FFT of the output slots, interior z planes stored.
//
// The two-pass lines of any_fft.cuh run in place: pass 1 straight from HBM
// into shared memory, pass 2 in place, the update where each mode lies (place
// p = (k1, k2) of a line holds frequency (a_out k1 + s_out k2) mod n2), then
// the same two passes mirrored, the last one straight back to HBM.  So no pass
// permutes its line and a block waits at four barriers.  Shared memory is
// [slot][place][column], each slot a row further within a 128-byte line than the
// one before, so that lanes over (column, place) and lanes over (column, slot)
// both read it without bank conflicts.
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

template <typename T>
constexpr int z_threads() {   // at most; FP64: fewer, larger threads, its pipe needs few warps
  return sizeof(T) == 4 ? 256 : 128;
}

template <typename T, int FORM, int CLS>
__global__ void __launch_bounds__(z_threads<T>(), CLS ? 1 : sizeof(T) == 4 ? 2 : 3)
    k_z_update(DevPlan P, cx<T>* spec, int64_t sstride, const ColJob* __restrict__ jobs, int nft, int lg) {
  constexpr int FIN = fields_in(FORM), FOUT = fields_out(FORM);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<T>* sm = reinterpret_cast<cx<T>*>(smem_raw);
  const ColJob J = jobs[blockIdx.x];
  const BoxDev& bx = P.boxes[J.box];
  const ShapeDev& sh = P.shapes[bx.shape];
  const int hx = sh.hx, n2 = bx.n[2], nm = J.nm;
  const int zst = bx.n[1] * hx;
  const int tx = 1 << lg, SP = z_slot_pitch(sizeof(cx<T>), n2, tx);
  const Line l(sh.az);
  const cx<T>* tw = cpool<T>(P) + sh.az.tw;
  cx<T>* g = spec + bx.soff + (int64_t)J.plane * hx + J.m0;
  const int c = threadIdx.x & (tx - 1), i0 = threadIdx.x >> lg, is = blockDim.x >> lg;
  const bool live = c < nm;
  grid_order(P.order);
  // pass 1 from HBM, lanes over (column, n2); slots >= nft already hold their
  // z spectrum (a cached constant current) and are placed as they are
  if (live) {
    const unsigned mr = line_magic(l.r2);
    with_radix<CLS>(l.r1, [&](auto rc) {
      for (int it = i0; it < nft * l.r2; it += is) {
        const int s = line_div(it, mr), n2i = it - s * l.r2;
        const cx<T>* gs = g + s * sstride + c;
        cx<T>* b = sm + s * SP + c;
        line_pass1<T, decltype(rc)::value, -1, true>(
            l, n2i, tw, [&](int i) { return gs[(int64_t)i * zst]; },
            [&](int k, int, cx<T> v) { b[(k * l.r2 + n2i) << lg] = v; });
      }
    });
    if constexpr (FIN > fields_in(kVacuum)) {
      constexpr int U = 4, NJ = 3;   // a current has three slots; 12 loads before any is stored
      if (nft + NJ == FIN)
        for (int p0 = i0; p0 < n2; p0 += U * is) {
          cx<T> v[U][NJ];
#pragma unroll
          for (int i = 0; i < U; ++i) {
            const int p = p0 + i * is, k1 = line_div(p, mr);
            const cx<T>* src = g + nft * sstride + (int64_t)l.freq(k1, p - k1 * l.r2) * zst + c;
#pragma unroll
            for (int q = 0; q < NJ; ++q)
              if (p < n2) v[i][q] = src[q * sstride];
          }
#pragma unroll
          for (int i = 0; i < U; ++i)
#pragma unroll
            for (int q = 0; q < NJ; ++q)
              if (p0 + i * is < n2) sm[(nft + q) * SP + ((p0 + i * is) << lg) + c] = v[i][q];
        }
    }
  }
  __syncthreads();
  // pass 2 in place, lanes over (column, slot)
  if (live) {
    const unsigned mf = line_magic(nft);
    with_radix<CLS>(l.r2, [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      for (int it = i0; it < nft * l.r1; it += is) {
        const int k1 = line_div(it, mf), s = it - k1 * nft;
        cx<T>* b = sm + s * SP + ((k1 * R) << lg) + c;
        cx<T> v[R];
#pragma unroll
        for (int j = 0; j < R; ++j) v[j] = b[j << lg];
        Dft<T, R, -1>::run(v);
#pragma unroll
        for (int j = 0; j < R; ++j) b[j << lg] = v[j];
      }
    });
  }
  __syncthreads();
  // update: column -> mode (mx, my), place -> mz
  {
    const unsigned mr = line_magic(l.r2);
    auto mode = [&](int col, int& mx, int& my) {
      mx = J.m0 + (col < nm ? col : nm - 1);
      my = J.plane + bx.yoff;
      while (mx >= hx) {
        mx -= hx;
        ++my;
      }
    };
    if constexpr (sizeof(T) == 4) {
      // two columns per thread in packed FP32
      const int cp = (threadIdx.x & (tx / 2 - 1)) * 2;
      if (cp < nm) {
        int mxa, mya, mxb, myb;
        mode(cp, mxa, mya);
        mode(cp + 1, mxb, myb);
        const ModeXY2 m = mode_xy2(mxa, mya, mxb, myb, sh, P);
        for (int p = threadIdx.x >> (lg - 1); p < n2; p += blockDim.x >> (lg - 1)) {
          const int k1 = line_div(p, mr);
          const ModeZ2 z = mode_z2(m, l.freq(k1, p - k1 * l.r2), sh, P);
          float2* b = sm + (p << lg) + cp;
          C2 v[spec_slots(FORM)];
#pragma unroll
          for (int s = 0; s < FIN; ++s) {
            const float4 q = *reinterpret_cast<const float4*>(b + s * SP);
            v[s] = C2{make_float2(q.x, q.z), make_float2(q.y, q.w)};
          }
          update_core2<FORM>(v, m.Kx, m.Ky, make_float2(z.kz, z.kz), m.px, m.py, pack2(z.pz, z.pz), m.pxy, z.q, P);
#pragma unroll
          for (int s = 0; s < FOUT; ++s)
            *reinterpret_cast<float4*>(b + s * SP) = make_float4(v[s].x.x, v[s].y.x, v[s].x.y, v[s].y.y);
        }
      }
    } else if (live) {
      int mx, my;
      mode(c, mx, my);
      const ModeXY<T> m = mode_xy<T>(mx, my, sh, P);
      for (int p = i0; p < n2; p += is) {
        const int k1 = line_div(p, mr);
        update_mode_z<T, FORM>(sm + (p << lg) + c, SP, m, l.freq(k1, p - k1 * l.r2), sh, P);
      }
    }
  }
  __syncthreads();
  // mirrored pass 2 in place, lanes over (column, slot)
  if (live) {
    const unsigned mf = line_magic(FOUT);
    with_radix<CLS>(l.r2, [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      for (int it = i0; it < FOUT * l.r1; it += is) {
        const int k1 = line_div(it, mf), s = it - k1 * FOUT;
        cx<T>* b = sm + s * SP + ((k1 * R) << lg) + c;
        cx<T> v[R];
#pragma unroll
        for (int j = 0; j < R; ++j) v[j] = b[j << lg];
        Dft<T, R, 1>::run(v);
        if (!l.wrap && k1) {
#pragma unroll
          for (int j = 1; j < R; ++j) v[j] = cmulc(v[j], tw[k1 * j]);
        }
#pragma unroll
        for (int j = 0; j < R; ++j) b[j << lg] = v[j];
      }
    });
  }
  __syncthreads();
  // mirrored pass 1 straight to HBM, lanes over (column, n2): only the
  // interior z planes, the inverse y pass reads no others
  if (live) {
    const unsigned mr = line_magic(l.r2);
    const int zlo = bx.ng_lo[2], nz = n2 - bx.ng_hi[2] - zlo;
    with_radix<CLS>(l.r1, [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      for (int it = i0; it < FOUT * l.r2; it += is) {
        const int s = line_div(it, mr), n2i = it - s * l.r2;
        const cx<T>* b = sm + s * SP + c;
        cx<T>* gs = g + s * sstride + c;
        cx<T> v[R];
#pragma unroll
        for (int k = 0; k < R; ++k) v[k] = b[(k * l.r2 + n2i) << lg];
        Dft<T, R, 1>::run(v);
        int i = l.a_in * n2i;
#pragma unroll
        for (int j = 0; j < R; ++j) {
          if ((unsigned)(i - zlo) < (unsigned)nz) gs[(int64_t)i * zst] = v[j];
          i = l.next(i, l.r2);
        }
      }
    });
  }
}

}  // namespace
}  // namespace psatd
