// Grid transfers of the multigrid cycles (Sec. 3.5), one coarse or fine point
// at a time, shared by the per-level launches (stencil.cu) and the cluster
// V-cycle (cluster.cu).
#pragma once

#include "common.cuh"
#include "point.cuh"

namespace bf {
namespace {

// ---------------------------------------------------------------------------
// Grid transfers (Sec. 3.5).
// Cell-centred restriction: mean of the 2^D children. Face restriction along
// its own axis: (1/4, 1/2, 1/4) on the faces 2I-1, 2I, 2I+1; across the other
// axes the mean of the two children. Both zero the coarse iterate. COH = true
// reads through L2, as in point.cuh.
// ---------------------------------------------------------------------------
template <int D, typename T, bool COH = false>
__device__ __forceinline__ T restrict_cell_val(const Geo& gf, const T* __restrict__ rf, int I, int J,
                                               int K) {
  long long f0 = gidx(gf, 2 * I, 2 * J, D == 3 ? 2 * K : 0);
  long long sy = gf.st[1], sz = gf.st[2];
  T s = ldm<COH>(rf + f0) + ldm<COH>(rf + f0 + 1);
  s += ldm<COH>(rf + f0 + sy);
  s += ldm<COH>(rf + f0 + sy + 1);
  if constexpr (D == 3) {
    s += ldm<COH>(rf + f0 + sz);
    s += ldm<COH>(rf + f0 + sz + 1);
    s += ldm<COH>(rf + f0 + sz + sy);
    s += ldm<COH>(rf + f0 + sz + sy + 1);
  }
  return s * (D == 3 ? T(0.125) : T(0.25));
}

template <int D, typename T, bool COH = false>
__device__ __forceinline__ void restrict_cell_at(const Geo& gf, const Geo& gc,
                                                 const T* __restrict__ rf, T* __restrict__ fc,
                                                 T* __restrict__ xc, int I, int J, int K) {
  long long c = gidx(gc, I, J, K);
  fc[c] = restrict_cell_val<D, T, COH>(gf, rf, I, J, K);
  xc[c] = T(0);
}

// one coarse face C (a stored face along d, a cell across it)
template <int D, int d, typename T, bool COH = false>
__device__ __forceinline__ T restrict_face_val(const Geo& gf, const Geo& gc,
                                               const T* __restrict__ rf, const int C[3]) {
  bool wallface = !gc.per[d] && (C[d] == 0 || (C[d] == gc.n[d] && d != gc.open));
  if (wallface) return T(0);
  constexpr int ta = (d == 0) ? 1 : 0;
  constexpr int tb = (D == 3) ? ((d == 2) ? 1 : 2) : -1;
  int nf = gf.n[d];
  int f[3] = {0, 0, 0};
  T s = T(0);
#pragma unroll
  for (int t2 = 0; t2 < (D == 3 ? 2 : 1); ++t2) {
#pragma unroll
    for (int t1 = 0; t1 < 2; ++t1) {
      f[ta] = 2 * C[ta] + t1;
      if constexpr (tb >= 0) f[tb] = 2 * C[tb] + t2;
      T along = T(0);
#pragma unroll
      for (int o = -1; o <= 1; ++o) {
        int q = 2 * C[d] + o;
        if (gf.per[d]) q = q < 0 ? q + nf : (q >= nf ? q - nf : q);
        if (d == gf.open && q > nf) q = nf - 1;   // even ghost beyond the outflow
        f[d] = q;
        T w = (o == 0) ? T(0.5) : T(0.25);
        along += w * ldm<COH>(rf + gidx(gf, f[0], f[1], f[2]));
      }
      s += along;
    }
  }
  return s * (D == 3 ? T(0.25) : T(0.5));
}

template <int D, int d, typename T, bool COH = false>
__device__ __forceinline__ void restrict_face_at(const Geo& gf, const Geo& gc,
                                                 const T* __restrict__ rf, T* __restrict__ fc,
                                                 T* __restrict__ xc, const int C[3]) {
  long long c = gidx(gc, C[0], C[1], C[2]);
  xc[c] = T(0);
  fc[c] = restrict_face_val<D, d, T, COH>(gf, gc, rf, C);
}

// 1D prolongation weights. Cell-centred axis: 3/4 on the parent, 1/4 on the
// next coarse cell toward the child; beyond a wall the mirror ghost
// (sign `mirror`) folds that 1/4 into the parent. Face axis: the coincident
// coarse face, or the mean of the two coarse faces around a midway face.
// The weights are exact binary fractions in any precision.
template <typename T>
__device__ __forceinline__ int prol_cell_1d(int i, int nc, int per, int mirror_lo, int mirror_hi,
                                            int idx[2], T w[2]) {
  int I = i >> 1;
  int J = I + ((i & 1) ? 1 : -1);
  idx[0] = I;
  w[0] = T(0.75);
  w[1] = T(0);
  if (per) {
    idx[1] = J < 0 ? J + nc : (J >= nc ? J - nc : J);
    w[1] = T(0.25);
    return 2;
  }
  if (J < 0 || J >= nc) {
    const int mirror = J < 0 ? mirror_lo : mirror_hi;
    w[0] = mirror > 0 ? T(1) : T(0.5);
    idx[1] = I;   // weight 0: any valid index
    return 1;
  }
  idx[1] = J;
  w[1] = T(0.25);
  return 2;
}
template <typename T>
__device__ __forceinline__ int prol_face_1d(int i, int nc, int per, int idx[2], T w[2]) {
  int I = i >> 1;
  w[1] = T(0);
  if ((i & 1) == 0) {
    idx[0] = I;   // a fine face index is below 2 nc, so I < nc
    idx[1] = I;   // weight 0: any valid index
    w[0] = T(1);
    return 1;
  }
  idx[0] = I;
  w[0] = T(0.5);
  idx[1] = (per && I + 1 == nc) ? 0 : I + 1;
  w[1] = T(0.5);
  return 2;
}

// separable tensor-product sum: x-rows first, then y, then z, each pair of
// terms as w1 t1 + (w0 t0) with one rounding of the product and one of the
// fused sum. Every axis takes two terms; a missing term has weight 0 and a
// valid index, and adding its exact zero leaves the sum unchanged, so the
// loops unroll fully and the index and weight arrays stay in registers.
template <typename T, bool COH = false>
__device__ __forceinline__ T prol_sum(const Geo& gc, const T* __restrict__ ec, const int idx[3][2],
                                      const T w[3][2]) {
  T col[2];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    T row[2];
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      long long r = gidx(gc, 0, idx[1][b], idx[2][c]);
      row[b] = pfma(w[0][1], ldm<COH>(ec + r + idx[0][1]), pmul(w[0][0], ldm<COH>(ec + r + idx[0][0])));
    }
    col[c] = pfma(w[1][1], row[1], pmul(w[1][0], row[0]));
  }
  return pfma(w[2][1], col[1], pmul(w[2][0], col[0]));
}

// the coarse correction at one fine cell fi
template <int D, typename T, bool COH = false>
__device__ __forceinline__ T prolong_cell_val(const Geo& gc, const T* __restrict__ ec,
                                              const int fi[3]) {
  int idx[3][2] = {{0, 0}, {0, 0}, {0, 0}};
  T w[3][2] = {{T(1), T(0)}, {T(1), T(0)}, {T(1), T(0)}};
  // the pressure correction mirrors evenly at walls and the inflow, oddly at
  // the outflow, where the pressure is held
#pragma unroll
  for (int a = 0; a < D; ++a)
    prol_cell_1d<T>(fi[a], gc.n[a], gc.per[a], +1, a == gc.open ? -1 : +1, idx[a], w[a]);
  return prol_sum<T, COH>(gc, ec, idx, w);
}

template <int D, typename T>
__device__ __forceinline__ void prolong_cell_at(const Geo& gf, const Geo& gc,
                                                const T* __restrict__ ec, T* __restrict__ xf,
                                                const int fi[3]) {
  const long long x = gidx(gf, fi[0], fi[1], fi[2]);
  xf[x] = padd(xf[x], prolong_cell_val<D, T>(gc, ec, fi));
}

// the coarse correction at one fine face fi of component d (not a wall face)
template <int D, int d, typename T, bool COH = false>
__device__ __forceinline__ T prolong_face_val(const Geo& gc, const T* __restrict__ ec,
                                              const int fi[3]) {
  int idx[3][2] = {{0, 0}, {0, 0}, {0, 0}};
  T w[3][2] = {{T(1), T(0)}, {T(1), T(0)}, {T(1), T(0)}};
#pragma unroll
  for (int a = 0; a < D; ++a) {
    if (a == d)
      prol_face_1d<T>(fi[a], gc.n[a], gc.per[a], idx[a], w[a]);
    else   // tangential velocity: odd at walls and the inflow, even beyond the outflow
      prol_cell_1d<T>(fi[a], gc.n[a], gc.per[a], -1, a == gc.open ? +1 : -1, idx[a], w[a]);
  }
  return prol_sum<T, COH>(gc, ec, idx, w);
}

template <int D, int d, typename T>
__device__ __forceinline__ void prolong_face_at(const Geo& gf, const Geo& gc,
                                                const T* __restrict__ ec, T* __restrict__ xf,
                                                const int fi[3]) {
  const long long x = gidx(gf, fi[0], fi[1], fi[2]);
  xf[x] = padd(xf[x], prolong_face_val<D, d, T>(gc, ec, fi));
}

}  // namespace
}  // namespace bf
