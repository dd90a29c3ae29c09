// The coarse levels of a V-cycle in one launch: one thread-block cluster per
// simulation, every iterate in distributed shared memory.
//
// A level of a few thousand to a few ten thousand cells keeps one launch per
// colour, component, residual and transfer far from any bound: 3 to 6 us each,
// nearly all latency. Here a cluster of C CTAs splits each level into slabs
// along the last axis (z; y in 2D). A CTA holds its slab of the iterate, the
// coefficients, right-hand sides and inverse diagonals in shared memory, red
// and black points of a row apart (a warp updates consecutive elements: no
// bank conflicts), with one halo plane on each side. A thread that updates a
// point of a boundary plane also stores it into the neighbour's halo plane
// (st.shared::cluster), so every read is local; the hardware cluster barrier
// separates the colour phases. Residuals and coarse iterates change levels
// through global memory (L2). The mixed-precision cycles solve the coarsest
// level in FP64, as the FP64 contexts do every level.
//
// Bound by latency: a phase costs a cluster barrier with release and acquire
// (0.36 us) and one pass of loads and a chain of some 20 operations, 0.5 us on a
// level of a few thousand cells, 1.5 us with 27,648 (by launches: 5 to 6 us for
// both colours on 32x32x64). A viscous V(2,2) cycle from a 24x24x48 level down
// takes 116 us against 208 us from 12x12x24 down in the 8-CTA kernel it replaced
// (iterates in L2) plus about 90 us of launches for the 24x24x48 level. Steps:
// 48x48x96 33.0 -> 18.2 ms, 144x144x288 (9x9x18 coarsest) 142 -> 107 ms, 2D 64x32
// 1.46 -> 0.74 ms.
//
// The point updates, residuals and transfers are those of the per-level
// launches, rounding for rounding, so an FP32 level gives the same bits either
// way; FP64 residuals have the flux form here, and agree to rounding. The cluster's
// size changes no bit.
#include <cuda_runtime.h>

#include <algorithm>

#include "common.cuh"
#include "point.cuh"
#include "transfer.cuh"

namespace bf {

namespace {

// Threads per CTA (768 and 1024 were slower on every level: fewer registers,
// dearer barriers).
constexpr int kClThreads = 512;
constexpr int kClMatThreads = 128;
constexpr int kClMatRows = 800;          // largest coarsest solve kept as a matrix
constexpr size_t kClSmem = 222 * 1024;   // dynamic shared memory of a CTA at most
// A level of at most this many cells runs on the cluster's first CTA alone: a
// block barrier takes 0.13 us, a cluster barrier with release and acquire
// 0.36 us (measured), and so few points gain nothing from more CTAs.
constexpr int kClSolo = 512;

__host__ __device__ inline unsigned cl_magic(int d) {
  return (unsigned)((0x100000000ull + (unsigned long long)d - 1) / (unsigned long long)d);
}
// q / d for q d < 2^32 (at most a few ten thousand points per CTA)
__device__ __forceinline__ int cl_div(int q, unsigned m, int d) {
  return d == 1 ? q : (int)__umulhi((unsigned)q, m);
}

// Lays a level out from element `base`; returns the end. inv: inverse
// diagonals are kept for the pressure too, and in two parts (FP64).
__host__ __device__ inline int cl_layout(int D, bool V, bool inv, const Geo& g, int C, int fs,
                                         int base, ClLv& v) {
  const int S = D - 1;
  if ((long long)g.n[0] * g.n[1] * g.n[2] <= kClSolo) C = 1;
  v.n0 = g.n[0];
  v.s0 = g.s[0];
  v.R = D == 3 ? g.n[1] : 1;
  v.sR = D == 3 ? g.s[1] : 1;
  v.nS = S == 2 ? g.n[2] : g.n[1];
  v.per0 = g.per[0];
  v.perR = D == 3 ? g.per[1] : 1;
  v.perS = S == 2 ? g.per[2] : g.per[1];
  v.RS = (v.s0 + 1) / 2;
  v.CP = v.RS * v.sR;
  v.PS = 2 * v.CP;
  v.nh = (v.n0 + 1) / 2;
  v.mnh = cl_magic(v.nh);
  v.mR = cl_magic(v.R);
  v.ms0 = cl_magic(v.s0);
  v.msR = cl_magic(v.sR);
  v.C = C;
  v.st1 = (int)g.st[1];
  v.st2 = (int)(S == 2 ? g.st[2] : g.st[1]);
  v.pc = (v.nS + C - 1) / C;
  v.na = (v.nS + v.pc - 1) / v.pc;
  v.last = v.nS - (v.na - 1) * v.pc;
  v.fs = fs;
  int o = base;
  const int nc = V ? D : 1;
  for (int d = 0; d < nc; ++d) {
    v.u[d] = o;
    o += (v.pc + 2) * v.PS;
  }
  if (V) {
    v.c = o;   // mu at centres: planes 0 .. pc
    o += (v.pc + 1) * v.PS;
    for (int q = 0; q < (D == 3 ? 3 : 1); ++q) {   // edges: plane pc + 1 where S is one axis
      const bool up = D == 2 || q >= 1;
      v.e[q] = o - v.PS;
      o += (v.pc + (up ? 1 : 0)) * v.PS;
    }
  } else {
    for (int a = 0; a < D; ++a) {
      v.e[a] = o - v.PS;
      o += (v.pc + (a == S ? 1 : 0)) * v.PS;
    }
  }
  for (int d = 0; d < 3; ++d) v.f[d] = v.g[d] = v.gl[d] = -1;   // not in shared memory
  if (fs)
    for (int d = 0; d < nc; ++d) {
      v.f[d] = o - v.PS;
      o += v.pc * v.PS;
      if (V || inv) {
        v.g[d] = o - v.PS;
        o += v.pc * v.PS;
      }
      if (inv) {
        v.gl[d] = o - v.PS;
        o += v.pc * v.PS;
      }
    }
  return o;
}

// the planes of one CTA of the level and its neighbours
__host__ __device__ inline void cl_rank(ClLv& v, int rank) {
  const bool in = rank < v.na;
  v.k0 = in ? rank * v.pc : v.nS;
  v.npl = in ? (rank == v.na - 1 ? v.last : v.pc) : 0;
  v.lo = in ? (rank > 0 ? rank - 1 : (v.perS ? v.na - 1 : -1)) : -1;
  v.hi = in ? (rank < v.na - 1 ? rank + 1 : (v.perS ? 0 : -1)) : -1;
  v.nlo = v.lo == v.na - 1 ? v.last : v.pc;
}

// Lays out levels from .. L - 1; returns their bytes (0: they do not fit). The
// first level keeps its right-hand sides in shared memory where all fits with
// them. The deeper ones always do, and so does the coarsest where it is the
// first and its right-hand side is rewritten in the slab: converted in a mixed
// cycle, without its mean for the pressure. nd > 0: the coarsest solve is a
// matrix of nd rows and holds only its right-hand side, from element u[0].
size_t cl_total(int D, bool fp64, bool V, const Geo* g, int L, int from, int C, int nd, ClLv* lv) {
  for (int f = 1; f >= (from == L - 1 && (!fp64 || !V) ? 1 : 0); --f) {
    size_t b = 0;
    for (int l = from; l < L; ++l) {
      const int el = fp64 || l == L - 1 ? 8 : 4;
      const int base = (int)(b / el);
      int end = cl_layout(D, V, el == 8, g[l], C, l == from ? f : 1, base, lv[l]);
      if (nd > 0 && l == L - 1) {
        lv[l].u[0] = base;
        end = base + nd;
      }
      b = ((size_t)end * el + 15) / 16 * 16;
      if (b > kClSmem) break;
    }
    if (b <= kClSmem) return b;
  }
  return 0;
}

template <typename T>
__device__ __forceinline__ T* cl_sm() {
  extern __shared__ __align__(16) unsigned char cl_raw[];
  return reinterpret_cast<T*>(cl_raw);
}

__device__ __forceinline__ void cl_sync() {
  asm volatile("barrier.cluster.arrive.release;\n\t"
               "barrier.cluster.wait.acquire;" ::: "memory");
}
// between the phases of a level
__device__ __forceinline__ void cl_phase_sync(const ClLv& v) {
  if (v.C > 1) cl_sync();
  else __syncthreads();
}
__device__ __forceinline__ void cl_store(float* p, int rank, float v) {
  unsigned a = (unsigned)__cvta_generic_to_shared(p), r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(r), "f"(v) : "memory");
}
__device__ __forceinline__ void cl_store(double* p, int rank, double v) {
  unsigned a = (unsigned)__cvta_generic_to_shared(p), r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(r), "d"(v) : "memory");
}

// store v at element idx (in local plane lp) and into the halo of the
// neighbour whose boundary plane it is
template <typename T>
__device__ __forceinline__ void cl_put(const ClLv& v, T* sm, int idx, int lp, T val) {
  sm[idx] = val;
  if (lp == 1 && v.lo >= 0) {
    if (v.C == 1) sm[idx + v.nlo * v.PS] = val;
    else cl_store(sm + idx + v.nlo * v.PS, v.lo, val);
  }
  if (lp == v.npl && v.hi >= 0) {
    if (v.C == 1) sm[idx - lp * v.PS] = val;
    else cl_store(sm + idx - lp * v.PS, v.hi, val);
  }
}

// A point of the slab: local index without its colour part, neighbour offsets
// (each step also flips the colour), wall flags, axis indices.
template <int D>
struct ClPt {
  int b, dp[3], dm[3];
  bool wp[3], wm[3];
  int ci[3], lp;
};
// PER: x or the row axis may be periodic. Without it a neighbour beyond a wall
// keeps its plain offset: it lies inside the slab's array and is not used.
template <int D, bool PER>
__device__ __forceinline__ void cl_point(const ClLv& v, int h, int par, int r, int lp, ClPt<D>& q) {
  constexpr int S = D - 1;
  const int i = 2 * h + par, k = v.k0 + lp - 1;
  q.b = lp * v.PS + r * v.RS + h;
  q.lp = lp;
  q.ci[0] = i;
  if constexpr (D == 3) q.ci[1] = r;
  q.ci[S] = k;
  if constexpr (D == 2) q.ci[2] = 0;
  const bool f0 = i == 0, l0 = i == v.n0 - 1;
  q.dp[0] = (PER && v.per0 && l0) ? -h : par;
  q.dm[0] = (PER && v.per0 && f0) ? (v.n0 - 1) >> 1 : par - 1;
  q.wp[0] = (!PER || !v.per0) && l0;
  q.wm[0] = (!PER || !v.per0) && f0;
  if constexpr (D == 3) {
    const bool f1 = r == 0, l1 = r == v.R - 1;
    q.dp[1] = (PER && v.perR && l1) ? -(v.R - 1) * v.RS : v.RS;
    q.dm[1] = (PER && v.perR && f1) ? (v.R - 1) * v.RS : -v.RS;
    q.wp[1] = (!PER || !v.perR) && l1;
    q.wm[1] = (!PER || !v.perR) && f1;
  }
  q.dp[S] = v.PS;
  q.dm[S] = -v.PS;
  q.wp[S] = !v.perS && k == v.nS - 1;
  q.wm[S] = !v.perS && k == 0;
}
template <int D>
__device__ __forceinline__ int cl_F(const ClLv& v, const ClPt<D>& q) {
  return q.ci[0] + (D == 3 ? v.st1 * q.ci[1] : 0) + v.st2 * q.ci[D - 1];
}

// f(h, parity, r, lp) over the owned points of one colour, numbered without
// gaps: a warp's lanes are full whatever the row length (an FP64 instruction
// costs the same for one lane as for 32)
template <class F>
__device__ __forceinline__ void cl_colour(const ClLv& v, int colour, F&& f) {
  const int np = v.npl * v.R * v.nh;
  for (int q = threadIdx.x; q < np; q += blockDim.x) {
    const int a = cl_div(q, v.mnh, v.nh), h = q - a * v.nh;
    const int lp0 = cl_div(a, v.mR, v.R), r = a - lp0 * v.R;
    const int par = (r + v.k0 + lp0 + colour) & 1;
    if (2 * h + par < v.n0) f(h, par, r, lp0 + 1);
  }
}
// ------------------------------------------------------------ point updates
// v_red and p_red (point.cuh) on the slab: u_d at its new value
template <int D, int d, typename T>
__device__ __forceinline__ T cl_v_update(const ClLv& v, const T* __restrict__ sm,
                                         const ClPt<D>& q, int own, int opp, T f, T idg, T idl,
                                         T ir) {
  const int dmd = q.dm[d];
  const T* ud = sm + v.u[d];
  const T mcp = sm[v.c + own], mcm = sm[v.c + opp + dmd];
  T cross = T(0), cep[2], cem[2];
  int n = 0;
#pragma unroll
  for (int e = 0; e < D; ++e) {
    if (e == d) continue;
    const T* ue = sm + v.u[e];
    const T* me = sm + v.e[pt_edge(d, e)];
    const T mep = me[opp + q.dp[e]], mem = me[own];
    cross = padd(cross, pfma(mep, psub(ue[opp + q.dp[e]], ue[own + q.dp[e] + dmd]),
                             -pmul(mem, psub(ue[own], ue[opp + dmd]))));
    cep[n] = mep;
    cem[n] = mem;
    ++n;
  }
  T off = pfma(pmul(T(2), mcm), ud[opp + dmd], pfma(pmul(T(2), mcp), ud[opp + q.dp[d]], cross));
  n = 0;
#pragma unroll
  for (int e = 0; e < D; ++e) {
    if (e == d) continue;
    if (!q.wp[e]) off = pfma(cep[n], ud[opp + q.dp[e]], off);
    if (!q.wm[e]) off = pfma(cem[n], ud[opp + q.dm[e]], off);
    ++n;
  }
  if constexpr (sizeof(T) == 4) return pmul(pfma(ir, off, f), idg);
  else return pt_quot(pfma(ir, off, f), idg, idl);
}

template <int D, typename T>
__device__ __forceinline__ void cl_p_terms(const ClLv& v, const T* __restrict__ sm,
                                           const ClPt<D>& q, int own, int opp, T& num, T& dg) {
  num = T(0);
  dg = T(0);
  const T* p = sm + v.u[0];
#pragma unroll
  for (int a = 0; a < D; ++a) {
    const T* b = sm + v.e[a];
    if (!q.wm[a]) {
      const T bb = b[own];
      num = pfma(bb, p[opp + q.dm[a]], num);
      dg = padd(dg, bb);
    }
    if (!q.wp[a]) {
      const T bb = b[opp + q.dp[a]];
      num = pfma(bb, p[opp + q.dp[a]], num);
      dg = padd(dg, bb);
    }
  }
}

// one colour of component d, or of the pressure; coef: ir or h^2
template <int D, int d, typename T, bool PER>
__device__ __forceinline__ void cl_v_phase(const ClLv& v, const T* __restrict__ f,
                                           const T* __restrict__ g, const T* __restrict__ gl,
                                           int colour, T ir) {
  T* sm = cl_sm<T>();
  cl_colour(v, colour, [&](int h, int par, int r, int lp) {
    ClPt<D> q;
    cl_point<D, PER>(v, h, par, r, lp, q);
    if (q.wm[d]) return;   // the wall face stays 0
    const int own = q.b + (colour ? v.CP : 0), opp = q.b + (colour ? 0 : v.CP);
    const T fv = v.fs ? sm[v.f[d] + own] : __ldg(f + cl_F(v, q));
    const T gv = v.fs ? sm[v.g[d] + own] : __ldg(g + cl_F(v, q));
    T lv = T(0);
    if constexpr (sizeof(T) == 8) lv = v.fs ? sm[v.gl[d] + own] : __ldg(gl + cl_F(v, q));
    cl_put(v, sm, v.u[d] + own, lp, cl_v_update<D, d, T>(v, sm, q, own, opp, fv, gv, lv, ir));
  });
  cl_phase_sync(v);
}

template <int D, typename T, bool PER>
__device__ __forceinline__ void cl_p_phase(const ClLv& v, const T* __restrict__ f,
                                           const T* __restrict__ g, const T* __restrict__ gl,
                                           int colour, T h2) {
  T* sm = cl_sm<T>();
  cl_colour(v, colour, [&](int h, int par, int r, int lp) {
    ClPt<D> q;
    cl_point<D, PER>(v, h, par, r, lp, q);
    const int own = q.b + (colour ? v.CP : 0), opp = q.b + (colour ? 0 : v.CP);
    const T fv = v.fs ? sm[v.f[0] + own] : __ldg(f + cl_F(v, q));
    T num, dg;
    cl_p_terms<D, T>(v, sm, q, own, opp, num, dg);
    T pv;
    if constexpr (sizeof(T) == 4) pv = px_final(num, dg, h2, fv);
    else pv = pt_quot(pfma(-h2, fv, num), v.fs ? sm[v.g[0] + own] : __ldg(g + cl_F(v, q)),
                      v.fs ? sm[v.gl[0] + own] : __ldg(gl + cl_F(v, q)));
    cl_put(v, sm, v.u[0] + own, lp, pv);
  });
  cl_phase_sync(v);
}

template <int D, typename T, bool V, bool PER>
__device__ __forceinline__ void cl_smooth(const ClLv& v, const LevelPtrs<T>& L, int n, T coef) {
  if (v.C == 1 && v.npl == 0) return;   // the first CTA's level
  for (int it = 0; it < n; ++it) {
    if constexpr (V) {
      for (int c = 0; c < 2; ++c)
        cl_v_phase<D, 0, T, PER>(v, L.uf[0], L.idg[0], L.idl[0], c, coef);
      for (int c = 0; c < 2; ++c)
        cl_v_phase<D, 1, T, PER>(v, L.uf[1], L.idg[1], L.idl[1], c, coef);
      if constexpr (D == 3)
        for (int c = 0; c < 2; ++c)
          cl_v_phase<D, 2, T, PER>(v, L.uf[2], L.idg[2], L.idl[2], c, coef);
    } else {
      for (int c = 0; c < 2; ++c) cl_p_phase<D, T, PER>(v, L.pf, L.pdg, L.pdl, c, coef);
    }
  }
}

// ---------------------------------------------------------------- residuals
template <int D, int d, typename T>
__device__ __forceinline__ void cl_v_res(const ClLv& v, const LevelPtrs<T>& L, const ClPt<D>& q,
                                         int own, int opp, T ir) {
  const T* sm = cl_sm<T>();
  const int F = cl_F(v, q);
  T r = T(0);
  if (!q.wm[d]) {
    const T* ud = sm + v.u[d];
    const int dmd = q.dm[d];
    const T u = ud[own];
    T W = vr_normal(sm[v.c + own], ud[opp + q.dp[d]], u, sm[v.c + opp + dmd], ud[opp + dmd]);
#pragma unroll
    for (int e = 0; e < D; ++e) {
      if (e == d) continue;
      const T* ue = sm + v.u[e];
      const T* me = sm + v.e[pt_edge(d, e)];
      const T up = q.wp[e] ? -u : ud[opp + q.dp[e]], um = q.wm[e] ? -u : ud[opp + q.dm[e]];
      W = vr_edge(W, u, me[opp + q.dp[e]], up, ue[opp + q.dp[e]], ue[own + q.dp[e] + dmd], me[own],
                  um, ue[own], ue[opp + dmd]);
    }
    r = vr_final(v.fs ? sm[v.f[d] + own] : __ldg(L.uf[d] + F), __ldg(L.m[d] + F), u, ir, W);
  }
  L.ur[d][F] = r;
}

template <int D, typename T, bool V, bool PER>
__device__ __forceinline__ void cl_residual(const ClLv& v, const LevelPtrs<T>& L, T coef) {
  const T* sm = cl_sm<T>();
  for (int colour = 0; colour < 2; ++colour)
    cl_colour(v, colour, [&](int h, int par, int r, int lp) {
      ClPt<D> q;
      cl_point<D, PER>(v, h, par, r, lp, q);
      const int own = q.b + (colour ? v.CP : 0), opp = q.b + (colour ? 0 : v.CP);
      if constexpr (V) {
        cl_v_res<D, 0, T>(v, L, q, own, opp, coef);
        cl_v_res<D, 1, T>(v, L, q, own, opp, coef);
        if constexpr (D == 3) cl_v_res<D, 2, T>(v, L, q, own, opp, coef);
      } else {
        T num, dg;
        cl_p_terms<D, T>(v, sm, q, own, opp, num, dg);
        const int F = cl_F(v, q);
        L.pr[F] = pr_final(v.fs ? sm[v.f[0] + own] : __ldg(L.pf + F), num, dg, sm[v.u[0] + own],
                           coef);
      }
    });
}

// ---------------------------------------------------------------- transfers
// the coarse level's right-hand side from the fine residual (global): into its
// slab (slab) and the global array, which holds every level's after a cycle as the
// launches leave it (the coarsest one's is read whole there by the pressure's mean
// and the matrix solve)
template <int D, typename T, typename TC, bool V>
__device__ __forceinline__ void cl_restrict(const ClLv& v, const Geo& gf, const Geo& gc,
                                            const LevelPtrs<T>& F, const LevelPtrs<T>& Lc,
                                            bool slab) {
  TC* sm = cl_sm<TC>();
  for (int colour = 0; colour < 2; ++colour)
    cl_colour(v, colour, [&](int h, int par, int r, int lp) {
      ClPt<D> q;
      cl_point<D, true>(v, h, par, r, lp, q);
      const int own = q.b + (colour ? v.CP : 0);
      if constexpr (V) {
        T w[D];
        w[0] = restrict_face_val<D, 0, T, true>(gf, gc, F.ur[0], q.ci);
        w[1] = restrict_face_val<D, 1, T, true>(gf, gc, F.ur[1], q.ci);
        if constexpr (D == 3) w[2] = restrict_face_val<D, 2, T, true>(gf, gc, F.ur[2], q.ci);
#pragma unroll
        for (int d = 0; d < D; ++d) {
          if (slab) sm[v.f[d] + own] = (TC)w[d];
          Lc.uf[d][cl_F(v, q)] = w[d];
        }
      } else {
        const T w = restrict_cell_val<D, T, true>(gf, F.pr, q.ci[0], q.ci[1], q.ci[2]);
        if (slab) sm[v.f[0] + own] = (TC)w;
        Lc.pf[cl_F(v, q)] = w;
      }
    });
}

// the slab's iterate to global memory
template <int D, typename T, typename TC, bool V>
__device__ __forceinline__ void cl_write(const ClLv& v, const LevelPtrs<T>& L) {
  const TC* sm = cl_sm<TC>();
  for (int colour = 0; colour < 2; ++colour)
    cl_colour(v, colour, [&](int h, int par, int r, int lp) {
      const int idx = lp * v.PS + r * v.RS + h + (colour ? v.CP : 0);
      const int F = 2 * h + par + (D == 3 ? v.st1 * r : 0) + v.st2 * (v.k0 + lp - 1);
      if constexpr (V) {
#pragma unroll
        for (int d = 0; d < D; ++d) L.u[d][F] = (T)sm[v.u[d] + idx];
      } else {
        L.p[F] = (T)sm[v.u[0] + idx];
      }
    });
}

// the coarse correction (global) added to the fine slab
template <int D, typename T, bool V>
__device__ __forceinline__ void cl_prolong(const ClLv& v, const Geo& gc, const LevelPtrs<T>& Lc) {
  T* sm = cl_sm<T>();
  for (int colour = 0; colour < 2; ++colour)
    cl_colour(v, colour, [&](int h, int par, int r, int lp) {
      ClPt<D> q;
      cl_point<D, true>(v, h, par, r, lp, q);
      const int own = q.b + (colour ? v.CP : 0);
      if constexpr (V) {
        if (!q.wm[0])
          cl_put(v, sm, v.u[0] + own, lp,
                 padd(sm[v.u[0] + own], prolong_face_val<D, 0, T, true>(gc, Lc.u[0], q.ci)));
        if (!q.wm[1])
          cl_put(v, sm, v.u[1] + own, lp,
                 padd(sm[v.u[1] + own], prolong_face_val<D, 1, T, true>(gc, Lc.u[1], q.ci)));
        if constexpr (D == 3)
          if (!q.wm[2])
            cl_put(v, sm, v.u[2] + own, lp,
                   padd(sm[v.u[2] + own], prolong_face_val<D, 2, T, true>(gc, Lc.u[2], q.ci)));
      } else {
        cl_put(v, sm, v.u[0] + own, lp,
               padd(sm[v.u[0] + own], prolong_cell_val<D, T, true>(gc, Lc.p, q.ci)));
      }
    });
}

// Fills a level's slab: coefficients; the iterate (from global memory with
// `iterate`, else 0); on the first level its right-hand side, converted from
// `F` (the FP32 arrays, where the FP64 coarsest level is the first) or L. A
// thread issues all loads of UN points before it stores any: a pass of one
// point per thread takes 0.9 us however little it loads.
template <int D, typename TC, typename T, bool V>
__device__ __forceinline__ void cl_load(const ClLv& v, const Geo& g, const LevelPtrs<TC>& L,
                                        const LevelPtrs<T>& F, bool first, bool iterate) {
  TC* sm = cl_sm<TC>();
  const int sS = D == 3 ? g.s[2] : g.s[1];
  constexpr int nc = V ? D : 1, ne = V ? (D == 3 ? 3 : 1) : D;
  constexpr int UN = sizeof(TC) == 8 ? 2 : 4;
  if (v.npl == 0) return;
  const int np = (v.npl + 2) * v.sR * v.s0;
  for (int q0 = threadIdx.x; q0 < np; q0 += UN * blockDim.x) {
    TC u[UN][nc], c[UN], e[UN][ne], f[UN][nc], gi[UN][nc], gl[UN][nc];
    int idx[UN], lpn[UN];
#pragma unroll
    for (int n = 0; n < UN; ++n) {
      const int q = q0 + n * (int)blockDim.x;
      const int a = cl_div(q, v.ms0, v.s0), i = q - a * v.s0;
      const int lp = cl_div(a, v.msR, v.sR), r = a - lp * v.sR;
      const int k = v.k0 + lp - 1;
      const int kw = v.perS ? (k < 0 ? k + v.nS : (k >= v.nS ? k - v.nS : k)) : k;
      const bool ok = q < np, in = ok && kw >= 0 && kw < sS;
      const bool own = ok && v.fs && lp >= 1 && lp <= v.npl;
      const int o = kw * v.st2 + r * v.st1 + i;
      lpn[n] = ok ? lp : -1;
      idx[n] = lp * v.PS + ((i + r + k) & 1) * v.CP + r * v.RS + (i >> 1);
#pragma unroll
      for (int d = 0; d < nc; ++d) u[n][d] = iterate && in ? (V ? L.u[d] : L.p)[o] : TC(0);
      if constexpr (V) c[n] = in && lp <= v.npl ? __ldg(L.muc + o) : TC(0);
#pragma unroll
      for (int m = 0; m < ne; ++m)
        e[n][m] = in && lp >= 1 ? __ldg((V ? L.mue[m] : L.beta[m]) + o) : TC(0);
#pragma unroll
      for (int d = 0; d < nc; ++d) {
        f[n][d] = own && first ? (TC)(V ? F.uf[d] : F.pf)[o] : TC(0);
        if constexpr (V) gi[n][d] = own ? __ldg(L.idg[d] + o) : TC(0);
        else if constexpr (sizeof(TC) == 8) gi[n][d] = own ? __ldg(L.pdg + o) : TC(0);
        if constexpr (sizeof(TC) == 8) gl[n][d] = own ? __ldg((V ? L.idl[d] : L.pdl) + o) : TC(0);
      }
    }
#pragma unroll
    for (int n = 0; n < UN; ++n) {
      if (lpn[n] < 0) continue;
      const int lp = lpn[n], x = idx[n];
#pragma unroll
      for (int d = 0; d < nc; ++d) sm[v.u[d] + x] = u[n][d];
      if constexpr (V)
        if (lp <= v.npl) sm[v.c + x] = c[n];
#pragma unroll
      for (int m = 0; m < ne; ++m) {   // plane npl + 1 where the slab axis is one of the two
        const bool up = V ? (D == 2 || m >= 1) : m == D - 1;
        if (lp >= 1 && (up || lp <= v.npl)) sm[v.e[m] + x] = e[n][m];
      }
      if (v.fs && lp >= 1 && lp <= v.npl) {
#pragma unroll
        for (int d = 0; d < nc; ++d) {
          if (first) sm[v.f[d] + x] = f[n][d];
          if constexpr (V || sizeof(TC) == 8) sm[v.g[d] + x] = gi[n][d];
          if constexpr (sizeof(TC) == 8) sm[v.gl[d] + x] = gl[n][d];
        }
      }
    }
  }
}

// The coarsest pressure problem is singular: its right-hand side (global, pf)
// loses its mean. Every CTA sums all of it in the same order.
template <int D, typename T>
__device__ __forceinline__ void cl_coarse_mean(const ClLv& v, const Geo& g, const T* pf,
                                               double* sh) {
  double* sm = cl_sm<double>();
  const int nc = g.n[0] * g.n[1] * g.n[2];
  double s = 0.0;
  for (int q = threadIdx.x; q < nc; q += kClThreads) {
    const int i = q % g.n[0], r = q / g.n[0], j = r % g.n[1], k = r / g.n[1];
    s += (double)__ldcg(pf + gidx(g, i, j, k));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  s = 0.0;
  for (int w = 0; w < kClThreads / 32; ++w) s += sh[w];
  const double mean = s / (double)nc;
  for (int colour = 0; colour < 2; ++colour)
    cl_colour(v, colour, [&](int h, int par, int r, int lp) {
      const int own = lp * v.PS + r * v.RS + h + (colour ? v.CP : 0);
      sm[v.f[0] + own] -= mean;
    });
  __syncthreads();
}

template <int D, typename T>
__device__ __forceinline__ const LevelPtrs<T>& cl_ptrs(const BMember& M, int l) {
  if constexpr (sizeof(T) == 4) return M.f[l];
  else return M.d[l];
}

// The coarsest solve as a matrix (see k_coarse_matrix): its rows are shared by
// the cluster's warps; each row's products are summed in one fixed order.
template <int D, typename T, bool V>
__device__ __forceinline__ void cl_matrix_solve(const Geo& g, const LevelPtrs<T>& L,
                                                const double* __restrict__ B, int n, double* fv,
                                                int C, int rank) {
  const int nc = g.n[0] * g.n[1] * g.n[2];
  auto at = [&](int q, int& d) {
    d = q / nc;
    const int c = q - d * nc, i = c % g.n[0], r = c / g.n[0];
    return (int)gidx(g, i, r % g.n[1], r / g.n[1]);
  };
  for (int q = threadIdx.x; q < n; q += blockDim.x) {
    int d;
    const int F = at(q, d);
    fv[q] = (double)__ldcg((V ? L.uf[d] : L.pf) + F);
  }
  __syncthreads();
  const int nw = blockDim.x >> 5, lane = threadIdx.x & 31;
  for (int row = rank * nw + (threadIdx.x >> 5); row < n; row += C * nw) {
    const double* __restrict__ b = B + (long long)row * n;
    double s = 0.0;
#pragma unroll 4
    for (int q = lane; q < n; q += 32) s = fma(__ldg(b + q), fv[q], s);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
      int d;
      const int F = at(row, d);
      (V ? L.u[d] : L.p)[F] = (T)s;
    }
  }
}

// T: the V-cycle's precision (FP32: the coarsest level in FP64). One cluster
// per listed member runs its levels from its tail level on, or the coarsest one.
template <int D, typename T, bool V, bool PER>
__global__ void __launch_bounds__(kClThreads, 1)
    k_cluster(const BMember* __restrict__ tab, const int* __restrict__ list, int nlist,
              const int* __restrict__ act, int coarse_only) {
  constexpr bool mixed = sizeof(T) == 4;
  __shared__ ClLv lvs[kMaxLevels];
  __shared__ double sh[32];
  unsigned C, rank;
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(C));
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  const int item = blockIdx.x / C;
  if (item >= nlist) return;
  const int m = list[item];
  if (act && !act[m]) return;   // the whole cluster leaves
  const BMember& M = tab[m];
  const int lc = M.L - 1, ls = coarse_only ? lc : M.tail;
  if (ls > lc) return;
  const double* __restrict__ cmat = M.cmat[V];
  const int nd = M.ncm[V];
  const bool dense = nd > 0;
  {   // the levels' layouts from the table
    const int* src = reinterpret_cast<const int*>(M.cl[coarse_only ? 1 : 0][V] + ls);
    int* dst = reinterpret_cast<int*>(lvs + ls);
    const int n = (lc - ls + 1) * (int)(sizeof(ClLv) / sizeof(int));
    for (int q = threadIdx.x; q < n; q += blockDim.x) dst[q] = __ldg(src + q);
  }
  __syncthreads();
  if ((int)threadIdx.x >= ls && (int)threadIdx.x <= lc) cl_rank(lvs[threadIdx.x], (int)rank);
  __syncthreads();
  for (int l = ls; l <= lc; ++l) {
    if (dense && l == lc) break;
    if (mixed && l == lc)
      cl_load<D, double, T, V>(lvs[l], M.g[l], M.d[l], cl_ptrs<D, T>(M, l), l == ls, false);
    else
      cl_load<D, T, T, V>(lvs[l], M.g[l], cl_ptrs<D, T>(M, l), cl_ptrs<D, T>(M, l), l == ls,
                          l == ls);
  }
  cl_sync();
  for (int l = ls; l < lc; ++l) {
    const ClLv v = lvs[l];
    const LevelPtrs<T>& L = cl_ptrs<D, T>(M, l);
    const T coef = V ? (T)M.ir[l] : (T)(M.g[l].h * M.g[l].h);
    cl_smooth<D, T, V, PER>(v, L, M.nu1, coef);
    cl_residual<D, T, V, PER>(v, L, V ? coef : (T)M.ih2[l]);
    const bool last = l + 1 == lc;
    if (v.C > 1 || lvs[l + 1].C > 1) cl_sync();
    else __syncthreads();
    const LevelPtrs<T>& Lc = cl_ptrs<D, T>(M, l + 1);
    if (mixed && last)
      cl_restrict<D, T, double, V>(lvs[l + 1], M.g[l], M.g[l + 1], L, Lc, !dense);
    else
      cl_restrict<D, T, T, V>(lvs[l + 1], M.g[l], M.g[l + 1], L, Lc, !(dense && last));
    if (last && (!V || dense)) cl_sync();   // every CTA's part is read
    else __syncthreads();
  }
  if (dense) {
    cl_matrix_solve<D, T, V>(M.g[lc], cl_ptrs<D, T>(M, lc), cmat, nd, cl_sm<double>() + lvs[lc].u[0],
                             (int)C, (int)rank);
  } else {
    const ClLv v = lvs[lc];
    if constexpr (!V) cl_coarse_mean<D, T>(v, M.g[lc], cl_ptrs<D, T>(M, lc).pf, sh);
    cl_smooth<D, double, V, PER>(v, M.d[lc], M.coarse_sweeps, V ? M.ir[lc] : M.g[lc].h * M.g[lc].h);
    cl_write<D, T, double, V>(v, cl_ptrs<D, T>(M, lc));
  }
  if (lc > ls) cl_sync();
  for (int l = lc - 1; l >= ls; --l) {
    const ClLv v = lvs[l];
    const LevelPtrs<T>& L = cl_ptrs<D, T>(M, l);
    cl_prolong<D, T, V>(v, M.g[l + 1], cl_ptrs<D, T>(M, l + 1));
    cl_phase_sync(v);
    cl_smooth<D, T, V, PER>(v, L, M.nu2, V ? (T)M.ir[l] : (T)(M.g[l].h * M.g[l].h));
    cl_write<D, T, T, V>(v, L);
    if (l > ls) {
      if (v.C > 1 || lvs[l - 1].C > 1) cl_sync();
      else __syncthreads();
    }
  }
}

// The coarsest solve starts from zero and its sweeps (after the pressure's
// mean removal) are linear, so for fixed coefficients it is a matrix: column q
// is its answer to the unit right-hand side q. Solves to a tolerance run tens
// of V-cycles per time step; with the matrix each of them replaces 96 dependent
// colour phases (about 0.5 us each) by one product. One block per column.
template <int D, bool V>
__global__ void __launch_bounds__(kClMatThreads)
    k_coarse_matrix(Geo g, LevelPtrs<double> L, int sweeps, double coef, double* __restrict__ B,
                    int n) {
  __shared__ ClLv lv;
  const int nc = g.n[0] * g.n[1] * g.n[2];
  const int col = blockIdx.x, d = col / nc, c = col - d * nc;
  const int ci[3] = {c % g.n[0], (c / g.n[0]) % g.n[1], c / (g.n[0] * g.n[1])};
  if (threadIdx.x == 0) {
    cl_layout(D, V, true, g, 1, 1, 0, lv);
    cl_rank(lv, 0);
  }
  __syncthreads();
  const ClLv v = lv;
  double* sm = cl_sm<double>();
  const bool wall = V && !g.per[d] && (d == 0 ? ci[0] : (d == 1 ? ci[1] : ci[2])) == 0;
  cl_load<D, double, double, V>(v, g, L, L, false, false);
  const double mean = V ? 0.0 : 1.0 / (double)nc;
  for (int colour = 0; colour < 2; ++colour)
    cl_colour(v, colour, [&](int h, int, int r, int lp) {
      const int idx = lp * v.PS + r * v.RS + h + (colour ? v.CP : 0);
      for (int e = 0; e < (V ? D : 1); ++e) sm[v.f[e] + idx] = -mean;
    });
  __syncthreads();
  if (threadIdx.x == 0 && !wall) {   // (a wall face's right-hand side is 0: its column is not read)
    const int r = D == 3 ? ci[1] : 0, k = ci[D - 1];
    sm[v.f[d] + (k + 1) * v.PS + ((ci[0] + r + k) & 1) * v.CP + r * v.RS + (ci[0] >> 1)] += 1.0;
  }
  __syncthreads();
  cl_smooth<D, double, V, true>(v, L, sweeps, coef);
  for (int colour = 0; colour < 2; ++colour)
    cl_colour(v, colour, [&](int h, int par, int r, int lp) {
      const int idx = lp * v.PS + r * v.RS + h + (colour ? v.CP : 0);
      const int q = 2 * h + par + g.n[0] * (r + (D == 3 ? g.n[1] : 1) * (lp - 1));
      for (int e = 0; e < (V ? D : 1); ++e)
        B[(long long)(e * nc + q) * n + col] = sm[v.u[e] + idx];
    });
}

template <int D, typename T, bool PER>
const void* cl_kernel_of(bool V) {
  return V ? (const void*)k_cluster<D, T, true, PER> : (const void*)k_cluster<D, T, false, PER>;
}
const void* cl_kernel(int D, bool fp64, bool V, bool per) {
  if (D == 3) {
    if (fp64) return per ? cl_kernel_of<3, double, true>(V) : cl_kernel_of<3, double, false>(V);
    return per ? cl_kernel_of<3, float, true>(V) : cl_kernel_of<3, float, false>(V);
  }
  if (fp64) return per ? cl_kernel_of<2, double, true>(V) : cl_kernel_of<2, double, false>(V);
  return per ? cl_kernel_of<2, float, true>(V) : cl_kernel_of<2, float, false>(V);
}

}  // namespace

size_t cl_bytes(int D, bool fp64, bool viscous, const Geo* g, int L, int from, int C, int nd,
                ClLv* lv) {
  ClLv own[kMaxLevels];
  return cl_total(D, fp64, viscous, g, L, from, C, nd, lv ? lv : own);
}

int cl_first_level(int D, bool fp64, const Geo* g, int L, long long cells, int C, const int nd[2]) {
  if (g[0].open >= 0 || cells <= 0) return L;
  for (int l = 0; l < L; ++l)
    if ((long long)g[l].n[0] * g[l].n[1] * g[l].n[2] <= cells &&
        cl_bytes(D, fp64, true, g, L, l, C, nd[1]) && cl_bytes(D, fp64, false, g, L, l, C, nd[0]))
      return l;
  return L;
}

// A matrix costs its build, n columns of the sweeps once per time step (about
// 0.1 ms for n = 384), and n^2 products per V-cycle: past 800 rows that is no
// longer less than the phases it replaces.
int cl_matrix_rows(int D, bool viscous, const Geo& g) {
  if (g.open >= 0) return 0;
  const long long n = (long long)g.n[0] * g.n[1] * g.n[2] * (viscous ? D : 1);
  ClLv v;
  if (n > kClMatRows || (size_t)cl_layout(D, viscous, true, g, 1, 1, 0, v) * 8 > kClSmem) return 0;
  return (int)n;
}

void launch_coarse_matrix(int D, bool viscous, const Geo& g, const LevelPtrs<double>& L, int sweeps,
                          double inv_re, double* B, int n, cudaStream_t s) {
  ClLv v;
  const size_t smem = (size_t)cl_layout(D, viscous, true, g, 1, 1, 0, v) * 8;
  const double coef = viscous ? inv_re / (g.h * g.h) : g.h * g.h;
  if (D == 3 && viscous) k_coarse_matrix<3, true><<<n, kClMatThreads, smem, s>>>(g, L, sweeps, coef, B, n);
  else if (D == 3) k_coarse_matrix<3, false><<<n, kClMatThreads, smem, s>>>(g, L, sweeps, coef, B, n);
  else if (viscous) k_coarse_matrix<2, true><<<n, kClMatThreads, smem, s>>>(g, L, sweeps, coef, B, n);
  else k_coarse_matrix<2, false><<<n, kClMatThreads, smem, s>>>(g, L, sweeps, coef, B, n);
}

int cl_max_ctas() {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(16);
  cfg.blockDim = dim3(kClThreads);
  cfg.dynamicSmemBytes = kClSmem;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = 16;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  int n = 0;
  const bool ok = cudaOccupancyMaxActiveClusters(&n, cl_kernel(3, false, true, true), &cfg) == cudaSuccess;
  if (!ok) cudaGetLastError();
  return ok && n >= 1 ? 16 : 8;
}

cudaError_t cl_setup() {
  for (int q = 0; q < 16; ++q) {
    const void* f = cl_kernel(q & 1 ? 3 : 2, (q & 2) != 0, (q & 4) != 0, (q & 8) != 0);
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  for (const void* f : {(const void*)k_coarse_matrix<3, true>, (const void*)k_coarse_matrix<3, false>,
                        (const void*)k_coarse_matrix<2, true>, (const void*)k_coarse_matrix<2, false>}) {
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClSmem);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

void launch_cluster(int D, bool fp64, bool viscous, bool per, const BMember* tab, const int* list, int nlist,
                    const int* act, bool coarse_only, int C, size_t smem, cudaStream_t s) {
  if (nlist <= 0) return;
  int only = coarse_only ? 1 : 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(nlist * C));
  cfg.blockDim = dim3(kClThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)C;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  void* args[] = {(void*)&tab, (void*)&list, (void*)&nlist, (void*)&act, (void*)&only};
  cudaLaunchKernelExC(&cfg, cl_kernel(D, fp64, viscous, per), args);
}

}  // namespace bf
