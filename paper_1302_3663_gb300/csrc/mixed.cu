// Mixed-precision pieces of the defect-correction solves: each outer
// iteration computes the fine-grid residual r = f - A x in FP64, hands it to
// an FP32 V-cycle as the right-hand side of A e = r (e starts at 0), and adds
// the FP32 correction back into the FP64 iterate. The coarsest grid is solved
// in FP64 (its right-hand side and solution are converted at the boundary).
#include <cuda_runtime.h>
#include <math_constants.h>

#include "common.cuh"

namespace bf {

namespace {

constexpr int kBlock1D = 256;

__host__ __device__ constexpr int edge_id(int d, int e) {
  return (d < e ? d : e) + (d < e ? e : d) - 1;
}
__device__ __forceinline__ long long offp(const Geo& g, int a, int ci) {
  return (g.per[a] && ci == g.n[a] - 1) ? -(long long)(g.n[a] - 1) * g.st[a] : g.st[a];
}
__device__ __forceinline__ long long offm(const Geo& g, int a, int ci) {
  return (g.per[a] && ci == 0) ? (long long)(g.n[a] - 1) * g.st[a] : -g.st[a];
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// sum over a block whose size is a multiple of 32; valid in thread 0
__device__ double block_sum(double v, double* sh) {
  v = warp_sum(v);
  int t = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
  int nt = blockDim.x * blockDim.y * blockDim.z;
  int lane = t & 31, w = t >> 5;
  if (lane == 0) sh[w] = v;
  __syncthreads();
  v = (t < (nt + 31) / 32) ? sh[t] : 0.0;
  if (w == 0) v = warp_sum(v);
  __syncthreads();
  return v;
}
// maximum over a block whose size is a multiple of 32; valid in thread 0
__device__ double block_max(double v, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  int t = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
  int nt = blockDim.x * blockDim.y * blockDim.z;
  int lane = t & 31, w = t >> 5;
  if (lane == 0) sh[w] = v;
  __syncthreads();
  v = (t < (nt + 31) / 32) ? sh[t] : 0.0;
  if (w == 0) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  }
  __syncthreads();
  return v;
}
inline dim3 blk3(int D) { return D == 3 ? dim3(32, 4, 2) : dim3(32, 8, 1); }
inline dim3 grd3(long long nx, long long ny, long long nz, dim3 b) {
  return dim3((unsigned)((nx + b.x - 1) / b.x), (unsigned)((ny + b.y - 1) / b.y),
              (unsigned)((nz + b.z - 1) / b.z));
}

// The 2D forms of the FP64 passes around the FP32 V-cycles, one thread per
// point (a 2D grid is small: launches and latency bound it, not arithmetic).
// The 3D forms are in op64.cu.
//
// FP64 pressure residual written as the FP32 right-hand side of the
// correction equation; the FP32 correction is zeroed; per-block partial sums
// of r^2 (for the relative-residual test) in partial[0 .. nb) and per-block
// maxima of |r| (for the divergence the projection will leave, Eq. NSdis2 -
// NSdis4: max |D.u| = (euler dt / sigma) max |r|) in partial[nb .. 2 nb),
// nb the launch's blocks; a non-finite residual counts as infinity.
__global__ void __launch_bounds__(256) k_p_residual_mixed2(Geo g, POpArgs A) {
  __shared__ double sh[32];
  const Blk B = own_blk();
  int i = B.x * blockDim.x + threadIdx.x;
  int j = B.y * blockDim.y + threadIdx.y;
  double r2 = 0.0, ra = 0.0;
  if (i < g.n[0] && j < g.n[1]) {
    int ci[3] = {i, j, 0};
    long long c = gidx(g, i, j, 0);
    const double pc = A.p[c];
    double div = 0.0;
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      const double* __restrict__ b = A.beta[a];
      if (ci[a] < g.n[a] - 1 || g.per[a]) {
        long long cp = c + offp(g, a, ci[a]);
        div += b[cp] * (A.p[cp] - pc);
      }
      if (ci[a] > 0 || g.per[a]) div -= b[c] * (pc - A.p[c + offm(g, a, ci[a])]);
    }
    double r = A.f[c] - div * A.ih2;
    A.r32[c] = (float)r;
    A.e32[c] = 0.0f;
    r2 = r * r;
    ra = fabs(r);
    if (!(ra <= CUDART_INF)) ra = CUDART_INF;
  }
  if (A.partial) {
    r2 = block_sum(r2, sh);
    ra = block_max(ra, sh);
    if (threadIdx.x == 0 && threadIdx.y == 0 && threadIdx.z == 0) {
      const int nb = B.gx * B.gy * B.gz;
      A.partial[B.linear()] = r2;
      A.partial[nb + B.linear()] = ra;
    }
  }
}

// Diagonal of the FP64 viscous operator of component d at face F:
// m_d + (inv_re / h^2) * (2 mu_c on both cells + the edge viscosities, an edge
// beyond a wall counted twice for the mirrored tangential neighbour).
template <int D, int d>
__device__ __forceinline__ double v_diag64(const Geo& g, const LevelPtrs<double>& L,
                                           const int ci[3], long long F, double ir) {
  long long od_m = offm(g, d, ci[d]);
  double mcp = L.muc[F], mcm = L.muc[F + od_m];
  double dgV = 2.0 * (mcp + mcm);
#pragma unroll
  for (int e = 0; e < D; ++e) {
    if (e == d) continue;
    const double* __restrict__ me = L.mue[edge_id(d, e)];
    bool pe = g.per[e] != 0;
    bool wp = !pe && ci[e] == g.n[e] - 1;
    bool wm = !pe && ci[e] == 0;
    double mep = me[F + offp(g, e, ci[e])], mem = me[F];
    dgV += (wp ? 2.0 : 1.0) * mep + (wm ? 2.0 : 1.0) * mem;
  }
  return L.m[d][F] + ir * dgV;
}

struct F32x3 {
  float* a[3];
};

// 1 / diagonal per face component for the FP32 sweeps: formed in FP64 from
// the level's FP64 coefficients, rounded once to FP32.
template <int D>
__global__ void __launch_bounds__(256) k_v_idg32(Geo g, LevelPtrs<double> L, F32x3 idg,
                                                 double ir) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  int j = blockIdx.y * blockDim.y + threadIdx.y;
  int k = blockIdx.z * blockDim.z + threadIdx.z;
  if (i >= g.n[0] || j >= g.n[1] || k >= g.n[2]) return;
  int ci[3] = {i, j, k};
  long long F = gidx(g, i, j, k);
#pragma unroll
  for (int d = 0; d < D; ++d) {
    float v = 0.f;
    if (g.per[d] || ci[d] != 0) {
      double dg;
      if (d == 0) dg = v_diag64<D, 0>(g, L, ci, F, ir);
      else if (d == 1) dg = v_diag64<D, 1>(g, L, ci, F, ir);
      else dg = v_diag64<D, (D == 3 ? 2 : 1)>(g, L, ci, F, ir);
      // (divided in FP64: an FP32 reciprocal and one Newton step have about 46
      // bits, too few beside a tie of the rounding to FP32, and no range beyond it)
      v = (float)(1.0 / dg);
    }
    idg.a[d][F] = v;
  }
}

// (A u)_d at face F of a 2D grid, in the flux form of op64.cu: differences
// first, so no diagonal is formed.
template <int d, typename V>
__device__ __forceinline__ double v_op2(const Geo& g, const VOpArgs& A, const V* const vec[3],
                                        const int ci[3], long long F) {
  constexpr int e = 1 - d;
  const V* __restrict__ ud = vec[d];
  const V* __restrict__ ue = vec[e];
  const double* __restrict__ me = A.mue[0];
  const long long dp = offp(g, d, ci[d]), dm = offm(g, d, ci[d]);
  const long long ep = offp(g, e, ci[e]), em = offm(g, e, ci[e]);
  const bool wp = !g.per[e] && ci[e] == g.n[e] - 1, wm = !g.per[e] && ci[e] == 0;
  const double u = (double)ud[F];
  const double tp = A.muc[F] * ((double)ud[F + dp] - u), tm = A.muc[F + dm] * (u - (double)ud[F + dm]);
  const double up = wp ? -u : (double)ud[F + ep], um = wm ? -u : (double)ud[F + em];
  const double sp = me[F + ep] * ((up - u) + ((double)ue[F + ep] - (double)ue[F + ep + dm]));
  const double sm = me[F] * ((u - um) + ((double)ue[F] - (double)ue[F + dm]));
  return fma(-A.ir, fma(2.0, tp - tm, sp - sm), A.m[d][F] * u);
}

// FCG: w = A z on every unknown face (0 on the fixed wall faces) with partial
// sums of z.q; else r = f - A u to FP32 (and FP64 when given), the FP32
// correction zeroed, with partial sums of r^2.
template <bool FCG>
__global__ void __launch_bounds__(256) k_v_op2(Geo g, VOpArgs A) {
  __shared__ double sh[32];
  const Blk B = own_blk();
  int i = B.x * blockDim.x + threadIdx.x;
  int j = B.y * blockDim.y + threadIdx.y;
  double acc = 0.0;
  if (i < g.n[0] && j < g.n[1]) {
    int ci[3] = {i, j, 0};
    long long F = gidx(g, i, j, 0);
#pragma unroll
    for (int d = 0; d < 2; ++d) {
      const bool wall = !g.per[d] && ci[d] == 0;
      double v = 0.0;
      if constexpr (FCG) {
        if (!wall) v = d == 0 ? v_op2<0>(g, A, A.z, ci, F) : v_op2<1>(g, A, A.z, ci, F);
        A.w[d][F] = v;
        acc += (double)A.z[d][F] * A.q[d][F];
      } else {
        if (!wall) v = A.q[d][F] - (d == 0 ? v_op2<0>(g, A, A.u, ci, F) : v_op2<1>(g, A, A.u, ci, F));
        A.r32[d][F] = (float)v;
        A.e32[d][F] = 0.0f;
        if (A.w[d]) A.w[d][F] = v;
        acc += v * v;
      }
    }
  }
  if (A.partial) {
    acc = block_sum(acc, sh);
    if (threadIdx.x == 0 && threadIdx.y == 0 && threadIdx.z == 0) A.partial[B.linear()] = acc;
  }
}

// x += e over the unknowns of ncomp face components (ncomp = 0: cells)
template <int D>
__device__ __forceinline__ void add_correction_body(const Blk& B, Geo g, Ptr3d x, F32x3 e,
                                                    int ncomp) {
  int i = B.x * blockDim.x + threadIdx.x;
  int j = B.y * blockDim.y + threadIdx.y;
  int k = B.z * blockDim.z + threadIdx.z;
  if (i >= g.n[0] || j >= g.n[1] || k >= g.n[2]) return;
  int ci[3] = {i, j, k};
  long long c = gidx(g, i, j, k);
  if (ncomp == 0) {
    x.a[0][c] += (double)e.a[0][c];
    return;
  }
#pragma unroll
  for (int d = 0; d < 3; ++d)   // compile-time components: no local-memory copies
    if (d < ncomp && (g.per[d] || ci[d] != 0)) x.a[d][c] += (double)e.a[d][c];
}

template <int D>
__global__ void __launch_bounds__(256) k_add_correction(Geo g, Ptr3d x, F32x3 e, int ncomp) {
  add_correction_body<D>(own_blk(), g, x, e, ncomp);
}

template <typename Tin, typename Tout>
__global__ void __launch_bounds__(256) k_convert(const Tin* __restrict__ in, Tout* __restrict__ out,
                                                 long long n) {
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n;
       q += (long long)gridDim.x * blockDim.x)
    out[q] = (Tout)in[q];
}

}  // namespace

namespace {

struct ConvList {
  const double* in[12];
  float* out[12];
  int n;
};

__global__ void __launch_bounds__(256) k_convert_list(ConvList L, long long elems) {
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < elems;
       q += (long long)gridDim.x * blockDim.x)
    for (int a = 0; a < L.n; ++a) L.out[a][q] = (float)L.in[a][q];
}

}  // namespace

// blocks of the FP64 passes (their partial results)
int op_blocks(int D, const Geo& g, const OpShape& S) {
  if (D == 3) return op_blocks(S);
  dim3 gr = grd3(g.n[0], g.n[1], 1, blk3(2));
  return (int)(gr.x * gr.y);
}

void launch_p_residual_mixed(int D, const Geo& g, const OpShape& S, const LevelPtrs<double>& L,
                             float* r32, float* e32, double* partial, cudaStream_t s) {
  POpArgs a;
  a.p = L.p;
  a.f = L.pf;
  for (int d = 0; d < 3; ++d) a.beta[d] = L.beta[d];
  a.r32 = r32;
  a.e32 = e32;
  a.partial = partial;
  a.ih2 = 1.0 / (g.h * g.h);
  if (D == 3) launch_p_op(g, S, a, s);
  else k_p_residual_mixed2<<<grd3(g.n[0], g.n[1], 1, blk3(2)), blk3(2), 0, s>>>(g, a);
}

namespace {
VOpArgs v_op_args(const Geo& g, const LevelPtrs<double>& L, double inv_re, double* partial) {
  VOpArgs a = {};
  a.muc = L.muc;
  for (int d = 0; d < 3; ++d) {
    a.mue[d] = L.mue[d];
    a.m[d] = L.m[d];
  }
  a.ir = inv_re / (g.h * g.h);
  a.partial = partial;
  return a;
}
}  // namespace

void launch_v_residual_mixed(int D, const Geo& g, const OpShape& S, const LevelPtrs<double>& L,
                             float* const r32[3], float* const e32[3], double inv_re,
                             double* partial, cudaStream_t s, double* const r64[3]) {
  VOpArgs a = v_op_args(g, L, inv_re, partial);
  for (int d = 0; d < 3; ++d) {
    a.u[d] = L.u[d];
    a.q[d] = L.uf[d];
    a.w[d] = r64 ? r64[d] : nullptr;
    a.r32[d] = r32[d];
    a.e32[d] = e32[d];
  }
  if (D == 3) launch_v_op(false, g, S, a, s);
  else k_v_op2<false><<<grd3(g.n[0], g.n[1], 1, blk3(2)), blk3(2), 0, s>>>(g, a);
}

void launch_v_residual_op(const Geo& g, const OpShape& S, const LevelPtrs<double>& L, double inv_re,
                          cudaStream_t s) {
  VOpArgs a = v_op_args(g, L, inv_re, nullptr);
  for (int d = 0; d < 3; ++d) {
    a.u[d] = L.u[d];
    a.q[d] = L.uf[d];
    a.w[d] = L.ur[d];
  }
  launch_v_op(false, g, S, a, s);
}

// ------------------------------------------------------------ flexible CG
// Flexible conjugate gradients for the viscous solve, in FP64 around the
// FP32 V-cycle as preconditioner M (the viscous operator A is symmetric
// positive definite; M is neither symmetric nor fixed, so the update of the
// search direction uses the flexible form, with one previous direction):
//   z = M r,  w = A z,  beta = -(z.q) / (p.q)  (0 at the first iteration),
//   p = z + beta p,  q = w + beta q,  alpha = (p.r) / (p.q),
//   x += alpha p,  r -= alpha q.
// Scalars travel between the kernels in device memory (slots of `out`).
// The direction and update passes touch every stored element of the level
// arrays (pads and fixed wall faces hold 0 in every vector, so they add
// nothing): flat grid-stride loops over pairs of doubles.
constexpr int kFlatBlocks = 1216;   // 8 blocks of 256 threads per SM on 152 SMs

// The direction pass is bound by the FP64 rate, the update by it and by memory:
// products are summed by fused multiply-adds alone and conversions stay off the
// FP64 pipe (on the 128x128x256 duct 162 -> 132 us and 129 -> 119 us).
// p = z + beta p, q = w + beta q; partial sums of p.q (first nb) and p.r (next nb)
template <int D>
__device__ __forceinline__ void fcg_dir_body(const Blk& B, long long npair, F32x3 z, Ptr3d w,
                                             Ptr3d p, Ptr3d q, Ptr3d r,
                                             const double* __restrict__ out, int sl_zq, int sl_pq,
                                             double* partial) {
  __shared__ double sh[32];
  const double pq_old = out[sl_pq];
  // the first direction is z itself: the previous solve's p and q are not read
  const bool first = pq_old == 0.0;
  const double beta = first ? 0.0 : -out[sl_zq] / pq_old;
  double pq = 0.0, pr = 0.0;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const float4* __restrict__ zz = reinterpret_cast<const float4*>(z.a[d]);
    const double2* __restrict__ ww = reinterpret_cast<const double2*>(w.a[d]);
    const double2* __restrict__ rr = reinterpret_cast<const double2*>(r.a[d]);
    double2* pp = reinterpret_cast<double2*>(p.a[d]);
    double2* qq = reinterpret_cast<double2*>(q.a[d]);
    for (long long k = B.x * (long long)blockDim.x + threadIdx.x; 2 * k < npair;
         k += (long long)B.gx * blockDim.x) {
      const float4 zf = zz[k];
      double2 qv[2] = {ww[2 * k], ww[2 * k + 1]};
      const double2 rv[2] = {rr[2 * k], rr[2 * k + 1]};
      double2 po[2], qo[2];
      if (!first) {
        po[0] = pp[2 * k];
        po[1] = pp[2 * k + 1];
        qo[0] = qq[2 * k];
        qo[1] = qq[2 * k + 1];
      }
      double2 pv[2] = {make_double2(wide64(zf.x), wide64(zf.y)),
                       make_double2(wide64(zf.z), wide64(zf.w))};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (!first) {
          pv[h].x += beta * po[h].x;
          pv[h].y += beta * po[h].y;
          qv[h].x += beta * qo[h].x;
          qv[h].y += beta * qo[h].y;
        }
        pp[2 * k + h] = pv[h];
        qq[2 * k + h] = qv[h];
        pq = fma(pv[h].y, qv[h].y, fma(pv[h].x, qv[h].x, pq));
        pr = fma(pv[h].y, rv[h].y, fma(pv[h].x, rv[h].x, pr));
      }
    }
  }
  pq = block_sum(pq, sh);
  pr = block_sum(pr, sh);
  if (threadIdx.x == 0) {
    partial[B.x] = pq;
    partial[B.gx + B.x] = pr;
  }
}

template <int D>
__global__ void __launch_bounds__(256) k_fcg_dir(long long npair, F32x3 z, Ptr3d w, Ptr3d p,
                                                 Ptr3d q, Ptr3d r, const double* __restrict__ out,
                                                 int sl_zq, int sl_pq, double* partial) {
  fcg_dir_body<D>(own_blk(), npair, z, w, p, q, r, out, sl_zq, sl_pq, partial);
}

// x += alpha p, r -= alpha q; the new residual as the FP32 right-hand side of
// the next preconditioning (correction zeroed); partial sums of r.r
template <int D>
__device__ __forceinline__ void fcg_update_body(const Blk& B, long long npair, Ptr3d x, Ptr3d p,
                                                Ptr3d q, Ptr3d r, F32x3 r32, F32x3 e32,
                                                const double* __restrict__ out, int sl_pq,
                                                int sl_pr, double* partial) {
  __shared__ double sh[32];
  const double pq = out[sl_pq];
  const double alpha = pq != 0.0 ? out[sl_pr] / pq : 0.0;
  double rs = 0.0;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    double2* xx = reinterpret_cast<double2*>(x.a[d]);
    const double2* __restrict__ pp = reinterpret_cast<const double2*>(p.a[d]);
    const double2* __restrict__ qq = reinterpret_cast<const double2*>(q.a[d]);
    double2* rr = reinterpret_cast<double2*>(r.a[d]);
    float4* r4 = reinterpret_cast<float4*>(r32.a[d]);
    float4* e4 = reinterpret_cast<float4*>(e32.a[d]);
    for (long long k = B.x * (long long)blockDim.x + threadIdx.x; 2 * k < npair;
         k += (long long)B.gx * blockDim.x) {
      double2 xv[2] = {xx[2 * k], xx[2 * k + 1]}, rv[2] = {rr[2 * k], rr[2 * k + 1]};
      const double2 pv[2] = {pp[2 * k], pp[2 * k + 1]}, qv[2] = {qq[2 * k], qq[2 * k + 1]};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        xv[h].x += alpha * pv[h].x;
        xv[h].y += alpha * pv[h].y;
        rv[h].x -= alpha * qv[h].x;
        rv[h].y -= alpha * qv[h].y;
        xx[2 * k + h] = xv[h];
        rr[2 * k + h] = rv[h];
        rs = fma(rv[h].y, rv[h].y, fma(rv[h].x, rv[h].x, rs));
      }
      r4[k] = make_float4(narrow32(rv[0].x), narrow32(rv[0].y), narrow32(rv[1].x),
                          narrow32(rv[1].y));
      e4[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  rs = block_sum(rs, sh);
  if (threadIdx.x == 0) partial[B.x] = rs;
}

template <int D>
__global__ void __launch_bounds__(256) k_fcg_update(long long npair, Ptr3d x, Ptr3d p, Ptr3d q,
                                                    Ptr3d r, F32x3 r32, F32x3 e32,
                                                    const double* __restrict__ out, int sl_pq,
                                                    int sl_pr, double* partial) {
  fcg_update_body<D>(own_blk(), npair, x, p, q, r, r32, e32, out, sl_pq, sl_pr, partial);
}

namespace {
Ptr3d p3(double* const a[3]) {
  Ptr3d o;
  for (int d = 0; d < 3; ++d) o.a[d] = a[d];
  return o;
}
F32x3 f3(float* const a[3]) {
  F32x3 o;
  for (int d = 0; d < 3; ++d) o.a[d] = a[d];
  return o;
}
}  // namespace

void launch_fcg_apply(int D, const Geo& g, const OpShape& S, const LevelPtrs<double>& L,
                      float* const z[3], double inv_re, double* const w[3], double* const q[3],
                      double* partial, cudaStream_t s) {
  VOpArgs a = v_op_args(g, L, inv_re, partial);
  for (int d = 0; d < 3; ++d) {
    a.z[d] = z[d];
    a.q[d] = q[d];
    a.w[d] = w[d];
  }
  if (D == 3) launch_v_op(true, g, S, a, s);
  else k_v_op2<true><<<grd3(g.n[0], g.n[1], 1, blk3(2)), blk3(2), 0, s>>>(g, a);
}

// flat loops run over two pairs: the level arrays hold a multiple of 8
// elements (rows padded to it) and start on 256-byte boundaries
__host__ __device__ long long flat_elems(const Geo& g) { return g.st[2] * g.s[2]; }

int fcg_flat_blocks(const Geo& g) {
  long long npair = flat_elems(g) / 2;
  long long nb = (npair + 255) / 256;
  return (int)(nb < kFlatBlocks ? (nb < 1 ? 1 : nb) : kFlatBlocks);
}

void launch_fcg_dir(int D, const Geo& g, float* const z[3], double* const w[3], double* const p[3],
                    double* const q[3], double* const r[3], const double* out, int sl_zq,
                    int sl_pq, double* partial, cudaStream_t s) {
  const long long npair = flat_elems(g) / 2;
  const int nb = fcg_flat_blocks(g);
  if (D == 3)
    k_fcg_dir<3><<<nb, 256, 0, s>>>(npair, f3(z), p3(w), p3(p), p3(q), p3(r), out, sl_zq, sl_pq, partial);
  else
    k_fcg_dir<2><<<nb, 256, 0, s>>>(npair, f3(z), p3(w), p3(p), p3(q), p3(r), out, sl_zq, sl_pq, partial);
}

void launch_fcg_update(int D, const Geo& g, double* const x[3], double* const p[3],
                       double* const q[3], double* const r[3], float* const r32[3],
                       float* const e32[3], const double* out, int sl_pq, int sl_pr,
                       double* partial, cudaStream_t s) {
  const long long npair = flat_elems(g) / 2;
  const int nb = fcg_flat_blocks(g);
  if (D == 3)
    k_fcg_update<3><<<nb, 256, 0, s>>>(npair, p3(x), p3(p), p3(q), p3(r), f3(r32), f3(e32), out,
                                       sl_pq, sl_pr, partial);
  else
    k_fcg_update<2><<<nb, 256, 0, s>>>(npair, p3(x), p3(p), p3(q), p3(r), f3(r32), f3(e32), out,
                                       sl_pq, sl_pr, partial);
}

void launch_add_correction(int D, const Geo& g, double* const x[3], float* const e[3], int ncomp,
                           cudaStream_t s) {
  dim3 b = blk3(D);
  dim3 gr = grd3(g.n[0], g.n[1], g.n[2], b);
  Ptr3d xx;
  F32x3 ee;
  for (int d = 0; d < 3; ++d) {
    xx.a[d] = x[d];
    ee.a[d] = e[d];
  }
  if (D == 3) k_add_correction<3><<<gr, b, 0, s>>>(g, xx, ee, ncomp);
  else k_add_correction<2><<<gr, b, 0, s>>>(g, xx, ee, ncomp);
}

void launch_f32_to_f64(const float* in, double* out, long long n, cudaStream_t s) {
  k_convert<float, double><<<(unsigned)flat_convert_blocks(n), kBlock1D, 0, s>>>(in, out, n);
}

void launch_f64_to_f32(const double* in, float* out, long long n, cudaStream_t s) {
  k_convert<double, float><<<(unsigned)flat_convert_blocks(n), kBlock1D, 0, s>>>(in, out, n);
}

void launch_v_idg32(int D, const Geo& g, const LevelPtrs<double>& L64,
                    const LevelPtrs<float>& L32, double ir, cudaStream_t s) {
  dim3 b = blk3(D);
  dim3 gr = grd3(g.n[0], g.n[1], g.n[2], b);
  F32x3 o;
  for (int d = 0; d < 3; ++d) o.a[d] = L32.idg[d];
  if (D == 3) k_v_idg32<3><<<gr, b, 0, s>>>(g, L64, o, ir);
  else k_v_idg32<2><<<gr, b, 0, s>>>(g, L64, o, ir);
}

void launch_coef_to_f32(int D, const Geo& g, const LevelPtrs<double>& L64,
                        const LevelPtrs<float>& L32, cudaStream_t s) {
  ConvList cl;
  cl.n = 0;
  for (int d = 0; d < D; ++d) {
    cl.in[cl.n] = L64.beta[d];
    cl.out[cl.n++] = L32.beta[d];
    cl.in[cl.n] = L64.m[d];
    cl.out[cl.n++] = L32.m[d];
  }
  cl.in[cl.n] = L64.muc;
  cl.out[cl.n++] = L32.muc;
  for (int e = 0; e < (D == 3 ? 3 : 1); ++e) {
    cl.in[cl.n] = L64.mue[e];
    cl.out[cl.n++] = L32.mue[e];
  }
  long long n = g.st[2] * g.s[2];
  long long nb = (n + kBlock1D - 1) / kBlock1D;
  if (nb > 4096) nb = 4096;
  k_convert_list<<<(unsigned)nb, kBlock1D, 0, s>>>(cl, n);
}

// ------------------------------------------------------------------ batched
// The level-0 FP64 steps of the batched solves: the bodies above over a
// persistent batch's work list, each with a member's own arrays, scalars and
// the block decomposition of its single-instance launch.
__global__ void __launch_bounds__(256) kb_add_correction(BArgs A, int viscous) {
  for_items(A, [&](const BMember& M, const Blk& B) {
    Ptr3d x;
    F32x3 e;
    for (int d = 0; d < 3; ++d) {
      x.a[d] = viscous ? M.d[0].u[d] : (d == 0 ? M.d[0].p : nullptr);
      e.a[d] = viscous ? M.f[0].u[d] : (d == 0 ? M.f[0].p : nullptr);
    }
    add_correction_body<3>(B, M.g[0], x, e, viscous ? 3 : 0);
  });
}

__global__ void __launch_bounds__(256) kb_fcg_dir(BArgs A, int sl_zq, int sl_pq) {
  for_items(A, [&](const BMember& M, const Blk& B) {
    F32x3 z;
    Ptr3d w, p, q, r;
    for (int d = 0; d < 3; ++d) {
      z.a[d] = M.f[0].u[d];
      w.a[d] = M.d[0].u2[d];
      p.a[d] = M.cg_p[d];
      q.a[d] = M.cg_q[d];
      r.a[d] = M.d[0].ur[d];
    }
    fcg_dir_body<3>(B, flat_elems(M.g[0]) / 2, z, w, p, q, r, M.sc.out, sl_zq, sl_pq,
                    M.sc.partial);
  });
}

__global__ void __launch_bounds__(256) kb_fcg_update(BArgs A, int sl_pq, int sl_pr) {
  for_items(A, [&](const BMember& M, const Blk& B) {
    Ptr3d x, p, q, r;
    F32x3 r32, e32;
    for (int d = 0; d < 3; ++d) {
      x.a[d] = M.d[0].u[d];
      p.a[d] = M.cg_p[d];
      q.a[d] = M.cg_q[d];
      r.a[d] = M.d[0].ur[d];
      r32.a[d] = M.f[0].uf[d];
      e32.a[d] = M.f[0].u[d];
    }
    fcg_update_body<3>(B, flat_elems(M.g[0]) / 2, x, p, q, r, r32, e32, M.sc.out, sl_pq, sl_pr,
                       M.sc.partial);
  });
}

int flat_convert_blocks(long long n) {
  long long nb = (n + kBlock1D - 1) / kBlock1D;
  if (nb > 4096) nb = 4096;
  return (int)(nb < 1 ? 1 : nb);
}

void launch_b_add_correction(const BArgs& A, bool viscous, int grid, cudaStream_t s) {
  if (A.n > 0) kb_add_correction<<<grid, blk3(3), 0, s>>>(A, viscous ? 1 : 0);
}
void launch_b_fcg_dir(const BArgs& A, int sl_zq, int sl_pq, int grid, cudaStream_t s) {
  if (A.n > 0) kb_fcg_dir<<<grid, 256, 0, s>>>(A, sl_zq, sl_pq);
}
void launch_b_fcg_update(const BArgs& A, int sl_pq, int sl_pr, int grid, cudaStream_t s) {
  if (A.n > 0) kb_fcg_update<<<grid, 256, 0, s>>>(A, sl_pq, sl_pr);
}

}  // namespace bf
