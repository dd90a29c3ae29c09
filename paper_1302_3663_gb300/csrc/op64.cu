// FP64 operator passes of the mixed-precision solves in 3D (no open axis):
// the flexible CG's w = A z, the viscous residual r = f - A u and the pressure
// residual, each with the reduction its solve needs.
//
// GB300 runs FP64 at 1/64 of the FP32 rate, so these passes are bound by
// their FP64 operations, not by memory. A face-by-face form computes every
// edge stress four times, every normal stress twice and every pressure flux
// twice. Here a block walks the planes of a chunk over a tile of columns,
// one thread per column; each thread forms the quantities its own point owns
// (three edge stresses, three normal stresses; three fluxes), hands those its
// neighbours need on through shared memory and carries those of the plane
// below in registers. About 42 FP64 operations per cell for the viscous
// operator instead of about 80, 13 instead of about 30 for the pressure, and
// one reduction per chunk instead of one per 256 points. w = A z on the
// 128x128x256 duct: 506 us with the FP64 pipe 74 % busy, against 665 us (86 %)
// face by face plus 34 us for an FP64 copy of z, which this form reads in FP32.
// The pressure's planes are short, so each is loaded while the one before is
// worked on: 147 us there and 269 us on 160x160x320 against 183 and 371 with
// the loads in front of their use. (The viscous planes hold four times the
// work; prefetching them towards L2 left 507 us at 507.)
#include <cuda_runtime.h>
#include <math_constants.h>

#include "common.cuh"

namespace bf {

namespace {

__device__ __forceinline__ double op_warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// sum over the block's kOpThreads threads; valid in thread 0
__device__ __forceinline__ double op_block_sum(double v, double* sh) {
  v = op_warp_sum(v);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    v = threadIdx.x < kOpThreads / 32 ? sh[threadIdx.x] : 0.0;
    v = op_warp_sum(v);
  }
  __syncthreads();
  return v;
}
__device__ __forceinline__ unsigned long long op_umax(unsigned long long a, unsigned long long b) {
  return a > b ? a : b;
}

__device__ __forceinline__ double op_wide(float f) { return wide64(f); }
__device__ __forceinline__ double op_wide(double f) { return f; }
// a sign flip on the integer pipe
__device__ __forceinline__ double op_neg_if(double v, bool neg) {
  return __hiloint2double(__double2hiint(v) ^ (neg ? (int)0x80000000u : 0), __double2loint(v));
}

// The column of a lane: c = 0 and c = ex + 1, r = 0 and r = ey + 1 are the
// halo of the tile's ex x ey own columns. `o` indexes the iterate (clamped at
// a wall, wrapped on a periodic axis), `om` the coefficients (the slot of the
// upper wall included).
struct Lane {
  int c, r, i, j, o, om;
  bool in, own, fx, fy;   // fx, fy: beyond a wall along x, y
};

__device__ __forceinline__ Lane op_lane(const Geo& g, const OpShape& S, int bx) {
  Lane q;
  const int w = S.TX + 2;
  q.r = threadIdx.x / w;
  q.c = threadIdx.x - q.r * w;
  const int i0 = (bx % S.nx) * S.TX, j0 = (bx / S.nx) * S.TY;
  const int ex = min(S.TX, g.n[0] - i0), ey = min(S.TY, g.n[1] - j0);
  q.i = i0 - 1 + q.c;
  q.j = j0 - 1 + q.r;
  q.in = q.c <= ex + 1 && q.r <= ey + 1;
  q.own = q.in && q.c >= 1 && q.c <= ex && q.r >= 1 && q.r <= ey;
  const bool ox = q.i < 0 || q.i >= g.n[0], oy = q.j < 0 || q.j >= g.n[1];
  q.fx = ox && !g.per[0];
  q.fy = oy && !g.per[1];
  const int iw = q.i < 0 ? q.i + g.n[0] : (q.i >= g.n[0] ? q.i - g.n[0] : q.i);
  const int jw = q.j < 0 ? q.j + g.n[1] : (q.j >= g.n[1] ? q.j - g.n[1] : q.j);
  const int ic = g.per[0] ? iw : min(max(q.i, 0), g.n[0] - 1);
  const int jc = g.per[1] ? jw : min(max(q.j, 0), g.n[1] - 1);
  const int im = g.per[0] ? iw : max(q.i, 0), jm = g.per[1] ? jw : max(q.j, 0);
  q.o = ic + (int)g.st[1] * jc;
  q.om = im + (int)g.st[1] * jm;
  return q;
}

// A velocity component's value at a lane's column and plane k with the mirror
// ghosts of the walls: odd for the tangential components, 0 for the normal one.
template <int d, typename T>
__device__ __forceinline__ double op_u(const Geo& g, const T* __restrict__ u, const Lane& q,
                                       int k) {
  const bool out = k < 0 || k >= g.n[2], fz = out && !g.per[2];
  const int kw = k < 0 ? k + g.n[2] : (k >= g.n[2] ? k - g.n[2] : k);
  const int kc = g.per[2] ? kw : min(max(k, 0), g.n[2] - 1);
  const bool nrm = d == 0 ? q.fx : (d == 1 ? q.fy : fz);
  if (nrm) return 0.0;
  const double v = op_wide(u[q.o + (int)g.st[2] * kc]);
  const bool neg = (d != 0 && q.fx) != ((d != 1 && q.fy) != (d != 2 && fz));
  return op_neg_if(v, neg);
}

// Viscous operator. With t_d = mu_c (u_d(+) - u_d) at centres and s_de =
// mu_de ((u_d - u_d(-e)) + (u_e - u_e(-d))) on edges,
//   V_d = 2 (t_d - t_d(-d)) + sum_e (s_de(+e) - s_de),   (A u)_d = m_d u_d - ir V_d.
// FCG: u is the FP32 correction z; w = A z, partial sums of z.q.
// else: r = f - A u to FP32 and the FP32 correction zeroed (when given), to w
// (when given), partial sums of r^2.
template <bool FCG>
__device__ __forceinline__ void v_op_body(const Blk& B, const Geo& g, const OpShape& S,
                                          const VOpArgs& a) {
  __shared__ double A[3][kOpThreads];
  __shared__ double E[5][kOpThreads];   // t_x, t_y, s_xy, s_xz, s_yz
  __shared__ double sh[32];
  const Lane q = op_lane(g, S, B.x);
  const int t = threadIdx.x, w = S.TX + 2;
  const int k0 = B.y * S.KC, k1 = min(k0 + S.KC, g.n[2]);
  const int st2 = (int)g.st[2];
  auto load = [&](int k, double u[3]) {
    if constexpr (FCG) {
      u[0] = op_u<0>(g, a.z[0], q, k);
      u[1] = op_u<1>(g, a.z[1], q, k);
      u[2] = op_u<2>(g, a.z[2], q, k);
    } else {
      u[0] = op_u<0>(g, a.u[0], q, k);
      u[1] = op_u<1>(g, a.u[1], q, k);
      u[2] = op_u<2>(g, a.u[2], q, k);
    }
  };
  // centres below a wall and above one are never used: clamped
  auto cell_plane = [&](int k) {
    const int kw = k < 0 ? k + g.n[2] : (k >= g.n[2] ? k - g.n[2] : k);
    return st2 * (g.per[2] ? kw : min(max(k, 0), g.n[2] - 1));
  };
  // edges on the upper wall have a slot of their own
  auto edge_plane = [&](int k) { return st2 * (g.per[2] && k >= g.n[2] ? k - g.n[2] : k); };
  double up[3] = {0.0, 0.0, 0.0};   // the column's values on the plane below
  double mcp = 0.0, sxzp = 0.0, syzp = 0.0, tzp = 0.0;
  double px = 0.0, py = 0.0, pz = 0.0;   // the in-plane part of V on the plane below
  double acc = 0.0;
  const bool mid = q.in && q.r >= 1, inner = mid && q.r <= S.TY;
  if (q.in) {
    load(k0 - 1, up);
    mcp = a.muc[q.om + cell_plane(k0 - 1)];
  }
  for (int k = k0; k <= k1; ++k) {
    double u[3] = {0.0, 0.0, 0.0}, mc = 0.0, mxy = 0.0, mxz = 0.0, myz = 0.0;
    double mF[3], qF[3];
    const int F = q.o + st2 * (k - 1);
    if (q.in) {
      load(k, u);
      const int ep = q.om + edge_plane(k);
      if (k < k1) {
        mc = a.muc[q.om + cell_plane(k)];
        if (mid) mxy = a.mue[0][ep];
      }
      if (inner) mxz = a.mue[1][ep];
      if (mid) myz = a.mue[2][ep];
      A[0][t] = u[0];
      A[1][t] = u[1];
      A[2][t] = u[2];
    }
    if (q.own && k > k0) {
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        mF[d] = a.m[d][F];
        qF[d] = a.q[d][F];
      }
    }
    __syncthreads();
    double tx = 0.0, ty = 0.0, sxy = 0.0, sxz = 0.0, syz = 0.0, tz = 0.0;
    if (q.in) {
      if (k < k1) {
        if (q.r <= S.TY) {
          ty = mc * (A[1][t + w] - u[1]);
          E[1][t] = ty;
        }
        if (inner && q.c <= S.TX) {
          tx = mc * (A[0][t + 1] - u[0]);
          E[0][t] = tx;
        }
        if (mid && q.c >= 1) {
          sxy = mxy * ((u[0] - A[0][t - w]) + (u[1] - A[1][t - 1]));
          E[2][t] = sxy;
        }
      }
      if (inner && q.c >= 1) {
        sxz = mxz * ((u[0] - up[0]) + (u[2] - A[2][t - 1]));
        E[3][t] = sxz;
        tz = mcp * (u[2] - up[2]);
      }
      if (mid) {
        syz = myz * ((u[1] - up[1]) + (u[2] - A[2][t - w]));
        E[4][t] = syz;
      }
    }
    __syncthreads();
    if (q.own) {
      if (k > k0) {   // the plane below is complete
        const double V[3] = {px + (sxz - sxzp), py + (syz - syzp), fma(2.0, tz - tzp, pz)};
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const bool wall = !g.per[d] && (d == 0 ? q.i == 0 : (d == 1 ? q.j == 0 : k == 1));
          const double Au = fma(-a.ir, V[d], mF[d] * up[d]);
          if constexpr (FCG) {
            a.w[d][F] = wall ? 0.0 : Au;
            acc = fma(up[d], qF[d], acc);
          } else {
            const double r = wall ? 0.0 : qF[d] - Au;
            if (a.r32[d]) {
              a.r32[d][F] = narrow32(r);
              a.e32[d][F] = 0.f;
            }
            if (a.w[d]) a.w[d][F] = r;
            acc = fma(r, r, acc);
          }
        }
      }
      if (k < k1) {
        px = fma(2.0, tx - E[0][t - 1], E[2][t + w] - sxy);
        py = fma(2.0, ty - E[1][t - w], E[2][t + 1] - sxy);
        pz = (E[3][t + 1] - sxz) + (E[4][t + w] - syz);
      }
    }
    sxzp = sxz;
    syzp = syz;
    tzp = tz;
    mcp = mc;
    up[0] = u[0];
    up[1] = u[1];
    up[2] = u[2];
  }
  if (a.partial) {
    acc = op_block_sum(acc, sh);
    if (t == 0) a.partial[B.linear()] = acc;
  }
}

// Pressure residual r = f - D.(beta D p) handed to FP32, the FP32 correction
// zeroed; per block the sum of r^2 in partial[0 .. nb) and the maximum of |r|
// (a non-finite residual counts as infinity) in partial[nb .. 2 nb). The
// maximum is taken on the bit patterns of |r|: the integer pipe is idle here.
__device__ __forceinline__ void p_op_body(const Blk& B, const Geo& g, const OpShape& S,
                                          const POpArgs& a) {
  __shared__ double A[kOpThreads];
  __shared__ double E[2][kOpThreads];
  __shared__ double sh[32];
  __shared__ unsigned long long shm[32];
  const Lane q = op_lane(g, S, B.x);
  const int t = threadIdx.x, w = S.TX + 2;
  const int k0 = B.y * S.KC, k1 = min(k0 + S.KC, g.n[2]);
  const int st2 = (int)g.st[2];
  const bool mid = q.in && q.r >= 1 && q.c >= 1;
  const bool wx = !g.per[0] && (q.i <= 0 || q.i >= g.n[0]);
  const bool wy = !g.per[1] && (q.j <= 0 || q.j >= g.n[1]);
  auto plane = [&](int k) {
    const int kw = k < 0 ? k + g.n[2] : (k >= g.n[2] ? k - g.n[2] : k);
    return st2 * (g.per[2] ? kw : min(max(k, 0), g.n[2] - 1));
  };
  struct Raw {
    double p, bx, by, bz, f;
  };
  auto load = [&](int k) {   // what the column needs of plane k (f: of the plane below)
    Raw r{0.0, 0.0, 0.0, 0.0, 0.0};
    if (q.in && k <= k1) {
      const int pk = plane(k);
      r.p = a.p[q.o + pk];
      if (k < k1 && mid) {
        if (!wx) r.bx = a.beta[0][q.om + pk];
        if (!wy) r.by = a.beta[1][q.om + pk];
      }
      if (q.own && (g.per[2] || (k > 0 && k < g.n[2]))) r.bz = a.beta[2][q.o + pk];
      if (q.own && k > k0) r.f = a.f[q.o + st2 * (k - 1)];
    }
    return r;
  };
  double pp = 0.0, part = 0.0, acc = 0.0;
  unsigned long long mx = 0ull;
  if (q.own) pp = a.p[q.o + plane(k0 - 1)];
  Raw v = load(k0);
  for (int k = k0; k <= k1; ++k) {
    A[t] = v.p;
    __syncthreads();
    const Raw nx = load(k + 1);   // in flight over this plane's work
    double fx = 0.0, fy = 0.0;
    if (mid && k < k1) {
      fx = v.bx * (v.p - A[t - 1]);
      fy = v.by * (v.p - A[t - w]);
      E[0][t] = fx;
      E[1][t] = fy;
    }
    __syncthreads();
    if (q.own) {
      const double dz = v.p - pp;
      if (k > k0) {
        const int F = q.o + st2 * (k - 1);
        const double r = fma(-a.ih2, fma(v.bz, dz, part), v.f);
        a.r32[F] = narrow32(r);
        a.e32[F] = 0.f;
        acc = fma(r, r, acc);
        mx = op_umax(mx, (unsigned long long)__double_as_longlong(r) & 0x7fffffffffffffffull);
      }
      if (k < k1) part = fma(-v.bz, dz, (E[0][t + 1] - fx) + (E[1][t + w] - fy));
    }
    pp = v.p;
    v = nx;
  }
  if (a.partial) {
    acc = op_block_sum(acc, sh);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = op_umax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((t & 31) == 0) shm[t >> 5] = mx;
    __syncthreads();
    if (t == 0) {
      for (int k = 1; k < kOpThreads / 32; ++k) mx = op_umax(mx, shm[k]);
      const double m = __longlong_as_double((long long)mx);
      const int nb = B.gx * B.gy * B.gz;
      a.partial[B.linear()] = acc;
      a.partial[nb + B.linear()] = m <= CUDART_INF ? m : CUDART_INF;
    }
    __syncthreads();
  }
}

template <bool FCG>
__global__ void __launch_bounds__(kOpThreads, 2)
    k_v_op(const __grid_constant__ Geo g, const __grid_constant__ OpShape S,
           const __grid_constant__ VOpArgs a) {
  v_op_body<FCG>(own_blk(), g, S, a);
}

__global__ void __launch_bounds__(kOpThreads, 2)
    k_p_op(const __grid_constant__ Geo g, const __grid_constant__ OpShape S,
           const __grid_constant__ POpArgs a) {
  p_op_body(own_blk(), g, S, a);
}

// The batched forms stage the member's geometry and pointers in shared
// memory: read there at each use, they cost no registers. Their items name a
// block by (tile along x, tile along y, chunk), each within 16 bits (op_grid3):
// the single launch's (tile, chunk), in the same order.
__device__ __forceinline__ Blk op_blk(const Blk& B) {
  return Blk{B.x + B.gx * B.y, B.z, 0, B.gx * B.gy, B.gz, 1};
}
template <bool FCG>
__global__ void __launch_bounds__(kOpThreads, 2) kb_v_op(BArgs A, int with_partial, int with_r64) {
  __shared__ Geo g;
  __shared__ OpShape S;
  __shared__ VOpArgs a;
  for_items(A, [&](const BMember& M, const Blk& B) {
    if (threadIdx.x == 0) {
      g = M.g[0];
      S = M.op;
      a.ir = M.ir[0];
      a.muc = M.d[0].muc;
      a.partial = with_partial ? M.sc.partial : nullptr;
      for (int d = 0; d < 3; ++d) {
        a.z[d] = M.f[0].u[d];
        a.u[d] = M.d[0].u[d];
        a.mue[d] = M.d[0].mue[d];
        a.m[d] = M.d[0].m[d];
        a.q[d] = FCG ? M.cg_q[d] : M.d[0].uf[d];
        a.w[d] = FCG ? M.d[0].u2[d] : (with_r64 ? M.d[0].ur[d] : nullptr);
        a.r32[d] = M.f[0].uf[d];
        a.e32[d] = M.f[0].u[d];
      }
    }
    __syncthreads();
    v_op_body<FCG>(op_blk(B), g, S, a);
  });
}

__global__ void __launch_bounds__(kOpThreads, 2) kb_p_op(BArgs A, int with_partial) {
  __shared__ Geo g;
  __shared__ OpShape S;
  __shared__ POpArgs a;
  for_items(A, [&](const BMember& M, const Blk& B) {
    if (threadIdx.x == 0) {
      g = M.g[0];
      S = M.op;
      a.ih2 = M.ih2[0];
      a.p = M.d[0].p;
      a.f = M.d[0].pf;
      for (int d = 0; d < 3; ++d) a.beta[d] = M.d[0].beta[d];
      a.r32 = M.f[0].pf;
      a.e32 = M.f[0].p;
      a.partial = with_partial ? M.sc.partial : nullptr;
    }
    __syncthreads();
    p_op_body(op_blk(B), g, S, a);
  });
}

}  // namespace

// Tile and chunk of a grid: the shape with the least FP64 work on the busiest
// of 152 SMs, two blocks resident on each, with (TX + 2)(TY + 2) lanes at
// most kOpThreads. A plane of a block issues 42 FP64 operations for every warp
// that holds lanes of the tile's own rows, 2 and 8 for the warps of the lower
// and upper halo row alone; a chunk costs one partial plane (about 0.5) more
// than it holds. A member's shape depends on its grid alone, so its partial
// sums are the same in a batch.
OpShape op_shape(const Geo& g) {
  OpShape best{};
  double bc = 1e300;
  for (int nx = 1; nx <= g.n[0]; ++nx) {
    const int TX = (g.n[0] + nx - 1) / nx, w = TX + 2;
    if (3 * w > kOpThreads) continue;
    if (TX < 16 && nx > 1) break;
    for (int TY = 1; TY <= g.n[1] && w * (TY + 2) <= kOpThreads; ++TY) {
      const int ny = (g.n[1] + TY - 1) / TY;
      if ((g.n[1] + ny - 1) / ny != TY) continue;
      const int lo = w / 32, hi = ((TY + 1) * w + 31) / 32, all = ((TY + 2) * w + 31) / 32;
      const double plane = 42.0 * (hi - lo) + 2.0 * lo + 8.0 * (all - hi) + 4.0;
      for (int KC = 2; KC <= 128; ++KC) {
        const int nc = (g.n[2] + KC - 1) / KC;
        const long long blocks = (long long)nx * ny * nc;
        const long long waves = (blocks + 303) / 304;
        const double load = blocks <= 152 ? 1.3 : 2.0 * (double)waves;
        const double c = load * (KC + 0.5) * plane;
        if (c < bc) {
          bc = c;
          best = OpShape{TX, TY, KC, nx, ny, nc};
        }
        if (KC >= g.n[2]) break;
      }
    }
  }
  return best;
}

int op_blocks(const OpShape& S) { return S.nx * S.ny * S.nc; }
dim3 op_grid3(const OpShape& S) { return dim3(S.nx, S.ny, S.nc); }

void launch_v_op(bool fcg, const Geo& g, const OpShape& S, const VOpArgs& a, cudaStream_t s) {
  const dim3 grid(S.nx * S.ny, S.nc);
  if (fcg) k_v_op<true><<<grid, kOpThreads, 0, s>>>(g, S, a);
  else k_v_op<false><<<grid, kOpThreads, 0, s>>>(g, S, a);
}

void launch_p_op(const Geo& g, const OpShape& S, const POpArgs& a, cudaStream_t s) {
  k_p_op<<<dim3(S.nx * S.ny, S.nc), kOpThreads, 0, s>>>(g, S, a);
}

void launch_b_v_residual_mixed(const BArgs& A, bool partial, bool r64, int grid, cudaStream_t s) {
  if (A.n > 0) kb_v_op<false><<<grid, kOpThreads, 0, s>>>(A, partial ? 1 : 0, r64 ? 1 : 0);
}
void launch_b_fcg_apply(const BArgs& A, int grid, cudaStream_t s) {
  if (A.n > 0) kb_v_op<true><<<grid, kOpThreads, 0, s>>>(A, 1, 0);
}
void launch_b_p_residual_mixed(const BArgs& A, bool partial, int grid, cudaStream_t s) {
  if (A.n > 0) kb_p_op<<<grid, kOpThreads, 0, s>>>(A, partial ? 1 : 0);
}

}  // namespace bf
