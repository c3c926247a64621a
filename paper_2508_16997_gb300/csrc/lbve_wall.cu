// lbve_wall.cu -- the edge pass before every step of instances with a solid
// mask or open columns (hand-written CUDA, sm_103a): one launch completes the
// wall nodes next to solid nodes and the two open columns.
//
// The pass is a few hundred to a few thousand nodes at the head of the step's
// serial chain (edge pass, then the tiles that read it), so its latency counts
// and not its traffic.  Each node is carried by four warps, one lattice each
// (they meet once, when the hydrodynamic warp publishes u), every operand is
// loaded before the first use without branches on the link pattern, and the
// interpolation weights come precomputed from the host: a float64 instruction
// costs a warp 64 cycles, and the weights took a float64 division per link.
// One thread per node and two launches took 16.8 + 8.8 us in float32 and 22.8 +
// 17.9 us in float64 (isolated, cold); this pass takes 7.0 and 8.8 us.
//
// Wall nodes (fluid nodes next to the mask).  For each wall link (x_b, i), i.e.
// x_b - e_i solid, the pass computes the population that arrives at x_b along
// e_i and stores it in the solid node's slot i, which is exactly where the step
// kernel's pull of x_b reads it.  So the fused step needs no wall logic for
// the mask: it pulls completed populations everywhere.
//   - Hydrodynamic lattice: linear interpolated bounce-back (Bouzidi,
//     Firdaouss & Lallemand 2001) at wall fraction q; q = 1/2 is half-way
//     bounce-back.  It stands in for the curved-wall scheme of Sec. 4.3.
//   - Conformation lattices: CNEBB (Sec. 3.3) with u_b from the completed
//     hydrodynamic populations; the closing rest population is written to
//     the node's own rest slot (only this node pulls it).
//   - Final step: the momentum-exchange force on the solid (eq_F_x) and the
//     CNEBB wall in/out amounts, float64, one record per wall node.
// Reads touch only fluid nodes' slots and writes only solid nodes' slots and
// the node's own rest slots (a warp writes a rest slot only of its own lattice,
// after the read by the same thread), so the threads never race.
//
// Open columns (Sec. 4.3 inlet/outlet).  The node's neighbour x_f (column 1 or
// nx - 2) is pulled and, on a wall row, completed (Zou-He, CNEBB) exactly as
// the step does; then every population of the open-column node follows by
// non-equilibrium extrapolation:
//   inlet:  f = f^eq(rho_f, u_in) - f^eq(rho_f, u_f) + f(x_f),
//           g = g^eq(A_in, u_in) - g^eq(phi_f, u_f) + g(x_f);
//   outlet: f = f^eq(1, u_f) - f^eq(rho_f, u_f) + f(x_f), g = g(x_f).
// The equilibrium differences are Hermite reconstructions of coefficient
// differences.  The result goes to the instance's colbuf, which the masked
// step reads in place of pulling these nodes.  No column node reads a slot that
// a wall node writes: the mask keeps three columns away from the ends, so its
// solid nodes lie beyond the pulls of x_f, and its wall nodes' rest slots too.
#include <cuda_runtime.h>

#include "lbve_internal.h"
#include "lbve_step.cuh"

namespace lbve {
namespace {

// D2Q9 velocities, opposites and weights (Sec. 3.1); with unrolled loops the
// index is a constant and these fold away.
__device__ __forceinline__ constexpr int ex(int i) {
  return (i == 1 || i == 5 || i == 8) ? 1 : ((i == 3 || i == 6 || i == 7) ? -1 : 0);
}
__device__ __forceinline__ constexpr int ey(int i) {
  return (i == 2 || i == 5 || i == 6) ? 1 : ((i == 4 || i == 7 || i == 8) ? -1 : 0);
}
__device__ __forceinline__ constexpr int opp(int i) {
  return i == 0 ? 0 : (i <= 4 ? (i + 1) % 4 + 1 : (i + 1) % 4 + 5);
}
__device__ __forceinline__ constexpr double wt(int i) {
  return i == 0 ? 4.0 / 9.0 : (i <= 4 ? 1.0 / 9.0 : 1.0 / 36.0);
}

constexpr int kEdgeNodes = 32, kEdgeThreads = 4 * kEdgeNodes;

template <typename R>
struct EdgeShared {  // flow of a block's nodes, from the hydrodynamic warp
  R rho[kEdgeNodes], ux[kEdgeNodes], uy[kEdgeNodes];
};

// CNEBB at a wall node, g: pulled populations, or (wall link i) the node's own
// post toward the wall.  Returns the sum (deviation) and completes g.
template <typename R>
__device__ __forceinline__ void cnebb_links(R g[9], R delta, R ux, R uy, int umask) {
  // phi_b = known pulled populations + own posts toward the wall
  R dphi = R(0);
#pragma unroll
  for (int i = 0; i < 9; ++i) dphi += g[i];
  const R phib = delta + dphi;
  // g_i = g_ibar + g^eq_i - g^eq_ibar = g_ibar + 6 w_i phi_b (e_i . u_b); the
  // opposite of a wall link is never one
  if constexpr (std::is_same<R, double>::value) {
    // the same with the products of opposite and diagonal links shared
    const double a = (2.0 / 3.0) * phib, b = (1.0 / 6.0) * phib;
    const double x = a * ux, y = a * uy, s = b * (ux + uy), d = b * (ux - uy);
    const double t[9] = {0.0, x, y, -x, -y, s, -d, -s, d};
#pragma unroll
    for (int i = 1; i < 9; ++i)
      if ((umask >> i) & 1) g[i] = g[opp(i)] + t[i];
  } else {
#pragma unroll
    for (int i = 1; i < 9; ++i)
      if ((umask >> i) & 1)
        g[i] = g[opp(i)] + (R)(6.0 * wt(i)) * phib * ((R)ex(i) * ux + (R)ey(i) * uy);
  }
  R rest = R(0);
#pragma unroll
  for (int i = 1; i < 9; ++i) rest += g[i];
  g[0] = dphi - rest;
}

// Wall node t, lattice `role` (0 hydrodynamic, 1 + l conformation l).
template <typename R, bool FINAL>
__device__ __forceinline__ void wall_node(const InstDev* __restrict__ insts,
                                          const WallDev* __restrict__ walls, int n, int t,
                                          int role, int lane, int parity,
                                          double* __restrict__ rec, EdgeShared<R>& sh) {
  const int4 head = t < n ? *reinterpret_cast<const int4*>(walls + t) : make_int4(-1, 0, 0, 0);
  const bool valid = head.x >= 0;
  const InstDev& D = insts[valid ? head.x : 0];
  const int k = head.y, umask = head.z, fmask = head.w;
  const int nx = D.nx, ny = D.ny, S = D.stride;
  const bool py = D.periodic_y != 0;
  R* __restrict__ p = (R*)D.pop[parity] + (size_t)(role == 0 ? 0 : 9 * role) * S;
  // node k + s e_i; mask nodes lie at least three rows from a flat wall, so
  // no neighbour leaves a walled domain
  int nb_m[9];
  R d[9];
  if (valid) {
    const int x = k % nx, y = k / nx;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      int xm = x - ex(i), ym = y - ey(i);
      xm = xm < 0 ? xm + nx : (xm >= nx ? xm - nx : xm);
      if (py) ym = ym < 0 ? ym + ny : (ym >= ny ? ym - ny : ym);
      nb_m[i] = ym * nx + xm;
    }
    // pulled population, or (wall link) the node's own post toward the wall
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const bool wall = i != 0 && ((umask >> i) & 1);
      d[i] = p[(size_t)(wall ? opp(i) : i) * S + (wall ? k : nb_m[i])];
    }
  }
  if (role == 0 && valid) {
    const WallDev& W = walls[t];
    const R Fx = D.force_field ? ((const R*)D.force)[k] : coef<R>(D, kCoefFx);
    const R Fy = D.force_field ? ((const R*)D.force)[S + k] : coef<R>(D, kCoefFy);
    // second interpolation operand: the next fluid node's post toward the wall
    // (q < 1/2; the own one where there is none) or the own post along e_i
    R a2[9], wa[9], wb[9];
#pragma unroll
    for (int i = 1; i < 9; ++i) {
      a2[i] = wa[i] = wb[i] = R(0);
      if ((umask >> i) & 1) {
        const bool below = (fmask >> (16 + i)) & 1;
        const int nb = nb_m[opp(i)];  // node k + e_i
        a2[i] = p[(size_t)(below ? opp(i) : i) * S + (below && ((fmask >> i) & 1) ? nb : k)];
        wa[i] = (R)W.a[i - 1];
        wb[i] = (R)W.b[i - 1];
      }
    }
    double fdx = 0.0, fdy = 0.0;
#pragma unroll
    for (int i = 1; i < 9; ++i) {
      if (!((umask >> i) & 1)) continue;
      const R fb = d[i];  // own post-collision toward the wall
      const R v = wa[i] * fb + wb[i] * a2[i];
      p[(size_t)i * S + nb_m[i]] = v;
      d[i] = v;
      if (FINAL) {
        // eq_F_x: e_ib (f^dagger_ib + f_i) over the links to the wall
        const double sum = 2.0 * wt(i) + (double)fb + (double)v;
        fdx -= ex(i) * sum;
        fdy -= ey(i) * sum;
      }
    }
    Flow<R> f;
    f.pull(d, Fx, Fy);
    sh.ux[lane] = f.ux;
    sh.uy[lane] = f.uy;
    if (FINAL) {
      double* r = rec + (size_t)t * kWallRec;
      r[0] = fdx;
      r[1] = fdy;
    }
  }
  __syncthreads();
  if (role > 0 && valid) {
    const int l = role - 1;
    const R delta = (l == 1) ? R(0) : R(1);
    double in = 0.0, out = 0.0;
    if (FINAL) {
#pragma unroll
      for (int i = 1; i < 9; ++i)
        if ((umask >> i) & 1) out += wt(i) * (double)delta + (double)d[i];
    }
    const R g0_old = d[0];
    cnebb_links<R>(d, delta, sh.ux[lane], sh.uy[lane], umask);
#pragma unroll
    for (int i = 1; i < 9; ++i)
      if ((umask >> i) & 1) {
        p[(size_t)i * S + nb_m[i]] = d[i];
        if (FINAL) in += wt(i) * (double)delta + (double)d[i];
      }
    p[k] = d[0];
    if (FINAL) {
      double* r = rec + (size_t)t * kWallRec;
      r[2 + l] = in + ((double)d[0] - (double)g0_old);
      r[5 + l] = out;
    }
  }
}

// Open-column node t, lattice `role`.
template <typename R>
__device__ __forceinline__ void column_node(const InstDev* __restrict__ insts,
                                            const ColTask* __restrict__ tasks, int n, int t,
                                            int role, int lane, int parity, EdgeShared<R>& sh) {
  const int4 head = t < n ? *reinterpret_cast<const int4*>(tasks + t) : make_int4(-1, 0, 0, 0);
  const bool valid = head.x >= 0;
  const InstDev& D = insts[valid ? head.x : 0];
  const int nx = D.nx, ny = D.ny, S = D.stride, y = head.y, side = head.z;
  const bool py = D.periodic_y != 0;
  const int xf = side == 0 ? 1 : nx - 2;
  const int rc = y * nx, k = rc + xf;
  const bool wb = valid && !py && y == 0, wt = valid && !py && y == ny - 1;
  const int l = role - 1;
  const R* __restrict__ src = (const R*)D.pop[parity] + (size_t)(role == 0 ? 0 : 9 * role) * S;
  R d[9], bx = R(0), by = R(0), phib = R(0), post[3] = {R(0), R(0), R(0)};
  if (valid) {
    int rm, rp;
    neighbour_rows(y, nx, ny, py, rm, rp);
    pull9<R>(src, S, rc, rm, rp, xf, xf - 1, xf + 1, d);
    if (side == 0) {
      const double* in = D.inlet;
      bx = (R)in[y];
      by = (R)in[ny + y];
      if (role > 0) phib = (R)in[(2 + l) * ny + y];
    }
    if (role > 0 && (wb || wt)) {
      // bottom wall: H = {4, 7, 8}; top wall: H = {2, 5, 6}
      post[0] = src[(wb ? 4 : 2) * S + k];
      post[1] = src[(wb ? 7 : 5) * S + k];
      post[2] = src[(wb ? 8 : 6) * S + k];
    }
  }
  if (role == 0 && valid) {
    const R Fx = D.force_field ? ((const R*)D.force)[k] : coef<R>(D, kCoefFx);
    const R Fy = D.force_field ? ((const R*)D.force)[S + k] : coef<R>(D, kCoefFy);
    if (wb || wt) zou_he<R>(d, Fx, Fy, wb);
    Flow<R> f;
    f.pull(d, Fx, Fy);
    sh.rho[lane] = f.rho;
    sh.ux[lane] = f.ux;
    sh.uy[lane] = f.uy;
  }
  __syncthreads();
  if (!valid) return;
  const R rho = sh.rho[lane], ux = sh.ux[lane], uy = sh.uy[lane];
  const int c = side * ny + y, ld = 2 * ny;
  R* __restrict__ cb = (R*)D.colbuf + (size_t)(role == 0 ? 0 : 9 * role) * ld + c;
  R e[9];
  if (role == 0) {
    if (side == 0) {
      reconstruct<R>(R(0), rho * (bx - ux), rho * (by - uy), rho * (bx * bx - ux * ux),
                     rho * (by * by - uy * uy), rho * (bx * by - ux * uy),
                     rho * (bx * bx * by - ux * ux * uy), rho * (bx * by * by - ux * uy * uy), e);
    } else {
      const R dr = R(1) - rho;  // density rho_0 = 1 at the outlet
      reconstruct<R>(dr, dr * ux, dr * uy, dr * ux * ux, dr * uy * uy, dr * ux * uy,
                     dr * ux * ux * uy, dr * ux * uy * uy, e);
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) cb[(size_t)i * ld] = d[i] + e[i];
    return;
  }
  if (wb || wt) {
    double win, wout;
    cnebb<R>(d, post[0], post[1], post[2], (l == 1) ? R(0) : R(1), ux, uy, wb, win, wout);
  }
  if (side == 0) {
    typename Arith<R>::Cde m;
    Arith<R>::moments(d, m);
    const R phif = ((l == 1) ? R(0) : R(1)) + m.dphi;
    reconstruct<R, false>(phib - phif, phib * bx - phif * ux, phib * by - phif * uy,
                          phib * bx * bx - phif * ux * ux, phib * by * by - phif * uy * uy,
                          phib * bx * by - phif * ux * uy, R(0), R(0), e);
#pragma unroll
    for (int i = 0; i < 9; ++i) cb[(size_t)i * ld] = d[i] + e[i];
  } else {
#pragma unroll
    for (int i = 0; i < 9; ++i) cb[(size_t)i * ld] = d[i];
  }
}

// The first wall_blocks blocks take the wall nodes, the rest the column nodes.
template <typename R, bool FINAL>
__global__ void __launch_bounds__(kEdgeThreads)
    edge_kernel(const InstDev* __restrict__ insts, const WallDev* __restrict__ walls, int n_walls,
                int wall_blocks, double* __restrict__ rec, const ColTask* __restrict__ tasks,
                int n_tasks, int parity) {
  __shared__ EdgeShared<R> sh;
  const int role = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if ((int)blockIdx.x < wall_blocks)
    wall_node<R, FINAL>(insts, walls, n_walls, blockIdx.x * kEdgeNodes + lane, role, lane, parity,
                        rec, sh);
  else
    column_node<R>(insts, tasks, n_tasks, (blockIdx.x - wall_blocks) * kEdgeNodes + lane, role,
                   lane, parity, sh);
}

template <typename R>
int launch_edges_t(const InstDev* d_insts, const WallDev* d_walls, double* d_rec, int n_walls,
                   const ColTask* d_tasks, int n_tasks, int parity, int flags, cudaStream_t st) {
  const int nw = (n_walls + kEdgeNodes - 1) / kEdgeNodes;
  const int nc = (n_tasks + kEdgeNodes - 1) / kEdgeNodes;
  if (nw + nc <= 0) return 0;
  if (flags & kFinal)
    edge_kernel<R, true><<<nw + nc, kEdgeThreads, 0, st>>>(d_insts, d_walls, n_walls, nw, d_rec,
                                                           d_tasks, n_tasks, parity);
  else
    edge_kernel<R, false><<<nw + nc, kEdgeThreads, 0, st>>>(d_insts, d_walls, n_walls, nw, d_rec,
                                                            d_tasks, n_tasks, parity);
  return cudaPeekAtLastError() == cudaSuccess ? 0 : -1;  // the caller reads and clears it
}

}  // namespace

int launch_edges(int prec, const InstDev* d_insts, const WallDev* d_walls, double* d_rec,
                 int n_walls, const ColTask* d_tasks, int n_tasks, int parity, int flags,
                 void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  if (prec == 0)
    return launch_edges_t<double>(d_insts, d_walls, d_rec, n_walls, d_tasks, n_tasks, parity,
                                  flags, st);
  return launch_edges_t<float>(d_insts, d_walls, d_rec, n_walls, d_tasks, n_tasks, parity, flags,
                               st);
}

}  // namespace lbve
