// lbve_step.cuh -- the fused coupled time step (hand-written CUDA, sm_103a).
//
// One CTA updates one tile of one instance.  Storage is structure-of-arrays,
// x fastest: 9 hydrodynamic planes then 3 x 9 conformation planes of
// post-collision populations, kept as deviations from the rest state
// (f_i - w_i, g^c_i - w_i delta_c), ping-pong between two buffers (pull
// scheme), plus 5 history planes (S_xx, S_xy, S_yy, ux, uy of the previous
// step) and an optional per-node body force.
//
// Per step, per node (paper Sec. 3):
//   pull-stream all 36 populations (eq_ev_f / eq_g0 left-hand sides);
//   complete wall rows: hydro wet-node bounce-back of the non-equilibrium part
//   (Zou-He, wall velocity 0), then CNEBB for each conformation lattice from
//   the node's own outgoing-to-wall post-collision slots (Sec. 3.3);
//   moments rho, u (eq_ev_f0), phi^c;
//   second-order finite differences of u, rho u_x^3, rho u_y^3 from a
//   one-node (two rows at walls) halo of moments held in shared memory;
//   Oldroyd-B stress (eq_kramer, eqb4) and source Phi_ab (Sec. 3.2);
//   TRT-RLB collisions of all four lattices, evaluated in Hermite moment
//   space: the regularised post-collision state is the projection onto
//   {1, H_a, H_ab, H_xxy, H_xyy} (the D2Q9 H_xxx, H_yyy vanish), so it is
//   rebuilt per direction from 8 (hydro) or 6 (conformation) coefficients.
//   This is algebraically identical to eq_ev_f / eq_g0 written per direction.
//
// Phase A computes rho, u on the tile plus halo into shared memory; phase B
// does the full update of the tile's own nodes.  Halo pulls hit L1/L2; each
// population is read from HBM once per step by the node that pulls it.
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

#include "lbve_df32.cuh"
#include "lbve_internal.h"
#include "lbve_linear.cuh"

#ifndef LBVE_FP32_MIN_BLOCKS
#define LBVE_FP32_MIN_BLOCKS 7
#endif

namespace lbve {

// Exact float -> double conversion by integer operations: GB300 converts
// float to double on its float64 pipe (64 cycles per warp instruction),
// integer operations issue every cycle.  Zero, subnormal, normal, infinite
// and NaN inputs (IEEE 754 binary32 -> binary64: exponent rebiased by
// 1023 - 127, fraction shifted by 29 bits; subnormals normalised).
__device__ __forceinline__ double f2d_exact(float f) {
  const uint32_t b = __float_as_uint(f);
  const uint64_t sign = (uint64_t)(b >> 31) << 63;
  const uint32_t e = (b >> 23) & 0xffu;
  const uint32_t m = b & 0x7fffffu;
  uint64_t r;
  if (e == 0xffu) {
    r = sign | 0x7ff0000000000000ull | ((uint64_t)m << 29);
  } else if (e != 0u) {
    r = sign | ((uint64_t)(e + 896u) << 52) | ((uint64_t)m << 29);
  } else if (m == 0u) {
    r = sign;
  } else {
    const int msb = 31 - __clz(m);  // 0..22: value 2^(msb - 149) (1 + fraction)
    r = sign | ((uint64_t)(msb + 874) << 52) | (((uint64_t)m << (52 - msb)) & 0xfffffffffffffull);
  }
  return __longlong_as_double((long long)r);
}
__device__ __forceinline__ double to_f64(float v) { return f2d_exact(v); }
__device__ __forceinline__ double to_f64(double v) { return v; }
__device__ __forceinline__ double to_f64(df32 v) { return f2d_exact(v.hi) + f2d_exact(v.lo); }

template <typename R>
struct HydroM {  // raw moments of the (deviation) populations
  R drho, jx, jy, pxx, pyy, pxy, qxxy, qxyy;
};
template <typename R>
struct CdeM {
  R dphi, jx, jy, pxx, pyy, pxy;
};

template <typename R>
__device__ __forceinline__ void hydro_moments(const R d[9], HydroM<R>& m) {
  const R s58 = (d[5] + d[6]) + (d[7] + d[8]);
  m.drho = ((d[0] + d[1]) + (d[2] + d[3])) + (d[4] + s58);
  m.jx = (d[1] - d[3]) + ((d[5] - d[6]) + (d[8] - d[7]));
  m.jy = (d[2] - d[4]) + ((d[5] + d[6]) - (d[7] + d[8]));
  m.pxx = (d[1] + d[3]) + s58;
  m.pyy = (d[2] + d[4]) + s58;
  m.pxy = (d[5] + d[7]) - (d[6] + d[8]);
  m.qxxy = (d[5] + d[6]) - (d[7] + d[8]);
  m.qxyy = (d[5] + d[8]) - (d[6] + d[7]);
}

template <typename R>
__device__ __forceinline__ void cde_moments(const R d[9], CdeM<R>& m) {
  const R s58 = (d[5] + d[6]) + (d[7] + d[8]);
  m.dphi = ((d[0] + d[1]) + (d[2] + d[3])) + (d[4] + s58);
  m.jx = (d[1] - d[3]) + ((d[5] - d[6]) + (d[8] - d[7]));
  m.jy = (d[2] - d[4]) + ((d[5] + d[6]) - (d[7] + d[8]));
  m.pxx = (d[1] + d[3]) + s58;
  m.pyy = (d[2] + d[4]) + s58;
  m.pxy = (d[5] + d[7]) - (d[6] + d[8]);
}

// Rebuild the nine (deviation) populations from Hermite coefficients:
//   d_i = w_i [ b0' + 3 e.b + 4.5 (H_xx bxx + 2 H_xy bxy + H_yy byy)
//               + 13.5 (H_xxy bxxy + H_xyy bxyy) ]
// with b0' the zeroth coefficient minus the rest value.
// Float32: the products with the weights are correctly rounded, w v =
// fmaf(v, w, v w_lo) with w + w_lo = 1/9 or 1/36 to 2^-48: multiplying by
// the rounded weights alone scales every moment the weights carry by
// sum_i fl(w_i) e_i e_i... = 1 + 7e-9 at every collision, a bias that the
// momentum (and the slowly relaxing conformation moments) accumulate over
// their relaxation times.  The rest population is taken as b0' minus the
// other eight, which equals its formula in exact arithmetic and keeps
// sum_i d_i = b0' up to unbiased rounding.  Float32 pairs keep the plain
// formula; float64 scales the coefficients by the weights and adds in fixed
// point (lattice_populations).
template <typename R>
__device__ __forceinline__ R wmul(R v, R w, R wlo) {
  if constexpr (sizeof(R) == 4)
    return fmaf(v, w, v * wlo);
  else
    return w * v;
}

// THIRD = false: without third-order coefficients (the conformation lattices).
// Float32 then adds the zero terms all the same: without them the compiler
// would contract the remaining products differently, and the roundings of
// float32 runs stay what they were.
template <typename R, bool THIRD = true>
__device__ __forceinline__ void reconstruct(R b0p, R bx, R by, R bxx, R byy, R bxy, R bxxy,
                                            R bxyy, R out[9]) {
  if constexpr (std::is_same<R, double>::value) {
    const double third = 1.0 / 3.0;
    lattice_populations<THIRD>(b0p * (1.0 / 9.0), bx * third, by * third, bxx * third, byy * third,
                               bxy, bxxy, bxyy, out);
  } else {
    const R w0 = R(4.0 / 9.0), w1 = R(1.0 / 9.0), w5 = R(1.0 / 36.0);
    // low parts of 1/9 and 1/36 below their float32 roundings
    constexpr float kW1lo = (float)(1.0 / 9.0 - (double)(float)(1.0 / 9.0));
    constexpr float kW5lo = (float)(1.0 / 36.0 - (double)(float)(1.0 / 36.0));
    const R w1lo = R(kW1lo), w5lo = R(kW5lo);
    const R s = bxx + byy;
    if constexpr (sizeof(R) == 8) out[0] = w0 * (b0p - lit<R>(1.5) * s);
    const R b13 = b0p + lit<R>(3.0) * bxx - lit<R>(1.5) * byy;
    R o13, o24, o57, o68;
    if constexpr (THIRD || sizeof(R) == 4) {
      o13 = lit<R>(3.0) * bx - lit<R>(4.5) * bxyy;
      o24 = lit<R>(3.0) * by - lit<R>(4.5) * bxxy;
      o57 = lit<R>(3.0) * (bx + by) + lit<R>(9.0) * (bxxy + bxyy);
      o68 = lit<R>(3.0) * (by - bx) + lit<R>(9.0) * (bxxy - bxyy);
    } else {
      o13 = lit<R>(3.0) * bx;
      o24 = lit<R>(3.0) * by;
      o57 = lit<R>(3.0) * (bx + by);
      o68 = lit<R>(3.0) * (by - bx);
    }
    out[1] = wmul<R>(b13 + o13, w1, w1lo);
    out[3] = wmul<R>(b13 - o13, w1, w1lo);
    const R b24 = b0p - lit<R>(1.5) * bxx + lit<R>(3.0) * byy;
    out[2] = wmul<R>(b24 + o24, w1, w1lo);
    out[4] = wmul<R>(b24 - o24, w1, w1lo);
    const R bd = b0p + lit<R>(3.0) * s;
    const R xy9 = lit<R>(9.0) * bxy;
    out[5] = wmul<R>((bd + xy9) + o57, w5, w5lo);
    out[7] = wmul<R>((bd + xy9) - o57, w5, w5lo);
    out[6] = wmul<R>((bd - xy9) + o68, w5, w5lo);
    out[8] = wmul<R>((bd - xy9) - o68, w5, w5lo);
    if constexpr (sizeof(R) == 4)
      out[0] = b0p - (((out[1] + out[3]) + (out[2] + out[4])) + ((out[5] + out[7]) + (out[6] + out[8])));
  }
}

// Pull the nine populations of one lattice arriving at (x, y): d_i(x) =
// post_i(x - e_i).  rm / rp are the row offsets of rows y-1 / y+1, or -1
// where that row is outside a walled domain (those directions stay unknown
// and are completed by the caller).
template <typename R>
__device__ __forceinline__ void pull9(const R* __restrict__ p, int S, int rc, int rm, int rp,
                                      int x, int xm, int xp, R d[9]) {
  d[0] = p[0 * S + rc + x];
  d[1] = p[1 * S + rc + xm];
  d[3] = p[3 * S + rc + xp];
  if (rm >= 0) {
    d[2] = p[2 * S + rm + x];
    d[5] = p[5 * S + rm + xm];
    d[6] = p[6 * S + rm + xp];
  } else {
    d[2] = d[5] = d[6] = R(0);
  }
  if (rp >= 0) {
    d[4] = p[4 * S + rp + x];
    d[7] = p[7 * S + rp + xp];
    d[8] = p[8 * S + rp + xm];
  } else {
    d[4] = d[7] = d[8] = R(0);
  }
}

// Hydrodynamic wet-node completion with zero wall velocity: sum e f = -F/2
// (so u = 0 through eq_ev_f0) and the wall-normal pair bounced back.  The
// paired weights are equal, so the formulas hold for deviations unchanged.
template <typename R>
__device__ __forceinline__ void zou_he(R d[9], R Fx, R Fy, bool bottom) {
  const R h = R(0.5) * (d[1] - d[3]);
  const R qx = R(0.25) * Fx, qy = R(0.25) * Fy;
  if (bottom) {
    d[2] = d[4];
    d[5] = d[7] - h - qx - qy;
    d[6] = d[8] + h + qx - qy;
  } else {
    d[4] = d[2];
    d[7] = d[5] + h + qx + qy;
    d[8] = d[6] - h - qx + qy;
  }
}

// CNEBB (Sec. 3.3) on deviations.  post_* are the node's own post-collision
// slots pointing toward the wall (H); the unknown directions U are their
// opposites.  phi_b = known incoming + sum_H post; unknown i gets
// g_i = g_ibar + (g^eq_i - g^eq_ibar) = g_ibar + 6 w_i phi_b (e_i . u_b);
// the rest population closes sum g = phi_b.  Returns the wall in/out amounts
// (full populations, float64).
template <typename R>
__device__ __forceinline__ void cnebb(R d[9], R post_a, R post_b, R post_c, R delta_c, R ubx,
                                      R uby, bool bottom, double& win, double& wout) {
  // bottom: H = {4, 7, 8}, U = {2, 5, 6};  top: H = {2, 5, 6}, U = {4, 7, 8}
  const R d0_old = d[0];
  R dphi;
  if (bottom) {
    dphi = ((d[0] + d[1]) + (d[3] + d[4])) + ((d[7] + d[8]) + ((post_a + post_b) + post_c));
  } else {
    dphi = ((d[0] + d[1]) + (d[3] + d[2])) + ((d[5] + d[6]) + ((post_a + post_b) + post_c));
  }
  const R phib = delta_c + dphi;
  const R a2 = R(6.0 / 9.0) * phib, a5 = R(6.0 / 36.0) * phib;
  if (bottom) {
    d[2] = d[4] + a2 * uby;
    d[5] = d[7] + a5 * (ubx + uby);
    d[6] = d[8] + a5 * (uby - ubx);
  } else {
    d[4] = d[2] - a2 * uby;
    d[7] = d[5] - a5 * (ubx + uby);
    d[8] = d[6] + a5 * (ubx - uby);
  }
  d[0] = dphi - (((d[1] + d[2]) + (d[3] + d[4])) + ((d[5] + d[6]) + (d[7] + d[8])));
  const double dc = to_f64(delta_c);
  wout = (to_f64(post_a) + to_f64(post_b) + to_f64(post_c)) + dc / 6.0;
  double added;
  if (bottom) added = to_f64(d[2]) + to_f64(d[5]) + to_f64(d[6]);
  else added = to_f64(d[4]) + to_f64(d[7]) + to_f64(d[8]);
  win = added + dc / 6.0 + (to_f64(d[0]) - to_f64(d0_old));
}

// One level of a transposed butterfly sum over a warp: each lane holds M
// partial sums; it keeps one half (the upper one when `up`), receives the
// partner's values of that half across lane distance o and adds them, so
// that after the levels 16, 8, 4, 2 (and a last pairwise sum across 1) lanes
// 2s and 2s + 1 hold the warp's total of value s, for 16 values with 16
// additions per lane instead of 5 per value.
template <int M>
__device__ __forceinline__ void fold_half(double* v, int o, bool up) {
#pragma unroll
  for (int j = 0; j < M / 2; ++j) {
    const double keep = up ? v[j + M / 2] : v[j];
    const double send = up ? v[j] : v[j + M / 2];
    v[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
  }
}

// Populations of one lattice at a node: pulled from the previous step
// (kModeStep) or the equilibrium of the staged initial fields (kModeInit).
template <typename R, int MODE>
struct PopSource;

template <typename R>
struct PopSource<R, kModeStep> {
  static __device__ __forceinline__ void hydro(const void* src, int S, int nx, int k, int rc,
                                               int rm, int rp, int x, int xm, int xp, R d[9]) {
    pull9<R>((const R*)src, S, rc, rm, rp, x, xm, xp, d);
  }
  static __device__ __forceinline__ void cde(const void* src, int l, int S, int nx, int k, int rc,
                                             int rm, int rp, int x, int xm, int xp, R d[9]) {
    pull9<R>((const R*)src + (size_t)(9 + 9 * l) * S, S, rc, rm, rp, x, xm, xp, d);
  }
};

template <typename R>
struct PopSource<R, kModeInit> {
  // staged fields: float64 [6][S] = rho, ux, uy, Axx, Axy, Ayy at node k
  static __device__ __forceinline__ void hydro(const void* src, int S, int nx, int k, int rc,
                                               int rm, int rp, int x, int xm, int xp, R d[9]) {
    const double* f = (const double*)src;
    const R r = (R)f[k], ux = (R)f[S + k], uy = (R)f[2 * S + k];
    // equilibrium (eq2): Hermite coefficients rho, rho u, rho uu, rho u_x^2 u_y, rho u_x u_y^2
    reconstruct<R>((R)(f[k] - 1.0), r * ux, r * uy, r * ux * ux, r * uy * uy, r * ux * uy,
                   r * ux * ux * uy, r * ux * uy * uy, d);
  }
  static __device__ __forceinline__ void cde(const void* src, int l, int S, int nx, int k, int rc,
                                             int rm, int rp, int x, int xm, int xp, R d[9]) {
    const double* f = (const double*)src;
    const R ux = (R)f[S + k], uy = (R)f[2 * S + k];
    const double A = f[(3 + l) * S + k];
    const R a = (R)A;
    const R ap = (R)(A - (l == 1 ? 0.0 : 1.0));
    // equilibrium (eq_geq): phi, phi u, phi uu
    reconstruct<R>(ap, a * ux, a * uy, a * ux * ux, a * uy * uy, a * ux * uy, R(0), R(0), d);
  }
};

// Row offsets of the rows y-1 and y+1 feeding the pull at row y (-1 outside
// a walled domain).
__device__ __forceinline__ void neighbour_rows(int y, int nx, int ny, bool py, int& rm, int& rp) {
  if (py) {
    rm = (y == 0 ? ny - 1 : y - 1) * nx;
    rp = (y == ny - 1 ? 0 : y + 1) * nx;
  } else {
    rm = y > 0 ? (y - 1) * nx : -1;
    rp = y < ny - 1 ? (y + 1) * nx : -1;
  }
}

template <typename R>
__device__ __forceinline__ R coef(const InstDev& D, int i);
template <>
__device__ __forceinline__ double coef<double>(const InstDev& D, int i) {
  return D.cd[i];
}
template <>
__device__ __forceinline__ float coef<float>(const InstDev& D, int i) {
  return D.cf[i];
}
template <>
__device__ __forceinline__ df32 coef<df32>(const InstDev& D, int i) {
  return df32(D.cf[i], D.cl[i]);
}

// Position of halo-ring slot q in the (TX+2) x (TY+2hy) region: hy rows
// above and hy rows below the tile (its TX columns), one column left and one
// right of it.  The region's four corner blocks are never computed: every
// difference stencil runs along a single axis, so no node reads them.
__device__ __forceinline__ void ring_slot(int q, int RW, int TY, int hy, int& lx, int& ly) {
  const int TX = RW - 2;
  if (q < hy * TX) {
    ly = q / TX;
    lx = 1 + q % TX;
  } else if ((q -= hy * TX) < hy * TX) {
    ly = hy + TY + q / TX;
    lx = 1 + q % TX;
  } else if ((q -= hy * TX) < TY) {
    lx = 0;
    ly = hy + q;
  } else {
    lx = RW - 1;
    ly = hy + q - TY;
  }
}

// Global node of region slot (lx, ly); false if it lies outside a walled domain.
__device__ __forceinline__ bool region_node(int lx, int ly, int x0, int y0, int hy, int nx,
                                            int ny, bool py, int& gx, int& gy) {
  gx = x0 - 1 + lx;
  gx = ((gx % nx) + nx) % nx;
  gy = y0 - hy + ly;
  if (py) {
    gy = ((gy % ny) + ny) % ny;
    return true;
  }
  return gy >= 0 && gy < ny;
}

// v wrapped into [0, n) when it lies less than one period outside it.
__device__ __forceinline__ int wrap_once(int v, int n) {
  return v < 0 ? v + n : (v >= n ? v - n : v);
}

// region_node for a kTileTX-wide tile of an instance with D.t32 set: its
// halo columns x0-1 .. x0+kTileTX and (periodic) rows y0-2 .. y0+TY+1 lie
// less than one period outside the domain (nx >= kTileTX; ny >= TY + 2 when
// periodic), so one conditional wrap replaces the modulo.
__device__ __forceinline__ bool region_node_once(int lx, int ly, int x0, int y0, int hy, int nx,
                                                 int ny, bool py, int& gx, int& gy) {
  gx = wrap_once(x0 - 1 + lx, nx);
  gy = y0 - hy + ly;
  if (py) {
    gy = wrap_once(gy, ny);
    return true;
  }
  return gy >= 0 && gy < ny;
}

// Conformation tensor and constitutive function F(A) of a node from its
// raw conformation deviations dphi_c (Sec. 2: eqb4 for Oldroyd-B, FENE-P,
// FENE-CR), F in deviation form F = f (A - I) + (f - a) I.
template <typename R, bool MASKED>
__device__ __forceinline__ void polymer_terms(const InstDev& D, R d0, R d1, R d2, R& Axx,
                                              R& Axy, R& Ayy, R& Fxx, R& Fxy, R& Fyy) {
  Axx = R(1) + d0;
  Axy = d1;
  Ayy = R(1) + d2;
  Fxx = d0;
  Fxy = d1;
  Fyy = d2;
  if (MASKED && D.model != 0) {  // other models run in the general variant only
    const R tr = Axx + Ayy;
    const R f = R(1) / (R(1) - tr * coef<R>(D, kCoefInvL2));
    const R a = D.model == 2 ? f : coef<R>(D, kCoefAfene);
    Fxx = f * d0 + (f - a);
    Fxy = f * d1;
    Fyy = f * d2 + (f - a);
  }
}

// a b + c with one rounding.  Written out in the float64 path, where a result
// must not depend on which product the compiler would contract (the CTA
// sizes and the one-lattice-per-warp kernel agree bit for bit).
__device__ __forceinline__ double mad(double a, double b, double c) { return fma(a, b, c); }

// 1 / v by one step of the cubically convergent iteration x (1 + e + e^2),
// e = 1 - v x (Householder's method), from the float32 approximate
// reciprocal: three float64 instructions where the division takes about nine.
// x is off by at most 2^-22 of its size (v truncated to 24 bits, the approximation
// within 2^-23), so the step leaves 2^-66 and the result is within 1/2 + 2^-12
// units of its last place (the division: 1/2; one of some 10^4 results
// differs from it, by one unit).  Outside [2^-100, 2^101) and for NaN it divides.
__device__ __forceinline__ double recip(double v) {
  const int hi = __double2hiint(v), lo = __double2loint(v);
  const unsigned e = ((unsigned)hi >> 20) & 0x7ffu;
  if (e - 923u > 200u) return 1.0 / v;
  // v rounded toward zero to float32, and its reciprocal back, by bit patterns
  const unsigned f = __funnelshift_l((unsigned)lo, (unsigned)(hi & 0x7fffffff) - (896u << 20), 3) |
                     ((unsigned)hi & 0x80000000u);
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(f)));
  const unsigned b = __float_as_uint(r);
  const double x = __hiloint2double(
      (int)((((b & 0x7fffffffu) >> 3) + (896u << 20)) | (b & 0x80000000u)), (int)(b << 29));
  const double t = fma(-v, x, 1.0);
  return fma(x, fma(t, t, t), x);
}

// Arithmetic of one node per storage precision: its moments, the differences
// of its neighbours' values, its source and its collisions up to the Hermite
// coefficients.  The general form (float32, float32 pairs) follows the paper's
// formulas; the float64 one below counts float64 instructions.
template <typename R>
struct Flow {  // rho, u of one node (eq_ev_f0)
  R rho, ux, uy;
  __device__ __forceinline__ void set(const HydroM<R>& m, R Fx, R Fy) {
    rho = R(1) + m.drho;
    const R irho = R(1) / rho;
    ux = (m.jx + lit<R>(0.5) * Fx) * irho;
    uy = (m.jy + lit<R>(0.5) * Fy) * irho;
  }
  __device__ __forceinline__ void pull(const R d[9], R Fx, R Fy) {
    HydroM<R> m;
    hydro_moments<R>(d, m);
    set(m, Fx, Fy);
  }
  __device__ __forceinline__ void rest() {
    rho = R(1);
    ux = uy = R(0);
  }
};

// The halo region of a tile in shared memory.
template <typename R, int N>
struct Region {
  R rho[N], ux[N], uy[N];
  __device__ __forceinline__ void put(int r, const Flow<R>& f) {
    rho[r] = f.rho;
    ux[r] = f.ux;
    uy[r] = f.uy;
  }
};

// G** = d_g u_b (G01 = dx uy), dP: d_x (rho ux^3), d_y (rho uy^3), dR: grad rho
// (eq_p_G form only).
template <typename R>
struct Grad {
  R G00, G01, G10, G11, dPx, dPy, dRx, dRy;
};

template <typename R>
struct Arith {
  using Hydro = HydroM<R>;
  using Cde = CdeM<R>;
  static __device__ __forceinline__ void moments(const R d[9], Hydro& m) { hydro_moments<R>(d, m); }
  static __device__ __forceinline__ void moments(const R d[9], Cde& m) { cde_moments<R>(d, m); }

  // Second-order differences at region slot ri (central inside, one-sided in
  // y on wall rows: rows y-2..y+2, only those a wall row needs are read).
  template <int N>
  static __device__ __forceinline__ void gradients(const Region<R, N>& Q, int ri, int RW, bool wb,
                                                   bool wt, const Flow<R>& f, bool density,
                                                   Grad<R>& G) {
    const auto half = lit<R>(0.5);
    G.G00 = half * (Q.ux[ri + 1] - Q.ux[ri - 1]);
    G.G01 = half * (Q.uy[ri + 1] - Q.uy[ri - 1]);
    const R cxp = Q.rho[ri + 1] * Q.ux[ri + 1] * Q.ux[ri + 1] * Q.ux[ri + 1];
    const R cxm = Q.rho[ri - 1] * Q.ux[ri - 1] * Q.ux[ri - 1] * Q.ux[ri - 1];
    G.dPx = half * (cxp - cxm);
    G.dRx = density ? half * (Q.rho[ri + 1] - Q.rho[ri - 1]) : R(0);
    const int a = wb ? ri : (wt ? ri - 2 * RW : ri), b = wb ? ri : (wt ? ri - RW : ri - RW);
    const int c = wb ? ri + RW : (wt ? ri : ri + RW), e = wb ? ri + 2 * RW : ri;
    const R r0 = f.rho, ux0 = f.ux, uy0 = f.uy;
    const R rm2 = Q.rho[a], uxm2 = Q.ux[a], uym2 = Q.uy[a];
    const R rm1 = Q.rho[b], uxm1 = Q.ux[b], uym1 = Q.uy[b];
    const R rp1 = Q.rho[c], uxp1 = Q.ux[c], uyp1 = Q.uy[c];
    const R rp2 = Q.rho[e], uxp2 = Q.ux[e], uyp2 = Q.uy[e];
    G.dRy = R(0);
    if (wb) {
      G.G10 = half * (lit<R>(-3) * ux0 + lit<R>(4) * uxp1 - uxp2);
      G.G11 = half * (lit<R>(-3) * uy0 + lit<R>(4) * uyp1 - uyp2);
      G.dPy = half * (lit<R>(-3) * (r0 * uy0 * uy0 * uy0) + lit<R>(4) * (rp1 * uyp1 * uyp1 * uyp1) -
                      rp2 * uyp2 * uyp2 * uyp2);
      if (density) G.dRy = half * (lit<R>(-3) * r0 + lit<R>(4) * rp1 - rp2);
    } else if (wt) {
      G.G10 = half * (lit<R>(3) * ux0 - lit<R>(4) * uxm1 + uxm2);
      G.G11 = half * (lit<R>(3) * uy0 - lit<R>(4) * uym1 + uym2);
      G.dPy = half * (lit<R>(3) * (r0 * uy0 * uy0 * uy0) - lit<R>(4) * (rm1 * uym1 * uym1 * uym1) +
                      rm2 * uym2 * uym2 * uym2);
      if (density) G.dRy = half * (lit<R>(3) * r0 - lit<R>(4) * rm1 + rm2);
    } else {
      G.G10 = half * (uxp1 - uxm1);
      G.G11 = half * (uyp1 - uym1);
      G.dPy = half * (rp1 * uyp1 * uyp1 * uyp1 - rm1 * uym1 * uym1 * uym1);
      if (density) G.dRy = half * (rp1 - rm1);
    }
  }

  // Zero differences along an axis (0: x, 1: y) between two solid nodes.
  static __device__ __forceinline__ void blocked(int axis, Grad<R>& G) {
    if (axis == 0) G.G00 = G.G01 = G.dPx = G.dRx = R(0);
    else G.G10 = G.G11 = G.dPy = G.dRy = R(0);
  }

  // One-sided differences along one axis next to the solid mask (same rule as
  // the central and wall-row differences: second order on the fluid side when
  // two fluid nodes lie there, else first order):
  //   t:     +1 toward +axis, -1 toward -axis (the fluid side)
  //   f:     the node; i1: region slot of its fluid neighbour at +t
  //   has2:  whether the node at +2t is fluid; w: its values
  template <int N>
  static __device__ __forceinline__ void one_sided(int axis, int t, const Region<R, N>& Q, int ri,
                                                   int i1, const Flow<R>& f, bool has2,
                                                   const Flow<R>& w, Grad<R>& G) {
    const R r0 = f.rho, ux0 = f.ux, uy0 = f.uy;
    const R r1 = Q.rho[i1], ux1 = Q.ux[i1], uy1 = Q.uy[i1];
    const R r2 = w.rho, u2x = w.ux, u2y = w.uy;
    const R v0 = axis == 0 ? ux0 : uy0, v1 = axis == 0 ? ux1 : uy1, v2 = axis == 0 ? u2x : u2y;
    const R c0 = r0 * v0 * v0 * v0, c1 = r1 * v1 * v1 * v1, c2 = r2 * v2 * v2 * v2;
    const R ts = (R)t;
    R dux, duy, dcube, drho;
    if (has2) {
      const R h = lit<R>(0.5) * ts;
      dux = h * (lit<R>(-3) * ux0 + lit<R>(4) * ux1 - u2x);
      duy = h * (lit<R>(-3) * uy0 + lit<R>(4) * uy1 - u2y);
      dcube = h * (lit<R>(-3) * c0 + lit<R>(4) * c1 - c2);
      drho = h * (lit<R>(-3) * r0 + lit<R>(4) * r1 - r2);
    } else {
      dux = ts * (ux1 - ux0);
      duy = ts * (uy1 - uy0);
      dcube = ts * (c1 - c0);
      drho = ts * (r1 - r0);
    }
    if (axis == 0) {
      G.G00 = dux;
      G.G01 = duy;
      G.dPx = dcube;
      G.dRx = drho;
    } else {
      G.G10 = dux;
      G.G11 = duy;
      G.dPy = dcube;
      G.dRy = drho;
    }
  }

  // Component l (xx, xy, yy) of the source Phi_ab of the conformation
  // equation (Sec. 3.2).
  static __device__ __forceinline__ R source(int l, const InstDev& D, R Axx, R Axy, R Ayy, R Fxx,
                                             R Fxy, R Fyy, const Grad<R>& G) {
    const R il = coef<R>(D, kCoefInvLam);
    const R G00 = G.G00, G01 = G.G01, G10 = G.G10, G11 = G.G11;
    const R div = G00 + G11;
    if (l == 0) return -Fxx * il + lit<R>(2) * (Axx * G00 + Axy * G10) + Axx * div;
    if (l == 1) return -Fxy * il + (Axx * G01 + Axy * G11) + (Axy * G00 + Ayy * G10) + Axy * div;
    return -Fyy * il + lit<R>(2) * (Axy * G01 + Ayy * G11) + Ayy * div;
  }

  // Hydrodynamic TRT-RLB collision (eq_ev_f, eq4, eq5, eq6, F_i): the Hermite
  // coefficients b0' (minus the rest value), b_x, b_y, b_xx, b_yy, b_xy,
  // b_xxy, b_xyy of the post-collision populations.
  static __device__ __forceinline__ void hydro_coefs(const InstDev& D, const Hydro& hm,
                                                     const Flow<R>& f, const Grad<R>& G, R Fxx,
                                                     R Fxy, R Fyy, R Fx, R Fy, R b[8]) {
    const R rho = f.rho, ux = f.ux, uy = f.uy;
    const R mpl = coef<R>(D, kCoefMupLam);
    const R txx = mpl * Fxx, txy = mpl * Fxy, tyy = mpl * Fyy;  // polymer stress (eq_kramer)
    const R cs2 = R(1.0 / 3.0);
    const R c1 = coef<R>(D, kCoefCs1), c2 = coef<R>(D, kCoefCs2);
    const R h1 = coef<R>(D, kCoefHs1), w1 = coef<R>(D, kCoefWs1);
    const R ruxx = rho * ux * ux, ruyy = rho * uy * uy, ruxy = rho * ux * uy;
    const R ruxxy = ruxx * uy, ruxyy = ruxy * uy;
    const R nxx = hm.pxx - cs2 * hm.drho - ruxx;   // A_xx^neq
    const R nyy = hm.pyy - cs2 * hm.drho - ruyy;   // A_yy^neq
    const R nxy = hm.pxy - ruxy;                   // A_xy^neq
    const R nxxy = hm.qxxy - cs2 * hm.jy - ruxxy;  // A_xxy^neq
    const R nxyy = hm.qxyy - cs2 * hm.jx - ruxyy;  // A_xyy^neq
    b[0] = hm.drho;
    b[1] = hm.jx + Fx;  // rho u + (1-1/tau)A_a + F-term
    b[2] = hm.jy + Fy;
    b[3] = ruxx + c1 * nxx - h1 * G.dPx - w1 * txx;
    b[4] = ruyy + c1 * nyy - h1 * G.dPy - w1 * tyy;
    b[5] = ruxy + c1 * nxy - w1 * txy;
    b[6] = ruxxy + c2 * nxxy;
    b[7] = ruxyy + c2 * nxyy;
  }

  // Conformation TRT-RLB collision of lattice l (eq_g0 with G~_i, F~_i and its
  // backward time difference): c0' (minus the rest value), c_x, c_y, c_xx, c_yy,
  // c_xy.  sl, so: the source now and one step back.
  template <bool MASKED>
  static __device__ __forceinline__ void cde_coefs(const InstDev& D, int l, const Cde& m,
                                                   const Flow<R>& f, R sl, R so, R uxo, R uyo,
                                                   R Fx, R Fy, const Grad<R>& G, R c[6]) {
    const R rho = f.rho, ux = f.ux, uy = f.uy;
    const R cs2 = R(1.0 / 3.0);
    const R ep = coef<R>(D, kCoefEp1), c2 = coef<R>(D, kCoefCp2), h1 = coef<R>(D, kCoefHp1);
    const R irho = R(1) / rho;
    const R uxx = ux * ux, uyy = uy * uy, uxy = ux * uy;
    // the force G~_i sees: F (eq_p_G_1) or F - c_s^2 grad rho (eq_p_G)
    const bool gt = MASKED && D.gtilde;
    const R Gx = gt ? Fx - cs2 * G.dRx : Fx, Gy = gt ? Fy - cs2 * G.dRy : Fy;
    const R phi = (l == 1 ? R(0) : R(1)) + m.dphi;
    const R Bx = m.jx - phi * ux, By = m.jy - phi * uy;
    const R Bxx = m.pxx - cs2 * m.dphi - phi * uxx;
    const R Byy = m.pyy - cs2 * m.dphi - phi * uyy;
    const R Bxy = m.pxy - phi * uxy;
    // small source terms first, one rounding at the magnitude of phi
    c[0] = m.dphi + (lit<R>(1.5) * sl - lit<R>(0.5) * so);
    const R pr = phi * irho;
    // (1 - 1/tau_p1) B = -B + ep B, kept split so float32 keeps the tiny
    // difference tau_p1 - 1/2 accurately
    c[1] = (phi * ux - Bx) + ep * Bx + h1 * (pr * Gx + ux * sl) +
           lit<R>(0.5) * h1 * (ux * sl - uxo * so);
    c[2] = (phi * uy - By) + ep * By + h1 * (pr * Gy + uy * sl) +
           lit<R>(0.5) * h1 * (uy * sl - uyo * so);
    c[3] = phi * uxx + c2 * Bxx;
    c[4] = phi * uyy + c2 * Byy;
    c[5] = phi * uxy + c2 * Bxy;
  }

  static __device__ __forceinline__ void hydro_populations(const R b[8], R out[9]) {
    reconstruct<R>(b[0], b[1], b[2], b[3], b[4], b[5], b[6], b[7], out);
  }
  static __device__ __forceinline__ void cde_populations(const R c[6], R out[9]) {
    reconstruct<R, false>(c[0], c[1], c[2], c[3], c[4], c[5], R(0), R(0), out);
  }
};

// ---- float64 ------------------------------------------------------------------------
// 167 float64 instructions per node beside the fixed-point sums (ncu; 418 with the
// general form), 772 us against 1,654 on 512^2 x 8 under ncu, the pipe 74 % active.
// The same formulas with fewer float64 instructions: rho u is j + F/2;
// second-order terms off c_s^2 come from the sums as three times their value;
// differences and cubes are shared (cubes in the region instead of the
// density, differences as twice their value); the diagonal second-order
// terms carry the weight 1/3 with which lattice_populations takes them
// (folded into the coefficients kCoefN1, kCoefWd, kCoefP2).
template <>
struct Flow<double> {
  double rho, irho, hx, hy, ux, uy;  // (hx, hy) = rho u
  template <typename M>
  __device__ __forceinline__ void set(const M& m, double Fx, double Fy) {
    rho = 1.0 + m.drho;
    irho = recip(rho);
    hx = mad(0.5, Fx, m.jx);
    hy = mad(0.5, Fy, m.jy);
    ux = hx * irho;
    uy = hy * irho;
  }
  __device__ __forceinline__ void pull(const double d[9], double Fx, double Fy) {
    Moments<double> m;
    lattice_moments<false>(d, m);
    set(m, Fx, Fy);
  }
  // rho u_x^3 / 3, rho u_y^3 / 3
  __device__ __forceinline__ double cube_x() const { return hx * (1.0 / 3.0) * ux * ux; }
  __device__ __forceinline__ double cube_y() const { return hy * (1.0 / 3.0) * uy * uy; }
  __device__ __forceinline__ void rest() {
    rho = irho = 1.0;
    hx = hy = ux = uy = 0.0;
  }
};

template <int N>
struct Region<double, N> {
  double rho[N], ux[N], uy[N], cx[N], cy[N];  // rho: read in the eq_p_G form only
  __device__ __forceinline__ void put(int r, const Flow<double>& f) {
    rho[r] = f.rho;
    ux[r] = f.ux;
    uy[r] = f.uy;
    cx[r] = f.cube_x();
    cy[r] = f.cube_y();
  }
};

// All twice the differences; the cubes' in units of Flow::cube_x.
template <>
struct Grad<double> {
  double D00, D01, D10, D11, dcx, dcy, dRx, dRy;
};

template <>
struct Arith<double> {
  struct Hydro {
    double drho, jx, jy, nxx, nyy, pxy, nxxy, nxyy;
  };
  struct Cde {
    double dphi, jx, jy, nxx, nyy, pxy;
  };
  static __device__ __forceinline__ void moments(const double d[9], Hydro& m) {
    Moments<double> s;
    lattice_moments<true>(d, s);
    m = Hydro{s.drho, s.jx, s.jy, s.nxx, s.nyy, s.pxy, s.nxxy, s.nxyy};
  }
  static __device__ __forceinline__ void moments(const double d[9], Cde& m) {
    Moments<double> s;
    lattice_moments<false>(d, s);
    m = Cde{s.drho, s.jx, s.jy, s.nxx, s.nyy, s.pxy};
  }

  // Twice the one-sided difference of a quantity from its value and those one
  // and two nodes inward, for an inward direction of +1.
  static __device__ __forceinline__ double inward(double q0, double q1, double q2) {
    return mad(4.0, q1, mad(-3.0, q0, -q2));
  }
  static __device__ __forceinline__ double along_y(const double* q, int ri, int RW, bool wb,
                                                   bool wt) {
    if (wb) return inward(q[ri], q[ri + RW], q[ri + 2 * RW]);
    if (wt) return -inward(q[ri], q[ri - RW], q[ri - 2 * RW]);
    return q[ri + RW] - q[ri - RW];
  }
  template <int N>
  static __device__ __forceinline__ void gradients(const Region<double, N>& Q, int ri, int RW,
                                                   bool wb, bool wt, const Flow<double>& f,
                                                   bool density, Grad<double>& G) {
    G.D00 = Q.ux[ri + 1] - Q.ux[ri - 1];
    G.D01 = Q.uy[ri + 1] - Q.uy[ri - 1];
    G.D10 = along_y(Q.ux, ri, RW, wb, wt);
    G.D11 = along_y(Q.uy, ri, RW, wb, wt);
    G.dcx = Q.cx[ri + 1] - Q.cx[ri - 1];
    G.dcy = along_y(Q.cy, ri, RW, wb, wt);
    G.dRx = density ? Q.rho[ri + 1] - Q.rho[ri - 1] : 0.0;
    G.dRy = density ? along_y(Q.rho, ri, RW, wb, wt) : 0.0;
  }
  static __device__ __forceinline__ void blocked(int axis, Grad<double>& G) {
    if (axis == 0) G.D00 = G.D01 = G.dcx = G.dRx = 0.0;
    else G.D10 = G.D11 = G.dcy = G.dRy = 0.0;
  }
  static __device__ __forceinline__ double side(int t, double q0, double q1, bool has2, double q2) {
    const double ts = (double)t;
    return has2 ? ts * inward(q0, q1, q2) : 2.0 * ts * (q1 - q0);
  }
  template <int N>
  static __device__ __forceinline__ void one_sided(int axis, int t, const Region<double, N>& Q,
                                                   int ri, int i1, const Flow<double>& f,
                                                   bool has2, const Flow<double>& w,
                                                   Grad<double>& G) {
    const double dux = side(t, f.ux, Q.ux[i1], has2, w.ux);
    const double duy = side(t, f.uy, Q.uy[i1], has2, w.uy);
    const double drho = side(t, f.rho, Q.rho[i1], has2, w.rho);
    if (axis == 0) {
      G.D00 = dux;
      G.D01 = duy;
      G.dcx = side(t, Q.cx[ri], Q.cx[i1], has2, w.cube_x());
      G.dRx = drho;
    } else {
      G.D10 = dux;
      G.D11 = duy;
      G.dcy = side(t, Q.cy[ri], Q.cy[i1], has2, w.cube_y());
      G.dRy = drho;
    }
  }

  static __device__ __forceinline__ double source(int l, const InstDev& D, double Axx, double Axy,
                                                  double Ayy, double Fxx, double Fxy, double Fyy,
                                                  const Grad<double>& G) {
    const double il = D.cd[kCoefInvLam], div2 = G.D00 + G.D11;
    if (l == 0) return mad(-il, Fxx, mad(Axx, mad(0.5, div2, G.D00), Axy * G.D10));
    if (l == 2) return mad(-il, Fyy, mad(Ayy, mad(0.5, div2, G.D11), Axy * G.D01));
    return mad(-il, Fxy, mad(0.5, mad(Axx, G.D01, Ayy * G.D10), Axy * div2));
  }

  // b_xx and b_yy come divided by 3.
  static __device__ __forceinline__ void hydro_coefs(const InstDev& D, const Hydro& m,
                                                     const Flow<double>& f, const Grad<double>& G,
                                                     double Fxx, double Fxy, double Fyy, double Fx,
                                                     double Fy, double b[8]) {
    const double kn = D.cd[kCoefN1], kh = D.cd[kCoefHs2], kw = D.cd[kCoefWd], kt = D.cd[kCoefN2];
    const double rxx = f.hx * (1.0 / 3.0) * f.ux, ryy = f.hy * (1.0 / 3.0) * f.uy;
    const double rxy = f.hx * f.uy, rxxy = rxy * f.ux, rxyy = rxy * f.uy;
    b[0] = m.drho;
    b[1] = m.jx + Fx;
    b[2] = m.jy + Fy;
    b[3] = mad(-kw, Fxx, mad(-kh, G.dcx, mad(kn, mad(-9.0, rxx, m.nxx), rxx)));
    b[4] = mad(-kw, Fyy, mad(-kh, G.dcy, mad(kn, mad(-9.0, ryy, m.nyy), ryy)));
    b[5] = mad(-D.cd[kCoefWx], Fxy, mad(D.cd[kCoefCs1], m.pxy - rxy, rxy));
    b[6] = mad(kt, mad(-3.0, rxxy, m.nxxy), rxxy);
    b[7] = mad(kt, mad(-3.0, rxyy, m.nxyy), rxyy);
  }

  // c_xx and c_yy come divided by 3.
  template <bool MASKED>
  static __device__ __forceinline__ void cde_coefs(const InstDev& D, int l, const Cde& m,
                                                   const Flow<double>& f, double sl, double so,
                                                   double uxo, double uyo, double Fx, double Fy,
                                                   const Grad<double>& G, double c[6]) {
    const double ep = D.cd[kCoefEp1], h1 = D.cd[kCoefHp1], kn = D.cd[kCoefP2];
    const double ux = f.ux, uy = f.uy;
    const bool gt = MASKED && D.gtilde;
    const double Gx = gt ? mad(-1.0 / 6.0, G.dRx, Fx) : Fx;
    const double Gy = gt ? mad(-1.0 / 6.0, G.dRy, Fy) : Fy;
    const double phi = l == 1 ? m.dphi : 1.0 + m.dphi;
    const double Bx = mad(-phi, ux, m.jx), By = mad(-phi, uy, m.jy);
    const double s15 = 1.5 * sl, s05 = 0.5 * so;
    c[0] = m.dphi + (s15 - s05);
    const double pr = phi * f.irho;
    c[1] = mad(h1, mad(pr, Gx, mad(ux, s15, -(uxo * s05))), mad(ep, Bx, mad(phi, ux, -Bx)));
    c[2] = mad(h1, mad(pr, Gy, mad(uy, s15, -(uyo * s05))), mad(ep, By, mad(phi, uy, -By)));
    const double ph = phi * (1.0 / 3.0);
    const double pxx = ph * (ux * ux), pyy = ph * (uy * uy), pxy = phi * (ux * uy);
    c[3] = mad(kn, mad(-9.0, pxx, m.nxx), pxx);
    c[4] = mad(kn, mad(-9.0, pyy, m.nyy), pyy);
    c[5] = mad(D.cd[kCoefCp2], m.pxy - pxy, pxy);
  }

  static __device__ __forceinline__ void hydro_populations(const double b[8], double out[9]) {
    lattice_populations<true>(b[0] * (1.0 / 9.0), b[1] * (1.0 / 3.0), b[2] * (1.0 / 3.0), b[3],
                              b[4], b[5], b[6], b[7], out);
  }
  static __device__ __forceinline__ void cde_populations(const double c[6], double out[9]) {
    lattice_populations<false>(c[0] * (1.0 / 9.0), c[1] * (1.0 / 3.0), c[2] * (1.0 / 3.0), c[3],
                               c[4], c[5], 0.0, 0.0, out);
  }
};

// Flow of node (gx, gy) at the current time: pull (or equilibrium at init),
// hydro wall completion, moments.
template <typename R, int MODE>
__device__ __forceinline__ void node_flow(const void* src, const R* __restrict__ force,
                                          bool ffield, R Fx0, R Fy0, int S, int nx, int ny,
                                          bool py, int gx, int gy, Flow<R>& f) {
  const int k = gy * nx + gx;
  int rm, rp;
  neighbour_rows(gy, nx, ny, py, rm, rp);
  const int xm = gx == 0 ? nx - 1 : gx - 1, xp = gx == nx - 1 ? 0 : gx + 1;
  const R Fx = ffield ? force[k] : Fx0;
  const R Fy = ffield ? force[S + k] : Fy0;
  R d[9];
  PopSource<R, MODE>::hydro(src, S, nx, k, gy * nx, rm, rp, gx, xm, xp, d);
  if (MODE == kModeStep && !py && (gy == 0 || gy == ny - 1)) zou_he<R>(d, Fx, Fy, gy == 0);
  f.pull(d, Fx, Fy);
}

// The collisions with the store of the 9 post-collision populations.
template <typename R>
__device__ __forceinline__ void collide_hydro(const InstDev& D, int k, int S, R* __restrict__ dst,
                                              const typename Arith<R>::Hydro& m, const Flow<R>& f,
                                              const Grad<R>& G, R Fxx, R Fxy, R Fyy, R Fx, R Fy) {
  R b[8], out[9];
  Arith<R>::hydro_coefs(D, m, f, G, Fxx, Fxy, Fyy, Fx, Fy, b);
  Arith<R>::hydro_populations(b, out);
#pragma unroll
  for (int i = 0; i < 9; ++i) dst[(size_t)i * S + k] = out[i];
}

template <typename R, bool MASKED>
__device__ __forceinline__ void collide_cde(const InstDev& D, int k, int S, R* __restrict__ dst,
                                            int l, const typename Arith<R>::Cde& m,
                                            const Flow<R>& f, R sl, R so, R uxo, R uyo, R Fx,
                                            R Fy, const Grad<R>& G) {
  R c[6], out[9];
  Arith<R>::template cde_coefs<MASKED>(D, l, m, f, sl, so, uxo, uyo, Fx, Fy, G, c);
  Arith<R>::cde_populations(c, out);
  R* dl = dst + (size_t)(9 + 9 * l) * S;
#pragma unroll
  for (int i = 0; i < 9; ++i) dl[(size_t)i * S + k] = out[i];
}

// Final-step record of one node: its float64 fields and its contributions to
// the tile's partial record.  lattice -1 writes everything; 0 the
// hydrodynamic part (rho, u, momentum, residual), 1..3 conformation lattice
// lattice - 1 (A component, its sum; the wall balance is the caller's).  The
// sums of rho, A_xx and A_yy are kept as deviations from their rest value 1
// (added per tile from its node count) and the residual is scaled by 1/U_c
// per tile: GB300 issues a float64 instruction only every 64 cycles per
// warp, so the final step keeps them few.
// Type of the per-node contributions to a tile's partial record: float32
// instances keep float32 values (and exact float32 pairs) until the warp
// totals, float64 instances float64 values.
template <typename R>
using PartT = typename std::conditional<sizeof(R) == 4, float, double>::type;

// ux_prev, uy_prev: the velocity fields of the previous final step at node
// k, read by the caller before the collision (unused at init)
template <typename R, int MODE>
__device__ __forceinline__ void final_node(const InstDev& D, int k, int S, int lattice, R drho,
                                           R rho, R ux, R uy, const R* dphi, PartT<R> ux_prev,
                                           PartT<R> uy_prev, PartT<R>* part, PartT<R>* plo) {
  double* fl = D.fields;
  bool finite = true;
  if (lattice <= 0) {
    const double dr = to_f64(drho);
    const double vx = to_f64(ux), vy = to_f64(uy);
    fl[k] = 1.0 + dr;
    fl[S + k] = vx;
    fl[2 * S + k] = vy;
    if constexpr (sizeof(R) == 4) {
      // in float32: the previous fields are float32 values
      const float res =
          (MODE == kModeStep) ? fmaxf(fabsf(ux - ux_prev), fabsf(uy - uy_prev)) : 0.f;
      // rho u exactly, as a float32 pair (product and its rounding error)
      const float px = rho * ux, py = rho * uy;
      part[kSumRho] = drho;
      part[kSumJx] = px;
      part[kSumJy] = py;
      plo[kSumJx] = fmaf(rho, ux, -px);
      plo[kSumJy] = fmaf(rho, uy, -py);
      part[kResid] = res;
      finite = isfinite(drho) && isfinite(ux) && isfinite(uy);
    } else {
      const double res =
          (MODE == kModeStep) ? fmax(fabs(vx - ux_prev), fabs(vy - uy_prev)) : 0.0;
      part[kSumRho] = dr;
      part[kSumJx] = to_f64(rho) * vx;
      part[kSumJy] = to_f64(rho) * vy;
      part[kResid] = res;
      finite = isfinite(dr) && isfinite(vx) && isfinite(vy);
    }
  }
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    if (lattice >= 0 && lattice != 1 + l) continue;
    const double d = to_f64(dphi[l]);
    fl[(3 + l) * S + k] = l == 1 ? d : 1.0 + d;
    if constexpr (sizeof(R) == 4) {
      part[kSumPhi + l] = dphi[l];
      finite = finite && isfinite(dphi[l]);
    } else {
      part[kSumPhi + l] = d;
      finite = finite && isfinite(d);
    }
  }
  if (!finite) part[kResid] = 0;
  part[kNonFinite] = finite ? 0 : 1;
}

// Final step: start the previous velocity fields of node k (the residual's
// operands) on their way to L2 with the node's other loads; they are read
// just before the collision.  Read only after the collision, each warp
// stalled there for a full HBM round trip, which made the final step of a
// large batch take 1.8 times as long; loaded with the populations, they
// cost more registers than they save.
__device__ __forceinline__ void prefetch_prev_u(const InstDev& D, int k, int S) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(D.fields + S + k));
  asm volatile("prefetch.global.L2 [%0];" ::"l"(D.fields + 2 * S + k));
}

// Source, both collisions, stores and final-step bookkeeping of one node
// whose populations are already reduced to (wall-completed) moments hm, cm[3];
// f, G: its flow and the differences; So, uo: source and velocity of the
// previous step (ignored at init).
// Writes the 36 post-collision populations and the 5 history values of node k;
// on the final step also the float64 fields and this node's partial sums.
template <typename R, int MODE, bool FINAL, bool MASKED>
__device__ __forceinline__ void collide_node(const InstDev& D, int k, int S, R* __restrict__ dst,
                                             R* __restrict__ hist,
                                             const typename Arith<R>::Hydro& hm,
                                             const typename Arith<R>::Cde* cm, const Flow<R>& f,
                                             const Grad<R>& G, R Fx, R Fy, R So0, R So1, R So2,
                                             R uxo, R uyo, PartT<R> ux_prev, PartT<R> uy_prev,
                                             PartT<R>* part, PartT<R>* plo) {
  // conformation tensor, constitutive function, source Phi_ab
  R Axx, Axy, Ayy, Fxx, Fxy, Fyy;
  polymer_terms<R, MASKED>(D, cm[0].dphi, cm[1].dphi, cm[2].dphi, Axx, Axy, Ayy, Fxx, Fxy, Fyy);
  R Sc[3], So[3] = {So0, So1, So2};
#pragma unroll
  for (int l = 0; l < 3; ++l) Sc[l] = Arith<R>::source(l, D, Axx, Axy, Ayy, Fxx, Fxy, Fyy, G);
  if (MODE != kModeStep) {
    // first step: the backward difference of the CDE source is zero
    So[0] = Sc[0];
    So[1] = Sc[1];
    So[2] = Sc[2];
    uxo = f.ux;
    uyo = f.uy;
  }
  collide_hydro<R>(D, k, S, dst, hm, f, G, Fxx, Fxy, Fyy, Fx, Fy);
#pragma unroll
  for (int l = 0; l < 3; ++l)
    collide_cde<R, MASKED>(D, k, S, dst, l, cm[l], f, Sc[l], So[l], uxo, uyo, Fx, Fy, G);

  hist[k] = Sc[0];
  hist[S + k] = Sc[1];
  hist[2 * S + k] = Sc[2];
  hist[3 * S + k] = f.ux;
  hist[4 * S + k] = f.uy;

  if (FINAL) {
    const R dphi[3] = {cm[0].dphi, cm[1].dphi, cm[2].dphi};
    final_node<R, MODE>(D, k, S, -1, hm.drho, f.rho, f.ux, f.uy, dphi, ux_prev, uy_prev, part,
                        plo);
  }
}

// Resident CTAs per SM the register budget is sized for: the float32 step
// is HBM-bound and wants more loads in flight; the float64 step is bound by
// the FP64 pipe.
// Masked tiles carry the mask's one-sided differences: 5 CTAs of 96 threads per
// SM (few of them run in another shape, launch_step_m).
#ifndef LBVE_FP32_MASKED_MIN_BLOCKS
#define LBVE_FP32_MASKED_MIN_BLOCKS 5
#endif
// Float64 CTAs: 256 threads two per SM (128 registers per thread).  The
// 64- and one-warp CTAs serve batches with fewer tiles than 4 and 2 per SM,
// so they are budgeted for that many and keep every value in registers.
// Float32 pairs: 3 CTAs per SM keep their registers (227 at most) without
// spills; 4 per SM spill a little and ran 1.4 % slower on the batched mix.
#ifndef LBVE_DF32_MIN_BLOCKS
#define LBVE_DF32_MIN_BLOCKS 3
#endif
template <typename R, bool MASKED, int NT>
struct MinBlocks {
  static constexpr int value =
      std::is_same<R, df32>::value
          ? LBVE_DF32_MIN_BLOCKS
          : sizeof(R) == 4 ? (MASKED ? LBVE_FP32_MASKED_MIN_BLOCKS : LBVE_FP32_MIN_BLOCKS)
                           : (NT <= 32 ? 2 : NT <= 64 ? 4 : 512 / NT);
};

// Open channels: nodes of the inlet (x = 0) and outlet (x = nx - 1) columns
// take their completed populations from the edge pass's colbuf during a
// step (the pull would miss the populations entering from outside).
__device__ __forceinline__ bool open_column(const InstDev& D, int gx) {
  return D.open_x && (gx == 0 || gx == D.nx - 1);
}
template <typename R>
__device__ __forceinline__ const R* colbuf_node(const InstDev& D, int gx, int gy) {
  return (const R*)D.colbuf + (gx == 0 ? 0 : D.ny) + gy;  // plane stride 2 ny
}

// Flow of region node (gx, gy) for the masked variant: open-column nodes
// from colbuf during a step, every other node as node_flow.
template <typename R, int MODE>
__device__ __forceinline__ void region_flow(const InstDev& D, const void* src,
                                            const R* __restrict__ force, bool ffield, R Fx0,
                                            R Fy0, int S, int nx, int ny, bool py, int gx,
                                            int gy, Flow<R>& f) {
  if (MODE == kModeStep && open_column(D, gx)) {
    const R* cb = colbuf_node<R>(D, gx, gy);
    const int ld = 2 * ny;
    R d[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) d[i] = cb[(size_t)i * ld];
    const int k = gy * nx + gx;
    const R Fx = ffield ? force[k] : Fx0, Fy = ffield ? force[S + k] : Fy0;
    f.pull(d, Fx, Fy);
    return;
  }
  node_flow<R, MODE>(src, force, ffield, Fx0, Fy0, S, nx, ny, py, gx, gy, f);
}

// Sum of two float32 pairs (hi + lo), renormalised (Knuth's two-sum of the
// high parts, the low parts added to its error, a fast two-sum at the end).
__device__ __forceinline__ void df_add(float& ah, float& al, float bh, float bl) {
  const float s = ah + bh, bv = s - ah;
  const float e = ((ah - (s - bv)) + (bh - bv)) + (al + bl);
  ah = s + e;
  al = e - (ah - s);
}

// One butterfly level (fold_half) on float32 pairs.
template <int M>
__device__ __forceinline__ void fold_half_df(float* h, float* l, int o, bool up) {
#pragma unroll
  for (int j = 0; j < M / 2; ++j) {
    const float kh = up ? h[j + M / 2] : h[j], kl = up ? l[j + M / 2] : l[j];
    const float sh = up ? h[j] : h[j + M / 2], sl = up ? l[j] : l[j + M / 2];
    const float rh = __shfl_xor_sync(0xffffffffu, sh, o), rl = __shfl_xor_sync(0xffffffffu, sl, o);
    h[j] = kh;
    l[j] = kl;
    df_add(h[j], l[j], rh, rl);
  }
}

// The tile's partial record of the final step in a fixed order: the 12
// sums by a transposed butterfly per warp, the residual (>= 0 and finite, so
// the order of its bit patterns is its numeric order) and the non-finite
// count as integers, then the warps in order and the rest values from the
// count of the tile's fluid nodes.  Every thread of the CTA calls it.  A
// float32 instance's values are float32 numbers or exact float32 pairs
// (part + plo), and its butterfly adds float32 pairs (a 48-bit sum; GB300
// issues a float64 addition only every 64 cycles per warp); the warp totals
// and everything after them are float64.  A float32 warp whose nodes carry no
// wall balance folds only the first 6 values (the order of the sum is fixed
// by the tile's own data, so totals stay reproducible).
template <int NT, typename P>
__device__ __forceinline__ void tile_partials(const InstDev& D, const TileDev& T, const P* part,
                                              const P* plo, bool active,
                                              double* __restrict__ partials,
                                              double (*s_red)[kPartial]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  static_assert(kNonFinite == 13 && kResid == 12, "12 sums, then residual and flag");
  double total;  // this lane's warp total of value slot
  double resid;  // the warp's largest residual
  int slot;   // the value slot this lane's total belongs to
  bool write;  // whether this lane writes it
  if constexpr (sizeof(P) == 4) {
    // a warp without wall nodes has zero wall balances (slots 6..11): its
    // butterfly sums the first 6 values only
    bool wall = false;
#pragma unroll
    for (int j = kWallIn; j < kResid; ++j) wall = wall || part[j] != 0.f || plo[j] != 0.f;
    if (__any_sync(0xffffffffu, wall)) {
      float h[16], l[16];
#pragma unroll
      for (int j = 0; j < 12; ++j) {
        h[j] = part[j];
        l[j] = plo[j];
      }
#pragma unroll
      for (int j = 12; j < 16; ++j) h[j] = l[j] = 0.f;
      fold_half_df<16>(h, l, 16, (lane & 16) != 0);
      fold_half_df<8>(h, l, 8, (lane & 8) != 0);
      fold_half_df<4>(h, l, 4, (lane & 4) != 0);
      fold_half_df<2>(h, l, 2, (lane & 2) != 0);
      const float rh = __shfl_xor_sync(0xffffffffu, h[0], 1);
      const float rl = __shfl_xor_sync(0xffffffffu, l[0], 1);
      df_add(h[0], l[0], rh, rl);
      total = f2d_exact(h[0]) + f2d_exact(l[0]);
      slot = (lane >> 1) & 15;
      write = (lane & 1) == 0 && slot < 12;
    } else {
      float h[8], l[8];
#pragma unroll
      for (int j = 0; j < 6; ++j) {
        h[j] = part[j];
        l[j] = plo[j];
      }
      h[6] = h[7] = l[6] = l[7] = 0.f;
      fold_half_df<8>(h, l, 16, (lane & 16) != 0);
      fold_half_df<4>(h, l, 8, (lane & 8) != 0);
      fold_half_df<2>(h, l, 4, (lane & 4) != 0);
#pragma unroll
      for (int o = 2; o > 0; o >>= 1) {
        const float rh = __shfl_xor_sync(0xffffffffu, h[0], o);
        const float rl = __shfl_xor_sync(0xffffffffu, l[0], o);
        df_add(h[0], l[0], rh, rl);
      }
      // value (lane >> 2) & 7; lanes 4m write it, lanes 4m + 1 the zero of wall slot 6 + m
      const int s8 = (lane >> 2) & 7;
      total = (lane & 3) == 1 ? 0.0 : f2d_exact(h[0]) + f2d_exact(l[0]);
      slot = (lane & 3) == 1 ? kWallIn + s8 : s8;
      write = (lane & 3) <= 1 && s8 < 6;
    }
    int rb = __float_as_int(part[kResid]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) rb = max(rb, __shfl_xor_sync(0xffffffffu, rb, o));
    resid = f2d_exact(__int_as_float(rb));
  } else {
    double v[16];
#pragma unroll
    for (int j = 0; j < 12; ++j) v[j] = part[j];
#pragma unroll
    for (int j = 12; j < 16; ++j) v[j] = 0.0;
    fold_half<16>(v, 16, (lane & 16) != 0);
    fold_half<8>(v, 8, (lane & 8) != 0);
    fold_half<4>(v, 4, (lane & 4) != 0);
    fold_half<2>(v, 2, (lane & 2) != 0);
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
    total = v[0];
    slot = (lane >> 1) & 15;
    write = (lane & 1) == 0 && slot < 12;
    long long rb = __double_as_longlong(part[kResid]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const long long ob = __shfl_xor_sync(0xffffffffu, rb, o);
      rb = ob > rb ? ob : rb;
    }
    resid = __longlong_as_double(rb);
  }
  const unsigned nf = __popc(__ballot_sync(0xffffffffu, part[kNonFinite] != P(0)));
  if (write) s_red[warp][slot] = total;
  if (lane == 0) {
    s_red[warp][kResid] = resid;
    s_red[warp][kNonFinite] = (double)nf;
  }
  const int nfluid = __syncthreads_count(active);
  if (threadIdx.x < 14) {
    const int j = threadIdx.x;
    double t = s_red[0][j];
    for (int w = 1; w < NT / 32; ++w) t = (j == kResid) ? fmax(t, s_red[w][j]) : t + s_red[w][j];
    if (j == kSumRho || j == kSumPhi || j == kSumPhi + 2) t += (double)nfluid;
    if (j == kResid) t *= D.inv_Uc;
    partials[(size_t)T.slot * kPartial + j] = t;
  }
}

// Programmatic dependent launch.  A step kernel lets the next one start as
// soon as all its CTAs run, and waits here for the previous one to complete
// before it touches anything that kernel writes; tile table and descriptors
// are constant over the steps and are read before.  Every CTA waits, also one
// with nothing to do: the completion of a kernel then implies that of all
// before it.
// The next kernel's launch and its CTAs' first dependent loads (tile, then
// descriptor) then hide behind the end of the one before: 3.53 -> 2.96 us per
// step on the five Wi-sweep channels in float32, 1.5 % on a 512^2 grid.  Not in
// float64: CTAs that arrive early share an SM with running ones, and two tiles
// of one step on one float64 pipe cost more (64^2 mill 6.6 -> 9.3 us; 6.7 with
// one CTA per SM).
template <typename R, int MODE, bool MASKED>
__host__ __device__ constexpr bool overlaps_steps() {
  return MODE == kModeStep && !MASKED && !std::is_same<R, double>::value;
}
__device__ __forceinline__ void start_next_kernel() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void wait_previous_kernel() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <typename R, int MODE, bool FINAL, bool MASKED, int NT>
__device__ __forceinline__ void process_tile(const InstDev* __restrict__ insts, const TileDev T,
                                             int parity, double* __restrict__ partials,
                                             Region<R, region_max(NT)>& Q,
                                             double (*s_red)[kPartial]) {
  const InstDev& D = insts[T.inst];
  const int nx = D.nx, ny = D.ny, S = D.stride, TX = D.TX, TY = D.TY, hy = D.hy;
  const bool py = D.periodic_y != 0;
  const void* src = D.pop[parity];
  const R* __restrict__ srcR = (const R*)src;
  R* __restrict__ dst = (R*)D.pop[parity ^ 1];
  const R* __restrict__ force = (const R*)D.force;
  const R* hist = (const R*)D.hist;
  const bool ffield = D.force_field != 0;
  const R Fx0 = coef<R>(D, kCoefFx), Fy0 = coef<R>(D, kCoefFy);
  const int RW = TX + 2;

  // ---- phase A --------------------------------------------------------------
  // Every load this thread needs -- one halo-ring node's hydro populations
  // and all of its own node's populations, history and force -- is issued
  // before any of them is used, so the tile's whole HBM traffic is in flight
  // together.  Own hydro and conformation populations are then reduced to
  // moments (walls completed first); rho and u go to shared memory.
  // Thread and halo-slot indices.  For plain kTileTX-wide tiles (D.t32) the
  // divisions by the width and the wraps use compile-time constants; the
  // arithmetic after this prologue is one code path for every width.
  const bool t32 = !MASKED && D.t32;
  int tx, ty;
  if (t32) {
    tx = threadIdx.x % kTileTX;
    ty = threadIdx.x / kTileTX;
  } else {
    tx = threadIdx.x % TX;
    ty = threadIdx.x / TX;
  }
  const bool in_tile = ty < TY;
  const int x = T.x0 + tx, y = T.y0 + ty;
  const bool inside = in_tile && (x < nx) && (y < ny);
  // solid-mask nodes (masked tiles only) take no part in the update
  // (rows 0..2 and ny-3.. of a walled domain and the three columns at open ends
  // carry no mask, so what follows here may look at the position alone and
  // the loads below need not wait for the mask); sxp..sym: blocked sides
  bool solid = false, sxp = false, sxm = false, syp = false, sym = false;
  const int ri = (ty + hy) * RW + tx + 1;  // this slot in the halo region
  const bool wb = inside && !py && y == 0, wt = inside && !py && y == ny - 1;
  // an open column's node arrives completed (colbuf): no wall completion there
  const bool ocol = MASKED && MODE == kModeStep && inside && open_column(D, x);
  if (MASKED && inside) {
    // a side is blocked by a solid node or, in an open channel, by the end of
    // the domain beyond the inlet / outlet column
    sxp = D.open_x && x == nx - 1;
    sxm = D.open_x && x == 0;
    if (const uint8_t* __restrict__ M = D.mask) {
      const int xp = x == nx - 1 ? 0 : x + 1, xm = x == 0 ? nx - 1 : x - 1;
      const int yp = y == ny - 1 ? (py ? 0 : y) : y + 1, ym = y == 0 ? (py ? ny - 1 : y) : y - 1;
      const uint8_t m0 = M[y * nx + x], m1 = M[y * nx + xp], m2 = M[y * nx + xm];
      const uint8_t m3 = M[yp * nx + x], m4 = M[ym * nx + x];
      solid = m0 != 0;
      sxp = sxp || m1 != 0;
      sxm = sxm || m2 != 0;
      // rows next to a flat wall carry no mask, so y +- 1 lies in the domain
      syp = !wb && !wt && m3 != 0;
      sym = !wb && !wt && m4 != 0;
    }
  }
  const bool active = inside && !solid;
  const bool wcomp = (wb || wt) && !ocol;
  const int nring = 2 * hy * TX + 2 * TY;  // the halo ring without its corners

  if (overlaps_steps<R, MODE, MASKED>()) wait_previous_kernel();

  // (1) first halo-ring node of this thread: issue its pull
  int ring_r = -1, rgx = 0, rgy = 0;
  R dr[9];
  if (threadIdx.x < nring) {
    int lx, ly;
    bool in_domain;
    if (t32) {
      ring_slot(threadIdx.x, kTileTX + 2, NT / kTileTX, hy, lx, ly);
      in_domain = region_node_once(lx, ly, T.x0, T.y0, hy, nx, ny, py, rgx, rgy);
    } else {
      ring_slot(threadIdx.x, RW, TY, hy, lx, ly);
      in_domain = region_node(lx, ly, T.x0, T.y0, hy, nx, ny, py, rgx, rgy);
    }
    if (in_domain) {
      ring_r = ly * RW + lx;
      if (MASKED && MODE == kModeStep && open_column(D, rgx)) {
        const R* cb = colbuf_node<R>(D, rgx, rgy);
#pragma unroll
        for (int i = 0; i < 9; ++i) dr[i] = cb[(size_t)i * 2 * ny];
      } else {
        int rm, rp;
        neighbour_rows(rgy, nx, ny, py, rm, rp);
        const int xm = rgx == 0 ? nx - 1 : rgx - 1, xp = rgx == nx - 1 ? 0 : rgx + 1;
        PopSource<R, MODE>::hydro(src, S, nx, rgy * nx + rgx, rgy * nx, rm, rp, rgx, xm, xp, dr);
      }
    }
  }

  // (2) own node: all 36 populations, force, history, wall slots
  R d[9], g[3][9], So[3] = {R(0), R(0), R(0)}, uxo = R(0), uyo = R(0), Fx = Fx0, Fy = Fy0;
  R post[3][3];  // own outgoing-to-wall post-collision slots (wall rows only)
  int k = 0;
  if (inside) {
    k = y * nx + x;
    int rm, rp;
    neighbour_rows(y, nx, ny, py, rm, rp);
    const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
    const int rc = y * nx;
    if (ocol) {
      const R* cb = colbuf_node<R>(D, x, y);
      const int ld = 2 * ny;
#pragma unroll
      for (int i = 0; i < 9; ++i) d[i] = cb[(size_t)i * ld];
#pragma unroll
      for (int l = 0; l < 3; ++l)
#pragma unroll
        for (int i = 0; i < 9; ++i) g[l][i] = cb[(size_t)(9 + 9 * l + i) * ld];
    } else {
      PopSource<R, MODE>::hydro(src, S, nx, k, rc, rm, rp, x, xm, xp, d);
#pragma unroll
      for (int l = 0; l < 3; ++l)
        PopSource<R, MODE>::cde(src, l, S, nx, k, rc, rm, rp, x, xm, xp, g[l]);
    }
    if (ffield) {
      Fx = force[k];
      Fy = force[S + k];
    }
    if (MODE == kModeStep) {
      So[0] = hist[k];
      So[1] = hist[S + k];
      So[2] = hist[2 * S + k];
      uxo = hist[3 * S + k];
      uyo = hist[4 * S + k];
      if (FINAL) prefetch_prev_u(D, k, S);
      if (wcomp) {
        // bottom wall: H = {4, 7, 8}; top wall: H = {2, 5, 6}
        const int h0 = wb ? 4 : 2, h1 = wb ? 7 : 5, h2 = wb ? 8 : 6;
#pragma unroll
        for (int l = 0; l < 3; ++l) {
          const R* own = srcR + (size_t)(9 + 9 * l) * S + k;
          post[l][0] = own[h0 * S];
          post[l][1] = own[h1 * S];
          post[l][2] = own[h2 * S];
        }
      }
    }
  }

  // (3) ring node moments
  if (ring_r >= 0) {
    const int rk = rgy * nx + rgx;
    const R rFx = ffield ? force[rk] : Fx0;
    const R rFy = ffield ? force[S + rk] : Fy0;
    if (MODE == kModeStep && !py && (rgy == 0 || rgy == ny - 1) &&
        !(MASKED && open_column(D, rgx)))
      zou_he<R>(dr, rFx, rFy, rgy == 0);
    Flow<R> f;
    f.pull(dr, rFx, rFy);
    Q.put(ring_r, f);
  }

  // (4) own moments; conformation walls completed with the node's own u
  typename Arith<R>::Hydro hm;
  typename Arith<R>::Cde cm[3];
  Flow<R> f;
  double wall_io[6] = {0, 0, 0, 0, 0, 0};
  if (active) {
    if (MODE == kModeStep && wcomp) zou_he<R>(d, Fx, Fy, wb);
    Arith<R>::moments(d, hm);
    f.set(hm, Fx, Fy);
    Q.put(ri, f);
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      if (MODE == kModeStep && wcomp) {
        const R delta = (l == 1) ? R(0) : R(1);
        cnebb<R>(g[l], post[l][0], post[l][1], post[l][2], delta, f.ux, f.uy, wb, wall_io[l],
                 wall_io[3 + l]);
      }
      Arith<R>::moments(g[l], cm[l]);
    }
  } else if (in_tile && !inside) {
    // slot outside the domain (ragged tile): it may still be a periodic
    // neighbour of an active node, so fill it with the wrapped node
    const int gx = t32 ? wrap_once(x, nx) : x % nx;
    const int gy = py ? (t32 ? wrap_once(y, ny) : y % ny) : y;
    if (gy < ny) {
      Flow<R> w;
      if constexpr (MASKED)
        region_flow<R, MODE>(D, src, force, ffield, Fx0, Fy0, S, nx, ny, py, gx, gy, w);
      else
        node_flow<R, MODE>(src, force, ffield, Fx0, Fy0, S, nx, ny, py, gx, gy, w);
      Q.put(ri, w);
    }
  }

  // (5) remaining ring nodes (only when the ring outnumbers the threads)
  for (int q = threadIdx.x + blockDim.x; q < nring; q += blockDim.x) {
    int lx, ly, gx, gy;
    ring_slot(q, RW, TY, hy, lx, ly);
    if (!region_node(lx, ly, T.x0, T.y0, hy, nx, ny, py, gx, gy)) continue;
    Flow<R> w;
    if constexpr (MASKED)
      region_flow<R, MODE>(D, src, force, ffield, Fx0, Fy0, S, nx, ny, py, gx, gy, w);
    else
      node_flow<R, MODE>(src, force, ffield, Fx0, Fy0, S, nx, ny, py, gx, gy, w);
    Q.put(ly * RW + lx, w);
  }
  __syncthreads();

  // ---- phase B: gradients, source, collisions, stores ----------------------
  PartT<R> part[FINAL ? 14 : 1], plo[FINAL ? 12 : 1];
#pragma unroll
  for (int j = 0; j < (FINAL ? 14 : 1); ++j) part[j] = 0;
#pragma unroll
  for (int j = 0; j < (FINAL ? 12 : 1); ++j) plo[j] = 0;

  if (active) {
    Grad<R> G;
    Arith<R>::gradients(Q, ri, RW, wb, wt, f, MASKED && D.gtilde, G);
    if constexpr (MASKED) {
      // one-sided differences where an axis neighbour is solid; the values
      // two nodes away come straight from the pulled populations (L2)
      const uint8_t* __restrict__ M = D.mask;
      if (sxp || sxm) {
        if (sxp && sxm) {
          Arith<R>::blocked(0, G);
        } else {
          const int t = sxp ? -1 : 1;
          const int i1 = t > 0 ? ri + 1 : ri - 1;
          const int x2 = (((x + 2 * t) % nx) + nx) % nx;
          const bool has2 = !(M && M[y * nx + x2] != 0);
          Flow<R> w;
          w.rest();
          if (has2)
            region_flow<R, MODE>(D, src, force, ffield, Fx0, Fy0, S, nx, ny, py, x2, y, w);
          Arith<R>::one_sided(0, t, Q, ri, i1, f, has2, w, G);
        }
      }
      if (syp || sym) {
        if (syp && sym) {
          Arith<R>::blocked(1, G);
        } else {
          const int t = syp ? -1 : 1;
          const int i1 = t > 0 ? ri + RW : ri - RW;
          int y2 = y + 2 * t;
          if (py) y2 = ((y2 % ny) + ny) % ny;
          const bool has2 = y2 >= 0 && y2 < ny && M[y2 * nx + x] == 0;
          Flow<R> w;
          w.rest();
          if (has2)
            region_flow<R, MODE>(D, src, force, ffield, Fx0, Fy0, S, nx, ny, py, x, y2, w);
          Arith<R>::one_sided(1, t, Q, ri, i1, f, has2, w, G);
        }
      }
    }
    if (FINAL) {
      if constexpr (sizeof(R) == 4) {
        if (wcomp) {
          // float32 pairs of the (float64) wall balances of a wall node
#pragma unroll
          for (int j = 0; j < 6; ++j) {
            const float hi = (float)wall_io[j];
            part[kWallIn + j] = hi;
            plo[kWallIn + j] = (float)(wall_io[j] - f2d_exact(hi));
          }
        }
      } else {
#pragma unroll
        for (int j = 0; j < 6; ++j) part[kWallIn + j] = wall_io[j];
      }
    }
    PartT<R> ux_prev = 0, uy_prev = 0;
    if (FINAL && MODE == kModeStep) {
      // prefetched into L2 above; read past L1 (nothing else touches these lines)
      ux_prev = (PartT<R>)__ldcg(D.fields + S + k);
      uy_prev = (PartT<R>)__ldcg(D.fields + 2 * S + k);
    }
    collide_node<R, MODE, FINAL, MASKED>(D, k, S, dst, (R*)D.hist_out, hm, cm, f, G, Fx, Fy, So[0],
                                         So[1], So[2], uxo, uyo, ux_prev, uy_prev, part, plo);
  } else if (FINAL && solid) {
    // a solid node reports zero fields and adds nothing to the totals
    const int ks = y * nx + x;
#pragma unroll
    for (int j = 0; j < 6; ++j) D.fields[(size_t)j * S + ks] = 0.0;
  }

  if (FINAL) tile_partials<NT, PartT<R>>(D, T, part, plo, active, partials, s_red);
}

// One CTA of NT threads per tile (NT a multiple of 32, at least 32, with
// TX * TY <= NT for every tile of the launch).  The plain variant leaves
// masked tiles to the masked one (which runs over a separate list of just
// those tiles).
template <typename R, int MODE, bool FINAL, bool MASKED, int NT, int MB>
__global__ void __launch_bounds__(NT, MB)
    step_kernel(const InstDev* __restrict__ insts, const TileDev* __restrict__ tiles,
                int parity, double* __restrict__ partials) {
  static_assert(NT % 32 == 0 && NT >= 32, "whole warps; the final-step reduction reads 14 lanes");
  __shared__ Region<R, region_max(NT)> Q;
  __shared__ double s_red[NT / 32][kPartial];
  constexpr bool kOverlap = overlaps_steps<R, MODE, MASKED>();
  if (kOverlap) start_next_kernel();
  const TileDev T = tiles[blockIdx.x];
  if (!MASKED && T.masked) {
    if (kOverlap) wait_previous_kernel();
    return;
  }
  process_tile<R, MODE, FINAL, MASKED, NT>(insts, T, parity, partials, Q, s_red);
}

// ---- float64 steps of tiny batches: one lattice per warp --------------------
//
// GB300 issues a float64 instruction only once every 64 cycles per warp, and
// a warp pays that for every instruction whatever the number of active
// lanes; four warps per SM saturate its float64 pipe.  A float64 batch too
// small to give every SM several warps is therefore bound by the float64
// instruction count of one thread's node, not by the number of nodes.  This
// variant spreads the update of each node over four warps: warp 0 carries
// the hydrodynamic lattice (pull, Zou-He, moments, rho and u, the gradients
// and the hydrodynamic collision), warp 1 + l the conformation lattice l
// (pull, CNEBB, moments, its component of Phi_ab and its collision); the
// warps meet in shared memory twice (rho, u; the three phi).  Every value is
// the same expression of the same operands as in process_tile, so the
// fields are bit-identical to those of the one-warp kernel.
//   Tiles of at most 32 nodes (TX * TY <= 32), plain tiles only (no mask, no
//   open column, Oldroyd-B with the eq_p_G_1 form of G~), time steps only
//   (the initialisation runs the one-warp kernel).
constexpr int kSplitThreads = 128;

template <bool FINAL>
__device__ __forceinline__ void process_tile_split(const InstDev* __restrict__ insts,
                                                   const TileDev T, int parity,
                                                   double* __restrict__ partials,
                                                   Region<double, region_max(32)>& Q,
                                                   double (*s_phi)[32], double* s_irho,
                                                   double (*s_red)[kPartial]) {
  using R = double;
  constexpr int MODE = kModeStep;
  const InstDev& D = insts[T.inst];
  const int nx = D.nx, ny = D.ny, S = D.stride, TX = D.TX, TY = D.TY, hy = D.hy;
  const bool py = D.periodic_y != 0;
  const void* src = D.pop[parity];
  const R* __restrict__ srcR = (const R*)src;
  R* __restrict__ dst = (R*)D.pop[parity ^ 1];
  const R* __restrict__ force = (const R*)D.force;
  const R* hist = (const R*)D.hist;
  const bool ffield = D.force_field != 0;
  const R Fx0 = coef<R>(D, kCoefFx), Fy0 = coef<R>(D, kCoefFy);
  const int RW = TX + 2;
  const int role = threadIdx.x >> 5, lane = threadIdx.x & 31;  // 0 hydro, 1 + l lattice l
  const int tx = lane % TX, ty = lane / TX;
  const bool in_tile = ty < TY;
  const int x = T.x0 + tx, y = T.y0 + ty;
  const bool inside = in_tile && (x < nx) && (y < ny);
  const bool active = inside;
  const int ri = (ty + hy) * RW + tx + 1;
  const bool wb = active && !py && y == 0, wt = active && !py && y == ny - 1;
  const bool wcomp = wb || wt;
  const int nring = 2 * hy * TX + 2 * TY;

  // ---- phase A: pulls -------------------------------------------------------
  // the halo ring's hydrodynamic pulls go to the conformation warps (their
  // own float64 work is the lighter one)
  const int q = threadIdx.x - 32;
  int ring_r = -1, rgx = 0, rgy = 0;
  R dr[9];
  if (role > 0 && q < nring) {
    int lx, ly;
    ring_slot(q, RW, TY, hy, lx, ly);
    if (region_node(lx, ly, T.x0, T.y0, hy, nx, ny, py, rgx, rgy)) {
      ring_r = ly * RW + lx;
      int rm, rp;
      neighbour_rows(rgy, nx, ny, py, rm, rp);
      const int xm = rgx == 0 ? nx - 1 : rgx - 1, xp = rgx == nx - 1 ? 0 : rgx + 1;
      PopSource<R, MODE>::hydro(src, S, nx, rgy * nx + rgx, rgy * nx, rm, rp, rgx, xm, xp, dr);
    }
  }
  const int l = role - 1;
  R d[9], post[3] = {R(0), R(0), R(0)}, So = R(0), uxo = R(0), uyo = R(0), Fx = Fx0, Fy = Fy0;
  int k = 0;
  if (active) {
    k = y * nx + x;
    int rm, rp;
    neighbour_rows(y, nx, ny, py, rm, rp);
    const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
    if (role == 0) {
      PopSource<R, MODE>::hydro(src, S, nx, k, y * nx, rm, rp, x, xm, xp, d);
      if (FINAL) prefetch_prev_u(D, k, S);
    } else {
      PopSource<R, MODE>::cde(src, l, S, nx, k, y * nx, rm, rp, x, xm, xp, d);
      So = hist[(size_t)l * S + k];
      uxo = hist[3 * S + k];
      uyo = hist[4 * S + k];
      if (wcomp) {
        const int h0 = wb ? 4 : 2, h1 = wb ? 7 : 5, h2 = wb ? 8 : 6;
        const R* own = srcR + (size_t)(9 + 9 * l) * S + k;
        post[0] = own[h0 * S];
        post[1] = own[h1 * S];
        post[2] = own[h2 * S];
      }
    }
    if (ffield) {
      Fx = force[k];
      Fy = force[S + k];
    }
  }
  // ring moments (a ring longer than the three conformation warps, which the
  // tile widths of the one-warp CTAs never make, is finished by warp 0 below)
  if (ring_r >= 0) {
    const int rk = rgy * nx + rgx;
    const R rFx = ffield ? force[rk] : Fx0;
    const R rFy = ffield ? force[S + rk] : Fy0;
    if (!py && (rgy == 0 || rgy == ny - 1)) zou_he<R>(dr, rFx, rFy, rgy == 0);
    Flow<R> w;
    w.pull(dr, rFx, rFy);
    Q.put(ring_r, w);
  }
  for (int qq = kSplitThreads - 32 + threadIdx.x; role == 0 && qq < nring; qq += 32) {
    int lx, ly, gx, gy;
    ring_slot(qq, RW, TY, hy, lx, ly);
    if (!region_node(lx, ly, T.x0, T.y0, hy, nx, ny, py, gx, gy)) continue;
    Flow<R> w;
    node_flow<R, MODE>(src, force, ffield, Fx0, Fy0, S, nx, ny, py, gx, gy, w);
    Q.put(ly * RW + lx, w);
  }
  // own hydrodynamic moments (warp 0), and the wrapped nodes of a ragged tile
  Arith<R>::Hydro hm;
  Flow<R> f;
  if (role == 0) {
    if (active) {
      if (wcomp) zou_he<R>(d, Fx, Fy, wb);
      Arith<R>::moments(d, hm);
      f.set(hm, Fx, Fy);
      Q.put(ri, f);
      s_irho[lane] = f.irho;
    } else if (in_tile) {
      const int gx = x % nx;
      const int gy = py ? y % ny : y;
      if (gy < ny) {
        Flow<R> w;
        node_flow<R, MODE>(src, force, ffield, Fx0, Fy0, S, nx, ny, py, gx, gy, w);
        Q.put(ri, w);
      }
    }
  }
  __syncthreads();

  // ---- conformation walls with the node's own u, moments -----------------------
  if (role > 0 && active) {
    f.ux = Q.ux[ri];
    f.uy = Q.uy[ri];
    f.irho = s_irho[lane];
    f.rho = R(1);  // not used by the conformation lattices
  }
  Arith<R>::Cde cm;
  double wall_in = 0.0, wall_out = 0.0;
  if (role > 0 && active) {
    if (wcomp) {
      const R delta = (l == 1) ? R(0) : R(1);
      cnebb<R>(d, post[0], post[1], post[2], delta, f.ux, f.uy, wb, wall_in, wall_out);
    }
    Arith<R>::moments(d, cm);
    s_phi[l][lane] = cm.dphi;
  }
  __syncthreads();

  // ---- phase B: gradients, source, this warp's collision, stores ---------------
  PartT<R> part[FINAL ? 14 : 1], plo[FINAL ? 12 : 1];
#pragma unroll
  for (int j = 0; j < (FINAL ? 14 : 1); ++j) part[j] = 0;
#pragma unroll
  for (int j = 0; j < (FINAL ? 12 : 1); ++j) plo[j] = 0;
  if (active) {
    Grad<R> G;
    Arith<R>::gradients(Q, ri, RW, wb, wt, f, false, G);
    R Axx, Axy, Ayy, Fxx, Fxy, Fyy;
    polymer_terms<R, false>(D, s_phi[0][lane], s_phi[1][lane], s_phi[2][lane], Axx, Axy, Ayy, Fxx,
                            Fxy, Fyy);
    if (role == 0) {
      double ux_prev = 0.0, uy_prev = 0.0;
      if (FINAL) {
        ux_prev = D.fields[S + k];
        uy_prev = D.fields[2 * S + k];
      }
      collide_hydro<R>(D, k, S, dst, hm, f, G, Fxx, Fxy, Fyy, Fx, Fy);
      R* hist_out = (R*)D.hist_out;
      hist_out[3 * S + k] = f.ux;
      hist_out[4 * S + k] = f.uy;
      if (FINAL)
        final_node<R, MODE>(D, k, S, 0, hm.drho, f.rho, f.ux, f.uy, nullptr, ux_prev, uy_prev,
                            part, plo);
    } else {
      const R sl = Arith<R>::source(l, D, Axx, Axy, Ayy, Fxx, Fxy, Fyy, G);
      collide_cde<R, false>(D, k, S, dst, l, cm, f, sl, So, uxo, uyo, Fx, Fy, G);
      ((R*)D.hist_out)[(size_t)l * S + k] = sl;
      if (FINAL) {
        const R dphi[3] = {s_phi[0][lane], s_phi[1][lane], s_phi[2][lane]};
        final_node<R, MODE>(D, k, S, role, R(0), f.rho, f.ux, f.uy, dphi, 0.0, 0.0, part, plo);
        part[kWallIn + l] = wall_in;
        part[kWallOut + l] = wall_out;
      }
    }
  }
  if (FINAL)
    tile_partials<kSplitThreads, double>(D, T, part, plo, active && role == 0, partials, s_red);
}

template <bool FINAL>
__global__ void __launch_bounds__(kSplitThreads, 4)
    step_kernel_split(const InstDev* __restrict__ insts, const TileDev* __restrict__ tiles,
                      int parity, double* __restrict__ partials) {
  __shared__ Region<double, region_max(32)> Q;
  __shared__ double s_phi[3][32], s_irho[32];
  __shared__ double s_red[kSplitThreads / 32][kPartial];
  const TileDev T = tiles[blockIdx.x];
  if (T.masked) return;
  process_tile_split<FINAL>(insts, T, parity, partials, Q, s_phi, s_irho, s_red);
}

}  // namespace lbve
