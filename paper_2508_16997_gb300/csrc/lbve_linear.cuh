// lbve_linear.cuh -- the linear parts of a float64 step (populations to
// moments, Hermite coefficients to populations) in 64-bit block fixed point.
//
// One SM retires a float64 instruction of a warp every 19.0 cycles, an integer
// instruction every 0.52 (measured with independent chains, 4 to 32 warps;
// both pipes run side by side).  A
// transform of nine populations is 21 to 23 additions, so it costs 400 to 440
// cycles on the float64 pipe.  In fixed point the values are aligned once to the
// largest exponent among them (11 integer instructions each), added exactly
// as 64-bit integers, and each result is rounded once to float64 (25
// instructions): 155 to 180 cycles on a pipe that is otherwise idle.  The step of
// the batched mix (64 instances) went from 2.54 to 1.19 ms with it.
//   Precision: the largest input's leading bit sits at bit 58, i.e. 6 bits
// below its last float64 bit are kept, and the sums are exact.  An input is
// truncated toward zero only where it is more than 2^6 smaller than the
// largest one, by less than 2^-58 of that one; the float64 additions replaced
// here round every partial sum at 2^-53 of its size.  Results round to nearest
// even.  Exact zeros stay zero.  Inputs of exponent 2^1009 and above
// (infinities and NaN among them) give NaN; bits below 2^-953 are cut off.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace lbve {

// ---- block fixed point -------------------------------------------------------
constexpr int kFixMinE = 128 << 20;   // smallest block exponent (in place, biased)
constexpr int kFixMaxE = 2032 << 20;  // from here on: not finite

// Exponent field of a float64 value, in place.
__device__ __forceinline__ int fix_exponent(double d) { return __double2hiint(d) & 0x7ff00000; }

// Block exponent of N values.
template <int N>
__device__ __forceinline__ int fix_block(const double* d) {
  int e = kFixMinE;
#pragma unroll
  for (int i = 0; i < N; ++i) e = max(e, fix_exponent(d[i]));
  return e;
}

// d in units of 2^(E - 1023 - 58), E the block exponent: magnitude below 2^59.
__device__ __forceinline__ int64_t fix_from(double d, int block) {
  const int hi = __double2hiint(d);
  const unsigned lo = (unsigned)__double2loint(d);
  const unsigned vh = __funnelshift_l(lo, (unsigned)hi, 11) | 0x80000000u;  // leading bit at 63
  const unsigned sh = (unsigned)(block + (5 << 20) - (hi & 0x7ff00000)) >> 20;
  uint64_t v = ((uint64_t)vh << 32) | (lo << 11);
  asm("shr.u64 %0, %1, %2;" : "=l"(v) : "l"(v), "r"(sh));  // 0 from 64 on
  const int64_t s = (int64_t)(hi >> 31);
  return ((int64_t)v ^ s) - s;
}

// v in those units times 2^SCALE, rounded to nearest even; nan: 0, or the
// bits of a NaN's high word.
template <int SCALE>
__device__ __forceinline__ double fix_to(int64_t v, int block, int nan) {
  const int s = (int)(v >> 63);
  const uint64_t a = (uint64_t)((v ^ (int64_t)s) - (int64_t)s);
  const int k = __clzll((long long)a);
  uint64_t w;
  asm("shl.b64 %0, %1, %2;" : "=l"(w) : "l"(a), "r"(k));  // leading bit at 63
  const uint64_t q = w >> 11;
  const unsigned up = (((unsigned)w & 0x7ffu) + ((unsigned)q & 1u) + 0x3ffu) >> 11;
  // bit 52 of q adds the implicit one to the exponent field
  const int t = a == 0 ? 0 : block + ((4 + SCALE) << 20) - (k << 20);
  const uint64_t r = q + ((uint64_t)(uint32_t)t << 32) + up;
  return __hiloint2double((int)(r >> 32) | (s & (int)0x80000000) | nan, (int)(uint32_t)r);
}

__device__ __forceinline__ int64_t twice_minus(int64_t a, int64_t b) { return a + a - b; }

// ---- the transforms ----------------------------------------------------------------
// Moments of the nine (deviation) populations of one lattice: the sum, the
// first moments, 3 sum e_x^2 d - sum d and its y counterpart (three times the
// second moment's part off c_s^2), sum e_x e_y d, and for the hydrodynamic
// lattice three times the third moments' parts off c_s^2.  23 additions
// (hydrodynamic) or 21.
template <typename T>
struct Moments {
  T drho, jx, jy, nxx, nyy, pxy, nxxy, nxyy;
};

template <typename T>
__device__ __forceinline__ void moment_sums(const T d[9], Moments<T>& m) {
  const T a13 = d[1] + d[3], b13 = d[1] - d[3], a24 = d[2] + d[4], b24 = d[2] - d[4];
  const T p57 = d[5] + d[7], m57 = d[5] - d[7], p68 = d[6] + d[8], m68 = d[6] - d[8];
  const T s = p57 + p68, xxy = m57 + m68, xyy = m57 - m68;
  const T pxx = a13 + s, pyy = a24 + s, zx = a24 + d[0], zy = a13 + d[0];
  m.drho = pxx + zx;
  m.jx = b13 + xyy;
  m.jy = b24 + xxy;
  m.nxx = twice_minus(pxx, zx);
  m.nyy = twice_minus(pyy, zy);
  m.pxy = p57 - p68;
  m.nxxy = twice_minus(xxy, b24);
  m.nxyy = twice_minus(xyy, b13);
}

// The nine populations of Hermite coefficients scaled to their weights:
//   a = b0/9, x = bx/3, y = by/3, xx = bxx/3, yy = byy/3, xy = bxy,
//   xxy = bxxy, xyy = bxyy (xxy, xyy only with THIRD);
// out[0] comes halved, out[1..4] doubled, out[5..8] times four.  Adding the
// pieces in this form takes no multiplication.  The scaled weights 1/9 and 1/3
// have the same relative rounding error (5.6e-17) as the products with 1/9 and
// 1/36 of the unscaled form.
template <typename T, bool THIRD>
__device__ __forceinline__ void population_sums(T a, T x, T y, T xx, T yy, T xy, T xxy, T xyy,
                                                T out[9]) {
  const T h = xx + yy, s = a + h;
  out[0] = twice_minus(a, h);
  const T e13 = twice_minus(a + xx, yy), e24 = twice_minus(a + yy, xx);
  const T o13 = THIRD ? twice_minus(x, xyy) : x + x, o24 = THIRD ? twice_minus(y, xxy) : y + y;
  out[1] = e13 + o13;
  out[3] = e13 - o13;
  out[2] = e24 + o24;
  out[4] = e24 - o24;
  const T xs = THIRD ? x + xyy : x, ys = THIRD ? y + xxy : y;
  const T e57 = s + xy, e68 = s - xy, o57 = xs + ys, o68 = ys - xs;
  out[5] = e57 + o57;
  out[7] = e57 - o57;
  out[6] = e68 + o68;
  out[8] = e68 - o68;
}

// ---- float64 values in and out ---------------------------------------------------
template <bool THIRD>
__device__ __forceinline__ void lattice_moments(const double d[9], Moments<double>& m) {
  const int e = fix_block<9>(d), nan = e >= kFixMaxE ? 0x7ff80000 : 0;
  int64_t v[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) v[i] = fix_from(d[i], e);
  Moments<int64_t> s;
  moment_sums<int64_t>(v, s);
  m.drho = fix_to<0>(s.drho, e, nan);
  m.jx = fix_to<0>(s.jx, e, nan);
  m.jy = fix_to<0>(s.jy, e, nan);
  m.nxx = fix_to<0>(s.nxx, e, nan);
  m.nyy = fix_to<0>(s.nyy, e, nan);
  m.pxy = fix_to<0>(s.pxy, e, nan);
  if (THIRD) {
    m.nxxy = fix_to<0>(s.nxxy, e, nan);
    m.nxyy = fix_to<0>(s.nxyy, e, nan);
  }
}

template <bool THIRD>
__device__ __forceinline__ void lattice_populations(double a, double x, double y, double xx,
                                                    double yy, double xy, double xxy, double xyy,
                                                    double out[9]) {
  const double c[8] = {a, x, y, xx, yy, xy, xxy, xyy};
  const int e = fix_block<THIRD ? 8 : 6>(c), nan = e >= kFixMaxE ? 0x7ff80000 : 0;
  int64_t v[8] = {0, 0, 0, 0, 0, 0, 0, 0}, o[9];
#pragma unroll
  for (int i = 0; i < (THIRD ? 8 : 6); ++i) v[i] = fix_from(c[i], e);
  population_sums<int64_t, THIRD>(v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7], o);
  out[0] = fix_to<1>(o[0], e, nan);
#pragma unroll
  for (int i = 1; i < 5; ++i) out[i] = fix_to<-1>(o[i], e, nan);
#pragma unroll
  for (int i = 5; i < 9; ++i) out[i] = fix_to<-2>(o[i], e, nan);
}

}  // namespace lbve
