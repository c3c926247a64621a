// lbve_linear.cuh -- the linear parts of a float64 step (populations to
// moments, Hermite coefficients to populations) in 64-bit block fixed point.
//
// One SM retires a float64 instruction of a warp every 19.0 cycles, an integer
// instruction every 0.52 (measured with independent chains, 4 to 32 warps;
// both pipes run side by side).  A
// transform of nine populations is 21 to 23 additions, so it costs 400 to 440
// cycles on the float64 pipe.  In fixed point the values are aligned once to the
// largest exponent among them (13 integer instructions each), added exactly
// as 64-bit integers, and each result is rounded once to float64 (25
// instructions), on a pipe that is otherwise idle.  The step of the batched mix
// (64 instances) went from 2.54 to 1.2 ms with it.
//   Precision: the largest input's leading bit sits at bit 58, i.e. 6 bits
// below its last float64 bit are kept, and the sums are exact.  An input more
// than 2^6 smaller than the largest one is rounded to nearest there, ties away
// from zero: by at most 2^-59 of the largest one, and on average by no more than
// half a last place of the input itself (the ties).  The float64 additions
// replaced here round every partial sum at 2^-53 of its size.  The rounding must
// not have a sign: with the bits cut off (half a unit toward zero on average), the
// zeroth coefficient beside rho u / 3 lost size at every collision and the density
// of slow flows was off.  Relative error of rho - 1 after 2000 steps of a
// hydrodynamic mill (quadruple precision as reference; float64 additions, cut
// off, rounded): 32^2 at Ma 0.01, Re 1: 5.7e-14, 1.2e-13, 5.0e-14; 32^2 at
// Ma 0.001, Re 0.1: 4.0e-13, 1.3e-12, 3.5e-13; 16^2 at Ma 0.001, Re 1: 1.6e-12,
// 2.3e-12, 1.6e-12.  Ties to even take 5 instructions more per input and no
// smaller error (5.0e-14, 3.2e-13, 1.5e-12; the mix 5 % slower).
// Results round to nearest even.  Exact zeros stay zero.  Inputs of exponent
// 2^1020 and above (infinities and NaN among them) give NaN, where float64
// additions would still have a finite sum up to 2^1024; below 2^-959 the last place
// is 2^-1017 whatever the largest value (kFixMinE).
//   The functions also compile for the host, where the tests compare them with
// exact arithmetic.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>

namespace lbve {

// ---- words of a float64 value, shifts that give 0 from 64 on ------------------
#define LBVE_HD __host__ __device__ __forceinline__
LBVE_HD int high_word(double d) {
#ifdef __CUDA_ARCH__
  return __double2hiint(d);
#else
  uint64_t b;
  std::memcpy(&b, &d, sizeof(b));
  return (int)(uint32_t)(b >> 32);
#endif
}
LBVE_HD unsigned low_word(double d) {
#ifdef __CUDA_ARCH__
  return (unsigned)__double2loint(d);
#else
  uint64_t b;
  std::memcpy(&b, &d, sizeof(b));
  return (unsigned)b;
#endif
}
LBVE_HD double from_words(int hi, unsigned lo) {
#ifdef __CUDA_ARCH__
  return __hiloint2double(hi, (int)lo);
#else
  const uint64_t b = ((uint64_t)(uint32_t)hi << 32) | lo;
  double d;
  std::memcpy(&d, &b, sizeof(d));
  return d;
#endif
}
LBVE_HD unsigned top_word(int hi, unsigned lo) {  // bits 21 to 52
#ifdef __CUDA_ARCH__
  return __funnelshift_l(lo, (unsigned)hi, 11);
#else
  return ((unsigned)hi << 11) | (lo >> 21);
#endif
}
LBVE_HD uint64_t shift_right(uint64_t v, unsigned n) {
#ifdef __CUDA_ARCH__
  asm("shr.u64 %0, %1, %2;" : "=l"(v) : "l"(v), "r"(n));
  return v;
#else
  return n < 64 ? v >> n : 0;
#endif
}
LBVE_HD uint64_t shift_left(uint64_t v, unsigned n) {
#ifdef __CUDA_ARCH__
  asm("shl.b64 %0, %1, %2;" : "=l"(v) : "l"(v), "r"(n));
  return v;
#else
  return n < 64 ? v << n : 0;
#endif
}
LBVE_HD int leading_zeros(uint64_t v) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)v);
#else
  return v == 0 ? 64 : __builtin_clzll(v);
#endif
}

// ---- block fixed point -------------------------------------------------------
// Smallest block exponent (in place, biased): the smallest result, a quarter of
// the unit 2^-1017, is still a normal number.
constexpr int kFixMinE = 64 << 20;
// Not finite from here on: the largest sum, that of n_xx over 15 inputs, would
// leave the range of float64.
constexpr int kFixMaxE = 2043 << 20;

// Exponent field of a float64 value, in place.
LBVE_HD int fix_exponent(double d) { return high_word(d) & 0x7ff00000; }

// Block exponent of N values.
template <int N>
LBVE_HD int fix_block(const double* d) {
  int e = kFixMinE;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const int f = fix_exponent(d[i]);
    e = f > e ? f : e;
  }
  return e;
}

// d in units of 2^(E - 1023 - 58), E the block exponent, rounded to nearest,
// ties away from zero: magnitude at most 2^59.  The shift leaves one bit more (the
// first of those dropped), which the last line adds to the magnitude: -r = ~r + 1.
LBVE_HD int64_t fix_from(double d, int block) {
  const int hi = high_word(d);
  const unsigned lo = low_word(d);
  const unsigned vh = top_word(hi, lo) | 0x80000000u;  // leading bit at 63
  const unsigned sh = ((unsigned)block + (4u << 20) - ((unsigned)hi & 0x7ff00000u)) >> 20;
  const uint64_t r = shift_right(((uint64_t)vh << 32) | (lo << 11), sh);
  const int64_t s = (int64_t)(hi >> 31);
  return (int64_t)((r ^ (uint64_t)s) + 1) >> 1;
}

// v in those units times 2^SCALE, rounded to nearest even; nan: 0, or the
// bits of a NaN's high word.
template <int SCALE>
LBVE_HD double fix_to(int64_t v, int block, int nan) {
  const int s = (int)(v >> 63);
  const uint64_t a = (uint64_t)((v ^ (int64_t)s) - (int64_t)s);
  const int k = leading_zeros(a);
  const uint64_t w = shift_left(a, (unsigned)k);  // leading bit at 63
  const uint64_t q = w >> 11;
  const unsigned up = (((unsigned)w & 0x7ffu) + ((unsigned)q & 1u) + 0x3ffu) >> 11;
  // bit 52 of q adds the implicit one to the exponent field
  const unsigned t = a == 0 ? 0u : (unsigned)block + ((4u + SCALE) << 20) - ((unsigned)k << 20);
  const uint64_t r = q + ((uint64_t)t << 32) + up;
  return from_words((int)(r >> 32) | (s & (int)0x80000000) | nan, (unsigned)r);
}

LBVE_HD int64_t twice_minus(int64_t a, int64_t b) { return a + a - b; }

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
LBVE_HD void moment_sums(const T d[9], Moments<T>& m) {
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
LBVE_HD void population_sums(T a, T x, T y, T xx, T yy, T xy, T xxy, T xyy, T out[9]) {
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
LBVE_HD void lattice_moments(const double d[9], Moments<double>& m) {
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
LBVE_HD void lattice_populations(double a, double x, double y, double xx, double yy, double xy,
                                 double xxy, double xyy, double out[9]) {
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

#undef LBVE_HD

}  // namespace lbve
