// Quotients in FP64, correctly rounded (parity mode rounds like the FP64
// reference), without the true division's operations: a true division takes
// about 10, and a cell has 55 of them on a pipe with 1/64 of the FP32 rate.
// Plain C++ too (compiled without contraction), so that it can be checked against
// the division on the host.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#include "lbe_two.cuh"  // LBE_HD

namespace lbe {

LBE_HD uint32_t hi_word(double a) {
#ifdef __CUDA_ARCH__
  return (uint32_t)__double2hiint(a);
#else
  uint64_t u;
  memcpy(&u, &a, 8);
  return (uint32_t)(u >> 32);
#endif
}
LBE_HD uint32_t lo_word(double a) {
#ifdef __CUDA_ARCH__
  return (uint32_t)__double2loint(a);
#else
  uint64_t u;
  memcpy(&u, &a, 8);
  return (uint32_t)u;
#endif
}
// 2^lo <= |a| < 2^(lo + n), by the exponent
LBE_HD bool exponent_in(double a, int lo, uint32_t n) {
  return ((hi_word(a) >> 20) & 0x7ffu) - (uint32_t)(1023 + lo) < n;
}
LBE_HD bool is_zero(double a) { return ((hi_word(a) << 1) | lo_word(a)) == 0u; }

#ifdef __CUDACC__
static __host__ __device__ __noinline__ double div_full(double a, double b) { return a / b; }
#else
static inline double div_full(double a, double b) { return a / b; }
#endif

// a / b for a divisor 2^-60 <= |b| < 2^60 whose rounded reciprocal y = RN(1/b) is
// at hand: Markstein's iteration (P. Markstein, IBM J. Res. Dev. 34, 1990).  If q
// is within one unit in the last place of a/b, the remainder r = a - b q is
// exact and RN(q + r y) = RN(a/b).  q = RN(a y) is that close where the
// residual |1 - b y| <= 2^-54 (kind 1: 3 operations); any other y needs one
// more iteration first (kind 2: 5).  Outside 2^-900 <= |a| < 2^900, where a
// remainder could underflow, the true division.
template <int KIND>
LBE_HD double div_by(double a, double b, double y) {
  const double q0 = a * y;
  double q = fma(fma(-b, q0, a), y, q0);
  if (KIND == 2) q = fma(fma(-b, q, a), y, q);
  if (exponent_in(a, -900, 1800u)) return q;
  // zero of the right sign (q is +0 for both)
  if (is_zero(a)) return q0;
  return div_full(a, b);
}
// a / fl(1/3), correctly rounded, in 2 operations.  fl(1/3) = (1 - 2^-54)/3, so
// the quotient is 3 a + 3 a 2^-54 (1 + 2^-54 + ...), and 3 a is a multiple of a
// quarter of the result's last place (ulp) while the second term lies between
// a quarter and a half of it: rounding that term to a product and adding it in
// one fused operation could miss a rounding boundary only where it is within
// 2^-53 of ulp/4 or ulp/2, that is for 3 a next to a power of two, where
// divisibility by 3 excludes the cases.  Below 2^-900 the true division.
LBE_HD double dv_cs2(double a) {
  const double q = fma(3.0, a, a * 0x1.8p-53);
  // (for a zero q is the zero of the same sign)
  if (((hi_word(a) >> 20) & 0x7ffu) < 123u && !is_zero(a)) return div_full(a, 1.0 / 3.0);
  return q;
}

// A divisor b: y = 1/b (FP64: rounded) and the kind: 1, 2 as above, 0 for b =
// 1, 4 for b = fl(1/3), 3 for the true division.
template <class C>
struct Den {
  C b, y;
  int kind;
};
LBE_HD double dv(double a, const Den<double>& d) {
  if (d.kind == 0) return a;
  if (d.kind == 4) return dv_cs2(a);
  return d.kind == 1 ? div_by<1>(a, d.b, d.y) : (d.kind == 2 ? div_by<2>(a, d.b, d.y) : a / d.b);
}
// The kind of a constant divisor b > 0 with y = RN(1/b) (on the host), and that
// of a cell's, which any y serves.
inline int constant_kind(double b, double y) {
  if (b == 1.0) return 0;
  if (b == 1.0 / 3.0) return 4;
  if (!exponent_in(b, -60, 120u)) return 3;
  return std::fabs(std::fma(-b, y, 1.0)) <= std::ldexp(1.0, -54) ? 1 : 2;
}
LBE_HD int cell_kind(double b) { return exponent_in(b, -60, 120u) ? 2 : 3; }

}  // namespace lbe
