// Correctly rounded FP64 division by a divisor that one launch shares (internal).
#pragma once

#include <cmath>

namespace saamg {

// a / c for one positive c and many a, with the bits of the IEEE division.  The FP64 pipe issues
// two lanes per clock and SM, and a general division is a dozen dependent instructions on it; with
// the correctly rounded reciprocal r = RN(1 / c) formed once on the host, one multiplication and
// two fused multiply-adds give RN(a / c) (Markstein's correction step; Brisebarre, Muller and
// Raina, "Accelerating correctly rounded floating-point division when the divisor is known in
// advance", IEEE Trans. Computers 53, 2004), as long as the remainder a - q c is exact.  Where c
// is a power of two, a * r is the quotient itself.  Every other operand -- zero, subnormal or
// huge a, infinities, NaN, an extreme c -- takes the division.
struct DivC {
  double c, r;
  int kind;  // 0: correction step, 1: c is a power of two, 2: always the division
};

inline DivC make_divc(double c) {
  DivC d;
  d.c = c;
  d.r = 1.0 / c;
  int e = 0;
  const bool fin = std::isfinite(c) && c > 0.0;
  const double m = fin ? std::frexp(c, &e) : 0.0;
  if (!fin || e < -400 || e > 400) d.kind = 2;
  else d.kind = m == 0.5 ? 1 : 0;
  return d;
}

__device__ __forceinline__ double div_by(double a, const DivC& d) {
  if (d.kind == 1) return __dmul_rn(a, d.r);
  const unsigned e = (static_cast<unsigned>(__double2hiint(a)) >> 20) & 0x7ffu;
  // 2^-511 <= |a| < 2^512: neither q nor the remainder leaves the normal range
  if (d.kind == 0 && e - 512u < 1023u) {
    const double q = __dmul_rn(a, d.r);
    return __fma_rn(__fma_rn(-d.c, q, a), d.r, q);
  }
  if (d.kind == 0 && (static_cast<unsigned long long>(__double_as_longlong(a)) << 1) == 0ull)
    return a;  // a zero keeps its sign
  return __ddiv_rn(a, d.c);
}

}  // namespace saamg
