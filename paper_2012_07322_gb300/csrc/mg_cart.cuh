// The 7-point FP64 Laplacian of equal spacings on the integer units.
//
// GB300 issues 2 FP64 operations per SM and clock against 64 integer ones, so
// an FP64 stencil is bound by its additions.  Here the seven values of a
// stencil become 64-bit integers aligned to the largest of their exponents
// (53 mantissa bits, 6 guard bits below, 4 bits of headroom above), the sum
// of the six neighbours minus six times the centre is taken exactly in
// integers, and one conversion, one multiply-add give f - c S.  Each value is
// cut below 2^-58 of the largest one, so the sum is off by less than 2^-54 of
// it before its own rounding; the flux form rounds every difference and every
// partial sum at 2^-53 of their magnitude.  (When all seven values have the
// same exponent, as away from zeros, nothing is cut and S is exact.)
#pragma once
#include "mg_dev.cuh"

namespace gmg {

// Signed mantissa with 6 guard bits, value = m 2^(e - 1081).
struct Fixed {
  long long m;
  int e;
};
__device__ __forceinline__ Fixed fix_decode(double v) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const int e = (int)((hi >> 20) & 0x7ffu);
  const unsigned mh = (hi & 0xfffffu) | (e ? 0x100000u : 0u);
  const unsigned long long a = (((unsigned long long)mh << 32) | lo) << 6;
  const long long s = (long long)((int)hi >> 31);
  Fixed o;
  o.m = ((long long)a ^ s) - s;
  o.e = e ? e : 1;
  return o;
}
__device__ __forceinline__ long long fix_align(const Fixed& v, int E) {
  const int s = E - v.e;
  return v.m >> (s < 63 ? s : 63);
}

// Exponent range handled: everything finite and not tiny (the scaled
// coefficient must be a normal number); others take the flux form.
constexpr int FIX_E_MIN = 128, FIX_E_MAX = 0x7fe;

// S = e + w + n + s + up + dn - 6 c, as S 2^(E - 1081); false when an
// operand is not finite or all are tiny (then nothing is computed).
__device__ __forceinline__ bool fix_sum(const Fixed& c, const Fixed& e, const Fixed& w, const Fixed& n, const Fixed& s,
                                        const Fixed& up, const Fixed& dn, long long& S, int& E) {
  E = max(max(max(c.e, e.e), max(w.e, n.e)), max(max(s.e, up.e), dn.e));
  if (E < FIX_E_MIN || E > FIX_E_MAX) return false;
  const long long a = fix_align(c, E);
  S = ((fix_align(e, E) + fix_align(w, E)) + (fix_align(n, E) + fix_align(s, E))) +
      ((fix_align(up, E) + fix_align(dn, E)) - ((a << 2) + (a << 1)));
  return true;
}
// cf 2^(E - 1081), cf a normal number of moderate size (1 / h^2).
__device__ __forceinline__ double fix_scale(double cf, int E) {
  return __hiloint2double(__double2hiint(cf) + ((E - 1081) << 20), __double2loint(cf));
}
// res = fv - cf S.
__device__ __forceinline__ bool fix_residual(const Fixed& c, const Fixed& e, const Fixed& w, const Fixed& n,
                                             const Fixed& s, const Fixed& up, const Fixed& dn, double cf, double fv,
                                             double& res) {
  long long S;
  int E;
  if (!fix_sum(c, e, w, n, s, up, dn, S, E)) return false;
  const int x = ((__double2hiint(cf) >> 20) & 0x7ff) + E - 1081;
  if (x < 1 || x > 2046) return false;
  res = fma(-fix_scale(cf, E), (double)S, fv);
  return true;
}

}  // namespace gmg
