// Exact sums of doubles (or floats) in 64-bit fixed point (sm_103a).
//
// GB300 executes two FP64 operations per clock and SM, 64 times fewer than
// integer ones, so sums of f's values run on the integer ALUs.  The values of
// one sum are aligned to the largest exponent among them, E: v = n 2^(E -
// 1079), |n| < 2^57, which holds all 53 bits of values down to 2^-4 of the
// largest (floats: all 24 bits down to 2^-33) and truncates smaller ones below
// 2^-56 of it (the moments' sums: two bits more): no more than the rounding of
// one double addition of the largest.  The sum of the aligned values times
// coefficients whose magnitudes sum to less than 64 is exact, and is rounded
// once, to 53 bits, when it
// becomes a double; a double evaluation rounds at each operation, at 2^-53 of
// its operands.  Sums whose largest exponent is outside [EMIN, EMAX]
// (non-finite, or beyond 1e-247 .. 1e264; for floats non-finite or below 1e-19)
// take a double evaluation.
#pragma once

#include "lbm_internal.cuh"

namespace lbm {
namespace fx {

constexpr int EMIN = 200, EMAX = 1900;
// S: 53-bit mantissas' top bit at bit 52 + S; n counts units of 2^(E - bias(S)).
// Sums of coefficients below 64 use SHIFT, plain sums of a cell's 15 values
// MOMENT_SHIFT, which truncates four times less (FP64 moments of 82 thousand
// noisy cells against quad precision, relative 2-norm of u: on one scale for
// all of a cell's sums SHIFT 9.0e-16, MOMENT_SHIFT 2.1e-16; on a scale per sum
// MOMENT_SHIFT 1.0e-16; double sums 5.3e-16).
constexpr int SHIFT = 4, MOMENT_SHIFT = 6;
constexpr int bias(int S) { return 1023 + 52 + S; }

// Magnitude pattern of a value (of a double its high word), which orders like
// the magnitudes' exponents, and the double-biased exponent E of the largest.
__device__ __forceinline__ int mag(double v) { return __double2hiint(v) & 0x7fffffff; }
__device__ __forceinline__ int mag(float v) { return __float_as_int(v) & 0x7fffffff; }
template <typename R>
__device__ __forceinline__ int exponent_of(int largest) {
  return sizeof(R) == 8 ? largest >> 20 : (largest >> 23) + (1023 - 127);
}
__device__ __forceinline__ bool in_range(int E) { return E >= EMIN && E <= EMAX; }
template <typename R>
__device__ __forceinline__ bool in_range_of(int E) {
  return sizeof(R) == 8 ? in_range(E) : E >= 64 + (1023 - 127) && E < 255 + (1023 - 127);
}

__device__ __forceinline__ long long aligned(unsigned long long n, unsigned sh, int sign_word) {
  asm("shr.u64 %0, %0, %1;" : "+l"(n) : "r"(sh));  // PTX clamps the shift at 64
  const long long s = sign_word >> 31;
  return ((long long)n ^ s) - s;
}

// v in units of 2^(E - bias(S)), truncated toward zero; E is in range and at
// least v's exponent (zeros and subnormals are shifted out).
template <int S = SHIFT>
__device__ __forceinline__ long long to_fixed(double v, int E) {
  const int h = __double2hiint(v);
  const unsigned l = (unsigned)__double2loint(v);
  const unsigned long long n = (((unsigned long long)(((unsigned)h & 0xfffffu) | 0x100000u) << 32) | l) << S;
  return aligned(n, (unsigned)(E - (mag(v) >> 20)), h);
}
template <int S = SHIFT>
__device__ __forceinline__ long long to_fixed(float v, int E) {
  const int b = __float_as_int(v);
  const unsigned long long n = (unsigned long long)(((unsigned)b & 0x7fffffu) | 0x800000u) << (S + 29);
  return aligned(n, (unsigned)(E - (1023 - 127) - (mag(v) >> 23)), b);
}

// The same for a value that a limiter compares and does not add: its exponent
// may be above E, and from 2^(E + 4) on it saturates at [2^59, 2^60) units, more
// than twice any difference of two values of exponents up to E.
__device__ __forceinline__ long long to_fixed_limiter(double v, int E) {
  constexpr int UP = 3;
  const int h = __double2hiint(v);
  const unsigned l = (unsigned)__double2loint(v);
  const unsigned long long n = (((unsigned long long)(((unsigned)h & 0xfffffu) | 0x100000u) << 32) | l) << (SHIFT + UP);
  return aligned(n, (unsigned)max(E + UP - (mag(v) >> 20), 0), h);
}

// n 2^(E - bias(S)), rounded to 53 bits (a tie away from zero).
template <int S = SHIFT>
__device__ __forceinline__ double from_fixed(long long n, int E) {
  const long long s = n >> 63;
  unsigned long long a = (unsigned long long)((n ^ s) - s);
  const int lz = __clzll((long long)a);
  a = a << (lz & 63);
  // top bit 63 - lz: biased exponent E - bias(S) + 1023 + 63 - lz, less one for
  // the mantissa's leading bit, which the sum below adds to it
  const unsigned e = (unsigned)(E - bias(S) + 1023 + 62 - lz);
  const unsigned long long q = (a >> 11) + ((a >> 10) & 1ull);  // a carry to 2^53 raises the exponent
  const unsigned hi = ((unsigned)(q >> 32) + (e << 20)) | ((unsigned)(s >> 32) & 0x80000000u);
  return a == 0 ? 0.0 : __hiloint2double((int)hi, (int)(unsigned)q);
}

// n in units 2^sh times as large, rounded down
__device__ __forceinline__ long long lowered(long long n, int sh) {
  asm("shr.s64 %0, %0, %1;" : "+l"(n) : "r"(sh));  // PTX clamps the shift at 64
  return n;
}

// rho, u and T of a cell's 15 values (relations e1-e3), the sums in fixed
// point: 28 of the FP64 operations a cell's moments take.  Each sum has the
// scale of its own values, so that none loses bits to a value it does not hold:
// the two of an axis in a momentum component, the six axis values in the
// energy, the eight diagonal ones, all in rho (on one scale for all, u had a
// median relative error of 2.5e-15 where f_0 is 1e3 times the rest, on these
// 1.0e-16, in double sums 4.6e-16; no difference in time on 256^3 moments or in
// the FP64 step).
template <typename R>
__device__ __forceinline__ void moments_fixed(const Model<double>& m, const R f[NV], double& rho, double& ux,
                                              double& uy, double& uz, double& T) {
  int pair[3], diag = mag(f[7]);
#pragma unroll
  for (int a = 0; a < 3; ++a) pair[a] = max(mag(f[1 + 2 * a]), mag(f[2 + 2 * a]));
#pragma unroll
  for (int i = 8; i < NV; ++i) diag = max(diag, mag(f[i]));
  const int axes = max(max(pair[0], pair[1]), pair[2]);
  const int smallest = min(min(pair[0], pair[1]), min(pair[2], diag));
  const int E = exponent_of<R>(max(max(axes, diag), mag(f[0])));
  if (!in_range_of<R>(E) || !in_range_of<R>(exponent_of<R>(smallest))) {
    double v[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = (double)f[i];
    moments(m, v, rho, ux, uy, uz, T);
    return;
  }
  auto sum = [](long long n, int e) { return from_fixed<MOMENT_SHIFT>(n, e); };
  const int EA = exponent_of<R>(axes), ED = exponent_of<R>(diag);
  long long sa = 0;
  double pa[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int e = exponent_of<R>(pair[a]);
    const long long p = to_fixed<MOMENT_SHIFT>(f[1 + 2 * a], e), q = to_fixed<MOMENT_SHIFT>(f[2 + 2 * a], e);
    pa[a] = sum(p - q, e);
    sa += lowered(p + q, EA - e);
  }
  long long n[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) n[i] = to_fixed<MOMENT_SHIFT>(f[7 + i], ED);
  const long long pp = n[0] + n[1], pm = n[2] + n[3], mp = n[4] + n[5], mm = n[6] + n[7];
  const long long sd = (pp + pm) + (mp + mm);
  const long long dz = ((n[0] + n[2]) + (n[4] + n[6])) - ((n[1] + n[3]) + (n[5] + n[7]));
  const long long n0 = to_fixed<MOMENT_SHIFT>(f[0], E);
  rho = sum(n0 + lowered(sa, E - EA) + lowered(sd, E - ED), E);
  const double px = fma(m.c1, pa[0], m.s * sum((pp + pm) - (mp + mm), ED));
  const double py = fma(m.c1, pa[1], m.s * sum((pp + mp) - (pm + mm), ED));
  const double pz = fma(m.c1, pa[2], m.s * sum(dz, ED));
  const double f0 = sizeof(R) == 8 ? (double)f[0] : sum(n0, E);
  const double en = fma(m.eta0sq, f0, fma(m.c1sq, sum(sa, EA), m.c2sq * sum(sd, ED)));
  const double ir = 1.0 / rho;
  ux = px * ir;
  uy = py * ir;
  uz = pz * ir;
  T = (en * ir - fma(ux, ux, fma(uy, uy, uz * uz))) * m.inv_b;
}

}  // namespace fx
}  // namespace lbm
