// Plain fused steps: one thread per interior cell, neighbours read straight
// from global memory.  Per cell and per velocity i (Secs. 2-3): moments ->
// f^eq -> NND convection along every axis with v_ia != 0 -> lambda_i
// Laplacian (i = 0..6) -> BGK + forward Euler, written to fout.
// step_plain_kernel is the single-precision cross-check variant;
// step_fp64_kernel is the double-precision path.
#include "fixed_sum.cuh"

namespace lbm {
namespace {

template <int SCHEME>
__global__ void __launch_bounds__(256) step_plain_kernel(const float* __restrict__ fin, float* __restrict__ fout,
                                                         Layout L, Model<float> m, unsigned* __restrict__ flags) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z;
  if (x >= L.nx || y >= L.ny) return;
  const long long c = L.at(x, y, z);
  const long long step[3] = {1, (long long)L.sx, L.plane};

  float f[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) f[i] = __ldg(fin + i * L.fs + c);

  float rho, ux, uy, uz, T;
  moments(m, f, rho, ux, uy, uz, T);
  {
    unsigned bad = 0u;
    if (!(rho > 0.f)) bad |= LBM_HEALTH_RHO;
    if (!(T > 0.f)) bad |= LBM_HEALTH_T;
    if (!(fabsf(rho) + fabsf(T) + fabsf(ux) + fabsf(uy) + fabsf(uz) < 1e30f)) bad |= LBM_HEALTH_NONFINITE;
    if (bad) atomicOr(flags, bad);
  }
  float feq[NV];
  equilibrium(m, rho, ux, uy, uz, T, feq);

#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const float* __restrict__ p = fin + i * L.fs + c;
    const float fc = f[i];
    float conv = 0.f, nb = 0.f;  // nb: the six neighbours' sum (dissipation, i <= 6)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int sg = vsign(i, a);
      const long long d = step[a];
      if (sg > 0) {
        const float m2 = __ldg(p - 2 * d), m1 = __ldg(p - d), p1 = __ldg(p + d);
        conv += grad_pos<SCHEME>(m2, m1, fc, p1);
        if (i <= 6) nb += p1 + m1;
      } else if (sg < 0) {
        const float m1 = __ldg(p - d), p1 = __ldg(p + d), p2 = __ldg(p + 2 * d);
        conv -= grad_neg<SCHEME>(m1, fc, p1, p2);
        if (i <= 6) nb += p1 + m1;
      } else if (i <= 6) {
        nb += __ldg(p + d) + __ldg(p - d);
      }
    }
    const float k = i == 0 ? 0.f : (i <= 6 ? m.k1 : m.k2);
    const float lam = i == 0 ? m.lam0 : (i <= 6 ? m.lam1 : 0.f);
    // f + dt/tau (f^eq - f) - (|v| dt/dx) conv + (lambda dt/dx^2)(nb - 6 f), with the
    // relaxation and the Laplacian's centre folded into keep = 1 - dt/tau - 6 lambda dt/dx^2;
    // conv holds sum_a sign(v_ia) * grad, the velocity magnitude is in k
    const float keep = i == 0 ? m.keep0 : (i <= 6 ? m.keep1 : m.keep2);
    float o = keep * fc + m.dt_tau * feq[i];
    if (i != 0) o -= k * conv;
    if (i <= 6) o += lam * nb;
    fout[i * L.fs + c] = o;
  }
}

// ---------------------------------------------------------------- double precision
//
// GB300 executes two FP64 operations per clock and SM, 64 times fewer than
// FP32 or integer ones, so the step is bound by the FP64 operations it needs
// and everything linear in f is taken off that pipe: the moments' sums, the
// convection's differences, minmods and sums, and the Laplacian, run in 64-bit
// fixed point (fixed_sum.cuh; the values aligned are those of a velocity's
// stencil, or of one of a cell's sums).  The largest sum, five times twice the convection of an
// axis velocity (|difference| <= 2, |minmod| <= |difference|) less its
// Laplacian, is at most 52 times the largest value (a diagonal velocity's
// convection 24 times).  256^3: 13.3 -> 4.2 ms per step (417 -> 112 FP64
// operations per cell; the FP64 pipe 84 -> 72 % busy, the integer ALUs 74 %:
// both near their rates); 300 x 80 x 80 with walls 1.68 -> 0.57 ms.
// Aligning by one multiplication where the values are within 2^4 of each other
// saves 900 of 3400 ALU instructions, but the cells at shocks and zero
// crossings send their warps through both forms (64^3 91 -> 104 us): not kept.
using fx::from_fixed;
using fx::in_range;
using fx::mag;
using fx::to_fixed;
using fx::to_fixed_limiter;

__device__ __forceinline__ long long clamp64(long long x, long long lo, long long hi) { return min(max(x, lo), hi); }

// Twice the one-sided gradient of Sec. 3 along one axis, upwind to downwind
// m2, m1, c, p1.  A negative velocity component's is the same with the axis
// reversed: -grad_neg(m1, c, p1, p2) = grad_pos(p2, p1, c, m1).
template <int SCHEME>
__device__ __forceinline__ long long grad2(long long m2, long long m1, long long c, long long p1) {
  const long long d = c - m1;
  if (SCHEME == LBM_SCHEME_UPWIND1) return 2 * d;
  if (SCHEME == LBM_SCHEME_UPWIND2) return 3 * d - (m1 - m2);
  const long long lo = min(d, 0ll), hi = max(d, 0ll);
  return 2 * d + (clamp64(p1 - c, lo, hi) - clamp64(m1 - m2, lo, hi));
}

// The same for three axes in double, for stencils outside the fixed-point range.
template <int SCHEME>
__device__ __noinline__ double conv2_double(double c, double x0, double x1, double x2, double y0, double y1, double y2,
                                            double z0, double z1, double z2) {
  return 2.0 * grad_pos<SCHEME>(x0, x1, c, x2) + 2.0 * grad_pos<SCHEME>(y0, y1, c, y2) +
         2.0 * grad_pos<SCHEME>(z0, z1, c, z2);
}

// Field offsets (32-bit, modulo 2^32: a field has fewer elements) of a cell's
// neighbours along one axis: [0..3] = -2, -1, +1, +2.
struct Nb {
  unsigned k[4];
};
__device__ __forceinline__ double at(const double* f, unsigned k) { return f[k]; }

// The values a velocity's update reads besides the cell's own, upwind to
// downwind m2, m1, p1 along each axis of a diagonal velocity; for an axis one
// m2, m1, p1 along its axis and the four lateral neighbours.  R..: reversed
// axes (negative components).
template <bool RX, bool RY, bool RZ>
__device__ __forceinline__ void diag_load(const double* f, const Nb& X, const Nb& Y, const Nb& Z,
                                          double v[9]) {
  v[0] = at(f, X.k[RX ? 3 : 0]); v[1] = at(f, X.k[RX ? 2 : 1]); v[2] = at(f, X.k[RX ? 1 : 2]);
  v[3] = at(f, Y.k[RY ? 3 : 0]); v[4] = at(f, Y.k[RY ? 2 : 1]); v[5] = at(f, Y.k[RY ? 1 : 2]);
  v[6] = at(f, Z.k[RZ ? 3 : 0]); v[7] = at(f, Z.k[RZ ? 2 : 1]); v[8] = at(f, Z.k[RZ ? 1 : 2]);
}
template <bool R>
__device__ __forceinline__ void axis_load(const double* f, const Nb& A, const Nb& B, const Nb& C,
                                          double v[9]) {
  v[0] = at(f, A.k[R ? 3 : 0]); v[1] = at(f, A.k[R ? 2 : 1]); v[2] = at(f, A.k[R ? 1 : 2]);
  v[3] = at(f, B.k[1]); v[4] = at(f, B.k[2]); v[5] = at(f, C.k[1]); v[6] = at(f, C.k[2]);
}

// The values that are added set the scale of a stencil.  m2 and p1 only bound
// the limited differences (NND), or do not enter (p1 of the upwind schemes, m2
// of the first-order one), so a large one costs the others no bits: with them
// in the scale, a neighbour K times the rest left the convection sum a relative
// error of K 2^-56.  UPWIND2 adds m2.
template <int SCHEME>
constexpr bool kAddsM2 = SCHEME == LBM_SCHEME_UPWIND2;
template <int SCHEME>
__device__ __forceinline__ long long fixed_m2(double v, int E) {
  return kAddsM2<SCHEME> ? to_fixed(v, E) : to_fixed_limiter(v, E);
}

// Twice the convection sum of a diagonal velocity.
template <int SCHEME>
__device__ __forceinline__ double diag_conv2(double c, const double v[9]) {
  int mx = mag(c);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    mx = max(mx, mag(v[3 * a + 1]));
    if (kAddsM2<SCHEME>) mx = max(mx, mag(v[3 * a]));
  }
  const int E = mx >> 20;
  if (!in_range(E)) return conv2_double<SCHEME>(c, v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7], v[8]);
  const long long n = to_fixed(c, E);
  long long s = 0;
#pragma unroll
  for (int a = 0; a < 3; ++a)
    s += grad2<SCHEME>(fixed_m2<SCHEME>(v[3 * a], E), to_fixed(v[3 * a + 1], E), n, to_fixed_limiter(v[3 * a + 2], E));
  return from_fixed(s, E);
}

// Convection and dissipation of an axis velocity.  With the dissipation term
// lambda_i = c1 dx / 10 (Sec. 3), so both terms are one multiple of lambda_i
// dt/dx^2 = |v| dt/(10 dx): returns 5 times twice the convection less the
// Laplacian, or twice the convection alone when the term is off.
template <int SCHEME>
__device__ __forceinline__ double axis_sum(double c, const double v[9], bool dissipation) {
  int mx = max(mag(c), mag(v[1]));
  if (kAddsM2<SCHEME>) mx = max(mx, mag(v[0]));
  if (dissipation) {
#pragma unroll
    for (int j = 2; j < 7; ++j) mx = max(mx, mag(v[j]));
  }
  const int E = mx >> 20;
  if (!in_range(E)) {
    const double conv2 = 2.0 * grad_pos<SCHEME>(v[0], v[1], c, v[2]);
    return dissipation ? 5.0 * conv2 - (((v[1] + v[2]) + (v[3] + v[4])) + (v[5] + v[6]) - 6.0 * c) : conv2;
  }
  const long long n = to_fixed(c, E), n1 = to_fixed(v[1], E), n2 = to_fixed_limiter(v[2], E);
  long long s = grad2<SCHEME>(fixed_m2<SCHEME>(v[0], E), n1, n, n2);
  if (dissipation) {
    s = 5 * s + 6 * n - (n1 + n2);
#pragma unroll
    for (int j = 3; j < 7; ++j) s -= to_fixed(v[j], E);
  }
  return from_fixed(s, E);
}

// The Laplacian of the rest velocity from its six neighbours.
__device__ __forceinline__ double rest_lap(double c, const double q[6]) {
  int mx = mag(c);
#pragma unroll
  for (int j = 0; j < 6; ++j) mx = max(mx, mag(q[j]));
  const int E = mx >> 20;
  if (!in_range(E)) return ((q[0] + q[1]) + (q[2] + q[3])) + (q[4] + q[5]) - 6.0 * c;
  long long s = -6 * to_fixed(c, E);
#pragma unroll
  for (int j = 0; j < 6; ++j) s += to_fixed(q[j], E);
  return from_fixed(s, E);
}

// Health bits of one cell.  The comparisons run on the values' high words;
// only a cell that is close to a limit takes the FP64 ones.
__device__ __forceinline__ unsigned health_fp64(double rho, double ux, double uy, double uz, double T) {
  const int hr = __double2hiint(rho), ht = __double2hiint(T);
  const int big = max(max(max(mag(rho), mag(T)), max(mag(ux), mag(uy))), mag(uz));
  if (hr >= 0x00100000 && ht >= 0x00100000 && big < (1023 + 97) << 20) return 0u;  // normal, below 2^97
  unsigned bad = 0u;
  if (!(rho > 0.0)) bad |= LBM_HEALTH_RHO;
  if (!(T > 0.0)) bad |= LBM_HEALTH_T;
  if (!(fabs(rho) + fabs(T) + fabs(ux) + fabs(uy) + fabs(uz) < 1e30)) bad |= LBM_HEALTH_NONFINITE;
  return bad;
}

// Offsets of cell `i` of `n` along an axis, its field offset k0 and the axis'
// element stride; periodic axes wrap here, others read the layers in memory.
__device__ __forceinline__ Nb neighbours(int i, int n, bool periodic, unsigned k0, unsigned stride) {
  Nb r;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    int o = j < 2 ? j - 2 : j - 1;
    if (periodic) {
      while (i + o < 0) o += n;
      while (i + o >= n) o -= n;
    }
    r.k[j] = k0 + (unsigned)o * stride;
  }
  return r;
}

// R1: dt = tau.  The velocities come in opposite pairs that share the even
// part of f^eq: three axis pairs and four diagonal ones, each a loop whose
// body serves all of its kind (the neighbour offsets and velocity components
// take turns), so the code stays short.  `parts` blocks share a row: 1, or 3
// (rest and axis pairs; two diagonal pairs each), each with the moments for
// itself.  kax, kdg: factors of axis_sum and diag_conv2.
template <int SCHEME, bool R1>
__global__ void __launch_bounds__(256, 3)
    step_fp64_kernel(const double* fin, double* __restrict__ fout, Layout L, Model<double> m, double kax,
                     double kdg, unsigned per, int parts, unsigned* __restrict__ flags) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = (blockIdx.y / parts) * blockDim.y + threadIdx.y;
  const int z = blockIdx.z, part = blockIdx.y % parts;
  // the axis pairs [0, a1) and diagonal pairs [d0, d1) of this part
  const int a1 = part == 0 ? 3 : 0;
  const int d0 = parts == 1 ? 0 : 2 * part - 2, d1 = parts == 1 ? 4 : 2 * part;
  chain_wait();
  if (x >= L.nx || y >= L.ny) return;
  const unsigned k0 = (unsigned)L.at(x, y, z);

  double rho, ux, uy, uz, T;
  {
    double f[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) f[i] = at(fin + i * L.fs, k0);
    fx::moments_fixed(m, f, rho, ux, uy, uz, T);
  }
  if (part == 0) {
    const unsigned bad = health_fp64(rho, ux, uy, uz, T);
    if (bad) atomicOr(flags, bad);
  }

  const Nb X = neighbours(x, L.nx, per & 1u, k0, 1u), Y = neighbours(y, L.ny, per & 2u, k0, (unsigned)L.sx),
           Z = neighbours(z, L.nz, per & 4u, k0, (unsigned)L.plane);
  // dt/tau f^eq + (1 - dt/tau) f
  auto relax = [&](double fe, double fc) { return R1 ? fe : fma(m.keep2, fc, m.dt_tau * fe); };

  if (part == 0) {
    const double c = at(fin, k0);
    const double fe = rho * (m.AR * T);
    const double q[6] = {at(fin, X.k[1]), at(fin, X.k[2]), at(fin, Y.k[1]), at(fin, Y.k[2]), at(fin, Z.k[1]), at(fin, Z.k[2])};
    fout[k0] = fma(m.lam0, rest_lap(c, q), relax(fe, c));
  }
  const double usq = fma(ux, ux, fma(uy, uy, uz * uz));
  {
    const double rA = rho * fma(m.AaT, T, fma(m.AaU, usq, m.Aa0));
    const double rB = rho * fma(m.BaT, T, fma(m.BaU, usq, m.Ba0));
    const double rD = rho * m.Da;
    const bool dissipation = m.lam1 != 0.0;
    Nb A = X, B = Y, C = Z;
    double ua = ux, ub = uy, uc = uz;
#pragma unroll 1
    for (int a = 0; a < a1; ++a) {
      const double w = m.c1 * ua, q = fma(rD, w * w, rA);
      const double* fp = fin + (1 + 2 * a) * L.fs;
      double* op = fout + (1 + 2 * a) * L.fs + k0;
      double v[9];
      double c = at(fp, k0);
      axis_load<false>(fp, A, B, C, v);
      *op = fma(kax, axis_sum<SCHEME>(c, v, dissipation), relax(fma(rB, w, q), c));
      fp += L.fs;
      c = at(fp, k0);
      axis_load<true>(fp, A, B, C, v);
      op[L.fs] = fma(kax, axis_sum<SCHEME>(c, v, dissipation), relax(fma(-rB, w, q), c));
      const Nb t = A;
      A = B;
      B = C;
      C = t;
      const double tu = ua;
      ua = ub;
      ub = uc;
      uc = tu;
    }
  }
  {
    const double rA = rho * fma(m.AdT, T, fma(m.AdU, usq, m.Ad0));
    const double rB = rho * fma(m.BdT, T, fma(m.BdU, usq, m.Bd0));
    const double rD = rho * m.Dd;
    Nb B = Y, C = Z;
    double uxy = ux + uy, uc = uz;
    // pairs (7 + k, 14 - k): signs (+,+,+), (+,+,-), (+,-,+), (+,-,-) and their opposites
#pragma unroll 1
    for (int k = 0; k < d1; ++k) {
      if (k >= d0) {
        const double w = m.s * (uxy + uc), q = fma(rD, w * w, rA);
        const double* fp = fin + (7 + k) * L.fs;
        double v[9];
        double c = at(fp, k0);
        diag_load<false, false, false>(fp, X, B, C, v);
        fout[(7 + k) * L.fs + k0] = fma(kdg, diag_conv2<SCHEME>(c, v), relax(fma(rB, w, q), c));
        fp = fin + (14 - k) * L.fs;
        c = at(fp, k0);
        diag_load<true, true, true>(fp, X, B, C, v);
        fout[(14 - k) * L.fs + k0] = fma(kdg, diag_conv2<SCHEME>(c, v), relax(fma(-rB, w, q), c));
      }
      // reverse z; after the second pair y as well
      auto reverse = [](Nb& n) {
        const Nb t = n;
        n.k[0] = t.k[3];
        n.k[1] = t.k[2];
        n.k[2] = t.k[1];
        n.k[3] = t.k[0];
      };
      reverse(C);
      uc = -uc;
      if (k == 1) {
        reverse(B);
        uxy = ux - uy;
      }
    }
  }
  chain_start();  // late: started early, the next step's blocks gather on the SMs that happen to have room
}

// The same with one pair of velocities per block (seven parts) and all loads
// issued before the moments' arithmetic: on a grid of a few hundred rows the
// step is one warp's latency, and the stencils' loads after the moments were a
// second trip to the L2 (150 x 1 x 1: 5.2 -> 4.3 us per step, 200 x 4 x 4: 6.3
// -> 5.9, with a scale per sum of the moments 6.0).
template <int SCHEME, bool R1>
__global__ void __launch_bounds__(32)
    step_fp64_pairs_kernel(const double* fin, double* __restrict__ fout, Layout L, Model<double> m,
                           double kax, double kdg, unsigned per, unsigned* __restrict__ flags) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y / 7, z = blockIdx.z, part = blockIdx.y % 7;
  const bool diag = part >= 3;
  const int ia = diag ? 4 + part : 1 + 2 * part, ib = diag ? 17 - part : 2 + 2 * part;  // the pair's velocities
  const unsigned k0 = (unsigned)L.at(x, y, z);
  const Nb X = neighbours(x, L.nx, per & 1u, k0, 1u), Y = neighbours(y, L.ny, per & 2u, k0, (unsigned)L.sx),
           Z = neighbours(z, L.nz, per & 4u, k0, (unsigned)L.plane);
  chain_wait();
  if (x >= L.nx) return;
  double f[NV], va[9], vb[9], r6[6];
#pragma unroll
  for (int i = 0; i < NV; ++i) f[i] = at(fin + i * L.fs, k0);
  const double *fa = fin + ia * L.fs, *fb = fin + ib * L.fs;
  if (diag) {
    const bool ry = part >= 5, rz = (part & 1) == 0;  // pairs (+,+,+), (+,+,-), (+,-,+), (+,-,-)
    const Nb B = {{Y.k[ry ? 3 : 0], Y.k[ry ? 2 : 1], Y.k[ry ? 1 : 2], Y.k[ry ? 0 : 3]}};
    const Nb C = {{Z.k[rz ? 3 : 0], Z.k[rz ? 2 : 1], Z.k[rz ? 1 : 2], Z.k[rz ? 0 : 3]}};
    diag_load<false, false, false>(fa, X, B, C, va);
    diag_load<true, true, true>(fb, X, B, C, vb);
  } else {
    const Nb A = part == 0 ? X : (part == 1 ? Y : Z), B = part == 0 ? Y : (part == 1 ? Z : X),
             C = part == 0 ? Z : (part == 1 ? X : Y);
    axis_load<false>(fa, A, B, C, va);
    axis_load<true>(fb, A, B, C, vb);
  }
  if (part == 0) {
    const Nb N[3] = {X, Y, Z};
#pragma unroll
    for (int j = 0; j < 6; ++j) r6[j] = at(fin, N[j / 2].k[1 + j % 2]);
  }
  const double ca = at(fa, k0), cb = at(fb, k0);

  double rho, ux, uy, uz, T;
  fx::moments_fixed(m, f, rho, ux, uy, uz, T);
  auto relax = [&](double fe, double fc) { return R1 ? fe : fma(m.keep2, fc, m.dt_tau * fe); };
  if (part == 0) {
    const unsigned bad = health_fp64(rho, ux, uy, uz, T);
    if (bad) atomicOr(flags, bad);
    fout[k0] = fma(m.lam0, rest_lap(f[0], r6), relax(rho * (m.AR * T), f[0]));
  }
  const double usq = fma(ux, ux, fma(uy, uy, uz * uz));
  double w, q, rB, ka, sa, sb;
  if (diag) {
    const double sy = part >= 5 ? ux - uy : ux + uy;
    w = m.s * ((part & 1) == 0 ? sy - uz : sy + uz);
    rB = rho * fma(m.BdT, T, fma(m.BdU, usq, m.Bd0));
    q = fma(rho * m.Dd, w * w, rho * fma(m.AdT, T, fma(m.AdU, usq, m.Ad0)));
    ka = kdg;
    sa = diag_conv2<SCHEME>(ca, va);
    sb = diag_conv2<SCHEME>(cb, vb);
  } else {
    w = m.c1 * (part == 0 ? ux : (part == 1 ? uy : uz));
    rB = rho * fma(m.BaT, T, fma(m.BaU, usq, m.Ba0));
    q = fma(rho * m.Da, w * w, rho * fma(m.AaT, T, fma(m.AaU, usq, m.Aa0)));
    ka = kax;
    sa = axis_sum<SCHEME>(ca, va, m.lam1 != 0.0);
    sb = axis_sum<SCHEME>(cb, vb, m.lam1 != 0.0);
  }
  fout[ia * L.fs + k0] = fma(ka, sa, relax(fma(rB, w, q), ca));
  fout[ib * L.fs + k0] = fma(ka, sb, relax(fma(-rB, w, q), cb));
  chain_start();
}

template <int SCHEME>
void launch_fp64(const double* fin, double* fout, const Layout& L, const Model<double>& m,
                 unsigned per, int parts, dim3 grid, dim3 block, unsigned* flags,
                 cudaStream_t st) {
  const double kax = m.lam1 != 0.0 ? -0.1 * m.k1 : -0.5 * m.k1;
  if (parts == 7)
    launch_chained(m.dt_tau == 1.0 ? step_fp64_pairs_kernel<SCHEME, true> : step_fp64_pairs_kernel<SCHEME, false>, grid,
                   block, 0, st, fin, fout, L, m, kax, -0.5 * m.k2, per, flags);
  else
    launch_chained(m.dt_tau == 1.0 ? step_fp64_kernel<SCHEME, true> : step_fp64_kernel<SCHEME, false>, grid, block, 0, st,
                   fin, fout, L, m, kax, -0.5 * m.k2, per, parts, flags);
}

}  // namespace

cudaError_t launch_step_plain(int scheme, const float* fin, float* fout, const Layout& L, const Model<float>& m,
                              unsigned* flags, cudaStream_t st) {
  dim3 block(32, 8, 1);
  dim3 grid((L.nx + 31) / 32, (L.ny + 7) / 8, L.nz);
  switch (scheme) {
    case LBM_SCHEME_NND: step_plain_kernel<LBM_SCHEME_NND><<<grid, block, 0, st>>>(fin, fout, L, m, flags); break;
    case LBM_SCHEME_UPWIND2: step_plain_kernel<LBM_SCHEME_UPWIND2><<<grid, block, 0, st>>>(fin, fout, L, m, flags); break;
    default: step_plain_kernel<LBM_SCHEME_UPWIND1><<<grid, block, 0, st>>>(fin, fout, L, m, flags); break;
  }
  return cudaGetLastError();
}

cudaError_t launch_step_fp64(int scheme, const double* fin, double* fout, const Layout& L, const Model<double>& m,
                             unsigned per, int num_sms, unsigned* flags, cudaStream_t st) {
  // Rows per block: 8 keep the y neighbours' rows in one SM's L1; a grid whose
  // rows fill fewer than two such blocks per SM spreads them one by one over
  // all SMs (4000 x 4 x 4, 13 warps per SM: 24 us against 30; from 21 warps per
  // SM on no difference).  Smaller still, a row's 5400 instructions in one warp
  // are the step's length, and its velocities go to several blocks (us per
  // step with 1 / 3 / 7 parts: 200 x 4 x 4, 0.7 warps per SM, 14.9 / 8.2 / 5.9;
  // 400 x 4 x 4, 1.4: 14.4 / 8.5 / 7.6; 800 x 4 x 4, 2.6: 14.5 / 10.0 / 12.5;
  // 2000 x 4 x 4, 6.6: 16.3 / 16.1 / 24.7).
  const long long warps = (long long)((L.nx + 31) / 32) * L.ny * L.nz;
  const int rows = warps >= 16LL * num_sms ? 8 : 1;
  const int parts = warps <= 2LL * num_sms ? 7 : (warps <= 6LL * num_sms ? 3 : 1);
  dim3 block(32, rows, 1);
  dim3 grid((L.nx + 31) / 32, (L.ny + rows - 1) / rows * parts, L.nz);
  switch (scheme) {
    case LBM_SCHEME_NND: launch_fp64<LBM_SCHEME_NND>(fin, fout, L, m, per, parts, grid, block, flags, st); break;
    case LBM_SCHEME_UPWIND2: launch_fp64<LBM_SCHEME_UPWIND2>(fin, fout, L, m, per, parts, grid, block, flags, st); break;
    default: launch_fp64<LBM_SCHEME_UPWIND1>(fin, fout, L, m, per, parts, grid, block, flags, st);
  }
  return cudaGetLastError();
}

}  // namespace lbm
