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
// fixed point (fixed_sum.cuh; the values aligned are a velocity's stencil, or
// a cell's 15 values).  The largest sum, five times twice the convection of an
// axis velocity (|difference| <= 2, |minmod| <= |difference|) less its
// Laplacian, is at most 52 times the largest value (a diagonal velocity's
// convection 24 times).  256^3: 13.3 -> 4.4 ms per step (417 -> about 130 FP64
// operations per cell; the FP64 pipe 84 -> 67 % busy, the integer ALUs 74 %:
// both near their rates); 300 x 80 x 80 with walls 1.68 -> 0.58 ms.
using fx::from_fixed;
using fx::in_range;
using fx::mag;
using fx::to_fixed;

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

// The same in double, for stencils outside the fixed-point range.
template <int SCHEME>
__device__ __noinline__ double conv2_double(double c, const double* v) {
  double s = 0.0;
  for (int a = 0; a < 3; ++a) s += 2.0 * grad_pos<SCHEME>(v[3 * a], v[3 * a + 1], c, v[3 * a + 2]);
  return s;
}

// Field offsets (32-bit, modulo 2^32: a field has fewer elements) of a cell's
// neighbours along one axis: [0..3] = -2, -1, +1, +2.
struct Nb {
  unsigned k[4];
};
__device__ __forceinline__ double at(const double* __restrict__ f, unsigned k) { return __ldg(f + k); }

// Twice the convection sum of a diagonal velocity: x, y, z neighbours; sx, sy, sz
// reverse an axis.
template <int SCHEME, bool RX, bool RY, bool RZ>
__device__ __forceinline__ double diag_conv2(const double* __restrict__ f, double c, const Nb& X, const Nb& Y,
                                             const Nb& Z) {
  double v[9] = {at(f, X.k[RX ? 3 : 0]), at(f, X.k[RX ? 2 : 1]), at(f, X.k[RX ? 1 : 2]),
                 at(f, Y.k[RY ? 3 : 0]), at(f, Y.k[RY ? 2 : 1]), at(f, Y.k[RY ? 1 : 2]),
                 at(f, Z.k[RZ ? 3 : 0]), at(f, Z.k[RZ ? 2 : 1]), at(f, Z.k[RZ ? 1 : 2])};
  int mx = mag(c);
#pragma unroll
  for (int j = 0; j < 9; ++j) mx = max(mx, mag(v[j]));
  const int E = mx >> 20;
  if (!in_range(E)) return conv2_double<SCHEME>(c, v);
  const long long n = to_fixed(c, E);
  long long s = 0;
#pragma unroll
  for (int a = 0; a < 3; ++a)
    s += grad2<SCHEME>(to_fixed(v[3 * a], E), to_fixed(v[3 * a + 1], E), n, to_fixed(v[3 * a + 2], E));
  return from_fixed(s, E);
}

// Convection and dissipation of an axis velocity along A (R: the negative
// one); B, C: the other axes.  With the dissipation term lambda_i = c1 dx / 10
// (Sec. 3), so both terms are one multiple of lambda_i dt/dx^2 = |v| dt/(10
// dx): returns 5 times twice the convection less the Laplacian, or twice the
// convection alone when the term is off.
template <int SCHEME, bool R>
__device__ __forceinline__ double axis_sum(const double* __restrict__ f, double c, const Nb& A, const Nb& B,
                                           const Nb& C, bool dissipation) {
  const double m2 = at(f, A.k[R ? 3 : 0]), m1 = at(f, A.k[R ? 2 : 1]), p1 = at(f, A.k[R ? 1 : 2]);
  const double q[4] = {at(f, B.k[1]), at(f, B.k[2]), at(f, C.k[1]), at(f, C.k[2])};
  int mx = max(max(mag(c), mag(m2)), max(mag(m1), mag(p1)));
#pragma unroll
  for (int j = 0; j < 4; ++j) mx = max(mx, mag(q[j]));
  const int E = mx >> 20;
  if (!in_range(E)) {
    const double conv2 = 2.0 * grad_pos<SCHEME>(m2, m1, c, p1);
    return dissipation ? 5.0 * conv2 - (((m1 + p1) + (q[0] + q[1])) + (q[2] + q[3]) - 6.0 * c) : conv2;
  }
  const long long n = to_fixed(c, E), n1 = to_fixed(m1, E), n2 = to_fixed(p1, E);
  long long s = grad2<SCHEME>(to_fixed(m2, E), n1, n, n2);
  if (dissipation) {
    s = 5 * s + 6 * n - (n1 + n2);
#pragma unroll
    for (int j = 0; j < 4; ++j) s -= to_fixed(q[j], E);
  }
  return from_fixed(s, E);
}

// The Laplacian of the rest velocity.
__device__ __forceinline__ double rest_lap(const double* __restrict__ f, double c, const Nb& X, const Nb& Y,
                                           const Nb& Z) {
  const double q[6] = {at(f, X.k[1]), at(f, X.k[2]), at(f, Y.k[1]), at(f, Y.k[2]), at(f, Z.k[1]), at(f, Z.k[2])};
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
// take turns), so the code stays short.  `parts` blocks share a row: 1; 3
// (rest and axis pairs; two diagonal pairs each); or 7 (one pair each, the
// first with the rest velocity), each with the moments for itself.  kax, kdg:
// factors of axis_sum and diag_conv2.
template <int SCHEME, bool R1>
__global__ void __launch_bounds__(256, 3)
    step_fp64_kernel(const double* __restrict__ fin, double* __restrict__ fout, Layout L, Model<double> m, double kax,
                     double kdg, unsigned per, int parts, unsigned* __restrict__ flags) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = (blockIdx.y / parts) * blockDim.y + threadIdx.y;
  const int z = blockIdx.z, part = blockIdx.y % parts;
  // the axis pairs [a0, a1) and diagonal pairs [d0, d1) of this part
  const int a0 = parts == 7 ? part : 0, a1 = parts == 1 ? 3 : (parts == 3 ? (part == 0 ? 3 : 0) : (part < 3 ? part + 1 : 0));
  const int d0 = parts == 1 ? 0 : (parts == 3 ? 2 * part - 2 : part - 3);
  const int d1 = parts == 1 ? 4 : (parts == 3 ? 2 * part : part - 2);
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
    fout[k0] = fma(m.lam0, rest_lap(fin, c, X, Y, Z), relax(fe, c));
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
      if (a >= a0) {
        const double w = m.c1 * ua, q = fma(rD, w * w, rA);
        const double* fp = fin + (1 + 2 * a) * L.fs;
        double* op = fout + (1 + 2 * a) * L.fs + k0;
        double c = at(fp, k0);
        *op = fma(kax, axis_sum<SCHEME, false>(fp, c, A, B, C, dissipation), relax(fma(rB, w, q), c));
        fp += L.fs;
        c = at(fp, k0);
        op[L.fs] = fma(kax, axis_sum<SCHEME, true>(fp, c, A, B, C, dissipation), relax(fma(-rB, w, q), c));
      }
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
        double c = at(fp, k0);
        fout[(7 + k) * L.fs + k0] =
            fma(kdg, diag_conv2<SCHEME, false, false, false>(fp, c, X, B, C), relax(fma(rB, w, q), c));
        fp = fin + (14 - k) * L.fs;
        c = at(fp, k0);
        fout[(14 - k) * L.fs + k0] =
            fma(kdg, diag_conv2<SCHEME, true, true, true>(fp, c, X, B, C), relax(fma(-rB, w, q), c));
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

template <int SCHEME>
void launch_fp64(const double* fin, double* fout, const Layout& L, const Model<double>& m,
                 unsigned per, int parts, dim3 grid, dim3 block, unsigned* flags,
                 cudaStream_t st) {
  const double kax = m.lam1 != 0.0 ? -0.1 * m.k1 : -0.5 * m.k1;
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
  // step with 1 / 3 / 7 parts: 200 x 4 x 4, 0.7 warps per SM, 14.9 / 8.2 / 6.3;
  // 400 x 4 x 4, 1.4: 14.4 / 8.5 / 7.7; 800 x 4 x 4, 2.6: 14.5 / 10.0 / 11.6;
  // 2000 x 4 x 4, 6.6: 16.3 / 16.3 / 24.9).
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
