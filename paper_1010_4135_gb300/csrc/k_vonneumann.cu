// Von Neumann amplification service (Sec. 3) for choosing run parameters.
//
// For a perturbation F exp(i k.x) of a uniform state (rho, u, T), one step
// multiplies F by the 15 x 15 complex matrix
//   G_ij = (1 - dt/tau - sum_a v_ia dt/dx phi_ia
//           + lambda_i dt sum_a (2 cos(k_a dx) - 2)/dx^2) delta_ij + dt/tau dfeq_i/df_j,
//   phi_ia = 1 - exp(-i k_a dx) for v_ia >= 0, exp(i k_a dx) - 1 otherwise
// (the paper's G with alpha~ = beta~ = 0), with the equilibrium Jacobian by
// the chain rule through (rho, u, T):
//   d rho/df_j = 1,  d u_a/df_j = (v_ja - u_a)/rho,
//   d T/df_j = (|v_j - u|^2 + eta_j^2 - b T)/(b rho),
// and the partial derivatives of f^eq_i = rho (A_i + B_i w_i + D_i w_i^2),
// w_i = v_i . u, with A_i, B_i affine in T and |u|^2 per velocity shell
// (Eq. "eq").  The service returns, per parameter set, the largest spectral
// radius max |omega| over a batch of states, wave-vector directions and
// wave numbers k dx = pi q / nk (q = 1 .. nk): the paper's stability measure.
//
// The eigenvalues come from a Householder reduction to upper Hessenberg form
// followed by the single-shift complex QR iteration with Wilkinson shifts,
// deflation at negligible subdiagonal entries and an exceptional shift after
// 10 and 20 iterations without one (the practical QR algorithm of Golub and
// Van Loan, Sec. 7.5, here without accumulating the transformations: only
// eigenvalues are needed, so each QR step acts on the unreduced diagonal block
// alone).  A matrix that has not converged after 30 n iterations reports +inf,
// which the caller reads as unstable.
//
// Bound by the FP64 pipe and, with few matrices per SM, by its latency: a
// request's 5760 matrices were 180 warps at one thread per matrix, about one
// per SM, each in a serial chain of FP64 operations (5.05 ms; now 1.72, the
// FP64 pipe 75 % busy).
// VT lanes share a matrix: they own columns in the transformations from the
// left, rows in those from the right, and repeat the scalar work (shifts,
// rotations) between them, with a synchronisation of the VT lanes at each
// rotation.  The matrices live in shared memory, VSTRIDE elements apart, so
// that the two matrices of a quarter warp use different banks.
#include <cmath>

#include "lbm_internal.cuh"

namespace lbm {
namespace {

constexpr int VN = NV;              // matrix order
constexpr int VN_THREADS = 32;      // one warp per block
constexpr int VSTRIDE = VN * VN + 3;  // elements between matrices
constexpr int VN_PARAMS = 7;        // c1, c2, eta0, gamma, dt, tau, dx
constexpr int VN_MAX_ITER = 30 * VN;

struct cd {
  double re, im;
};
__device__ __forceinline__ cd mk(double r, double i) { return {r, i}; }
__device__ __forceinline__ cd operator+(cd a, cd b) { return {a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ cd operator-(cd a, cd b) { return {a.re - b.re, a.im - b.im}; }
__device__ __forceinline__ cd operator*(cd a, cd b) { return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }
__device__ __forceinline__ cd operator*(double s, cd a) { return {s * a.re, s * a.im}; }
__device__ __forceinline__ cd cconj(cd a) { return {a.re, -a.im}; }
__device__ __forceinline__ double norm2(cd a) { return fma(a.re, a.re, a.im * a.im); }
__device__ __forceinline__ double cabs(cd a) { return hypot(a.re, a.im); }
// acc + a b and acc - a b
__device__ __forceinline__ cd fmadd(cd a, cd b, cd acc) {
  return {fma(a.re, b.re, fma(-a.im, b.im, acc.re)), fma(a.re, b.im, fma(a.im, b.re, acc.im))};
}
__device__ __forceinline__ cd fmsub(cd a, cd b, cd acc) {
  return {fma(-a.re, b.re, fma(a.im, b.im, acc.re)), fma(-a.re, b.im, fma(-a.im, b.re, acc.im))};
}
__device__ __forceinline__ double cabs1(cd a) { return fabs(a.re) + fabs(a.im); }
__device__ __forceinline__ cd csqrt_(cd a) {
  const double r = cabs(a);
  if (r == 0.0) return {0.0, 0.0};
  const double t = sqrt(0.5 * (r + fabs(a.re)));
  return a.re >= 0.0 ? cd{t, a.im / (2.0 * t)} : cd{fabs(a.im) / (2.0 * t), copysign(t, a.im)};
}

// Matrix of this thread's group of VT lanes (4 or 8), row-major; g is the thread's place
// in the group, mask the group's lanes of the warp.
template <int VT_>
struct Mat {
  static constexpr int VT = VT_;
  cd* m;
  int g;
  unsigned mask;
  __device__ cd& at(int r, int c) const { return m[r * VN + c]; }
  __device__ void sync() const { __syncwarp(mask); }
  // sum and maximum over the group, the same value in every lane
  __device__ double sum(double v) const {
#pragma unroll
    for (int o = VT / 2; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o);
    return v;
  }
  __device__ int max(int v) const {
#pragma unroll
    for (int o = VT / 2; o > 0; o >>= 1) v = ::max(v, __shfl_xor_sync(mask, v, o));
    return v;
  }
  __device__ double max(double v) const {
#pragma unroll
    for (int o = VT / 2; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(mask, v, o));
    return v;
  }
};

// The discrete velocities (Sec. 2) in the library's order: 0 rest; 1..6 +-c1
// along x, y, z; 7..14 (c2/sqrt 3)(sx, sy, sz), signs +++, ++-, ..., ---.
__device__ void velocity(int i, double c1, double s, double v[3]) {
  v[0] = v[1] = v[2] = 0.0;
  if (i == 0) return;
  if (i <= 6) {
    v[(i - 1) / 2] = ((i - 1) % 2 == 0) ? c1 : -c1;
    return;
  }
  const int k = i - 7;
  v[0] = (k & 4) ? -s : s;
  v[1] = (k & 2) ? -s : s;
  v[2] = (k & 1) ? -s : s;
}

// Per-velocity coefficients of Eq. "eq": A = A0 + AT T + AU u^2, B = B0 + BT T
// + BU u^2, D.
__device__ void shell(int i, double c1, double c2, double eta0, double b, double co[7]) {
  const double c12 = c1 * c1, c22 = c2 * c2, e2 = eta0 * eta0;
  if (i == 0) {
    co[0] = 0.0; co[1] = (b - 3.0) / e2; co[2] = 0.0; co[3] = co[4] = co[5] = co[6] = 0.0;
  } else if (i <= 6) {
    const double ka = 1.0 / (6.0 * (c12 - c22)), kb = 1.0 / (2.0 * c12 * (c12 - c22));
    co[0] = -c22 * ka; co[1] = ((b - 3.0) * c22 / e2 + 3.0) * ka; co[2] = c22 / c12 * ka;
    co[3] = -c22 * kb; co[4] = (b + 2.0) * kb; co[5] = kb; co[6] = 1.0 / (2.0 * c12 * c12);
  } else {
    const double kd = 1.0 / (8.0 * (c22 - c12)), ke = 3.0 / (8.0 * c22 * (c22 - c12));
    co[0] = -c12 * kd; co[1] = ((b - 3.0) * c12 / e2 + 3.0) * kd; co[2] = (3.0 * c12 - c22) / (2.0 * c22) * kd;
    co[3] = -c12 * ke; co[4] = (b + 2.0) * ke; co[5] = ke; co[6] = 9.0 / (16.0 * c22 * c22);
  }
}

// G(k) of the state st = (rho, u1, u2, u3, T) and parameters p into M; each
// lane writes rows g, g + VT, ...
template <class Mat>
__device__ void build_g(const Mat& M, const double* st, const double* p, const double kv[3], int dissipation) {
  constexpr int VT = Mat::VT;
  const double c1 = p[0], c2 = p[1], eta0 = p[2], gamma = p[3], dt = p[4], tau = p[5], dx = p[6];
  const double b = 2.0 / (gamma - 1.0), s = c2 / sqrt(3.0);
  const double rho = st[0], u[3] = {st[1], st[2], st[3]}, T = st[4];
  const double usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  const double r = dt / tau, ir = 1.0 / rho, ibr = 1.0 / (b * rho);
  double cs[3], sn[3];
  for (int a = 0; a < 3; ++a) sincos(kv[a] * dx, &sn[a], &cs[a]);
#pragma unroll 1
  for (int i = M.g; i < VN; i += VT) {
    double vi[3], co[7];
    velocity(i, c1, s, vi);
    shell(i, c1, c2, eta0, b, co);
    const double w = vi[0] * u[0] + vi[1] * u[1] + vi[2] * u[2];
    const double A = co[0] + co[1] * T + co[2] * usq, B = co[3] + co[4] * T + co[5] * usq, D = co[6];
    const double f_rho = A + B * w + D * w * w;
    const double f_T = rho * (co[1] + co[4] * w) * ibr;  // with the factor of d T/df_j
    double f_u[3];                                       // with the factor of d u/df_j
    for (int a = 0; a < 3; ++a)
      f_u[a] = rho * ((2.0 * co[2] + 2.0 * co[5] * w) * u[a] + (B + 2.0 * D * w) * vi[a]) * ir;
#pragma unroll 1
    for (int j = 0; j < VN; ++j) {
      // columns of the chain rule: (v_ja - u_a), |v_j - u|^2 + eta_j^2 - b T
      double vj[3];
      velocity(j, c1, s, vj);
      const double d0 = vj[0] - u[0], d1 = vj[1] - u[1], d2 = vj[2] - u[2];
      const double e = fma(d0, d0, fma(d1, d1, d2 * d2)) + ((j == 0 ? eta0 * eta0 : 0.0) - b * T);
      const double J = fma(f_T, e, fma(f_u[0], d0, fma(f_u[1], d1, fma(f_u[2], d2, f_rho))));
      M.at(i, j) = mk(r * J, 0.0);
    }
    // diagonal: relaxation, convection (first-order upwind phase), dissipation
    const double lam = !dissipation ? 0.0 : (i == 0 ? c1 * dx : (i <= 6 ? c1 * dx / 10.0 : 0.0));
    cd d = mk(1.0 - r, 0.0);
    for (int a = 0; a < 3; ++a) {
      // phi = 1 - e^{-i th} = (1 - cos th) + i sin th ; e^{i th} - 1 = (cos th - 1) + i sin th
      const cd phi = vi[a] >= 0.0 ? mk(1.0 - cs[a], sn[a]) : mk(cs[a] - 1.0, sn[a]);
      d = d - (vi[a] * dt / dx) * phi;
      d = d + mk(lam * dt * (2.0 * cs[a] - 2.0) / (dx * dx), 0.0);
    }
    M.at(i, i) = M.at(i, i) + d;
  }
  M.sync();
}

// Spectral radius of M (destroyed), or +inf if the QR iteration does not
// converge or M is not finite; the same value in every lane.  rot: VN rotations of the group.
struct Rot {
  cd s;
  double c;
};
template <class Mat>
__device__ double spectral_radius(const Mat& M, Rot* rot) {
  constexpr int VT = Mat::VT;
  const int n = VN, g = M.g;
  // Entries far from 1 are scaled by a power of two (exact): the products of
  // four entries below (two squared norms) then stay in range.
  int largest = 0;  // high word of the largest component
  for (int r = g; r < n; r += VT)
    for (int c = 0; c < n; ++c)
      largest = max(largest, max(__double2hiint(M.at(r, c).re) & 0x7fffffff, __double2hiint(M.at(r, c).im) & 0x7fffffff));
  const int e2 = (M.max(largest) >> 20) - 1023;
  const int scale = e2 < 1024 && (e2 > 64 || e2 < -64) ? e2 : 0;
  if (scale != 0) {
    for (int r = g; r < n; r += VT)
      for (int c = 0; c < n; ++c) M.at(r, c) = mk(scalbn(M.at(r, c).re, -scale), scalbn(M.at(r, c).im, -scale));
    M.sync();
  }
  // Householder reduction to upper Hessenberg form (similarity, eigenvalues kept)
#pragma unroll 1
  for (int k = 0; k + 2 < n; ++k) {
    double part = 0.0;  // squared norm below the subdiagonal
    for (int i = k + 2 + g; i < n; i += VT) part += norm2(M.at(i, k));
    const double tail = M.sum(part);
    if (tail == 0.0) continue;  // the column is already in Hessenberg form
    const cd x0 = M.at(k + 1, k);
    const double p0 = norm2(x0), alpha = sqrt(tail + p0), ax0 = sqrt(p0);
    const cd phase = ax0 > 0.0 ? mk(x0.re / ax0, x0.im / ax0) : mk(1.0, 0.0);
    // v = x + phase alpha e1 (stored in column k below the diagonal), beta = 2 / |v|^2
    const cd v0 = x0 + alpha * phase;
    const double beta = 2.0 / (tail + norm2(v0));
    M.sync();
    if (g == 0) M.at(k + 1, k) = v0;
    M.sync();
    for (int j = k + 1 + g; j < n; j += VT) {  // left: rows k+1..n-1 of columns k+1..n-1
      cd sum = mk(0.0, 0.0);
      for (int i = k + 1; i < n; ++i) sum = fmadd(cconj(M.at(i, k)), M.at(i, j), sum);
      sum = beta * sum;
      for (int i = k + 1; i < n; ++i) M.at(i, j) = fmsub(M.at(i, k), sum, M.at(i, j));
    }
    M.sync();
    for (int r = g; r < n; r += VT) {  // right: columns k+1..n-1 of every row
      cd sum = mk(0.0, 0.0);
      for (int i = k + 1; i < n; ++i) sum = fmadd(M.at(r, i), M.at(i, k), sum);
      sum = beta * sum;
      for (int i = k + 1; i < n; ++i) M.at(r, i) = fmsub(sum, cconj(M.at(i, k)), M.at(r, i));
    }
    M.sync();
    // the reflected column: -phase alpha e1
    if (g == 0) M.at(k + 1, k) = (-alpha) * phase;
    for (int i = k + 2 + g; i < n; i += VT) M.at(i, k) = mk(0.0, 0.0);
    M.sync();
  }
  // shifted QR on the unreduced diagonal blocks, eigenvalues only.  A
  // subdiagonal entry is negligible below ulp times its diagonal neighbours
  // or ulp times the matrix norm: the iteration's backward error is of that
  // size anyway, and without the norm floor a cluster of tiny eigenvalues
  // (those of G for dt = tau are O(Courant number)) is never split off
  const double ulp = 2.220446049250313e-16;
  const double TINY = 1e-220;  // |x| = 1e-110 beside a norm of 2^-64 at least
  double nrm = 0.0;
  for (int r = g; r < n; r += VT)
    for (int c = r > 0 ? r - 1 : 0; c < n; ++c) nrm = fmax(nrm, cabs1(M.at(r, c)));
  const double floor_small = ulp * M.max(nrm);
  const int shift = __ffs((int)M.mask) - 1;
  double radius = 0.0;
  int hi = n - 1, its = 0, total = 0;
#pragma unroll 1
  while (hi >= 0) {
    int l = 0;  // start of the unreduced block that ends at hi: VT entries are looked at together
    for (int top = hi; top > 0; top -= VT) {
      const int i = top - g;
      bool small = false;
      if (i > 0) {
        const double tst = cabs1(M.at(i - 1, i - 1)) + cabs1(M.at(i, i));
        small = cabs1(M.at(i, i - 1)) <= fmax(ulp * tst, floor_small);
      }
      const unsigned found = (__ballot_sync(M.mask, small) >> shift) & ((1u << VT) - 1u);
      if (found) {
        l = top - (__ffs((int)found) - 1);
        break;
      }
    }
    if (l > 0 && g == 0) M.at(l, l - 1) = mk(0.0, 0.0);
    if (l == hi) {  // a 1 x 1 block: an eigenvalue
      const double e = cabs(M.at(hi, hi));
      if (!(e <= 1e300)) return INFINITY;  // non-finite: reported as unstable
      radius = fmax(radius, e);
      --hi;
      its = 0;
      continue;
    }
    if (++total > VN_MAX_ITER) return INFINITY;
    ++its;
    // Wilkinson shift: the eigenvalue of the trailing 2 x 2 block nearer its last entry
    const cd a = M.at(hi - 1, hi - 1), bq = M.at(hi - 1, hi), c = M.at(hi, hi - 1), d = M.at(hi, hi);
    cd mu;
    if (its == 10 || its == 20) {  // exceptional shift
      mu = d + mk(0.75 * cabs1(c), 0.0);
    } else {
      const cd half = 0.5 * (a - d);
      const cd disc = csqrt_(half * half + bq * c);
      const cd m1 = d + half + disc, m2 = d + half - disc;
      mu = cabs1(m1 - d) <= cabs1(m2 - d) ? m1 : m2;
    }
    M.sync();
    for (int j = l + g; j <= hi; j += VT) M.at(j, j) = M.at(j, j) - mu;
    M.sync();
#pragma unroll 1
    for (int j = l; j < hi; ++j) {
      // rotation of rows j, j+1 that takes (x, y) to (|(x, y)|, 0) times x's phase
      const cd x = M.at(j, j), y = M.at(j + 1, j);
      const double px = norm2(x), pn = px + norm2(y);
      double cg = 1.0;
      cd sg = mk(0.0, 0.0);
      // |y| is above ulp times the matrix' norm, so px pn is a normal number
      if (px >= TINY) {
        const double rs = rsqrt(px * pn);  // 1 / (|x| |(x, y)|)
        cg = px * rs;
        sg = rs * (x * cconj(y));
      } else if (pn >= TINY) {  // x is nothing beside y: exchange the rows
        cg = 0.0;
        sg = mk(1.0, 0.0);
      }
      if (g == 0) rot[j] = {sg, cg};
      M.sync();
      for (int col = j + g; col <= hi; col += VT) {
        const cd t1 = M.at(j, col), t2 = M.at(j + 1, col);
        M.at(j, col) = fmadd(sg, t2, cg * t1);
        M.at(j + 1, col) = fmsub(cconj(sg), t1, cg * t2);
      }
      M.sync();
    }
    for (int r = l + g; r <= hi; r += VT) {  // the rows of R times the rotations' adjoints
      int j = r - 1 > l ? r - 1 : l;
      cd t1 = M.at(r, j);
      for (; j < hi; ++j) {
        const cd t2 = M.at(r, j + 1), sj = rot[j].s;
        const double cj = rot[j].c;
        M.at(r, j) = fmadd(cconj(sj), t2, cj * t1);
        t1 = fmsub(sj, t1, cj * t2);
      }
      M.at(r, hi) = t1;
    }
    M.sync();
    for (int j = l + g; j <= hi; j += VT) M.at(j, j) = M.at(j, j) + mu;
    M.sync();
  }
  return scalbn(radius, scale);
}

// Item t of the batch: parameter set t / per_param, then state, direction and
// wave number; out[p] is the max over its items (atomic max of the bit
// patterns, which order like the values for non-negative doubles).
template <int VT>
__global__ void __launch_bounds__(VN_THREADS)
    vn_kernel(const double* __restrict__ states, int nstates, const double* __restrict__ params, int nparams,
              const double* __restrict__ dirs, int ndirs, int nk, int dissipation,
              unsigned long long* __restrict__ out) {
  constexpr int VN_MATS = VN_THREADS / VT;
  __shared__ __align__(16) cd mats[VN_MATS * VSTRIDE];
  __shared__ Rot rots[VN_MATS][VN];
  const long long per_param = (long long)nstates * ndirs * nk;
  const int slot = threadIdx.x / VT;
  const long long t = (long long)blockIdx.x * VN_MATS + slot;
  if (t >= per_param * nparams) return;
  const int p = (int)(t / per_param);
  long long rem = t % per_param;
  const int s = (int)(rem / ((long long)ndirs * nk));
  rem %= (long long)ndirs * nk;
  const int d = (int)(rem / nk), q = (int)(rem % nk);
  const double* dv = dirs + 3 * d;
  const double dn = sqrt(dv[0] * dv[0] + dv[1] * dv[1] + dv[2] * dv[2]);
  const double dx = params[VN_PARAMS * p + 6];
  const double kdx = 3.141592653589793 * (q + 1) / nk;
  const double kv[3] = {dv[0] / dn * kdx / dx, dv[1] / dn * kdx / dx, dv[2] / dn * kdx / dx};
  Mat<VT> M{mats + slot * VSTRIDE, (int)threadIdx.x % VT, ((1u << VT) - 1u) << (slot * VT)};
  build_g(M, states + 5 * s, params + VN_PARAMS * p, kv, dissipation);
  const double rad = spectral_radius(M, rots[slot]);
  if (M.g == 0) atomicMax(out + p, (unsigned long long)__double_as_longlong(rad));
}

}  // namespace

cudaError_t launch_vn_max_growth(const double* states, int nstates, const double* params, int nparams,
                                 const double* dirs, int ndirs, int nk, int dissipation, double* out,
                                 cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(double) * nparams, st);
  if (e != cudaSuccess) return e;
  int device = 0, num_sms = 0;
  e = cudaGetDevice(&device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, device);
  if (e != cudaSuccess) return e;
  // Lanes per matrix: with fewer than 16 matrices per SM four lanes leave too
  // few warps to cover the FP64 pipe's latency, with more eight repeat too much
  // scalar work (us: 1920 matrices 1448 with four, 1031 with eight; 5760
  // matrices 1723 and 2050; one lane each 4980 and 5054, two 2378 and 2449).
  const long long items = (long long)nstates * ndirs * nk * nparams;
  auto run = [&](auto kernel, int mats) {
    kernel<<<(unsigned)((items + mats - 1) / mats), VN_THREADS, 0, st>>>(states, nstates, params, nparams, dirs, ndirs, nk,
                                                                        dissipation,
                                                                        reinterpret_cast<unsigned long long*>(out));
  };
  if (items < 16LL * num_sms) run(vn_kernel<8>, VN_THREADS / 8);
  else run(vn_kernel<4>, VN_THREADS / 4);
  return cudaGetLastError();
}

}  // namespace lbm
