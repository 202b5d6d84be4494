// Boundary fill, initialisation, moments, pack/unpack and the FP64
// conservation reduction.  Initialisation and moments compute in double
// precision whatever the storage type of f; the boundary fill computes in the
// storage precision (its results are stored at that precision).
#include "fixed_sum.cuh"
#include "pair_math.cuh"

namespace lbm {
namespace {

// A double rounded to the nearest float (ties to even) on the integer ALUs:
// the conversion instruction runs on the FP64 pipe, which bounds the kernels
// here.  Values outside the normal float range take the instruction.
__device__ __noinline__ float narrow_any(double v) { return (float)v; }  // out of line: inline it would run always
__device__ __forceinline__ double narrow(double v, double) { return v; }
__device__ __forceinline__ float narrow(double v, float) {
  const int h = __double2hiint(v);
  const unsigned l = (unsigned)__double2loint(v);
  const unsigned m = (unsigned)h & 0x7fffffffu;
  if (m < (897u << 20) || m >= (1150u << 20)) return narrow_any(v);  // below 2^-126, or 2^127 and above
  const unsigned b = __funnelshift_l(l, m - (896u << 20), 3);
  const unsigned r = b + (((l & 0x1fffffffu) + 0x0fffffffu + (b & 1u)) >> 29);
  return __uint_as_float(r | ((unsigned)h & 0x80000000u));
}

template <typename R>
__device__ __forceinline__ void store_cell(R* __restrict__ f, long long fs, long long idx, const double v[NV]) {
#pragma unroll
  for (int i = 0; i < NV; ++i) f[i * fs + idx] = narrow(v[i], R());
}

// Running sums of two float lanes, each held as an unevaluated pair hi + lo
// (about 44 significant bits), in packed arithmetic.  add() keeps hi the
// rounded running sum and adds its rounding error (exact: the error-free sum
// of two floats) to lo; renorm() folds lo back into hi (|hi| >= |lo|, so the
// fast two-sum is exact) and is called every few adds, so lo stays of order
// 2^-24 |hi| and n additions lose about n * 2^-48 relative.
struct DFloat2 {
  float2 hi = {0.f, 0.f}, lo = {0.f, 0.f};
  __device__ __forceinline__ void add(float2 x) {
    const float2 s = pm::add(hi, x), bp = pm::sub(s, hi);
    const float2 e = pm::add(pm::sub(hi, pm::sub(s, bp)), pm::sub(x, bp));
    hi = s;
    lo = pm::add(lo, e);
  }
  __device__ __forceinline__ void renorm() {
    const float2 s = pm::add(hi, lo);
    lo = pm::sub(lo, pm::sub(s, hi));
    hi = s;
  }
  __device__ __forceinline__ double value() const {
    return ((double)hi.x + (double)lo.x) + ((double)hi.y + (double)lo.y);
  }
};

// Moments and equilibrium of the boundary fill.  In single precision they are
// the pair kernel's (pair_math.cuh), so that a layer comes out the same
// whether the fill writes it or the pair kernel forms it (WtDesc).
__device__ __forceinline__ void fill_macros(const Model<double>& m, const double v[NV], double M[5]) {
  moments(m, v, M[0], M[1], M[2], M[3], M[4]);
}
__device__ __forceinline__ void fill_macros(const Model<float>& m, const float v[NV], float M[5]) {
  float2 F[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) F[i] = pm::bc2(v[i]);
  const pm::Mom r = pm::moments<false>(m, RecoverDesc(), F, nullptr, 0, 0, true, true);
  M[0] = r.rho.x; M[1] = r.ux.x; M[2] = r.uy.x; M[3] = r.uz.x; M[4] = r.T.x;
}
__device__ __forceinline__ void fill_feq(const Model<double>& m, const double M[5], double e[NV]) {
  equilibrium(m, M[0], M[1], M[2], M[3], M[4], e);
}
__device__ __forceinline__ void fill_feq(const Model<float>& m, const float M[5], float e[NV]) {
  pm::Mom r = {pm::bc2(M[0]), pm::bc2(M[1]), pm::bc2(M[2]), pm::bc2(M[3]), pm::bc2(M[4])};
  r.usq = pm::fma2(r.ux, r.ux, pm::fma2(r.uy, r.uy, pm::mul(r.uz, r.uz)));
#pragma unroll
  for (int i = 0; i < NV; ++i) e[i] = pm::feq(m, r, i).x;
}

// One thread per (face position): writes the two node layers outside a face.
// blockIdx.y = face (2*axis + hi); faces whose bit is clear in `mask` are
// skipped.  Sec. 4(2) boundary rules, ghost f = f^eq.  M is the arithmetic
// type (the storage type of f: ghost values are stored at that precision).
template <typename R, typename M>
__global__ void fill_kernel(R* __restrict__ f, Layout L, Model<M> m, BcDesc bc, unsigned mask) {
  chain_start();
  chain_wait();
  const int face = blockIdx.y;
  if (!((mask >> face) & 1u)) return;
  const int axis = face >> 1, hi = face & 1;
  // cross-section coordinates (s1 fastest) and the element stride along the face normal
  const int n1 = axis == 0 ? L.ny : L.nx;
  const int n2 = axis == 2 ? L.ny : L.nz;
  const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= (long long)n1 * n2) return;
  const int s1 = (int)(p % n1), s2 = (int)(p / n1);
  const long long base = axis == 0 ? L.at(0, s1, s2) : (axis == 1 ? L.at(s1, 0, s2) : L.at(s1, s2, 0));
  const long long step = axis == 0 ? 1LL : (axis == 1 ? (long long)L.sx : L.plane);
  const int N = axis == 0 ? L.nx : (axis == 1 ? L.ny : L.nz);
  const int kind = bc.kind[face];
  const int g1 = hi ? N : -1, g2 = hi ? N + 1 : -2;
  const long long i1 = base + g1 * step, i2 = base + g2 * step;
  if (kind == LBM_BC_PERIODIC) {
    const long long r1 = base + (((g1 % N) + N) % N) * step, r2 = base + (((g2 % N) + N) % N) * step;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const R v1 = f[i * L.fs + r1], v2 = f[i * L.fs + r2];
      f[i * L.fs + i1] = v1;
      f[i * L.fs + i2] = v2;
    }
    return;
  }
  M G1[5], G2[5];
  if (kind == LBM_BC_FIXED) {
#pragma unroll
    for (int k = 0; k < 5; ++k) G1[k] = G2[k] = (M)bc.fixed[face][k];
  } else {
    const long long m0 = base + (hi ? N - 1 : 0) * step;
    M v[NV], M0[5];
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = (M)f[i * L.fs + m0];
    fill_macros(m, v, M0);
    if (kind == LBM_BC_EXTRAPOLATE) {
      const long long m1 = base + (hi ? N - 2 : 1) * step;
      M M1[5];
#pragma unroll
      for (int i = 0; i < NV; ++i) v[i] = (M)f[i * L.fs + m1];
      fill_macros(m, v, M1);
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        G1[k] = M(2) * M0[k] - M1[k];
        G2[k] = M(2) * G1[k] - M0[k];
      }
    } else {  // LBM_BC_REFLECT: the normal velocity is component 1 + axis
#pragma unroll
      for (int k = 0; k < 5; ++k) G1[k] = G2[k] = M0[k];
      const M un = axis == 0 ? M0[1] : (axis == 1 ? M0[2] : M0[3]);
      if (axis == 0) { G1[1] = M(0); G2[1] = -un; }
      if (axis == 1) { G1[2] = M(0); G2[2] = -un; }
      if (axis == 2) { G1[3] = M(0); G2[3] = -un; }
    }
  }
  M e[NV];
  fill_feq(m, G1, e);
#pragma unroll
  for (int i = 0; i < NV; ++i) f[i * L.fs + i1] = (R)e[i];
  fill_feq(m, G2, e);
#pragma unroll
  for (int i = 0; i < NV; ++i) f[i * L.fs + i2] = (R)e[i];
}

__device__ __forceinline__ bool cell_of(const Layout& L, long long k, int& x, int& y, int& z) {
  if (k >= L.ncell()) return false;
  const unsigned q = (unsigned)k, r = q / (unsigned)L.nx;  // a field has fewer than 2^32 cells
  x = (int)(q - r * (unsigned)L.nx);
  z = (int)(r / (unsigned)L.ny);
  y = (int)(r - (unsigned)z * (unsigned)L.ny);
  return true;
}

// f^eq of one cell in double precision (Eq. "eq"), rho folded into the
// shells' coefficients and opposite velocities sharing their even part: 60
// FP64 operations against 77 velocity by velocity.
__device__ __forceinline__ void feq_fp64(const Model<double>& m, double rho, double ux, double uy, double uz, double T,
                                         double e[NV]) {
  const double usq = fma(ux, ux, fma(uy, uy, uz * uz));
  e[0] = rho * (m.AR * T);
  {
    const double rA = rho * fma(m.AaT, T, fma(m.AaU, usq, m.Aa0)), rB = rho * fma(m.BaT, T, fma(m.BaU, usq, m.Ba0));
    const double rD = rho * m.Da;
    const double u3[3] = {ux, uy, uz};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const double w = m.c1 * u3[a], q = fma(rD, w * w, rA);
      e[1 + 2 * a] = fma(rB, w, q);
      e[2 + 2 * a] = fma(-rB, w, q);
    }
  }
  const double rA = rho * fma(m.AdT, T, fma(m.AdU, usq, m.Ad0)), rB = rho * fma(m.BdT, T, fma(m.BdU, usq, m.Bd0));
  const double rD = rho * m.Dd;
  const double sxy = ux + uy, dxy = ux - uy;
  const double t4[4] = {sxy + uz, sxy - uz, dxy + uz, dxy - uz};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double w = m.s * t4[k], q = fma(rD, w * w, rA);
    e[7 + k] = fma(rB, w, q);
    e[14 - k] = fma(-rB, w, q);
  }
}

template <typename R>
__global__ void init_kernel(R* __restrict__ f, Layout L, Model<double> m, const double* __restrict__ rho,
                            const double* __restrict__ u, const double* __restrict__ T) {
  const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  int x, y, z;
  if (!cell_of(L, k, x, y, z)) return;
  const long long n = L.ncell();
  double e[NV];
  feq_fp64(m, rho[k], u[k], u[n + k], u[2 * n + k], T[k], e);
  store_cell(f, L.fs, L.at(x, y, z), e);
}

// One thread per cell; the sums run in fixed point (fixed_sum.cuh), so of the
// FP64 pipe's work the 15 conversions from float and half of the moments'
// operations go.
template <typename R>
__global__ void __launch_bounds__(256) moments_kernel(const R* __restrict__ f, Layout L, Model<double> m,
                                                      double* __restrict__ rho, double* __restrict__ u,
                                                      double* __restrict__ T) {
  const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  int x, y, z;
  if (!cell_of(L, k, x, y, z)) return;
  const long long n = L.ncell(), at = L.at(x, y, z);
  R v[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) v[i] = f[i * L.fs + at];
  double r, ux, uy, uz, t;
  fx::moments_fixed(m, v, r, ux, uy, uz, t);
  rho[k] = r;
  u[k] = ux;
  u[n + k] = uy;
  u[2 * n + k] = uz;
  T[k] = t;
}

template <typename R>
__global__ void pack_kernel(const R* __restrict__ f, Layout L, R* __restrict__ dense) {
  const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  int x, y, z;
  if (!cell_of(L, k, x, y, z)) return;
  const long long n = L.ncell(), idx = L.at(x, y, z);
#pragma unroll
  for (int i = 0; i < NV; ++i) dense[i * n + k] = f[i * L.fs + idx];
}

template <typename R>
__global__ void unpack_kernel(R* __restrict__ f, Layout L, const R* __restrict__ dense) {
  const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  int x, y, z;
  if (!cell_of(L, k, x, y, z)) return;
  const long long n = L.ncell(), idx = L.at(x, y, z);
#pragma unroll
  for (int i = 0; i < NV; ++i) f[i * L.fs + idx] = dense[i * n + k];
}

// Two x-columns of every (y, z) row and field against a dense [15][nz][ny][2]
// array: to_dense = 1 copies the interior columns next to the x face `side`
// (x = 0, 1 or nx-2, nx-1) out, to_dense = 0 writes the two layers outside it
// (x = -2, -1 or nx, nx+1).  One thread per (field, row, column).
template <typename R>
__global__ void halo_kernel(R* __restrict__ f, Layout L, int side, int to_dense, R* __restrict__ dense) {
  const long long rows = (long long)L.ny * L.nz;
  const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= rows * 2 * NV) return;
  const int j = (int)(k & 1);
  const long long r = (k >> 1) % rows;
  const int i = (int)((k >> 1) / rows);
  const int y = (int)(r % L.ny), z = (int)(r / L.ny);
  const int x = to_dense ? (side ? L.nx - 2 + j : j) : (side ? L.nx + j : -2 + j);
  const long long at = (long long)i * L.fs + L.at(x, y, z);
  if (to_dense) dense[k] = f[at];
  else f[at] = dense[k];
}

// conservation sums: blocks of 12 warps, 4 row slots x 3 groups of 5 fields
constexpr int RED_GROUPS = 3, RED_GF = NV / RED_GROUPS, RED_ROWS = 4;
constexpr int RED_THREADS = 32 * RED_GROUPS * RED_ROWS;
static_assert(RED_GROUPS * RED_GF == NV, "field groups cover the 15 fields");

// Per-field accumulation of one thread's cells, four floats or two doubles at
// a time: double for double storage; for float storage error-free double-float
// pairs, converted to double at the end (GB300's FP64 rate would make a
// per-value conversion and double add the bottleneck of this memory-bound
// reduction).  `largest` follows the values' magnitudes, on the integer ALUs
// for doubles (a double comparison runs on the FP64 pipe); a NaN shows in the
// sum.
template <typename R, int N>
struct FieldAcc;
template <int N>
struct FieldAcc<double, N> {
  // the two values of a load, then up to FOLD such sums, then those: a lane's
  // chain of additions, and its rounding where all values are alike, does not
  // grow with the grid (256^3, uniform values, 432 of them per lane, relative
  // error of the total, 400 values: rms 5.9e-15, worst 1.2e-14 in one chain;
  // 5.6e-16, 1.5e-15 so)
  static constexpr int FOLD = 32;
  double s[N], total[N];
  int largest = 0, loads = 0;
  __device__ FieldAcc() {
#pragma unroll
    for (int i = 0; i < N; ++i) s[i] = total[i] = 0.0;
  }
  __device__ __forceinline__ void add(int i, const double v[2]) {
    s[i] += v[0] + v[1];
    largest = max(largest, max(fx::mag(v[0]), fx::mag(v[1])));
  }
  __device__ __forceinline__ void renorm() {
    if (++loads % FOLD != 0) return;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      total[i] += s[i];
      s[i] = 0.0;
    }
  }
  __device__ __forceinline__ double value(int i) const { return total[i] + s[i]; }
  __device__ __forceinline__ bool in_range() const { return true; }
  // a NaN or infinity has a high word above every finite one
  __device__ __forceinline__ bool bad() const { return !(__hiloint2double(largest, 0) < 1e300); }
};
template <int N>
struct FieldAcc<float, N> {
  DFloat2 s[N];
  float largest = 0.f;
  __device__ __forceinline__ void add(int i, const float v[4]) {
    s[i].add(make_float2(v[0], v[1]));
    s[i].add(make_float2(v[2], v[3]));
#pragma unroll
    for (int k = 0; k < 4; ++k) largest = fmaxf(largest, fabsf(v[k]));
  }
  __device__ __forceinline__ void renorm() {
#pragma unroll
    for (int i = 0; i < N; ++i) s[i].renorm();
  }
  __device__ __forceinline__ double value(int i) const { return s[i].value(); }
  __device__ __forceinline__ bool in_range() const { return !(largest >= 1e30f); }  // 2^27 such values stay finite
  __device__ __forceinline__ bool bad() const { return !(largest < 3.0e38f); }
};

// 16-byte vector loads of float / double rows (read once: streaming hint).
__device__ __forceinline__ void load16(const float* p, float v[4]) {
  const float4 q = __ldcs(reinterpret_cast<const float4*>(p));
  v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
__device__ __forceinline__ void load16(const double* p, double v[2]) {
  const double2 q = __ldcs(reinterpret_cast<const double2*>(p));
  v[0] = q.x; v[1] = q.y;
}

// Deterministic FP64 global sums of (rho, rho u, E) over interior cells.  The
// moments are linear in f, so the kernel sums each field f_i over the cells
// and combines the 15 field totals at the end: mass = sum_i F_i, momentum =
// sum_i v_i F_i, energy = sum_i (v_i^2 + eta_i^2) F_i.  Each warp takes whole
// x rows (rows b * RED_ROWS + slot, stepping by gridDim.x * RED_ROWS) and one
// group of five fields, three warps per row slot; a lane reads 16 bytes of
// each of its five fields per x step (a warp: 512 contiguous bytes per
// field), all five loads issued before the first add.  Few registers per
// thread let many warps, and so many bytes, be in flight per SM.  Values
// past the row end are masked to zero.  Warps reduce by a fixed shuffle
// tree, blocks by warp order, and the last block to finish sums the
// per-block totals with 256 of its threads in a fixed split (16 strided
// partial sums per field, then in order).  The order never depends on
// timing, so the result is bitwise reproducible for a given grid.
template <typename R>
__global__ void __launch_bounds__(RED_THREADS) conserved_kernel(const R* __restrict__ f, Layout L, Model<double> m,
                                                                double* __restrict__ partials,
                                                                unsigned* __restrict__ counter,
                                                                double* __restrict__ result,
                                                                unsigned* __restrict__ flags) {
  constexpr int WARPS = RED_THREADS / 32;
  __shared__ double wsum[WARPS][16];
  __shared__ double part[16][16];
  __shared__ bool last;
  FieldAcc<R, RED_GF> acc;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int grp = warp % RED_GROUPS, slot = warp / RED_GROUPS;
  const int nrows = L.ny * L.nz;
  const int nr = gridDim.x * RED_ROWS;
  constexpr int VW = 16 / (int)sizeof(R);  // elements per 16-byte load
  const R* fg = f + (long long)grp * RED_GF * L.fs;
  auto each = [&](auto take) {  // every vector of this lane, masked past the row end
    for (int r = blockIdx.x * RED_ROWS + slot; r < nrows; r += nr) {
      // interior rows start at x = OX (a multiple of 8 elements): 16-byte aligned
      const R* row = fg + L.at(0, r % L.ny, r / L.ny);
      for (int x0 = lane * VW; x0 < L.nx; x0 += 32 * VW) {
        // the last vector may reach up to VW - 1 elements past the row end,
        // into the row's halo and padding (inside the buffer); masked below
        R v[RED_GF][VW];
#pragma unroll
        for (int i = 0; i < RED_GF; ++i) load16(row + i * L.fs + x0, v[i]);
        if (x0 + VW > L.nx) {
#pragma unroll
          for (int i = 0; i < RED_GF; ++i)
#pragma unroll
            for (int k = 0; k < VW; ++k)
              if (x0 + k >= L.nx) v[i][k] = R(0);
        }
        take(v);
      }
    }
  };
  each([&](const R(&v)[RED_GF][VW]) {
#pragma unroll
    for (int i = 0; i < RED_GF; ++i) acc.add(i, v[i]);
    acc.renorm();
  });
  double sums[RED_GF];
#pragma unroll
  for (int i = 0; i < RED_GF; ++i) sums[i] = acc.value(i);
  if (!acc.in_range()) {
    // float sums of such values may have left the float range: once more in double
#pragma unroll
    for (int i = 0; i < RED_GF; ++i) sums[i] = 0.0;
    each([&](const R(&v)[RED_GF][VW]) {
#pragma unroll
      for (int k = 0; k < VW; ++k)
#pragma unroll
        for (int i = 0; i < RED_GF; ++i) sums[i] += (double)v[i][k];
    });
  }
  bool bad = acc.bad();
#pragma unroll
  for (int i = 0; i < RED_GF; ++i) bad = bad || fx::mag(sums[i]) > 0x7ff00000;  // a NaN, on the integer ALUs
  if (bad) atomicOr(flags, (unsigned)LBM_HEALTH_NONFINITE);
#pragma unroll
  for (int i = 0; i < RED_GF; ++i) {
    double v = sums[i];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if (lane == 0) wsum[warp][grp * RED_GF + i] = v;
  }
  // the other groups' fields of this warp are zero (adding them is exact)
  if (lane < NV && (lane < grp * RED_GF || lane >= (grp + 1) * RED_GF)) wsum[warp][lane] = 0.0;
  __syncthreads();
  if (threadIdx.x < NV) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) t += wsum[w][threadIdx.x];
    partials[blockIdx.x * 16 + threadIdx.x] = t;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = (atomicAdd(counter, 1u) == gridDim.x - 1);
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (threadIdx.x < 256) {
    // field i, strided part j of 16; the partials are read through L2 (the
    // other blocks' writes are ordered before their counter increments),
    // eight loads in flight per step of the fixed-order sum
    const int i = threadIdx.x & 15, j = threadIdx.x >> 4;
    double t = 0.0;
    if (i < NV) {
      unsigned b = j;
      for (; b + 7 * 16 < gridDim.x; b += 8 * 16) {
        double v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = __ldcg(partials + (b + q * 16) * 16 + i);
#pragma unroll
        for (int q = 0; q < 8; ++q) t += v[q];
      }
      for (; b < gridDim.x; b += 16) t += __ldcg(partials + b * 16 + i);
    }
    part[j][i] = t;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double F[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      F[i] = 0.0;
      for (int j = 0; j < 16; ++j) F[i] += part[j][i];
    }
    const double sa = ((F[1] + F[2]) + (F[3] + F[4])) + (F[5] + F[6]);
    const double sd = ((F[7] + F[8]) + (F[9] + F[10])) + ((F[11] + F[12]) + (F[13] + F[14]));
    result[0] = F[0] + sa + sd;
    result[1] = m.c1 * (F[1] - F[2]) + m.s * (((F[7] + F[8]) + (F[9] + F[10])) - ((F[11] + F[12]) + (F[13] + F[14])));
    result[2] = m.c1 * (F[3] - F[4]) + m.s * (((F[7] + F[8]) + (F[11] + F[12])) - ((F[9] + F[10]) + (F[13] + F[14])));
    result[3] = m.c1 * (F[5] - F[6]) + m.s * (((F[7] + F[9]) + (F[11] + F[13])) - ((F[8] + F[10]) + (F[12] + F[14])));
    result[4] = m.eta0sq * F[0] + m.c1sq * sa + m.c2sq * sd;
    *counter = 0u;
  }
}

inline int blocks_for(long long n, int threads) { return (int)((n + threads - 1) / threads); }

}  // namespace

cudaError_t launch_fill(int prec, void* f, const Layout& L, const Model<double>& md, const Model<float>& mf,
                        const BcDesc& bc, unsigned mask, cudaStream_t st) {
  if (!mask) return cudaSuccess;
  long long cmax = 1;
  const long long cnt[3] = {(long long)L.ny * L.nz, (long long)L.nx * L.nz, (long long)L.nx * L.ny};
  for (int a = 0; a < 3; ++a)
    if (((mask >> (2 * a)) & 3u) && cnt[a] > cmax) cmax = cnt[a];
  dim3 grid((unsigned)((cmax + 127) / 128), 6);
  if (prec == LBM_FP64) return launch_chained(fill_kernel<double, double>, grid, 128, 0, st, (double*)f, L, md, bc, mask);
  return launch_chained(fill_kernel<float, float>, grid, 128, 0, st, (float*)f, L, mf, bc, mask);
}

cudaError_t launch_init(int prec, void* f, const Layout& L, const Model<double>& m, const double* rho, const double* u,
                        const double* T, cudaStream_t st) {
  const int b = blocks_for(L.ncell(), 256);
  if (prec == LBM_FP64) init_kernel<double><<<b, 256, 0, st>>>((double*)f, L, m, rho, u, T);
  else init_kernel<float><<<b, 256, 0, st>>>((float*)f, L, m, rho, u, T);
  return cudaGetLastError();
}

cudaError_t launch_moments(int prec, const void* f, const Layout& L, const Model<double>& m, double* rho, double* u,
                           double* T, cudaStream_t st) {
  const int b = blocks_for(L.ncell(), 256);
  if (prec == LBM_FP64) moments_kernel<double><<<b, 256, 0, st>>>((const double*)f, L, m, rho, u, T);
  else moments_kernel<float><<<b, 256, 0, st>>>((const float*)f, L, m, rho, u, T);
  return cudaGetLastError();
}

cudaError_t launch_pack(int prec, const void* f, const Layout& L, void* dense, cudaStream_t st) {
  const int b = blocks_for(L.ncell(), 256);
  if (prec == LBM_FP64) pack_kernel<double><<<b, 256, 0, st>>>((const double*)f, L, (double*)dense);
  else pack_kernel<float><<<b, 256, 0, st>>>((const float*)f, L, (float*)dense);
  return cudaGetLastError();
}

cudaError_t launch_unpack(int prec, void* f, const Layout& L, const void* dense, cudaStream_t st) {
  const int b = blocks_for(L.ncell(), 256);
  if (prec == LBM_FP64) unpack_kernel<double><<<b, 256, 0, st>>>((double*)f, L, (const double*)dense);
  else unpack_kernel<float><<<b, 256, 0, st>>>((float*)f, L, (const float*)dense);
  return cudaGetLastError();
}

cudaError_t launch_halo(int prec, void* f, const Layout& L, int side, int to_dense, void* dense, cudaStream_t st) {
  const int b = blocks_for((long long)L.ny * L.nz * 2 * NV, 256);
  if (prec == LBM_FP64) halo_kernel<double><<<b, 256, 0, st>>>((double*)f, L, side, to_dense, (double*)dense);
  else halo_kernel<float><<<b, 256, 0, st>>>((float*)f, L, side, to_dense, (float*)dense);
  return cudaGetLastError();
}

cudaError_t launch_conserved(int prec, const void* f, const Layout& L, const Model<double>& m, double* partials,
                             int max_blocks, unsigned* counter, double* result, unsigned* flags, cudaStream_t st) {
  // about eight rows per row slot, and no more blocks than run at once: a
  // block's reduction at its end is some 300 FP64 operations per warp (256^3
  // FP32, us per call: 2048 blocks 287, 455 blocks 239)
  int b = blocks_for((long long)L.ny * L.nz, 8 * RED_ROWS);
  if (b > max_blocks) b = max_blocks;
  if (b < 1) b = 1;
  if (prec == LBM_FP64)
    conserved_kernel<double><<<b, RED_THREADS, 0, st>>>((const double*)f, L, m, partials, counter, result, flags);
  else
    conserved_kernel<float><<<b, RED_THREADS, 0, st>>>((const float*)f, L, m, partials, counter, result, flags);
  return cudaGetLastError();
}

}  // namespace lbm
