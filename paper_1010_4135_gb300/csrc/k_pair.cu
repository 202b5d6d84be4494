// Tiled single-precision fused step, two x-adjacent cells per thread.
//
// Same plane ring as step_tiled_kernel (one 4D TMA copy per z plane into an
// mbarrier-tracked ring; see tma_ring.cuh), but each thread of a 32 x 8 tile
// owns the cell pair (x, x+1).  The pair is loaded with one 64-bit shared load
// per field and neighbour row, and everything that is the same arithmetic for
// both cells runs as packed f32x2 operations (FADD2, FMUL2, FFMA2), which
// halves the instructions the schedulers issue.
//
// Per interface the NND minmod is evaluated once: minmod(x, d) is x clamped
// to [min(d, 0), max(d, 0)], the two minmods of one cell share d, the pair
// shares the minmod of its middle x-interface, and the minmod of each
// z-interface is carried from plane z to plane z+1.  The Laplacian centre
// and the relaxation are folded into one coefficient per velocity shell:
//   f_new = keep_i f + (dt/tau) f^eq - (|v| dt/dx) C + (lambda_i dt/dx^2) S,
// with S the sum of the six neighbours and keep_i = 1 - dt/tau - 6 lambda_i dt/dx^2.
//
// The v_z < 0 velocities need plane z+2 for one term.  It is added when plane
// z+1 is worked on (part[] below), so a plane needs one plane of look-ahead,
// not two: two of the four ring slots hold copies in flight where it was one
// (together with the boundary code taken out of the loop, 256^3: 418 -> 385 us
// per step, 77 % of the measured copy bandwidth).
//
// Boundary layers (WtDesc): the planes of a periodic z axis are read where
// they are; the layers of reflecting faces and of extrapolating x faces are
// formed by the threads at the face when they read them, from the moments
// they hold anyway (two packed equilibria for a thread's pair, against a
// store, a separate pass or a re-read of the new state: reading a unit's own
// stores back cost 26 us per unit with a face, 383 -> 448 us on 256^3); and
// the kernel writes the periodic x and y images of the state it produces with
// the values themselves, so the next step needs no separate fill for them.
#include "pair_math.cuh"
#include "tma_ring.cuh"

namespace lbm {
namespace {

using ring::mbar_init;
using ring::mbar_expect_tx;
using ring::mbar_wait;
using ring::tma_load_plane;

// Tile geometry of the pair kernel: a TX x TY column of cells, one thread per
// cell pair (x, x+1), and a four-plane ring: cell plane z reads ring planes z
// (its x / y neighbours) and z+1 while z+2 and z+3 land.
template <int TX_, int TY_>
struct PairGeo {
  static constexpr int TX = TX_, TY = TY_, NSLOT = 4;
  static constexpr int BX = TX + 2 * TMA_LEFT, BY = TY + 4;  // tile with its halo
  static constexpr int PL = BX * BY;                          // floats per field in one plane tile
  static constexpr int SLOT_BYTES = NV * PL * 4;              // bytes one TMA copy delivers
  static constexpr int SLOT_STRIDE = (SLOT_BYTES + 127) / 128 * 128;
  static constexpr int SMEM = NSLOT * SLOT_STRIDE + NSLOT * 8;  // slots, then the mbarriers
  static constexpr int PX = TX / 2;                           // threads along x
  static constexpr int THREADS = PX * TY;
  // CTAs per SM that the shared memory allows (228 KB per SM, 1 KB reserved
  // per CTA, the batched kernel's 8-byte work-queue slot rounded to 128)
  static constexpr int CTAS_PER_SM = 233472 / (SMEM + 128 + 1024);
  static_assert(CTAS_PER_SM >= 1, "ring fits one CTA");
  static_assert(THREADS % 32 == 0, "whole warps");
  static_assert(PX == 16 || PX == 32,
                "64-bit shared loads: a half warp (one 128-byte wavefront) reads one contiguous tile row");
  static_assert(BX * 4 % 16 == 0 && BX <= 256, "TMA box inner extent: a 16-byte multiple, at most 256");
  static_assert(TX % 32 == 0, "tile rows start on 32-byte sectors (OX is a multiple of 8)");
};
// 32 x 8 tiles (the single-cell tiled kernel's box, 40 x 12): two CTAs of 4
// warps per SM.  With two planes in flight an L2 prefetch of later ones only
// adds L2 lookups (256^3, us per step: 385; one plane ahead 401, two 399,
// three 410 and more; with one plane in flight it was needed: 475 against 488).
// Larger tiles re-read fewer halo cells, but leave one CTA per SM: 64 x 8 in
// two halves 426, 32 x 16 415, 32 x 24 and 64 x 12 in three slots with 12
// warps of 168 registers 437 and 434.
using Geo = PairGeo<ring::TX, ring::TY>;
static_assert(Geo::BX == ring::BX && Geo::BY == ring::BY, "Geo shares the tiled kernel's tensor map");

using pm::bc2;
using pm::ld2;

// Forms of the kernel.  The plane loop is about as long as the instruction
// caches serve at full rate: code that few units or few grids run costs all
// units that carry it (256^3, us per step: the layers of x faces in the loop
// 14, those of y and z walls 20, the FP64 recovery 17; the boundary code in a
// second copy of the loop, for the units at a boundary only, 30 more than in
// the one loop).  So a launch takes the form with the parts its grids need.
// FULL: every tile lies inside the grid (nx and ny multiples of the tile), so
// the activity tests fold away.  R1: dt = tau (dt/tau = 1, keep_2 = 0).  RD:
// FP64 temperature recovery.  XF, WALL: layers of extrapolating / reflecting
// x faces, of reflecting y and z faces, formed as they are read.  FEW: some
// grid has fewer than four rows and periodic y, so its rows have several images
// (the others' rows keep their one address; found by walking a grid's rows, the
// images cost every grid of the launch: 256^3 with dt = tau/2 3468 us, now 427,
// beside 200 x 3 x 3 in a batch 3496, now 414).
template <bool FULL_, bool R1_, bool RD_, bool XF_, bool WALL_, bool FEW_>
struct Opt {
  static constexpr bool FULL = FULL_, R1 = R1_, RD = RD_, XF = XF_, WALL = WALL_, FEW = FEW_;
};

// One z-march unit: the TX x TY column at (x0, y0), planes z0 .. z0+nzc-1.
// Plane j of the unit is the ring's plane number jb + j (slot (jb+j) % NSLOT,
// phase parity ((jb+j) / NSLOT) & 1), so consecutive units of a CTA keep
// using the same barriers; jb advances by the unit's plane count.  All
// threads of the CTA call it together; timed_out is uniform.
template <int SCHEME, class G, class O>
__device__ __forceinline__ void pair_unit(const CUtensorMap* tin, const float* fin,
                                          float* __restrict__ fout, const Layout& L, const Model<float>& m,
                                          const WtDesc& wt, const RecoverDesc& rd, int x0, int y0, int z0,
                                          int nzc,
                                          unsigned* __restrict__ flags, unsigned char* smem, uint64_t* bars,
                                          unsigned& jb, bool& timed_out, unsigned wait_limit) {
  constexpr int NSLOT = G::NSLOT, PL = G::PL, BX = G::BX;
  const int tid = threadIdx.x;
  const int tx = tid % G::PX, ty = tid / G::PX;
  const int x = x0 + 2 * tx, y = y0 + ty;
  const bool act0 = O::FULL || ((x < L.nx) && (y < L.ny));
  const bool act1 = O::FULL || ((x + 1 < L.nx) && (y < L.ny));
  // ring planes 0 .. nzc+1 are the padded planes z0+2 .. z0+nzc+3 (interior
  // z0 .. z0+nzc+1); cell plane k reads ring planes k and k+1
  const int nplanes = nzc + 2;
  // interior plane z of the grid or its two z layers; a periodic z axis has no
  // layers: its planes are read where they are (WtDesc)
  auto zplane = [&](int z) {
    if (!wt.per[2]) return z;
    while (z < 0) z += L.nz;
    while (z >= L.nz) z -= L.nz;
    return z;
  };

  // copy ring plane j (interior z0 + j, padded two more) into its slot
  int issued = 0;  // thread 0 only
  auto issue = [&](int j) {
    const unsigned g = jb + (unsigned)j;
    float* dst = reinterpret_cast<float*>(smem + (g % NSLOT) * G::SLOT_STRIDE);
    mbar_expect_tx(&bars[g % NSLOT], G::SLOT_BYTES);
    tma_load_plane(dst, tin, x0 + OX - TMA_LEFT, y0, zplane(z0 + j) + 2, &bars[g % NSLOT]);
    issued = j + 1;
  };
  if (tid == 0) {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    for (int j = 0; j < NSLOT && j < nplanes; ++j) issue(j);
  }
  auto slot = [&](int j) {
    return reinterpret_cast<const float*>(smem + ((jb + (unsigned)j) % NSLOT) * G::SLOT_STRIDE);
  };
  // waits for data use wait_limit; the drain after a timeout uses the full limit
  auto arrived = [&](int j) {
    const unsigned g = jb + (unsigned)j;
    return mbar_wait(&bars[g % NSLOT], (g / NSLOT) & 1u, wait_limit);
  };
  auto drained = [&](int j) {
    const unsigned g = jb + (unsigned)j;
    return mbar_wait(&bars[g % NSLOT], (g / NSLOT) & 1u);
  };

  const int c = (ty + 2) * BX + TMA_LEFT + 2 * tx;  // own pair in a plane tile (even: 8-byte aligned)
  const long long gbase = L.at(x, y, z0);

  float2 h1[NV], h2[NV], carry[NV];
  const long long below1 = L.at(x, y, zplane(z0 - 1)), below2 = L.at(x, y, zplane(z0 - 2));
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    h1[i] = act0 ? ld2(fin + i * L.fs + below1) : make_float2(0.f, 0.f);
    h2[i] = act0 ? ld2(fin + i * L.fs + below2) : make_float2(0.f, 0.f);
    carry[i] = make_float2(0.f, 0.f);
  }

  unsigned bad = 0u;
  // ring planes 0 and 1 must have landed; the outcome is made uniform by the barrier
  {
    bool ok = arrived(0);
    ok = arrived(1) && ok;
    timed_out = __syncthreads_or(!ok) != 0;
  }
  if (O::WALL && wt.zlo && z0 < 2 && !timed_out && act0) {
    // the layers below a reflecting z-lo face, from the grid's plane 0
    const float* P0 = slot(0);
    float2 v[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = z0 == 0 ? ld2(P0 + i * PL + c) : h1[i];
    const pm::Mom r = pm::moments<false>(m, rd, v, P0, c, PL, act0, act1);
    const pm::Mom e1 = pm::wall_layer<2>(r, false), e2 = pm::wall_layer<2>(r, true);
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      h2[i] = pm::feq(m, z0 == 0 ? e2 : e1, i);
      if (z0 == 0) h1[i] = pm::feq(m, e1, i);
    }
  }
  if (!timed_out && SCHEME == LBM_SCHEME_NND) {
    const float* P0 = slot(0);
#pragma unroll
    for (int i = 0; i < NV; ++i) carry[i] = pm::carry0(i, h2[i], h1[i], ld2(P0 + i * PL + c));
  }

  // The v_z < 0 velocities' update of a plane needs the z difference one plane
  // further up than anything else does (pm::deferred), so it is finished and
  // stored a plane late: part[i] holds it without its last term.  Cell plane k
  // then reads ring planes k and k+1 only, and of the four slots two (not one)
  // hold copies in flight.
  float2 part[NV];

  // Besides the own pair of plane k (F, below), the planes below are carried
  // in registers only where a field needs them: h1 for the Laplacian of
  // f_0..f_6 and the z stencil of the axis velocities, the lower z difference
  // (dz) for the diagonal velocities with v_z > 0 (NND), and h2 for the
  // second-order upwind scheme.
  constexpr bool DZ = SCHEME == LBM_SCHEME_NND;
  float2 dz[NV];
  if (!timed_out && DZ) {
    const float* Q0 = slot(0);
#pragma unroll
    for (int i = 7; i < NV; ++i)
      if (vsign(i, 2) > 0) dz[i] = pm::sub(ld2(Q0 + i * PL + c), h1[i]);
  }
  // health: running minima of rho and T and a running sum of rho + T of each
  // cell of the pair, judged once at the end of the unit.  A non-finite rho or
  // T makes the sum non-finite, and so does a non-finite velocity: T is
  // (E/rho - u^2)/b, -inf or NaN when u^2 is inf or NaN.
  float2 hmin_rho = make_float2(INFINITY, INFINITY), hmin_T = hmin_rho, hsum = make_float2(0.f, 0.f);
  // periodic images of this pair (element offsets from its own index, 0 = none):
  // one per axis, or several y ones in a grid of fewer than four rows (few)
  unsigned img_y = 0, img_x = 0;
  const bool few = O::FEW && wt.per[1] && L.ny < 4;
  if (act0) {
    if (!few && wt.per[1]) img_y = (unsigned)L.sx * (unsigned)(y < 2 ? L.ny : (y >= L.ny - 2 ? -L.ny : 0));
    if (wt.per[0]) img_x = (unsigned)(x == 0 ? L.nx : (x == L.nx - 2 ? -L.nx : 0));
  }
  // store the pair's new values of plane k, the deferred fields (late) or the others, and their images
  auto store = [&](const float2(&out)[NV], int k, bool late) {
    // the pair's element offset within a field: below 2^32 (the host rejects
    // longer fields), so the fields' stores share one 32-bit offset
    const unsigned g = (unsigned)gbase + (unsigned)k * (unsigned)L.plane;
    auto put = [&](unsigned at) {
      if (act1) {
#pragma unroll
        for (int i = 0; i < NV; ++i)
          if (pm::deferred<SCHEME>(i) == late) *reinterpret_cast<float2*>(fout + i * L.fs + at) = out[i];
      } else if (act0) {
#pragma unroll
        for (int i = 0; i < NV; ++i)
          if (pm::deferred<SCHEME>(i) == late) fout[i * L.fs + at] = out[i].x;
      }
    };
    put(g);
    if (img_y | img_x) {
      if (img_y) put(g + img_y);
      if (img_x) put(g + img_x);
    }
    if (few && act0) {
#pragma unroll 1
      for (int j = 0; j < 4; ++j) {  // the four layers: -2, -1, ny, ny + 1
        const int q = j < 2 ? j - 2 : L.ny + j - 2;
        if ((q - y) % L.ny == 0) put(g + (unsigned)(q - y) * (unsigned)L.sx);
      }
    }
  };
  // faces whose layers are formed here, from the moments of the cells at the
  // face, at the moment they are read (WtDesc)
  const bool at_xlo = O::XF && wt.xlo && x == 0 && act0, at_xhi = O::XF && wt.xhi && x == L.nx - 2 && act0;
  const bool at_ylo = O::WALL && wt.ylo && y == 0 && act0, at_yhi = O::WALL && wt.yhi && y == L.ny - 1 && act0;
  const bool tile_y = O::WALL && ((wt.ylo && y0 == 0) || (wt.yhi && y0 + G::TY >= L.ny));
  // the pair's own values of the plane: loaded once for the first plane, then
  // carried from the previous plane's z-neighbour loads, so that the moments
  // of a plane start without waiting on shared memory (256^3: 0.4206 ->
  // 0.4173 ms per step, although the register rotation adds instructions)
  float2 F[NV];
  if (!timed_out) {
    const float* Q0 = slot(0);
#pragma unroll
    for (int i = 0; i < NV; ++i) F[i] = ld2(Q0 + i * PL + c);
  }
  for (int k = 0; k < nzc && !timed_out; ++k) {
    const float* P0 = slot(k);
    const float* P1 = slot(k + 1);
    float2 Z1[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) Z1[i] = ld2(P1 + i * PL + c);

    // moments (relations e1-e3), health, equilibrium and the per-field update
    const pm::Mom r = pm::moments<O::RD>(m, rd, F, P0, c, PL, act0, act1);
    {
      // the layers take the FP32 moments, as the fill forms them, also where
      // the cell's own were recovered in FP64
      auto face_moments = [&]() { return O::RD && rd.on ? pm::moments<false>(m, rd, F, P0, c, PL, act0, act1) : r; };
      // layers beyond the faces this pair touches: into the plane tile's halo
      // (x: read by this thread only; y: by the row above or below too, a row
      // of this warp), or in place of the plane above
      if (O::XF && (at_xlo | at_xhi)) {
#pragma unroll 1
        for (int lo = 0; lo < 2; ++lo) {
          if (!(lo ? at_xlo : at_xhi)) continue;
          float* t = const_cast<float*>(P0) + c + (lo ? -2 : 2);
          const pm::Mom e = pm::x_layers(face_moments(), lo ? wt.xlo : wt.xhi, lo);
#pragma unroll
          for (int i = 0; i < NV; ++i) *reinterpret_cast<float2*>(t + i * PL) = pm::feq(m, e, i);
        }
      }
      if (O::WALL && tile_y) {
        if (at_ylo | at_yhi) {
#pragma unroll 1
          for (int q = 0; q < 4; ++q) {  // lo inner, lo outer, hi inner, hi outer
            if (!(q < 2 ? at_ylo : at_yhi)) continue;
            float* t = const_cast<float*>(P0) + c + (q < 2 ? -1 - q : q - 1) * BX;
            const pm::Mom e = pm::wall_layer<1>(face_moments(), q & 1);
#pragma unroll
            for (int i = 0; i < NV; ++i) *reinterpret_cast<float2*>(t + i * PL) = pm::feq(m, e, i);
          }
        }
        __syncwarp();
      }
      // in every form, although only WALL ones can take it: compiled out of
      // the others it makes them slower (us: 256^3, 150 steps, 59942, without
      // 60169; 128^3, 150 steps, 9358, 9406; four served grids 17919, 18105)
      if (wt.zhi && z0 + k == L.nz - 1) {
        const pm::Mom e = pm::wall_layer<2>(face_moments(), false);
#pragma unroll
        for (int i = 0; i < NV; ++i) Z1[i] = pm::feq(m, e, i);
      }
    }
    hmin_rho = make_float2(fminf(hmin_rho.x, r.rho.x), fminf(hmin_rho.y, r.rho.y));
    hmin_T = make_float2(fminf(hmin_T.x, r.T.x), fminf(hmin_T.y, r.T.y));
    hsum = pm::add(hsum, pm::add(r.rho, r.T));
    // out: this plane's fields, and the deferred ones of the plane below
    float2 out[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const float2 o = pm::field_update<SCHEME, BX, DZ, O::R1>(m, i, P0 + i * PL + c, F[i], Z1[i], h1[i], h2[i],
                                                               carry[i], dz[i], pm::feq(m, r, i));
      if (pm::deferred<SCHEME>(i)) {
        out[i] = pm::tail(m, i, dz[i], part[i]);
        part[i] = o;
      } else {
        out[i] = o;
      }
    }
    store(out, k, false);
    if (k > 0) store(out, k - 1, true);
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      if (SCHEME == LBM_SCHEME_UPWIND2) h2[i] = h1[i];
      h1[i] = F[i];
      F[i] = Z1[i];
    }
    // ring plane k+2 (needed next step) must have landed; the barrier also
    // marks plane k as retired, so its slot takes plane k + NSLOT (releasing
    // the slots warp by warp, with no barrier, was slower: 390 us against 383)
    if (__syncthreads_or(!arrived(k + 2))) {
      timed_out = true;
      break;
    }
    if (tid == 0 && k + NSLOT < nplanes) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      issue(k + NSLOT);
    }
  }

  // the last plane's deferred fields, from ring plane nzc+1 (landed: the last step waited for it)
  if (nzc > 0 && !timed_out) {
    const float* P1 = slot(nzc + 1);
    float2 out[NV], top[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i)
      if (pm::deferred<SCHEME>(i)) top[i] = ld2(P1 + i * PL + c);
    const int over = z0 + nzc - (L.nz - 1);  // 0, 1: ring plane nzc+1 is the first, second layer above the grid
    if (O::WALL && wt.zhi && over >= 0) {
      // a reflecting z-hi face's, from the grid's last plane (still in its slot)
      const float* P0 = slot(nzc - over);
      float2 v[NV];
#pragma unroll
      for (int i = 0; i < NV; ++i) v[i] = ld2(P0 + i * PL + c);
      const pm::Mom e = pm::wall_layer<2>(pm::moments<false>(m, rd, v, P0, c, PL, act0, act1), over == 1);
#pragma unroll
      for (int i = 0; i < NV; ++i)
        if (pm::deferred<SCHEME>(i)) top[i] = pm::feq(m, e, i);
    }
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      if (!pm::deferred<SCHEME>(i)) continue;
      const float2 Z1 = top[i];
      out[i] = pm::tail(m, i, SCHEME == LBM_SCHEME_NND ? pm::mmc2(pm::sub(Z1, F[i]), carry[i]) : Z1, part[i]);
    }
    store(out, nzc - 1, true);
  }
  if (nzc > 0 && !timed_out) {
    const float mr[2] = {hmin_rho.x, hmin_rho.y}, mt[2] = {hmin_T.x, hmin_T.y}, hs[2] = {hsum.x, hsum.y};
    const bool on[2] = {act0, act1};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (!on[h]) continue;
      if (!(mr[h] > 0.f)) bad |= LBM_HEALTH_RHO;
      if (!(mt[h] > 0.f)) bad |= LBM_HEALTH_T;
      if (!(fabsf(hs[h]) < 1e30f)) bad |= LBM_HEALTH_NONFINITE;
    }
  }
  if (tid == 0 && timed_out) atomicOr(flags, (unsigned)LBM_HEALTH_TIMEOUT);
  if (bad) atomicOr(flags, bad);
  if (timed_out) {
    // leave no copy in flight: the newest plane of each slot is waited for (bounded)
    if (tid == 0) {
      for (int j = max(0, issued - NSLOT); j < issued; ++j) drained(j);
    }
    __syncthreads();
  }
  jb += (unsigned)nplanes;
}

template <int SCHEME, class G, class O>
__global__ void __launch_bounds__(G::THREADS, G::CTAS_PER_SM)
    step_pair_kernel(const __grid_constant__ CUtensorMap tin, const float* fin, float* __restrict__ fout,
                     Layout L, Model<float> m, WtDesc wt, RecoverDesc rd, ZSched zs, unsigned* __restrict__ flags,
                     unsigned wait_limit) {
  extern __shared__ __align__(128) unsigned char smem[];
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + G::NSLOT * G::SLOT_STRIDE);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int s = 0; s < G::NSLOT; ++s) mbar_init(&bars[s], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  chain_wait();
  unsigned jb = 0;
  bool timed_out = false;
  pair_unit<SCHEME, G, O>(&tin, fin, fout, L, m, wt, rd, blockIdx.x * G::TX, blockIdx.y * G::TY, zs.z0(blockIdx.z),
                          zs.len(blockIdx.z, L.nz), flags, smem, bars, jb, timed_out, wait_limit);
  chain_start();  // late: started early, the next step's CTAs pair up on the SMs that have room first
}

// Persistent batched step: two CTAs per SM take the units of every grid in
// the descriptor table (the long chunks of all grids, then the short ones;
// grid-major, then z chunk, then tile; each unit one
// z-march of a TX x TY column of one grid) from a work queue, one atomic
// increment per unit, so fast and slow CTAs balance.  Every CTA overshoots
// the queue once; the last CTA to finish resets the queue for the next
// launch (stream order), which keeps the launch replayable in a CUDA graph.
template <int SCHEME, class G, class O>
__global__ void __launch_bounds__(G::THREADS, G::CTAS_PER_SM)
    step_pair_batch_kernel(const __grid_constant__ BatchTable tab) {
  extern __shared__ __align__(128) unsigned char smem[];
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + G::NSLOT * G::SLOT_STRIDE);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int s = 0; s < G::NSLOT; ++s) mbar_init(&bars[s], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  chain_wait();
  unsigned jb = 0;
  bool timed_out = false;
  __shared__ long long next;
  for (;;) {
    if (threadIdx.x == 0) next = (long long)atomicAdd(tab.queue, 1ull);
    __syncthreads();
    const long long u = next;
    __syncthreads();
    if (u >= tab.total_units || timed_out) break;
    int e = 0;
    const bool late = u >= tab.long_units;
    while (e + 1 < tab.n && u >= (late ? tab.item[e + 1].first_short : tab.item[e + 1].first_long)) ++e;
    const BatchItem& it = tab.item[e];
    const long long local = u - (late ? it.first_short : it.first_long);
    const long long per_chunk = (long long)it.tiles_x * it.tiles_y;
    const int chunk = (int)(local / per_chunk) + (late ? it.zs.nbig : 0);
    const int t = (int)(local % per_chunk);
    // the unit's descriptors as locals: read through the runtime index e, the
    // table's constants would otherwise be re-loaded at every use in the plane
    // loop (256^3 alone: 0.497 -> 0.469 ms; eight 128^3: 0.556 -> 0.525 ms)
    const Layout L = it.L;
    const Model<float> m = it.m;
    const WtDesc wt = it.wt;
    const RecoverDesc rd = it.rd;
    const ZSched zs = it.zs;
    pair_unit<SCHEME, G, O>(&tab.map[e], it.fin, it.fout, L, m, wt, rd, (t % it.tiles_x) * G::TX,
                            (t / it.tiles_x) * G::TY, zs.z0(chunk), zs.len(chunk, L.nz), it.flags, smem, bars, jb,
                            timed_out, tab.wait_limit);
  }
  chain_start();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(tab.done, 1u) == gridDim.x - 1) {
      *tab.queue = 0ull;
      *tab.done = 0u;
      __threadfence();
    }
  }
}

// What the forms go by, over all grids of a launch.
struct Need {
  bool full = true, r1 = true, rd = false, xf = false, wall = false, few = false;
  void add(const Layout& L, const Model<float>& m, const WtDesc& wt, const RecoverDesc& r) {
    full = full && L.nx % Geo::TX == 0 && L.ny % Geo::TY == 0;
    r1 = r1 && m.dt_tau == 1.0f && m.keep2 == 0.0f;
    rd = rd || r.on;
    xf = xf || wt.xlo || wt.xhi;
    wall = wall || wt.ylo || wt.yhi || wt.zlo || wt.zhi;
    few = few || (wt.per[1] && L.ny < 4);
  }
};

// The forms that exist: NND with dt = tau and no recovery (every run of the
// paper) has one per boundary need; NND with another relaxation time or with
// recovery has one for whole and one for cut tiles, each with x faces (256^3,
// us per step against the form with all parts: dt = tau/2 387, 427; recovery
// 398, 505); everything else (the upwind schemes, 368 and 375; walls or few
// rows with either of those; both walls and few rows) one form with all parts.
using FullPlain = Opt<true, true, false, false, false, false>;
using FullFaces = Opt<true, true, false, true, false, false>;
using Plain = Opt<false, true, false, false, false, false>;
using Faces = Opt<false, true, false, true, false, false>;
using Walls = Opt<false, true, false, true, true, false>;
using FewRows = Opt<false, true, false, true, false, true>;
using FullRelax = Opt<true, false, false, true, false, false>;
using Relax = Opt<false, false, false, true, false, false>;
using FullRecover = Opt<true, false, true, true, false, false>;
using Recover = Opt<false, false, true, true, false, false>;
using General = Opt<false, false, true, true, true, true>;

template <int SCHEME, class F>
void with_form(const Need& n, F f) {
  if constexpr (SCHEME == LBM_SCHEME_NND) {
    if (!n.few && !n.wall && (n.rd || !n.r1)) {
      if (n.rd) return n.full ? f(FullRecover()) : f(Recover());
      return n.full ? f(FullRelax()) : f(Relax());
    }
    if (n.r1 && !n.rd && !(n.few && n.wall)) {
      if (n.few) return f(FewRows());
      if (n.wall) return f(Walls());
      if (n.full) return n.xf ? f(FullFaces()) : f(FullPlain());
      return n.xf ? f(Faces()) : f(Plain());
    }
  }
  f(General());
}

template <int SCHEME, class... O>
cudaError_t set_attributes() {
  const void* fn[] = {(const void*)step_pair_kernel<SCHEME, Geo, O>..., (const void*)step_pair_batch_kernel<SCHEME, Geo, O>...};
  cudaError_t e = cudaSuccess;
  for (const void* f : fn)
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, Geo::SMEM);
  return e;
}

template <int SCHEME>
void launch_scheme(const CUtensorMap& map, const float* fin, float* fout, const Layout& L, const Model<float>& m,
                   const WtDesc& wt, const RecoverDesc& rd, const ZSched& zs, unsigned* flags, unsigned wait_limit,
                   cudaStream_t st) {
  dim3 grid((L.nx + Geo::TX - 1) / Geo::TX, (L.ny + Geo::TY - 1) / Geo::TY, zs.nch);
  Need need;
  need.add(L, m, wt, rd);
  with_form<SCHEME>(need, [&](auto o) {
    launch_chained(step_pair_kernel<SCHEME, Geo, decltype(o)>, grid, Geo::THREADS, Geo::SMEM, st, map, fin, fout, L, m, wt,
                   rd, zs, flags, wait_limit);
  });
}

template <int SCHEME>
void launch_batch_scheme(const BatchTable& tab, int grid, cudaStream_t st) {
  Need need;
  for (int e = 0; e < tab.n; ++e) need.add(tab.item[e].L, tab.item[e].m, tab.item[e].wt, tab.item[e].rd);
  with_form<SCHEME>(need, [&](auto o) {
    launch_chained(step_pair_batch_kernel<SCHEME, Geo, decltype(o)>, grid, Geo::THREADS, Geo::SMEM, st, tab);
  });
}

}  // namespace

cudaError_t prepare_pair_kernels() {
  cudaError_t e = set_attributes<LBM_SCHEME_NND, FullPlain, FullFaces, Plain, Faces, Walls, FewRows, FullRelax, Relax,
                                 FullRecover, Recover, General>();
  if (e == cudaSuccess) e = set_attributes<LBM_SCHEME_UPWIND2, General>();
  if (e == cudaSuccess) e = set_attributes<LBM_SCHEME_UPWIND1, General>();
  return e;
}

PairShape pair_shape() { return {Geo::TX, Geo::TY, Geo::CTAS_PER_SM}; }

cudaError_t launch_step_pair_batch(int scheme, const BatchTable& tab, int grid, cudaStream_t st) {
  switch (scheme) {
    case LBM_SCHEME_NND: launch_batch_scheme<LBM_SCHEME_NND>(tab, grid, st); break;
    case LBM_SCHEME_UPWIND2: launch_batch_scheme<LBM_SCHEME_UPWIND2>(tab, grid, st); break;
    default: launch_batch_scheme<LBM_SCHEME_UPWIND1>(tab, grid, st);
  }
  return cudaGetLastError();
}

cudaError_t launch_step_pair(int scheme, const CUtensorMap& map, const float* fin, float* fout, const Layout& L,
                             const Model<float>& m, const WtDesc& wt, const RecoverDesc& rd, const ZSched& zs,
                             unsigned* flags, unsigned wait_limit, cudaStream_t st) {
  switch (scheme) {
    case LBM_SCHEME_NND: launch_scheme<LBM_SCHEME_NND>(map, fin, fout, L, m, wt, rd, zs, flags, wait_limit, st); break;
    case LBM_SCHEME_UPWIND2:
      launch_scheme<LBM_SCHEME_UPWIND2>(map, fin, fout, L, m, wt, rd, zs, flags, wait_limit, st);
      break;
    default: launch_scheme<LBM_SCHEME_UPWIND1>(map, fin, fout, L, m, wt, rd, zs, flags, wait_limit, st);
  }
  return cudaGetLastError();
}

// 1/x as the FP32 step kernels form the inverse density (pm::rcp2), two
// values per thread; an odd tail pads its second lane with 1.
__global__ void __launch_bounds__(256) reciprocal_kernel(const float* __restrict__ x, float* __restrict__ y,
                                                         long long n) {
  const long long stride = 2LL * gridDim.x * blockDim.x;
  for (long long i = 2LL * ((long long)blockIdx.x * blockDim.x + threadIdx.x); i < n; i += stride) {
    const bool two = i + 1 < n;
    const float2 r = pm::rcp2(make_float2(x[i], two ? x[i + 1] : 1.f));
    y[i] = r.x;
    if (two) y[i + 1] = r.y;
  }
}

cudaError_t launch_reciprocal_fp32(const float* x, float* y, long long n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const long long pairs = (n + 1) / 2;
  const int blocks = (int)std::min<long long>((pairs + 255) / 256, 152LL * 8);
  reciprocal_kernel<<<blocks, 256, 0, st>>>(x, y, n);
  return cudaGetLastError();
}

}  // namespace lbm
