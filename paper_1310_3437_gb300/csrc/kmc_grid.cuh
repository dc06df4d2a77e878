// kmc_grid.cuh -- per-step search grid and the guard bands of the binary32
// pre-tests, computed on the device by a few warps per simulation.
//
// Cell size.  A candidate pair has |r| <= d_min + |v| t* < d0 + |v_i - v_j| dt
// <= d0 + (s_i + s_j) dt with s = |v| (Sec. 2: the partner must reach its distance
// of closest approach within the next time step).  With every particle at most S
// fast, cells at least d0 + 2 S dt wide hold each partner in the same or a
// neighbouring cell (Sec. 2: 26 neighbours in 3D).  With stencil K the cell is 1/K of
// that and K cells are searched on each side.  The width gets a relative margin m
// for the binary32 cell assignment, and cell_scale >= 1 only enlarges it.
//
// Speed split.  The fastest particle sets S = vmax, although nearly all particles
// are much slower.  The grid may instead be sized for a threshold S1 < vmax: the
// particles faster than S1 ("fast") are sorted into a second population.  Slow-slow
// pairs are searched on the S1 grid as above; every fast particle searches c cells
// on each side, c = ceil((d0 + 2 vmax dt) / w), over both populations (fast-fast
// pairs once, by the lower index).  Each candidate pair is still tested exactly
// once.  S1 is chosen per step from the number of particles above a few trial
// thresholds (counted by the push of the previous step) with a cost estimate.
// None of this can change a result, only the amount of work.  An axis with fewer
// than 2K+1 cells becomes a single cell (searched once, no duplicate neighbours).
#pragma once

#include "kmc_internal.cuh"

namespace kmc {

__device__ __forceinline__ float f_up(double x) { return __double2float_ru(x); }

// The builder runs on one warp per simulation between the push and the next step's
// count, so its latency is in every step: what takes it is the length of the chain of
// dependent operations, and on this part a binary64 division or square root is a chain
// of about 560 or 595 cycles and a 64-bit integer division of 440 (a binary32 one: 35).
// Hence: the cell counts and the cost estimates in binary32 (only the speed depends on
// the choice; the margins of the cell width cover the rounding, see plan_cells), square
// roots as upper bounds from the rounded-up binary32 root, per-axis values on a lane
// each, every parameter read before the first use of any, and the guard bands, which the
// count does not need, left to the scan (compute_guards).  One simulation, record and grid:
// 35 -> 4.8 us at 4096 particles, 47 -> 5.3 us at 2^20.
struct CellPlan {
  int nc[3];
  float m;
  uint32_t col_shift, col_tz, nkeys;
  bool ok;
};

// Mean particles per cell from which the binary32 path searches with tiles.  On the same grid
// the two are close: slow pairs of a step at 2^21 particles, rows against tiles, tube at 1 per
// cell 165 and 175 us, at 4.8 180 and 198; plane at 2.5 102 and 117; box at 4.1 226 and 212, at
// 8.4 268 and 250; blast at 5.8 319 and 249, at 13 393 and 308.  But the line also sets the
// grid: the row search's time hardly depends on the filling (its rows are trimmed to the
// particle's reach), the tiled one's on the cells, so with tiles the speed split takes fuller
// cells and fewer fast particles.  Whole passes with the line at 2.5, 3.5, 5, 7 and 10: four
// steps of the 2^24 tube 13.11, 13.12, 13.10, 13.52 and 14.39 ms, of 10^7 particles in the
// plane 5.83, 5.83, 5.84, 6.04 and 6.35, eight of a box of 262 k 1.033, 1.045, 1.058, 1.083 and
// 1.041 (which search takes how much of it changes from line to line); a request of 50 k, a
// 2^20 job, an ensemble of 30 and a 2^21 blast are the same within 1 %.
constexpr float kTileOccupancy = 3.5f;

// an upper bound of sqrt(x) for x >= 0, within 2^-19 of it
__device__ __forceinline__ double sqrt_up(float x) {
  return (double)__fsqrt_ru(x) * (1.0 + 0x1p-20);
}

// x 2^e for a positive x, e in the place of a high word's exponent; 0 below the normal range
__device__ __forceinline__ double times_2(double x, int e) {
  const int hi = __double2hiint(x) + e;
  return hi < 0x00100000 ? 0.0 : __hiloint2double(hi, __double2loint(x));
}

// cells for search radius h (before the stencil split); key space capped by max_keys.
// Along x the radius is split into K * kxm cells (kxm = 2: narrow cells along the rows
// of the row search), along y and z into K.  In binary32: the quotient is within 4 u32
// of the exact one, so a cell is at least h (1 + m) (1 - 5 u32) / Ka wide, and the
// binary32 cell assignment needs 8 u32 nmax of the margin m >= 1e-4 + 16 u32 nmax.
__device__ inline CellPlan plan_cells(const float ext[3], float h, int K, uint64_t max_keys,
                                      int kxm = 1) {
  CellPlan p;
  p.ok = false;
  p.m = 0.0f;
  p.col_shift = 0;
  p.col_tz = 1;
  p.nkeys = 1;
  p.nc[0] = p.nc[1] = p.nc[2] = 1;
  for (int attempt = 0; attempt < 64; ++attempt) {
    // margin for binary32 cell assignment: index error <= 4 u32 n per particle
    const float ih = 1.0f / h;
    const float q0 = ext[0] * (float)(K * kxm) * ih, q1 = ext[1] * (float)K * ih,
                q2 = ext[2] * (float)K * ih;
    const float nmax = fminf(fmaxf(q0, fmaxf(q1, q2)), 65535.0f);
    p.m = 1e-4f + 16.0f * 0x1p-24f * nmax;
    const float shrink = 1.0f / (1.0f + p.m);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int Ka = a == 0 ? K * kxm : K;
      const float q = (a == 0 ? q0 : a == 1 ? q1 : q2) * shrink;
      int c = q > 65535.0f ? 65535 : (int)q;  // q >= 0: the conversion is the floor
      if (c < 2 * Ka + 1) c = 1;
      p.nc[a] = c;
    }
    // key space of the tiled column order: T x T Morton tiles, T = 2^t <= 8
    const uint32_t ny = (uint32_t)p.nc[1], nz = (uint32_t)p.nc[2];
    const uint32_t small = ny < nz ? ny : nz;
    const uint32_t t = small >= 8u ? 3u : small >= 4u ? 2u : small >= 2u ? 1u : 0u;
    const uint32_t ty = (ny + (1u << t) - 1u) >> t, tz = (nz + (1u << t) - 1u) >> t;
    const uint64_t nkeys = ((uint64_t)(ty * tz) << (2 * t)) * (uint64_t)p.nc[0];
    if (nkeys <= max_keys) {
      p.col_shift = t;
      p.col_tz = tz;
      p.nkeys = (uint32_t)nkeys;
      p.ok = true;
      return p;
    }
    h *= 1.25f;  // coarsen until the key space fits
  }
  return p;
}

// Cost estimates for the choice of the split threshold, in units of one pair test of
// the row search (measured on GB300 at 2^24 particles, 6.6 ps; only the ratios matter).
// A slow particle in the row search: its trimmed half-stencil, about 5 tests per particle
// per cell (rho = particles per cell of width w), and its set-up (about 6 tests' time).  In
// tiles (107 ps at 7 per cell, 262 at about 45): 0.65 rho + 11.5, with binary64 records 23
// (162 ps at 1.2 per cell).  A fast particle: its reach-trimmed stencil (about 1.4 times the
// sphere of radius R_f) at 1.4 tests' time per test plus 10 per (y, z) column it walks, three
// times that with binary64 tests.  (With the row search's cost for well filled cells and the
// fast search 1.4 times as dear, too many particles were fast: 10 steps of a 2^21 blast 10.4
// against 9.55 ms, of an ensemble of 30 2.50 against 2.41, 2^24 tube 12.97 against 12.57.)
__device__ inline float slow_cost(float n, float rho, bool fp32) {
  if (!fp32) return n * (0.65f * rho + 23.0f);
  return n * (rho < kTileOccupancy ? 5.0f * rho + 6.0f : 0.65f * rho + 11.5f);
}
__device__ inline float fast_cost(float nfast, float rho, float rf_cells, float ncol, bool fp32) {
  const float tests = rho * 1.4f * 4.18879f * rf_cells * rf_cells * rf_cells;
  return nfast * (fp32 ? 1.0f : 3.0f) * (1.4f * tests + 10.0f * ncol);
}

// extent along x: the box, or the upper wall at the start of the step (particles are below it)
__device__ __forceinline__ double extent_x(int bc, double box, double x0, double up, double dt,
                                           uint64_t step) {
  if (bc != KMC_REFLECT) return box;
  const double X = x0 - up * ((double)step * dt);
  return X > 0.0 ? X : box;
}

// Trial thresholds of the speed split, fractions of the bound V of max |v| (squares
// rounded down), with their particle counts cleared for the next count: lane t the
// threshold t.
__device__ inline void set_split_thresholds(SimDev& s, float vmax2_bound, uint32_t lane) {
  if (lane >= (uint32_t)kSplitTrials) return;
  const double fV = (double)split_frac((int)lane) * sqrt_up(vmax2_bound);
  s.d.split_thr[lane] = __double2float_rd(fV * fV);
  s.d.split_cnt[lane] = 0;
}

// Called by all 32 lanes of a warp: lane t < kSplitTrials estimates the cost of
// trial threshold t, all lanes choose alike, lanes 0..2 take one axis each and lane 0
// writes the rest of the grid.
__device__ inline void compute_grid(SimDev& s, float vmax2_bound, uint64_t step, bool have_counts,
                                    uint32_t lane) {
  constexpr uint32_t kAll = 0xFFFFFFFFu;
  // ---- parameters, all loads in flight together --------------------------------
  const int K = s.K, search_kernel = s.search_kernel, split_ok = s.split_ok;
  const uint32_t n = s.n, cell_cap = s.cell_cap;
  const bool fp32 = s.precision == KMC_GUARDED_FP32;
  const double d0 = s.d0, dt = s.dt, cell_scale = s.cell_scale;
  const float min_occ = (float)s.split_min_occ;
  const double box0 = s.box[0], box1 = s.box[1], box2 = s.box[2];
  const int bc0 = s.bc[0], bc1 = s.bc[1], bc2 = s.bc[2];
  const double x0 = s.piston_x0, up = s.piston_u;
  const bool can_split = split_ok && have_counts;
  const uint32_t my_trial = lane < (uint32_t)kSplitTrials ? lane : 0u;
  const float my_thr = s.d.split_thr[my_trial];
  const float my_nfast = (float)s.d.split_cnt[my_trial];

  const double scale = cell_scale > 1.0 ? cell_scale : 1.0;
  const double V = sqrt_up(vmax2_bound);  // upper bound of max |v|
  const double Rfull = d0 + 2.0 * V * dt;
  const double ext0 = extent_x(bc0, box0, x0, up, dt, step);
  const float extf[3] = {(float)ext0, (float)box1, (float)box2};
  const bool per[3] = {bc0 == KMC_PERIODIC, bc1 == KMC_PERIODIC, bc2 == KMC_PERIODIC};
  const float Rf = f_up(Rfull);

  // ---- split threshold: estimated pair-test cost of each trial (one lane each) --
  bool my_feasible = false;
  float my_cost = 0.0f;
  if (lane < (uint32_t)kSplitTrials) {
    const int t = (int)lane;
    do {
    if (t > 0 && !can_split) break;
    // trial thresholds were set from the previous step's bound; the slow cell must
    // cover the threshold actually used for classification (a binary32 square)
    const double S1 = t == 0 ? V : sqrt_up(my_thr);
    if (t > 0 && !(S1 < V)) break;
    const float hs = f_up((d0 + 2.0 * S1 * dt) * scale);
    const CellPlan p = plan_cells(extf, hs, K, (uint64_t)cell_cap / (t == 0 ? 1 : 2));
    if (!p.ok) break;
    const float rho = (float)n / ((float)p.nc[0] * (float)p.nc[1] * (float)p.nc[2]);
    if (t == 0) {
      my_cost = slow_cost((float)n, rho, fp32);
      my_feasible = true;
      break;
    }
    if (split_ok == 1 && rho < min_occ) break;
    // fast stencil: c cells on each side per split axis; periodic axes must hold it,
    // and no axis may be a one-cell periodic axis (no minimum-image test there)
    float ncol = 1.0f, iwmax = 0.0f;
    bool fits = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if (p.nc[a] == 1) {
        if (per[a]) fits = false;
        continue;
      }
      const float iw = (float)p.nc[a] / extf[a];
      iwmax = fmaxf(iwmax, iw);
      // the final grid below rounds this count up in the same way
      int c = (int)ceilf(Rf * (1.0f + p.m) * iw * (1.0f + 1e-6f));
      if (c < K) c = K;
      if (per[a] && p.nc[a] < 2 * c + 2) fits = false;
      if (a > 0) ncol *= (2.0f * c + 1.0f);
    }
    if (!fits) break;
    // a fast particle's reach, its speed taken just above the threshold
    const float rf = (float)(d0 + (1.15 * S1 + V) * dt);
    const float rf_cells = iwmax > 0.0f ? rf * iwmax : 1.0f;
    my_cost = slow_cost((float)n - my_nfast, rho, fp32) + fast_cost(my_nfast, rho, rf_cells, ncol, fp32);
    my_feasible = true;
    } while (false);
  }
  const uint32_t fmask = __ballot_sync(kAll, my_feasible);
  int best = 0;
  if (split_ok == 2) {
    // forced: cycle through the feasible trial thresholds step by step
    const int want = (int)(step % (uint64_t)(kSplitTrials - 1));
    for (int d = 0; d < kSplitTrials - 1; ++d) {
      const int t = 1 + (want + d) % (kSplitTrials - 1);
      if ((fmask >> t) & 1u) { best = t; break; }
    }
  } else {
    float cost = __shfl_sync(kAll, my_cost, 0);
#pragma unroll
    for (int t = 1; t < kSplitTrials; ++t) {
      const float ct = __shfl_sync(kAll, my_cost, t);
      if (((fmask >> t) & 1u) && ct < 0.95f * cost) { best = t; cost = ct; }
    }
  }
  const bool split = best > 0;
  const float thr = __shfl_sync(kAll, my_thr, best);
  const float s1sq = split ? thr : 0.0f;
  const double S1 = split ? sqrt_up(s1sq) : V;
  // trial thresholds for the next step (counted by the push of this step)
  set_split_thresholds(s, vmax2_bound, lane);

  const float hs = f_up((d0 + 2.0 * S1 * dt) * scale);
  const uint64_t max_keys = (uint64_t)cell_cap / (split ? 2 : 1);
  CellPlan p = plan_cells(extf, hs, K, max_keys);
  // search for the slow population: tiles where cells are well filled (and always in
  // binary64), lane per particle along its rows in sparse cells and for one-cell periodic
  // axes (the tiled search walks those per particle, in binary64 only)
  const float occ = (float)n / ((float)p.nc[0] * (float)p.nc[1] * (float)p.nc[2]);
  bool cp = false;
#pragma unroll
  for (int a = 0; a < 3; ++a) cp = cp || (p.nc[a] == 1 && per[a]);
  int mode = MODE_TILES;
  if (search_kernel == KMC_SEARCH_PARTICLE) mode = MODE_PARTICLE;
  else if (fp32 && (cp || search_kernel == KMC_SEARCH_ROW ||
                    (search_kernel == 0 && occ < kTileOccupancy)))
    mode = MODE_ROWS;
  int kx = K;
  if (mode == MODE_ROWS && p.nc[0] > 1) {
    // rows of half-width cells: each particle's row is trimmed to its reach in
    // half-cell steps (the grid is otherwise the same)
    const CellPlan q = plan_cells(extf, hs, K, max_keys, 2);
    if (q.ok && q.nc[0] > 1 && q.nc[1] == p.nc[1] && q.nc[2] == p.nc[2]) {
      p = q;
      kx = 2 * K;
    }
  }
  // per axis (lanes 0..2; the other lanes repeat lane 2)
  const int ax = lane < 2u ? (int)lane : 2;
  const int my_nc = ax == 0 ? p.nc[0] : ax == 1 ? p.nc[1] : p.nc[2];
  const float my_iw = (float)my_nc / (ax == 0 ? extf[0] : ax == 1 ? extf[1] : extf[2]);
  const int Ka = ax == 0 ? kx : K;
  int my_cfast = 0;
  if (split && my_nc != 1) {
    // at least Rfull (1 + m) / w cells: the product is within 4 u32 of it
    my_cfast = (int)ceilf(Rf * (1.0f + p.m) * my_iw * (1.0f + 1e-6f));
    if (my_cfast < Ka) my_cfast = Ka;
  }
  Grid& g = s.d.grid;
  if (lane < 3u) {
    g.nc[lane] = my_nc;
    g.cfast[lane] = my_cfast;
    g.inv_wf[lane] = my_nc == 1 ? 0.0f : my_iw;
  }
  if (lane != 0) return;  // lane 0 writes the rest
  if (!p.ok) s.d.status |= ST_CELL_OVERFLOW;
  g.split = split ? 1u : 0u;
  g.split_t = best;
  g.s1sq = s1sq;
  g.mode = mode;
  g.kx = kx;
  g.col_shift = p.col_shift;
  g.col_tz = p.col_tz;
  g.nkeys = p.nkeys;
  g.K = K;
  g.m = p.m;
}

// A reflecting wall turns a particle back once a step and a periodic axis wraps it once, so one
// that crosses the whole box within a step can end it outside.  The cell assignment takes it
// into the nearest cell; the tiled search's frames do not hold it.  From the step after the
// first in which some particle may have done so (sim_create: from the first step if one starts
// beyond the wall's position) that search goes without its filter.  No particle moves faster
// than 1.5 V before the walls act, V the step's bound of max |v|: a collision leaves a speed
// of at most sqrt(v_a^2 + v_b^2), in a mixture of at most 3 V.
__device__ inline void watch_box(SimDev& s, uint32_t lane) {
  const int ax = lane < 2u ? (int)lane : 2;
  const int bc = s.bc[ax];
  const double dt = s.dt, up = s.piston_u;
  const uint64_t step = s.d.step;
  double room = s.box[ax], go = (s.mix ? 3.01 : 1.5) * sqrt_up(s.d.vmax2) * dt;
  if (ax == 0 && bc == KMC_REFLECT) {
    room = s.piston_x0 - up * ((double)step * dt);
    go += 2.0 * fabs(up) * dt;
  }
  const bool out = bc != KMC_ABSORB && !(ax == 2 && s.planar) && !(go <= room);
  if (__any_sync(0xFFFFFFFFu, out) && lane == 0 && s.d.loose_from > step + 1) s.d.loose_from = step + 1;
}

// The guard bands of the step's pre-tests, from the grid that compute_grid chose.  Only the
// searches need them, so they are worked out while the cells are counted up: in the chain of
// the grid builder they took 5 us of every step, in a block of their own in the scan nothing
// that shows (6.1 us at 4096 particles with and without).  All 32 lanes of a warp; part 0
// sets the sphere tests and the reaches, part 1 the other tests' bands (one warp for both
// took 6.8 us, longer than the scan of a small simulation), part 2 watches the box.
__device__ __noinline__ inline void compute_guards(SimDev& s, uint32_t part, uint32_t lane) {
  if (part == 2u) return watch_box(s, lane);
  constexpr uint32_t kAll = 0xFFFFFFFFu;
  const double u32 = 0x1p-24, u64 = 0x1p-53;
  Grid& g = s.d.grid;
  // ---- per axis (lanes 0..2; the other lanes repeat lane 2) ---------------------
  // Error of the binary32 separation against the binary64 one, per component (the
  // binary32 mirror holds box coordinates and velocities, each rounded once):
  //   multi-cell axis: both coordinates (u32 L each), a periodic image shifts one
  //     side by the rounded box length (u32 L) and that sum is rounded (u32 L); the
  //     difference itself rounds with u32 |r|: 4 u32 L + u32 rb, plus 8 u64 L for the
  //     binary64 separation's own rounding;
  //   one-cell axis (minimum image in binary32): u32 * 6.1 * extent + 8 u64 L.
  // Velocity difference: 4.1 u32 V.  Component bounds: |r_k| <= rb_k, |v_k| <= 2V.
  const int ax = lane < 2u ? (int)lane : 2;
  const int my_nc = g.nc[ax], my_cfast = g.cfast[ax], Ka = ax == 0 ? g.kx : g.K;
  const double m = (double)g.m;
  const double my_box = s.box[ax];
  const int my_bc = s.bc[ax], my_bc0 = s.bc[0];
  const double d0 = s.d0, dt = s.dt, d0sq = s.d0sq, x0 = s.piston_x0, up = s.piston_u;
  const uint64_t step = s.d.step;
  const float vmax2_bound = s.d.vmax2, s1sq = g.s1sq;
  const bool loose = s.d.loose_from <= step;
  const bool split = g.split != 0u;
  const double V = sqrt_up(vmax2_bound);  // upper bound of max |v|
  const double S1 = split ? sqrt_up(s1sq) : V;
  const double my_ext = ax == 0 ? extent_x(my_bc, my_box, x0, up, dt, step) : my_box;
  const double my_w = my_nc == 1 ? my_ext : my_ext / (double)my_nc;
  const double L = my_box > my_ext ? my_box : my_ext;
  const int Ke = my_cfast > Ka ? my_cfast : Ka;
  // half extent of a tile's frame along the axis, for a run in one cell (kmc_search.cu): the
  // high word, which orders positive values
  const int my_fr = __double2hiint((my_nc == 1 ? 0.5 : g.K == 1 ? 1.5 : 2.5) * my_w);
  double my_e, my_rb;
  if (my_nc == 1) {
    my_e = 6.1 * u32 * L + 8.0 * u64 * L;
    my_rb = my_bc == KMC_PERIODIC ? 0.5 * L * (1.0 + 8.0 * u32) + 2.0 * my_e : L;
  } else {
    my_rb = (Ke + 1.0 + 2.0 * m) * my_w;
    my_e = u32 * (4.0 * L + my_rb) * (1.0 + 1e-3) + 8.0 * u64 * L;
  }
  if (part == 0u && lane < 3u) {
    g.wf[lane] = (float)my_w;
    g.Lf[lane] = (float)my_box;
    g.halfLf[lane] = (float)(0.5 * my_box);
    g.tief[lane] = f_up(4.0 * my_e);
  }
  const double e0 = __shfl_sync(kAll, my_e, 0), e1 = __shfl_sync(kAll, my_e, 1),
               e2 = __shfl_sync(kAll, my_e, 2);
  const double b0 = __shfl_sync(kAll, my_rb, 0), b1 = __shfl_sync(kAll, my_rb, 1),
               b2 = __shfl_sync(kAll, my_rb, 2);
  const double L0 = __shfl_sync(kAll, L, 0), L1 = __shfl_sync(kAll, L, 1),
               L2 = __shfl_sync(kAll, L, 2);
  const int f0 = __shfl_sync(kAll, my_fr, 0), f1 = __shfl_sync(kAll, my_fr, 1),
            f2 = __shfl_sync(kAll, my_fr, 2);
  if (lane != 0) return;  // lane 0 writes the rest

  const double dt2 = dt * dt;
  const double er = fmax(e0, fmax(e1, e2)), rbmax = fmax(b0, fmax(b1, b2));
  const double Lmax = fmax(L0, fmax(L1, L2));
  // The power of two at or below the smallest frame of the tiled search (the largest of the
  // three half extents and of S1 dt) is the unit in which squares of lengths are brought to
  // binary32, so that they stay inside its range in whatever unit the caller measures lengths.
  // (On exponents, the bits from 20 of the high word: the binary64 pipe has two lanes.)
  const int frame = max(max(f0, f1), max(f2, __double2hiint(S1 * dt)));
  // (2^-90 to 2^90, and no reach of the fast particles 2^60 times as large)
  const bool sane = frame >= 0x3A500000 && frame < 0x45900000 &&
                    __double2hiint(rbmax) < frame + (60 << 20);
  const int ue = sane ? (frame & 0x7FF00000) - 0x3FF00000 : 0;
  const double q0 = times_2(b0, -ue), q1 = times_2(b1, -ue), q2 = times_2(b2, -ue);
  const double rn = sane ? times_2(sqrt_up(fmaxf(f_up((q0 * q0 + q1 * q1) + q2 * q2), 1e-38f)) *
                                       (1.0 + 1e-6), ue)
                         : 1.7320508075688773 * (1.0 + 1e-6) * rbmax;
  const double V2 = V * V, rnV2 = rn * 2.0 * V;
  const double ev = 4.1 * u32 * V;
  const double g3 = 3.0 * u32 / (1.0 - 3.0 * u32);
  const double g3d = 3.0 * u64 / (1.0 - 3.0 * u64);
  const double g2 = 2.0 * u32 / (1.0 - 2.0 * u32);
  const double up2 = 1.0 + 2.0 * u32, up4 = 1.0 + 4.0 * u32;
  const double rel40 = 1.0 + 0x1p-40;
  const double s3 = 1.7320508075688772 * (1.0 + 1e-15);
  const double bslack = 7.0 * ev * V + 3.0 * ev * ev;  // |v|^2 - |v~|^2 slack, absolute
  if (part == 0u) {
    // ---- binary64 sphere pre-test: R > c0 + c1 B  =>  not a candidate ----------
    // Exactly, |r|^2 |v|^2 = (r.v)^2 + |r x v|^2, so |r|^2 = t*^2 |v|^2 + d_min^2 <
    // dt^2 |v|^2 + d0^2 for a candidate; with the roundings of the test this holds
    // with a relative slack below 30 u64, far inside the 2^-40 used here.
    g.c0 = d0sq * ((1.0 + 0x1p-40) * (1.0 + 0x1p-50));
    g.c1 = dt2 * ((1.0 + 0x1p-40) * (1.0 + 0x1p-50));
    // row trimming: a slow-slow candidate has |r| < d0 + (|v_i| + |v_j|) dt <= d0 + 2 S1 dt
    const double S1dt = S1 * dt;
    const double reach = (d0 + 2.0 * S1dt) * (1.0 + 1e-6);
    g.row_r2 = f_up(reach * reach * (1.0 + 1e-6));
    // per particle: (i, j) with j slow has |r| < d0 + (|v_i| + |v_j|) dt <= d0 + S1 dt + |v_i| dt
    g.row_a = f_up((d0 + S1dt) * (1.0 + 1e-6));
    g.row_b = f_up(dt * (1.0 + 1e-6));
    g.fast_a = f_up((d0 + V * dt) * (1.0 + 1e-6));
    g.row_eps = f_up(16.0 * u32 * Lmax);
    g.row_pad = f_up(4.0 * u32 * Lmax);
    // sphere test
    const double c0 = (rel40 * (d0sq + dt2 * bslack) + 2.0 * s3 * er * rn) * (1.0 + g3);
    g.s_c0 = f_up(c0 * up2);
    g.s_c1 = f_up(dt2 * (rel40 * (1.0 + g3) / (1.0 - g3) * up2));
    // pair filter of the tiled search (kmc_search.cu, "Error of the filter"): the sphere
    // test's constant with three times the separation error er, and the slack of
    // velocities rounded to 11 bits, 2^-7 (dt S1)^2; in squares of the unit.  tile_k is dt
    // with at least the root of the sphere test's factor on dt^2.
    const double c = (rel40 * (d0sq + dt2 * bslack) + 8.0 * s3 * er * rn + 27.0 * er * er) *
                         ((1.0 + g3) * up2) + 0x1p-7 * 1.001 * dt2 * S1 * S1;
    g.tile_k = f_up(dt * (rel40 * (1.0 + g3) / (1.0 - g3) * up2));
    g.s1f = f_up(S1);
    // The filter runs where its operands cannot leave binary16 and binary32: every particle in
    // its cell (watch_box; the third warp sets it for the steps after this), a frame of
    // ordinary size, a threshold below eight of its squares (not a gas in one cell much smaller
    // than d0), and dt neither past binary32 nor so much above the frame that scaled
    // velocities overflow (2^127 and 2^100).
    const int ce = (__double2hiint(c) >> 20) - 2 * (ue >> 20);  // exponent of c in unit^2
    const bool filter = sane && !loose && ce < 1023 + 3 &&
                        __double2hiint(dt) < min(0x46300000 + ue, 0x47E00000);
    g.tile_unit = filter ? __uint_as_float((uint32_t)((ue >> 20) + 127) << 23) : 0.0f;
    g.tile_c = !filter ? 0.0f : ce < 1023 - 60 ? 0x1p-60f : f_up(times_2(c, -2 * ue));
    return;
  }
  // the upper x wall at the end of the step, for the push (never -0.0)
  s.d.wall_x = my_bc0 == KMC_PERIODIC
                   ? 0.0
                   : __dadd_rn(__dsub_rn(x0, __dmul_rn(up, __dmul_rn((double)(step + 1), dt))), 0.0);
  // approach test (t* >= 0): |A~ - A64| <= a_g
  const double Ga = (s3 * (ev * rn + 2.0 * V * er) + rnV2 * (g3 * 1.01 + g3d)) * (1.0 + 1e-3);
  g.a_g = f_up(Ga);
  // time test (t* < dt): X~ = A~ - dt B~ > t_g  =>  A64 >= dt B64
  const double Ex = u32 * (rnV2 * 1.01 + dt * V2 * 8.16);
  const double Gt = (Ex + Ga + dt * (8.1 * g3 * V2 + bslack)) * (1.0 + 1e-3);
  g.t_g = f_up(Gt);
  g.dtf = (float)dt;
  // distance test (d_min < d0): |w~| >= w_e + d0 sqrt(B_up)  =>  W64 >= d0^2 B64
  const double ew = 2.0 * (rbmax * ev + 2.0 * V * er) * 1.001 + rbmax * V * (4.04 * g2 + 8.0 * u64);
  g.w_e = f_up(s3 * ew * up4);
  g.b_rel = f_up((1.0 / (1.0 - g3)) * (1.0 + g3d) * up2);
  g.b_abs = f_up(bslack * ((1.0 + g3d) * up2));
  // 1 / sqrt(1 - g3d) <= 1 + g3d
  g.d0up = f_up(d0 * (rel40 * (1.0 + g3d) * up4 * (1.0 + 4.0 * u32)));
  g.w_rel = f_up((1.0 + g3) * up4);
}

}  // namespace kmc
