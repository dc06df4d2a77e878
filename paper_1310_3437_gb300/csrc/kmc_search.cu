// kmc_search.cu -- neighbourhood search for collision candidates (Sec. 2: every
// particle of a bin is compared with the particles of its own and the neighbouring
// bins; the cost is O(B * N_bin^2 / P), eq. "eff").
//
// Each unordered pair is tested once: particle p meets the "forward half" of its
// stencil (own cell with j > p, then the cells whose offset (dz, dy, dx) is
// lexicographically positive).  The search does no division: it only culls pairs that
// provably fail the paper's criteria and emits the survivors; kmc_match.cu re-tests
// every survivor with the exact binary64 predicate.
//
//   k_search_rows32 slow pairs, binary32, sparse cells: a lane per particle along its rows.
//   k_search_tiles  slow pairs, well filled cells and binary64: 32 x 32 tiles of pairs
//                   through one quadratic form on the tensor cores, then the tests of the
//                   precision on what that leaves.
//   k_search_fast   the fast particles of the speed split, a warp each.
//   k_search        slow pairs with a thread per particle (kmc_params.search_kernel = 1).
//
//   KMC_FP64          binary64 sphere test |r|^2 > d0^2 + dt^2 |v|^2 (+2^-40 slack), then
//                     the binary64 approach and time tests.
//   KMC_GUARDED_FP32  binary32 on box coordinates: sphere test, then approach, time and
//                     distance tests, each widened by a guard band that bounds the
//                     binary32 error (kmc_grid.cuh derives the bands).
// A pair that passes the binary64 predicate is never culled by either variant, so
// both variants produce exactly the candidate list of the binary64 definition.
#include <cuda_fp16.h>

#include <algorithm>

#include "kmc_internal.cuh"

namespace kmc {

struct Own32 {
  float ox, oy, oz, vx, vy, vz;
};

// Two binary32 values in one 64-bit register, and the packed (f32x2) arithmetic of
// sm_100-class GPUs on them: each half is rounded exactly as the scalar operation.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 r, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

__device__ __forceinline__ void min_image_f(float& r, float halfL, float L, float tie, bool& keep) {
  float ar = fabsf(r);
  if (fabsf(ar - halfL) <= tie) keep = true;
  else if (ar > halfL) r = r > 0.f ? r - L : r + L;
}

// block-uniform: does any simulation of the batch run this step with the given search
// (mode < 0: the fast-particle search, i.e. any simulation under the speed split)?
__device__ __forceinline__ bool batch_uses(const Batch& B, int mode) {
  bool any = false;
  for (int q = threadIdx.x; q < B.nsims; q += blockDim.x) {
    const SimDev& t = B.sim(q);
    any = any || (sim_active(t) && (mode < 0 ? t.d.grid.split != 0u : t.d.grid.mode == mode));
  }
  return __syncthreads_or(any) != 0;
}

// Conservative binary64 approach and time pre-tests on a sphere survivor.  The search
// computes r = x_j - x_i, v = v_j - v_i, |v|^2 and r.v with the same operations as the
// exact test (k_refine), so rv is its value bit for bit; the exact test needs
// t* = fl(-rv / vv) >= 0 and < dt.  Dropped here only when that provably fails:
//   rv > vv 2^-1000: -rv / vv <= -2^-1000 (too large to round to -0.0, which would
//     count as >= 0), so t* < 0;
//   -rv >= fl(fl(dt vv)(1 + 2^-48)) >= dt vv (1 + 2^-50): fl(-rv / vv) >= dt.
// (vv >= 2^-900 here; rounding of the two thresholds only makes the drops rarer.)
__device__ __forceinline__ bool f64_cannot_approach(double rv, double vv, double dt) {
  return rv > dmul(vv, 0x1p-1000) || -rv >= dmul(dmul(dt, vv), 1.0 + 0x1p-48);
}

constexpr int kCellWarps = 8;   // warps per block of the warp-wise searches
constexpr int kWarpBuf = 64;    // emitted pairs staged per warp

struct Guard32 {
  float c0, c1, ag, tg, dtf, d0up, brel, babs, we, wrel;
};

__device__ __forceinline__ Guard32 guard_of(const Grid& g) {
  Guard32 q;
  q.c0 = g.s_c0; q.c1 = g.s_c1; q.ag = g.a_g; q.tg = g.t_g; q.dtf = g.dtf;
  q.d0up = g.d0up; q.brel = g.b_rel; q.babs = g.b_abs; q.we = g.w_e; q.wrel = g.w_rel;
  return q;
}

// exact guarded test of one pair on the sphere survivors (rare path)
__device__ __forceinline__ bool full_test32(const Guard32& q, float rx, float ry, float rz,
                                            float vx, float vy, float vz, float Bv) {
  const float A = -fmaf(rz, vz, fmaf(ry, vy, rx * vx));
  if (A < -q.ag) return false;
  if (fmaf(-q.dtf, Bv, A) > q.tg) return false;
  const float w0 = fmaf(ry, vz, -(rz * vy));
  const float w1 = fmaf(rz, vx, -(rx * vz));
  const float w2 = fmaf(rx, vy, -(ry * vx));
  const float W = fmaf(w2, w2, fmaf(w1, w1, w0 * w0));
  const float thr = fmaf(q.d0up, sqrtf(fmaf(Bv, q.brel, q.babs)), q.we);
  return !(W > thr * thr * q.wrel);
}

// The same test behind a real call: inlined, the compiler predicates it into every
// lane's instruction stream (about 30 instructions per pair although only the rare
// sphere survivors need it); as a call it issues only when some lane of the warp
// takes the branch.
__device__ __noinline__ bool full_test32_call(const Guard32& q, float rx, float ry, float rz,
                                              float vx, float vy, float vz, float Bv) {
  return full_test32(q, rx, ry, rz, vx, vy, vz, Bv);
}

// Emission from divergent lanes: a shared-memory counter per warp; entries that do
// not fit in the warp's buffer go straight to the global list.
__device__ __forceinline__ void emit_lane(uint2* buf, uint32_t* count, SimDev& s, uint32_t i,
                                          uint32_t j) {
  uint32_t pos = atomicAdd(count, 1u);
  if (pos < (uint32_t)kWarpBuf) {
    buf[pos] = make_uint2(i, j);
  } else {
    uint32_t g = atomicAdd(&s.d.n_raw, 1u);
    if (g < s.edge_cap) s.edge[g] = make_uint2(i, j);
    else atomicOr(&s.d.status, ST_EDGE_OVERFLOW);
  }
}

// warp-uniform: move the buffered pairs to the global list
__device__ __forceinline__ void flush_lanes(uint2* buf, uint32_t* count, SimDev& s, uint32_t lane) {
  __syncwarp();
  uint32_t c = *count;
  c = c < (uint32_t)kWarpBuf ? c : (uint32_t)kWarpBuf;
  if (c) {
    uint32_t base = 0;
    if (lane == 0) base = atomicAdd(&s.d.n_raw, c);
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    for (uint32_t k = lane; k < c; k += 32) {
      uint32_t g = base + k;
      if (g < s.edge_cap) s.edge[g] = buf[k];
      else atomicOr(&s.d.status, ST_EDGE_OVERFLOW);
    }
  }
  __syncwarp();
  if (lane == 0) *count = 0;
  __syncwarp();
}

// --------------------------------------------------------------------------- //
// Thread per particle: the lane of particle p walks the cells of its forward half
// stencil.  The search of kmc_params.search_kernel = 1, and of every simulation that has
// a one-cell periodic axis (fewer than 2K + 1 cells), where each separation needs the
// minimum image.  Returns the pairs tested.
template <int PREC, int K>
__device__ __noinline__ unsigned long long particle_walk(SimDev& s, uint32_t p, uint2* buf,
                                                         uint32_t* cnt) {
  const Grid& g = s.d.grid;
  const int cur = s.d.parity ^ 1;
  const uint32_t* __restrict__ cs = s.cell_start;
  const int nx = g.nc[0], ny = g.nc[1], nz = g.nc[2];
  const int Kx = nx == 1 ? 0 : K, Ky = ny == 1 ? 0 : K, Kz = nz == 1 ? 0 : K;
  const bool px = s.bc[0] == KMC_PERIODIC, py = s.bc[1] == KMC_PERIODIC,
             pz = s.bc[2] == KMC_PERIODIC;
  unsigned long long tests = 0;
  // the particle's cell, recomputed as the sort computed it
  const int cx = cell_coord(g, 0, s.x[cur][0][p]), cy = cell_coord(g, 1, s.x[cur][1][p]),
            cz = cell_coord(g, 2, s.x[cur][2][p]);
  // own record
  double xo[3] = {0, 0, 0}, vo[3] = {0, 0, 0};
  Own32 o32 = {0, 0, 0, 0, 0, 0};
  const double* __restrict__ X0 = s.x[cur][0];
  const double* __restrict__ X1 = s.x[cur][1];
  const double* __restrict__ X2 = s.x[cur][2];
  const double* __restrict__ V0 = s.v[cur][0];
  const double* __restrict__ V1 = s.v[cur][1];
  const double* __restrict__ V2 = s.v[cur][2];
  const float4* __restrict__ MM = s.mir;
  if (PREC == KMC_FP64) {
    xo[0] = X0[p]; xo[1] = X1[p]; xo[2] = X2[p];
    vo[0] = V0[p]; vo[1] = V1[p]; vo[2] = V2[p];
  } else {
    float4 a;
    float2 b;
    mirror_load(MM, p, a, b);
    o32 = {a.x, a.y, a.z, a.w, b.x, b.y};
  }
  // one-cell periodic axes need the minimum image explicitly
  const bool cp0 = nx == 1 && px, cp1 = ny == 1 && py, cp2 = nz == 1 && pz;
  const double L0 = s.box[0], L1 = s.box[1], L2 = s.box[2];
  const Guard32 q = guard_of(g);

  // a neighbour reached across a periodic boundary is seen as its image: wrap
  // flags -1 (below 0) or +1 (at or above the extent) per axis
  for (int dz = 0; dz <= Kz; ++dz) {
    int qz = cz + dz, wz = 0;
    if (qz >= nz) {
      if (!pz) break;
      qz -= nz;
      wz = 1;
    }
    for (int dy = (dz == 0 ? 0 : -Ky); dy <= Ky; ++dy) {
      int qy = cy + dy, wy = 0;
      if (qy < 0) {
        if (!py) continue;
        qy += ny;
        wy = -1;
      } else if (qy >= ny) {
        if (!py) continue;
        qy -= ny;
        wy = 1;
      }
      const uint32_t colbase = col_code(g, (uint32_t)qy, (uint32_t)qz) * (uint32_t)nx;
      const int dx0 = (dz == 0 && dy == 0) ? 0 : -Kx;
      for (int dx = dx0; dx <= Kx; ++dx) {
        int qx = cx + dx, wx = 0;
        if (qx < 0) {
          if (!px) continue;
          qx += nx;
          wx = -1;
        } else if (qx >= nx) {
          if (!px) continue;
          qx -= nx;
          wx = 1;
        }
        const uint32_t key = colbase + (uint32_t)qx;
        uint32_t beg = __ldg(cs + key), end = __ldg(cs + key + 1);
        if (dz == 0 && dy == 0 && dx == 0) beg = p + 1;
        if (beg >= end) continue;
        tests += end - beg;
        if (PREC == KMC_FP64) {
          for (uint32_t j = beg; j < end; ++j) {
            double r0 = dsub(__ldg(X0 + j), xo[0]);
            double r1 = dsub(__ldg(X1 + j), xo[1]);
            double r2 = dsub(__ldg(X2 + j), xo[2]);
            if (px) r0 = min_image(r0, L0, s.half_box[0]);
            if (py) r1 = min_image(r1, L1, s.half_box[1]);
            if (pz) r2 = min_image(r2, L2, s.half_box[2]);
            double g0 = dsub(__ldg(V0 + j), vo[0]);
            double g1 = dsub(__ldg(V1 + j), vo[1]);
            double g2 = dsub(__ldg(V2 + j), vo[2]);
            double R = dadd(dadd(dmul(r0, r0), dmul(r1, r1)), dmul(r2, r2));
            double Bv = dadd(dadd(dmul(g0, g0), dmul(g1, g1)), dmul(g2, g2));
            if (Bv >= 0x1p-900 && R > dadd(g.c0, dmul(g.c1, Bv))) continue;
            if (Bv >= 0x1p-900 &&
                f64_cannot_approach(dadd(dadd(dmul(r0, g0), dmul(r1, g1)), dmul(r2, g2)), Bv, s.dt))
              continue;
            emit_lane(buf, cnt, s, p, j);
          }
        } else {
          // own coordinates moved by the image shift (j seen at x_j + w L)
          const float sx = o32.ox - (float)wx * g.Lf[0];
          const float sy = o32.oy - (float)wy * g.Lf[1];
          const float sz = o32.oz - (float)wz * g.Lf[2];
          for (uint32_t j = beg; j < end; ++j) {
            float4 a;
            float2 b;
            mirror_load(MM, j, a, b);
            float rx = a.x - sx, ry = a.y - sy, rz = a.z - sz;
            bool keep = false;
            // minimum image on one-cell periodic axes; near the tie the two
            // images are both possible in binary64: keep the pair unculled
            if (cp0) min_image_f(rx, g.halfLf[0], g.Lf[0], g.tief[0], keep);
            if (cp1) min_image_f(ry, g.halfLf[1], g.Lf[1], g.tief[1], keep);
            if (cp2) min_image_f(rz, g.halfLf[2], g.Lf[2], g.tief[2], keep);
            const float gx = a.w - o32.vx, gy = b.x - o32.vy, gz = b.y - o32.vz;
            const float R = fmaf(rz, rz, fmaf(ry, ry, rx * rx));
            const float Bv = fmaf(gz, gz, fmaf(gy, gy, gx * gx));
            if (keep || (R <= fmaf(q.c1, Bv, q.c0) && full_test32(q, rx, ry, rz, gx, gy, gz, Bv)))
              emit_lane(buf, cnt, s, p, j);
          }
        }
      }
    }
  }
  return tests;
}

template <int PREC, int K>
__global__ void __launch_bounds__(kTile) k_search(Batch B) {
  __shared__ uint2 wbuf[kTile / 32][kWarpBuf];
  __shared__ uint32_t wcount[kTile / 32];
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  if (lane == 0) wcount[warp] = 0;
  __syncwarp();
  // grid-stride over tiles of kTile particles (an occupancy-sized grid)
  const uint32_t ntiles = B.ptiles;
  for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int k = find_sim(B.ptile, B.nsims, tile);
    SimDev& s = B.sim(k);
    if (s.d.grid.mode != MODE_PARTICLE) continue;
    // the status word can change while the search runs (a full pair buffer): one answer
    if (!__all_sync(0xFFFFFFFFu, sim_active(s))) continue;
    const uint32_t p = (tile - B.tile0(B.ptile, k)) * kTile + threadIdx.x;
    // with the speed split only the slow population (keys below nkeys) is searched here;
    // particles that left through absorbing walls sit after every cell key
    const uint32_t nslow = (s.d.grid.split || s.absorb) ? __ldg(s.cell_start + s.d.grid.nkeys) : s.n;
    unsigned long long tests = 0;
    if (p < nslow) tests = particle_walk<PREC, K>(s, p, wbuf[warp], &wcount[warp]);
    flush_lanes(wbuf[warp], &wcount[warp], s, lane);
    for (int o = 16; o > 0; o >>= 1) tests += __shfl_down_sync(0xFFFFFFFFu, tests, o);
    if (lane == 0 && tests) atomicAdd(&s.d.pair_tests, tests);
  }
}

// --------------------------------------------------------------------------- //
// Row search (binary32), for sparsely filled cells.  One lane per slow particle i,
// 32 consecutive particles (cell order) per warp.  With the mirror in box
// coordinates a stencil row -- the 2K+1 cells along x of one forward (y, z) column,
// or in i's own column the cells from its own on with only j > i -- is one
// contiguous range of partners; a row that crosses a periodic x boundary splits
// into two pieces, the far one seen through its image.  Each lane lists its
// non-empty pieces in shared memory and then walks them as one sequence of tests,
// one test per iteration, so no per-cell loop and no per-cell shift remain.  The
// warp runs as many iterations as its busiest lane needs.  Rows split only on a
// periodic x axis (PX); without one the piece lists take half the shared memory,
// which leaves more of the SM's L1 to cache the partner records.
// SHARED (few particles, see shift_of): 2^shift warps take the same 32 particles, warp w of
// them the columns c with c mod 2^shift = w.
template <int K, bool PX>
struct RowLayout {
  static constexpr int kCols = 1 + K + K * (2 * K + 1);  // own column + forward columns
  static constexpr int kPieces = PX ? 2 * kCols : kCols; // a row splits at most once
  static constexpr int kWarps = kTile / 32;
  static constexpr size_t kPieceBytes = (size_t)kWarps * kPieces * 32 * sizeof(uint2);
  static constexpr size_t kCodeBytes = (size_t)kWarps * kPieces * 32;
  static constexpr size_t kBytes = kPieceBytes + kCodeBytes + (size_t)kWarps * kWarpBuf * sizeof(uint2);
};

// image flags of a piece: bit 0 / 1 = seen at +L / -L along x, bits 2-3 y, bits 4-5 z
__device__ __forceinline__ uint32_t image_code(int wx, int wy, int wz) {
  return (uint32_t)(wx > 0) | ((uint32_t)(wx < 0) << 1) | ((uint32_t)(wy > 0) << 2) |
         ((uint32_t)(wy < 0) << 3) | ((uint32_t)(wz > 0) << 4) | ((uint32_t)(wz < 0) << 5);
}

template <int K, bool PX, bool SHARED>
__global__ void __launch_bounds__(kTile, 4) k_search_rows32(Batch B, uint32_t shift) {
  using RL = RowLayout<K, PX>;
  constexpr int NP = RL::kPieces;
  extern __shared__ __align__(16) unsigned char rows_smem[];
  __shared__ uint32_t wcount[RL::kWarps];
  __shared__ Guard32 sq;
  __shared__ float4 shift_tab[64];  // image shift (x, y, z) of each image code
  __shared__ int s_live;            // the current simulation runs this step
  // grid-stride over tiles of kTile particles: the kernel is launched every step on an
  // occupancy-sized grid and exits at once when the step runs another search
  if (!batch_uses(B, MODE_ROWS)) return;
  const uint32_t parts = SHARED ? 1u << shift : 1u, units = B.ptiles * parts;
  int kcur = -1;  // simulation whose constants the shared tables hold
  // The warp's pair tests and emitted pairs go to the simulation's counters only when
  // the simulation changes, the staging buffer is half full, or at the end: per-tile
  // atomics on these two counters from every warp serialise in L2.  The running
  // counts live in shared memory (registers are the row search's limit).
  __shared__ unsigned long long wtests[RL::kWarps];
  auto warp_buf = [&]() {
    return reinterpret_cast<uint2*>(rows_smem + RL::kPieceBytes + RL::kCodeBytes) +
           (size_t)(threadIdx.x >> 5) * kWarpBuf;
  };
  auto warp_flush = [&](SimDev& f) {
    const uint32_t w = threadIdx.x >> 5, l = threadIdx.x & 31u;
    flush_lanes(warp_buf(), &wcount[w], f, l);
    if (l == 0 && wtests[w]) atomicAdd(&f.d.pair_tests, wtests[w]);
    if (l == 0) wtests[w] = 0;
    __syncwarp();
  };
  if ((threadIdx.x & 31u) == 0) {
    wcount[threadIdx.x >> 5] = 0;
    wtests[threadIdx.x >> 5] = 0;
  }
  __syncwarp();
  for (uint32_t unit = blockIdx.x; unit < units; unit += gridDim.x) {
    const uint32_t tile = SHARED ? unit >> shift : unit;
    const int k = find_sim(B.ptile, B.nsims, tile);
    SimDev& s = B.sim(k);
    // launch-fixed fields only: the barriers below depend on it
    if (!sim_scheduled(s) || s.d.grid.mode != MODE_ROWS || (s.bc[0] == KMC_PERIODIC) != PX)
      continue;
    const Grid& g = s.d.grid;
    // The shared constants change only with the simulation (block-uniform: every warp
    // walks the same tiles), so the warps of a block need not wait for each other at
    // every tile: each runs on to its part of the next tile.
    if (k != kcur) {
      if (kcur >= 0) warp_flush(B.sim(kcur));  // staged pairs and counts of the last one
      __syncthreads();  // every warp is done with the previous simulation's constants
      if (threadIdx.x == 0) {
        sq = guard_of(g);
        // the status word, read once per simulation and block (the search itself can set
        // it: a full pair buffer only stops the stores, which are bounds-checked)
        s_live = sim_active(s) ? 1 : 0;
      }
      if (threadIdx.x < 64) {
        const uint32_t c = threadIdx.x;
        const float w0 = (float)((int)(c & 1u) - (int)((c >> 1) & 1u));
        const float w1 = (float)((int)((c >> 2) & 1u) - (int)((c >> 3) & 1u));
        const float w2 = (float)((int)((c >> 4) & 1u) - (int)((c >> 5) & 1u));
        shift_tab[c] = make_float4(w0 * g.Lf[0], w1 * g.Lf[1], w2 * g.Lf[2], 0.f);
      }
      __syncthreads();
      kcur = k;
    }
    if (!s_live) continue;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t nslow = (g.split || s.absorb) ? __ldg(s.cell_start + g.nkeys) : s.n;
    const uint32_t part = SHARED ? warp & (parts - 1u) : 0u;
    uint32_t p = (tile - B.tile0(B.ptile, k)) * kTile + threadIdx.x;
    if (SHARED) p = p - warp * 32u + (unit & (parts - 1u)) * (kTile >> shift) + (warp >> shift) * 32u;
    if (p - lane >= nslow) continue;  // the whole warp is past the slow population
    uint2* pc = reinterpret_cast<uint2*>(rows_smem) + (size_t)warp * NP * 32;
    uint8_t* cd = rows_smem + RL::kPieceBytes + (size_t)warp * NP * 32;
    uint2* buf = warp_buf();
    uint32_t* cnt = &wcount[warp];

    const bool valid = p < nslow;
    const int nx = g.nc[0], ny = g.nc[1], nz = g.nc[2];
    // along x the grid may have narrower cells under the row search (kx per radius)
    const int Kx = nx == 1 ? 0 : g.kx, Ky = ny == 1 ? 0 : K, Kz = nz == 1 ? 0 : K;
    constexpr bool px = PX;
    const bool py = s.bc[1] == KMC_PERIODIC, pz = s.bc[2] == KMC_PERIODIC;
    // one-cell periodic axes need the minimum image explicitly
    const bool cp0 = nx == 1 && px, cp1 = ny == 1 && py, cp2 = nz == 1 && pz;
    const bool any_cp = cp0 || cp1 || cp2;
    const uint32_t* __restrict__ cs = s.cell_start;
    const float4* __restrict__ MM = s.mir;

    // 1. the lane's non-empty pieces, column by column
    int np = 0;
    uint32_t total = 0, iters = 0;  // tests; iterations of up to two tests of one piece
    Own32 o = {0, 0, 0, 0, 0, 0};
    int cx = 0, cy = 0, cz = 0;
    if (valid) {
      float4 a;
      float2 b;
      mirror_load(MM, p, a, b);
      o = {a.x, a.y, a.z, a.w, b.x, b.y};
      // the particle's cell, recomputed from the mirror as the sort computed it
      cx = cell_coord_f(g, 0, a.x);
      cy = cell_coord_f(g, 1, a.y);
      cz = cell_coord_f(g, 2, a.z);
    }
    // Nearly every warp lies in one (y, z) column (a column holds thousands of
    // particles in cell order).  Then the forward columns are the same for all lanes:
    // lane c works out column c (whether it exists, its key base, its image code)
    // once for the warp.  Lane 0 is valid whenever any lane is.
    const int cy0 = __shfl_sync(0xFFFFFFFFu, cy, 0), cz0 = __shfl_sync(0xFFFFFFFFu, cz, 0);
    const bool uni = __all_sync(0xFFFFFFFFu, !valid || (cy == cy0 && cz == cz0));
    uint32_t ctab = kNone, ctag = 0;
    if (uni && lane < (uint32_t)RL::kCols) {
      const int c = (int)lane;
      const int dz = c <= K ? 0 : 1 + (c - K - 1) / (2 * K + 1);
      const int dy = c == 0 ? 0 : (c <= K ? c : (c - K - 1) % (2 * K + 1) - K);
      int qz = cz0 + dz, wz = 0, qy = cy0 + dy, wy = 0;
      bool ok = !(dz > Kz || dy > Ky || dy < -Ky);
      if (qz >= nz) { ok = ok && pz; qz -= nz; wz = 1; }
      if (qy < 0) { ok = ok && py; qy += ny; wy = -1; }
      else if (qy >= ny) { ok = ok && py; qy -= ny; wy = 1; }
      if (ok) {
        ctab = col_code(g, (uint32_t)qy, (uint32_t)qz) * (uint32_t)nx;
        ctag = (uint32_t)(wy & 3) | ((uint32_t)(wz & 3) << 2);
      }
    }
    {
      // row trimming: the part of each row within the reach of this particle.  A
      // column whose cells lie farther than the reach in (y, z) is skipped; in the
      // others only the cells with x within sqrt(reach^2 - d^2) are kept (d the
      // column's distance in (y, z), taken from the cell edges and rounded down; the
      // x extent rounded up).  Rows that cross a periodic x boundary keep their full
      // length on the crossing side.
      // the reach of this particle: |v_i| from its binary32 velocity (each component
      // within u32 of the binary64 one, the sum of squares within 3 u32, the square
      // root within 3 ulp; the argument kept normal, which only enlarges it) times
      // 1 + 4e-6 bounds |v_i| from above; the products and the square get 1e-6 each.
      // The smaller of this and the common reach holds.
      const float sv2 = fmaxf(fmaf(o.vz, o.vz, fmaf(o.vy, o.vy, o.vx * o.vx)), 1e-30f);
      // (the square root from the approximate reciprocal root: 3 ulp, inside the margin)
      const float si = sv2 * rsqrtf(sv2) * 1.000004f;
      const float Ri = fmaf(si, g.row_b, g.row_a) * 1.000001f;
      const float R2 = fminf(g.row_r2, Ri * Ri * 1.000001f);
      const float eps = g.row_eps, pad = g.row_pad;
      const float wyf = g.wf[1], wzf = g.wf[2], ivx = g.inv_wf[0];
#pragma unroll
      for (int c = 0; c < RL::kCols; ++c) {
        if (SHARED && ((uint32_t)c & (parts - 1u)) != part) continue;
        const int dz = c <= K ? 0 : 1 + (c - K - 1) / (2 * K + 1);
        const int dy = c == 0 ? 0 : (c <= K ? c : (c - K - 1) % (2 * K + 1) - K);
        // the column's key base and image flags (warp table, or this lane's own)
        uint32_t colb, wtag;
        if (uni) {
          colb = __shfl_sync(0xFFFFFFFFu, ctab, c);
          wtag = __shfl_sync(0xFFFFFFFFu, ctag, c);
          if (colb == kNone) continue;
        } else {
          if (dz > Kz || dy > Ky || dy < -Ky) continue;
          int qz = cz + dz, wz = 0;
          if (qz >= nz) {
            if (!pz) continue;
            qz -= nz;
            wz = 1;
          }
          int qy = cy + dy, wy = 0;
          if (qy < 0) {
            if (!py) continue;
            qy += ny;
            wy = -1;
          } else if (qy >= ny) {
            if (!py) continue;
            qy -= ny;
            wy = 1;
          }
          colb = col_code(g, (uint32_t)qy, (uint32_t)qz) * (uint32_t)nx;
          wtag = (uint32_t)(wy & 3) | ((uint32_t)(wz & 3) << 2);
        }
        if (!valid) continue;
        const int wy = (wtag & 3u) == 3u ? -1 : (int)(wtag & 3u);
        const int wz = (int)((wtag >> 2) & 3u);
        float d2 = 0.f;
        if (dy != 0) {
          const float e = dy > 0 ? (float)(cy + dy) * wyf - o.oy : o.oy - (float)(cy + dy + 1) * wyf;
          const float el = fmaxf(e - eps, 0.f);
          d2 = el * el;
        }
        if (dz != 0) {  // forward columns only: dz > 0
          const float e = (float)(cz + dz) * wzf - o.oz;
          const float el = fmaxf(e - eps, 0.f);
          d2 = fmaf(el, el, d2);
        }
        d2 *= 0.9999995f;
        if (d2 >= R2) continue;
        // x extent sqrt(R2 - d2) from the approximate reciprocal square root (at most
        // 2 ulp off, 3 ulp with the product), widened by 33 ulp; the argument is kept
        // normal, which only widens it
        const float t2 = fmaxf(R2 - d2, 1e-30f);
        const float ex = fmaf(t2 * rsqrtf(t2), 1.000004f, pad);
        int xa = c == 0 ? cx : cx - Kx, xb = cx + Kx;  // cells of the row, unwrapped
        if (Kx > 0) {
          const int ta = (int)floorf((o.ox - ex) * ivx), tb = (int)floorf((o.ox + ex) * ivx);
          if (ta >= 0 && ta > xa) xa = ta;
          if (tb <= nx - 1 && tb < xb) xb = tb;
          if (xb < xa) continue;
        }
        {
          const int a0 = xa < 0 ? 0 : xa, b0 = xb >= nx ? nx - 1 : xb;
          const uint32_t jb = c == 0 ? p + 1 : __ldg(cs + colb + a0);
          const uint32_t je = __ldg(cs + colb + b0 + 1);
          if (je > jb) {
            pc[np * 32 + lane] = make_uint2(jb, je);
            cd[np * 32 + lane] = (uint8_t)image_code(0, wy, wz);
            ++np;
            total += je - jb;
            iters += ((je + 1u) >> 1) - (jb >> 1);  // pair slots
          }
        }
        if (px && xa < 0) {  // cells [xa + nx, nx) seen through the image at -L
          const uint32_t jb = __ldg(cs + colb + xa + nx), je = __ldg(cs + colb + nx);
          if (je > jb) {
            pc[np * 32 + lane] = make_uint2(jb, je);
            cd[np * 32 + lane] = (uint8_t)image_code(-1, wy, wz);
            ++np;
            total += je - jb;
            iters += ((je + 1u) >> 1) - (jb >> 1);  // pair slots
          }
        }
        if (px && xb >= nx) {  // cells [0, xb - nx] seen through the image at +L
          const uint32_t jb = __ldg(cs + colb), je = __ldg(cs + colb + xb - nx + 1);
          if (je > jb) {
            pc[np * 32 + lane] = make_uint2(jb, je);
            cd[np * 32 + lane] = (uint8_t)image_code(1, wy, wz);
            ++np;
            total += je - jb;
            iters += ((je + 1u) >> 1) - (jb >> 1);  // pair slots
          }
        }
      }
    }

    // 2. walk the pieces in pair slots of the mirror, two tests per iteration (a half
    //    outside the piece masked), the binary32 pre-tests in packed f32x2 arithmetic
    const uint32_t T = __reduce_max_sync(0xFFFFFFFFu, any_cp ? total : iters);
    uint32_t j = 0, je = 0;
    int r = 0;
    float sx = o.ox, sy = o.oy, sz = o.oz;
    if (np > 0) {
      const uint2 q = pc[lane];
      const float4 sh = shift_tab[cd[lane]];
      j = q.x;
      je = q.y;
      sx = o.ox - sh.x;
      sy = o.oy - sh.y;
      sz = o.oz - sh.z;
    }
    const float c0 = g.s_c0, c1 = g.s_c1;
    if (any_cp) {
      // one-cell periodic axes (thin slabs): one test per iteration with the minimum image
      for (uint32_t t = 0; t < T; ++t) {
        if (j < je) {
          float4 a;
          float2 b;
          mirror_load(MM, j, a, b);
          float rx = a.x - sx, ry = a.y - sy, rz = a.z - sz;
          bool keep = false;
          if (cp0) min_image_f(rx, g.halfLf[0], g.Lf[0], g.tief[0], keep);
          if (cp1) min_image_f(ry, g.halfLf[1], g.Lf[1], g.tief[1], keep);
          if (cp2) min_image_f(rz, g.halfLf[2], g.Lf[2], g.tief[2], keep);
          const float gx = a.w - o.vx, gy = b.x - o.vy, gz = b.y - o.vz;
          const float R = fmaf(rz, rz, fmaf(ry, ry, rx * rx));
          const float Bv = fmaf(gz, gz, fmaf(gy, gy, gx * gx));
          if (keep || (R <= fmaf(c1, Bv, c0) && full_test32_call(sq, rx, ry, rz, gx, gy, gz, Bv)))
            emit_lane(buf, cnt, s, p, j);
          if (++j == je && r + 1 < np) {
            ++r;
            const uint2 q = pc[r * 32 + lane];
            const float4 sh = shift_tab[cd[r * 32 + lane]];
            j = q.x;
            je = q.y;
            sx = o.ox - sh.x;
            sy = o.oy - sh.y;
            sz = o.oz - sh.z;
          }
        }
      }
    } else {
      const f32x2 C0 = pack2(c0, c0), C1 = pack2(c1, c1);
      const f32x2 VX = pack2(o.vx, o.vx), VY = pack2(o.vy, o.vy), VZ = pack2(o.vz, o.vz);
      f32x2 SX = pack2(sx, sx), SY = pack2(sy, sy), SZ = pack2(sz, sz);
      // the piece [j, je) in pair slots: slot k holds particles 2k and 2k + 1, three
      // 16-byte loads give each component of both already paired; a half outside the
      // piece (its first slot's lower, its last slot's upper half) is masked
      const ulonglong2* __restrict__ MP = reinterpret_cast<const ulonglong2*>(MM);
      uint32_t k = j >> 1, ke = (je + 1u) >> 1;
      for (uint32_t t = 0; t < T; ++t) {
        if (k < ke) {
          const ulonglong2* rec = MP + 3 * (size_t)k;
          const ulonglong2 Q0 = __ldg(rec), Q1 = __ldg(rec + 1), Q2 = __ldg(rec + 2);
          const f32x2 rx = sub2(Q0.x, SX), ry = sub2(Q0.y, SY), rz = sub2(Q1.x, SZ);
          const f32x2 gx = sub2(Q1.y, VX), gy = sub2(Q2.x, VY), gz = sub2(Q2.y, VZ);
          const f32x2 R = fma2(rz, rz, fma2(ry, ry, mul2(rx, rx)));
          const f32x2 Bv = fma2(gz, gz, fma2(gy, gy, mul2(gx, gx)));
          const f32x2 bound = fma2(C1, Bv, C0);
          float R0, R1, T0, T1;
          unpack2(R, R0, R1);
          unpack2(bound, T0, T1);
          const uint32_t j0 = 2u * k;
          const bool s0 = j0 >= j && R0 <= T0, s1 = j0 + 1u < je && R1 <= T1;
          if (s0 || s1) {  // rare: a sphere survivor
            float rx0, rx1, ry0, ry1, rz0, rz1, gx0, gx1, gy0, gy1, gz0, gz1, B0, B1;
            unpack2(rx, rx0, rx1);
            unpack2(ry, ry0, ry1);
            unpack2(rz, rz0, rz1);
            unpack2(gx, gx0, gx1);
            unpack2(gy, gy0, gy1);
            unpack2(gz, gz0, gz1);
            unpack2(Bv, B0, B1);
            if (s0 && full_test32_call(sq, rx0, ry0, rz0, gx0, gy0, gz0, B0))
              emit_lane(buf, cnt, s, p, j0);
            if (s1 && full_test32_call(sq, rx1, ry1, rz1, gx1, gy1, gz1, B1))
              emit_lane(buf, cnt, s, p, j0 + 1u);
          }
          if (++k == ke && r + 1 < np) {
            ++r;
            const uint2 q = pc[r * 32 + lane];
            const float4 sh = shift_tab[cd[r * 32 + lane]];
            j = q.x;
            je = q.y;
            k = j >> 1;
            ke = (je + 1u) >> 1;
            SX = pack2(o.ox - sh.x, o.ox - sh.x);
            SY = pack2(o.oy - sh.y, o.oy - sh.y);
            SZ = pack2(o.oz - sh.z, o.oz - sh.z);
          }
        }
      }
    }
    __syncwarp();
    if (*cnt >= (uint32_t)(kWarpBuf / 2)) flush_lanes(buf, cnt, s, lane);
    unsigned long long tests = total;
    for (int off = 16; off > 0; off >>= 1) tests += __shfl_down_sync(0xFFFFFFFFu, tests, off);
    if (lane == 0) wtests[warp] += tests;
  }
  if (kcur >= 0) warp_flush(B.sim(kcur));
}

// --------------------------------------------------------------------------- //
// Tiled search of the slow pairs.  A warp takes 32 consecutive particles i (cell order)
// and all partners that any of them can have: for a run of lanes in one (y, z) column
// these are one contiguous range of the order per forward column (the cells along x from
// K below the first lane's to K above the last lane's; in the own column from the first
// lane's particle on), plus the wrapped part on a periodic x axis.  The ranges are laid
// end to end and taken 32 partners j at a time, a lane each.  The sphere test of all
// 32 x 32 pairs is one quadratic form,
//   |a_i - a_j|^2 - |b_i - b_j|^2 = s_i + s_j - 2 a_i.a_j + 2 b_i.b_j,  s = |a|^2 - |b|^2,
// a the position and b = dt v, both relative to the run's middle and scaled by a power of
// two so that |a|, |b| <= 1: an inner product of 16 terms, which eight
// mma.sync.m16n8k16 (binary16 operands, binary32 sums) form for the whole tile.  Every
// position is the sum of two binary16 values (22 bits), so are s_i and s_j; the
// velocities are one.  The sign of (form - threshold) is a bit of a lane's survivor mask,
// shifted in by one funnel shift per accumulator.  Survivors go to a per-warp queue, and
// the tests of the precision run on 32 of them at a time with every lane busy: cell
// offset (each pair at exactly one image), then the binary32 sphere and full guarded
// tests on the mirror, or the binary64 sphere, approach and time tests on the state.  The
// filter only saves them work: what it drops they would drop.  In a step whose lengths or
// threshold are outside what the operands can hold (compute_guards) it passes every pair
// (binary64: the lanes walk their particles' cells as the thread-per-particle search does).
//
// Error of the filter, in the scaled units.  A candidate has (kmc_grid.cuh)
// |a_i - a_j|^2 <= c + |b_i - b_j|^2 for the exact binary32 coordinates, with c the
// scaled constant of the sphere test with 3 er for the separation, since here the
// coordinates are rounded once more relative to the run's middle.  The rounding of b to
// 11 bits moves |b_i - b_j|^2 by at most 14 2^-11 b^2 < 2^-7 b^2 (both in tile_c).  The
// rest, with the components of a and |b| at most 1, the threshold at most 2 and u = 2^-24:
// dropped and rounded low parts 18 u, s and its halves 44 u, the inner product (16 products,
// exact in binary32, whose partial sums are at most 14, added with truncation) 448 u;
// 2^-14 = 1024 u is taken.
//
// SHARED (few particles, see shift_of): 2^shift warps take the same 32 particles, warp w of
// them the tiles w, w + 2^shift, ... of every run.
//
// What bounds it: issue slots.  A tile costs 8 mma (2 cycles of the SM's tensor cores
// each), 32 funnel shifts (half rate), about 75 instructions to pack the 32 partners and
// about 30 per turn of survivors, so it pays where most of a tile's 1024 pairs are pairs
// that have to be tested: see kTileOccupancy (kmc_grid.cuh).  Measured, slow pairs of one
// step: 10^8 particles at 7 per cell 16.0 ms with the row search, 10.5 ms with tiles; an
// ensemble of 30 boxes and tubes 336 (warp per cell and rows) -> 226 us; binary64 at 2^20
// 3.11 ms (thread per particle, every pair in binary64) -> 0.167 ms.  Packing the partners
// once per block or in the sort, 64 partners at a time, and records fetched ahead were no
// faster: the bookkeeping per run and column, not the packing, fills the issue slots.
constexpr int kPlane = 36;  // uint4 per plane of packed records: 32 and 4 of padding, so
                            // that the two planes lie in different shared-memory banks
constexpr float kFar = 60000.0f;  // form of an absent row or column: above any threshold
constexpr int kRunCells = 64;     // cells along x that the lanes of a run may span

template <int K>
struct TileWarp {
  static constexpr int kCols = 1 + K + K * (2 * K + 1);  // own column + forward columns
  static constexpr int kPieces = 3 * kCols;              // a range and its two wrapped parts
  uint4 rec[2 * kPlane];       // packed records: the rows, then 32 partners at a time
  uint32_t start[kPieces + 1]; // pieces: first slot, first partner, image code
  uint32_t first[kPieces + 1];
  uint32_t code[kPieces + 1];
  uint2 info[32];              // the partners' indices and image codes
  uint2 queue[64];             // survivors: row particle and partner
  uint32_t qcode[64];          // and the partner's image code
  uint2 buf[kWarpBuf];         // emitted pairs
  uint32_t count;
};

// image code of a piece: bits 0-1 x, 2-3 y, 4-5 z (1: seen at +L, 2: at -L), bit 6: own
// column
constexpr uint32_t kImages = 63u, kOwnColumn = 64u;
__device__ __forceinline__ float image_shift(uint32_t code, float L) {
  return (code & 1u) ? L : ((code & 2u) ? -L : 0.0f);
}

__device__ __forceinline__ uint32_t half_bits(__half2 h) { return *reinterpret_cast<uint32_t*>(&h); }
__device__ __forceinline__ uint32_t half_pair(float lo, float hi) {
  return half_bits(__floats2half2_rn(lo, hi));
}

// The 16 terms as 8 words w0..w7 of two; words c and c + 4 belong to the lanes with
// lane % 4 == c of the matrix fragments and lie side by side: plane 0 holds
// (w0, w4, w1, w5), plane 1 (w2, w6, w3, w7).
//   row:     (-2xh -2xh) (-2yh -2yh) (-2zh -2zh) (1 1)   | (-2xl sh) (-2yl 2bx) (-2zl 2by) (sl 2bz)
//   partner: (xh xl)     (yh yl)     (zh zl)     (sh sl) | (xh 1)    (yh bx)    (zh by)    (1 bz)
// with s = |a|^2 - |b|^2 of the rounded b, and the row's s less the threshold.  An absent
// row or partner is all zero but for its s = kFar and the partner's 1.
__device__ __forceinline__ void store_row(uint4* rec, uint32_t at, float ax, float ay, float az,
                                          float bx, float by, float bz, float T, bool in) {
  const __half2 hb = __floats2half2_rn(bx, by), hz = __floats2half2_rn(bz, 0.0f);
  bx = __low2float(hb); by = __high2float(hb); bz = __low2float(hz);
  const float s = in ? fmaf(ax, ax, fmaf(ay, ay, az * az)) - fmaf(bx, bx, fmaf(by, by, bz * bz)) - T
                     : kFar;
  const float m = in ? -2.0f : 0.0f;
  ax *= m; ay *= m; az *= m;
  bx *= -m; by *= -m; bz *= -m;
  const __half2 hxy = __floats2half2_rn(ax, ay), hzs = __floats2half2_rn(az, s);
  uint4 u, w;
  u.x = half_bits(__low2half2(hxy));
  u.y = half_pair(ax - __low2float(hxy), s);
  u.z = half_bits(__high2half2(hxy));
  u.w = half_pair(ay - __high2float(hxy), bx);
  w.x = half_bits(__low2half2(hzs));
  w.y = half_pair(az - __low2float(hzs), by);
  w.z = in ? 0x3C003C00u : 0u;
  w.w = half_pair(s - __high2float(hzs), bz);
  rec[at] = u;
  rec[kPlane + at] = w;
}
__device__ __forceinline__ void store_partner(uint4* rec, uint32_t at, float ax, float ay, float az,
                                              float bx, float by, float bz, float far) {
  const __half2 hxy = __floats2half2_rn(ax, ay), hb = __floats2half2_rn(bx, by),
                hzb = __floats2half2_rn(az, bz);
  bx = __low2float(hb); by = __high2float(hb); bz = __high2float(hzb);
  const float s = (fmaf(ax, ax, fmaf(ay, ay, az * az)) + far) - fmaf(bx, bx, fmaf(by, by, bz * bz));
  const __half2 one = __floats2half2_rn(1.0f, 1.0f);
  uint4 u, w;
  u.x = half_pair(ax, ax - __low2float(hxy));
  u.y = half_bits(__lows2half2(hxy, one));
  u.z = half_pair(ay, ay - __high2float(hxy));
  u.w = half_bits(__halves2half2(__high2half(hxy), __low2half(hb)));
  w.x = half_pair(az, az - __low2float(hzb));
  w.y = half_bits(__halves2half2(__low2half(hzb), __high2half(hb)));
  w.z = half_pair(s, s - __half2float(__float2half_rn(s)));
  w.w = half_bits(__highs2half2(one, hzb));
  rec[at] = u;
  rec[kPlane + at] = w;
}

__device__ __forceinline__ void mma_form(float d[4], const uint32_t a[4], uint2 b) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%10, %10, %10, %10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y), "f"(0.0f));
}

// The bits of a lane's mask where the partner comes after the row, in a tile whose partner
// 0 is the particle after row 0 (the own column: each pair once, no particle with itself).
// The lane holds rows frag + 8 L (L = 0..3) and partners 8 n + 2 quad + e (n = 0..3, e = 0,
// 1), bit 31 - (8 n + 2 L + e).
__device__ __forceinline__ uint32_t later_bits(uint32_t frag, uint32_t quad) {
  uint32_t bits = 0;
#pragma unroll
  for (uint32_t at = 0; at < 32; ++at) {
    const uint32_t row = frag + 8u * ((at >> 1) & 3u), col = 8u * (at >> 3) + 2u * quad + (at & 1u);
    if (1u + col > row) bits |= 0x80000000u >> at;
  }
  return bits;
}

// The bits of a lane's mask where row and partner are the same particle, partner 0 of the
// tile being row `first` of the warp: equal for the one e that makes first + 2 quad + e -
// frag = 8 k, and there for L = n + k.
__device__ __forceinline__ uint32_t self_bits(uint32_t first, uint32_t frag, uint32_t quad) {
  const int u = (int)(first + 2u * quad - frag);
  const int e = u & 1, k = (u + e) >> 3;
  if ((u + e) & 7) return 0u;
  uint32_t bits = 0;
#pragma unroll
  for (int n = 0; n < 4; ++n)
    if (n + k >= 0 && n + k < 4) bits |= 0x80000000u >> (8 * n + 2 * (n + k) + e);
  return bits;
}

// binary32 record of a particle (FP64: its state rounded once, as the mirror would hold it)
template <int PREC>
__device__ __forceinline__ Own32 record32(const SimDev& s, const float4* __restrict__ M,
                                          int cur, uint32_t p) {
  if (PREC == KMC_FP64)
    return {d2f_rn(__ldg(s.x[cur][0] + p)), d2f_rn(__ldg(s.x[cur][1] + p)),
            d2f_rn(__ldg(s.x[cur][2] + p)), d2f_rn(__ldg(s.v[cur][0] + p)),
            d2f_rn(__ldg(s.v[cur][1] + p)), d2f_rn(__ldg(s.v[cur][2] + p))};
  float4 a;
  float2 b;
  mirror_load(M, p, a, b);
  return {a.x, a.y, a.z, a.w, b.x, b.y};
}

// the tests of the precision on one survivor: particle i (a row), partner j
template <int PREC, int K>
__device__ __noinline__ void test_survivor(SimDev& s, uint2* buf, uint32_t* cnt, uint2 ij,
                                           uint32_t code) {
  const Grid& g = s.d.grid;
  const uint32_t i = ij.x, j = ij.y;
  const int cur = s.d.parity ^ 1, nx = g.nc[0], Kx = nx == 1 ? 0 : K;
  const Own32 o = record32<PREC>(s, s.mir, cur, j), q = record32<PREC>(s, s.mir, cur, i);
  // every pair at exactly one image: the partner's cell, seen through this image, lies in
  // the row's stencil; in the own column only forward cells and later particles
  const int d = cell_coord_f(g, 0, o.ox) + ((code & 1u) ? nx : ((code & 2u) ? -nx : 0)) -
                cell_coord_f(g, 0, q.ox);
  if (d > Kx || d < -Kx) return;
  if ((code & kOwnColumn) && (d < 0 || (d == 0 && j <= i))) return;
  bool emit;
  if (PREC == KMC_FP64) {
    double r[3], v[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      r[a] = dsub(__ldg(s.x[cur][a] + j), __ldg(s.x[cur][a] + i));
      if (s.bc[a] == KMC_PERIODIC) r[a] = min_image(r[a], s.box[a], s.half_box[a]);
      v[a] = dsub(__ldg(s.v[cur][a] + j), __ldg(s.v[cur][a] + i));
    }
    const double R = dadd(dadd(dmul(r[0], r[0]), dmul(r[1], r[1])), dmul(r[2], r[2]));
    const double Bv = dadd(dadd(dmul(v[0], v[0]), dmul(v[1], v[1])), dmul(v[2], v[2]));
    emit = !(Bv >= 0x1p-900 && R > dadd(g.c0, dmul(g.c1, Bv)));
    if (emit && Bv >= 0x1p-900 &&
        f64_cannot_approach(dadd(dadd(dmul(r[0], v[0]), dmul(r[1], v[1])), dmul(r[2], v[2])), Bv, s.dt))
      emit = false;
  } else {
    // own coordinates moved by the image shift (j seen at x_j + w L)
    const float rx = o.ox - (q.ox - image_shift(code, g.Lf[0]));
    const float ry = o.oy - (q.oy - image_shift(code >> 2, g.Lf[1]));
    const float rz = o.oz - (q.oz - image_shift(code >> 4, g.Lf[2]));
    const float gx = o.vx - q.vx, gy = o.vy - q.vy, gz = o.vz - q.vz;
    const float R = fmaf(rz, rz, fmaf(ry, ry, rx * rx));
    const float Bv = fmaf(gz, gz, fmaf(gy, gy, gx * gx));
    emit = R <= fmaf(g.s_c1, Bv, g.s_c0) &&
           full_test32(guard_of(g), rx, ry, rz, gx, gy, gz, Bv);
  }
  if (emit) emit_lane(buf, cnt, s, i, j);
}

template <int PREC, int K, bool SHARED>
__global__ void __launch_bounds__(kTile, 4) k_search_tiles(Batch B, uint32_t shift) {
  using TW = TileWarp<K>;
  constexpr uint32_t kAll = 0xFFFFFFFFu;
  constexpr int kCols = TW::kCols;
  __shared__ TW tw[kTile / 32];
  if (!batch_uses(B, MODE_TILES)) return;
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  TW& w = tw[warp];
  if (lane == 0) w.count = 0;
  __syncwarp();
  // The warps of a block never wait for each other.  Survivors, pair counts and emitted
  // pairs are kept per warp until 32 (survivors) or half a buffer (pairs) are there, the
  // simulation changes, or the end: per-tile atomics from every warp would serialise in L2.
  unsigned long long tests = 0;
  uint32_t queued = 0;
  int kcur = -1;
  auto finish = [&](SimDev& f) {
    if (lane < queued) test_survivor<PREC, K>(f, w.buf, &w.count, w.queue[lane], w.qcode[lane]);
    queued = 0;
    flush_lanes(w.buf, &w.count, f, lane);
    if (lane == 0 && tests) atomicAdd(&f.d.pair_tests, tests);
    tests = 0;
  };
  const uint32_t frag = lane >> 2, quad = lane & 3u, later = later_bits(frag, quad);
  // this lane's two words of record r: plane quad / 2, half quad % 2
  const uint2* words = reinterpret_cast<const uint2*>(w.rec + (quad >> 1) * kPlane) + (quad & 1u);
  constexpr uint32_t kWarps = kTile / 32;
  const uint32_t parts = SHARED ? 1u << shift : 1u, step = gridDim.x * kWarps;
  const uint32_t units = B.ptiles * kWarps * parts;
  for (uint32_t unit = SHARED ? blockIdx.x + gridDim.x * warp : blockIdx.x * kWarps + warp;
       unit < units; unit += step) {
    const uint32_t part = unit & (parts - 1u), rows = SHARED ? unit >> shift : unit, tile = rows / kWarps;
    const int k = find_sim(B.ptile, B.nsims, tile);
    SimDev& s = B.sim(k);
    if (k != kcur) {
      if (kcur >= 0) finish(B.sim(kcur));
      kcur = k;
    }
    // the status word can change while the search runs (a full pair buffer): one answer
    if (!__all_sync(kAll, sim_active(s)) || s.d.grid.mode != MODE_TILES) continue;
    const Grid& g = s.d.grid;
    const uint32_t* __restrict__ cs = s.cell_start;
    const uint32_t nslow = (g.split || s.absorb) ? __ldg(cs + g.nkeys) : s.n;
    const uint32_t p0 = (rows - B.tile0(B.ptile, k) * kWarps) * 32u, p = p0 + lane;
    if (p0 >= nslow) continue;
    const bool valid = p < nslow;
    const int nx = g.nc[0], ny = g.nc[1], nz = g.nc[2], cur = s.d.parity ^ 1;
    const int Kx = nx == 1 ? 0 : K, Ky = ny == 1 ? 0 : K, Kz = nz == 1 ? 0 : K;
    const bool px = s.bc[0] == KMC_PERIODIC, py = s.bc[1] == KMC_PERIODIC,
               pz = s.bc[2] == KMC_PERIODIC;
    if (PREC == KMC_FP64 && (g.tile_unit == 0.0f || (nx == 1 && px) || (ny == 1 && py) ||
                             (nz == 1 && pz))) {
      // No filter (lengths may be past binary32), or a one-cell periodic axis: the minimum
      // image of every pair (binary32: row search)
      if (part != 0u) continue;
      unsigned long long t = valid ? particle_walk<PREC, K>(s, p, w.buf, &w.count) : 0ull;
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(kAll, t, o);
      tests += t;
      flush_lanes(w.buf, &w.count, s, lane);
      continue;
    }
    const float4* __restrict__ MM = s.mir;
    Own32 o = {0, 0, 0, 0, 0, 0};
    int cx = 0, cy = 0, cz = 0;
    if (valid) {
      o = record32<PREC>(s, MM, cur, p);
      // the particle's cell, recomputed as the sort computed it
      cx = cell_coord_f(g, 0, o.ox);
      cy = cell_coord_f(g, 1, o.oy);
      cz = cell_coord_f(g, 2, o.oz);
    }
    // runs of lanes in one column (in cell order: consecutive lanes, cells ascending)
    unsigned todo = __ballot_sync(kAll, valid);
    while (todo) {
      const int lead = __ffs((int)todo) - 1;
      const int y = __shfl_sync(kAll, cy, lead), z = __shfl_sync(kAll, cz, lead);
      const int x0 = __shfl_sync(kAll, cx, lead);
      const unsigned run =
          todo & __ballot_sync(kAll, valid && cy == y && cz == z && cx - x0 < kRunCells);
      todo &= ~run;
      const int x1 = __shfl_sync(kAll, cx, 31 - __clz((int)run));

      // 1. the pieces: lane c takes forward column c
      uint32_t jb = 0, len = 0, code = 0, jb1 = 0, len1 = 0, jb2 = 0, len2 = 0;
      if (lane < (uint32_t)kCols) {
        const int c = (int)lane;
        const int dz = c <= K ? 0 : 1 + (c - K - 1) / (2 * K + 1);
        const int dy = c == 0 ? 0 : (c <= K ? c : (c - K - 1) % (2 * K + 1) - K);
        int qy = y + dy, qz = z + dz;
        bool ok = dz <= Kz && dy <= Ky && dy >= -Ky;
        if (qz >= nz) { ok = ok && pz; qz -= nz; code |= 16u; }
        if (qy < 0) { ok = ok && py; qy += ny; code |= 8u; }
        else if (qy >= ny) { ok = ok && py; qy -= ny; code |= 4u; }
        if (c == 0) code |= kOwnColumn;
        if (ok) {
          const uint32_t* col = cs + col_code(g, (uint32_t)qy, (uint32_t)qz) * (uint32_t)nx;
          const int xa = c == 0 ? x0 : x0 - Kx, xb = x1 + Kx;
          jb = __ldg(col + (xa < 0 ? 0 : xa));
          const uint32_t je = __ldg(col + (xb >= nx ? nx : xb + 1));
          if (c == 0) jb = max(jb, p0 + (uint32_t)lead + 1u);
          len = je > jb ? je - jb : 0u;
          if (px && xa < 0) {  // cells [xa + nx, nx) seen at -L
            jb1 = __ldg(col + xa + nx);
            len1 = __ldg(col + nx) - jb1;
          }
          if (px && xb >= nx) {  // cells [0, xb - nx] seen at +L
            jb2 = __ldg(col);
            len2 = __ldg(col + xb - nx + 1) - jb2;
          }
        } else {
          code &= ~kImages;
        }
      }
      const uint32_t my_slots = len + len1 + len2;
      uint32_t slots = my_slots;
#pragma unroll
      for (int d = 1; d < kCols; d <<= 1) {
        const uint32_t u = __shfl_up_sync(kAll, slots, d);
        if (lane >= (uint32_t)d) slots += u;
      }
      const uint32_t total = __shfl_sync(kAll, slots, kCols - 1);
      if (total <= 32u * part) continue;
      if (part == 0u) tests += (unsigned long long)__popc(run) * total;
      // Plain: no piece is seen through an image.  The five pieces of K = 1 then stay in
      // registers; otherwise they go to shared memory.
      const bool plain =
          K == 1 && !__any_sync(kAll, (code & kImages) != 0u || len1 != 0u || len2 != 0u);
      uint32_t s1 = 0, s2 = 0, s3 = 0, s4 = 0, o0 = 0, o1 = 0, o2 = 0, o3 = 0, o4 = 0, pieces = 0;
      if (plain) {
        const uint32_t first = slots - my_slots, off = jb - first;
        s1 = __shfl_sync(kAll, first, 1); s2 = __shfl_sync(kAll, first, 2);
        s3 = __shfl_sync(kAll, first, 3); s4 = __shfl_sync(kAll, first, 4);
        o0 = __shfl_sync(kAll, off, 0); o1 = __shfl_sync(kAll, off, 1);
        o2 = __shfl_sync(kAll, off, 2); o3 = __shfl_sync(kAll, off, 3);
        o4 = __shfl_sync(kAll, off, 4);
      } else {
        const uint32_t my_cnt = (len ? 1u : 0u) + (len1 ? 1u : 0u) + (len2 ? 1u : 0u);
        uint32_t cnt = my_cnt;
#pragma unroll
        for (int d = 1; d < kCols; d <<= 1) {
          const uint32_t u = __shfl_up_sync(kAll, cnt, d);
          if (lane >= (uint32_t)d) cnt += u;
        }
        pieces = __shfl_sync(kAll, cnt, kCols - 1);
        uint32_t at = cnt - my_cnt, st = slots - my_slots;
        auto put = [&](uint32_t b, uint32_t n, uint32_t c) {
          if (!n) return;
          w.start[at] = st;
          w.first[at] = b;
          w.code[at] = c;
          st += n;
          ++at;
        };
        put(jb, len, code);
        put(jb1, len1, code | 2u);
        put(jb2, len2, code | 1u);
      }

      // 2. the run's frame: origin in its middle, scale the power of two that brings
      // the extents and dt |v| to at most 1
      const float wx = g.wf[0], wy = g.wf[1], wz = g.wf[2];
      float ox = 0.5f * (float)(x0 + x1 + 1) * wx, oy = ((float)y + 0.5f) * wy,
            oz = ((float)z + 0.5f) * wz;
      const float kv = g.tile_k;
      const float M = 1.01f * fmaxf(fmaxf((0.5f * (float)(x1 - x0 + 1) + (float)Kx) * wx,
                                          (0.5f + (float)Ky) * wy),
                                    fmaxf((0.5f + (float)Kz) * wz, kv * g.s1f));
      float sc = __uint_as_float((253u - (__float_as_uint(M) >> 23)) << 23);  // 2^-(e+1)
      const bool filter = PREC == KMC_FP64 || g.tile_unit != 0.0f;
      if (!filter) sc = ox = oy = oz = 0.0f;  // operands zero, threshold 2^-14: every pair passes
      // (the unit is at most the frame: the product is a power of two of at most 1/2)
      const float su = sc * g.tile_unit;
      const float T = fmaf(su * su, g.tile_c * 1.000001f, 0x1p-14f);
      const float kb = filter ? kv * sc : 0.0f;
      store_row(w.rec, lane, fmaf(o.ox, sc, -ox * sc), fmaf(o.oy, sc, -oy * sc),
                fmaf(o.oz, sc, -oz * sc), o.vx * kb, o.vy * kb, o.vz * kb, T, (run >> lane) & 1u);
      __syncwarp();
      uint32_t A[2][4];
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        const uint2 lo = words[2 * (16 * t + frag)], hi = words[2 * (16 * t + 8 + frag)];
        A[t][0] = lo.x; A[t][1] = hi.x; A[t][2] = lo.y; A[t][3] = hi.y;
      }
      __syncwarp();  // the rows are read before the first partners take their place

      // 3. the tiles
      for (uint32_t base = 32u * part; base < total; base += 32u * parts) {
        const uint32_t slot = base + lane;
        uint32_t j, jc = 0;
        float qx = -ox * sc, qy = -oy * sc, qz = -oz * sc;
        if (plain) {
          uint32_t off = o0;
          jc = kOwnColumn;
          if (slot >= s1) { off = o1; jc = 0; }
          if (slot >= s2) off = o2;
          if (slot >= s3) off = o3;
          if (slot >= s4) off = o4;
          j = slot + off;
        } else {
          // P is the piece that holds slot `base`; the pieces starting inside the tile (at
          // most 31, each non-empty, among P + 1 .. P + 31) mark their first slot in one OR
          uint32_t P = 0;
#pragma unroll
          for (uint32_t q = 0; q < (uint32_t)TW::kPieces; q += 32)
            P += __popc(__ballot_sync(kAll, q + lane < pieces && w.start[q + lane] <= base));
          --P;
          const uint32_t st = P + lane < pieces ? w.start[P + lane] : kNone;
          const uint32_t bit = (st > base && st - base < 32u) ? 1u << (st - base) : 0u;
          const uint32_t marks = __reduce_or_sync(kAll, bit);
          const uint32_t pi = P + __popc(marks & (kAll >> (31u - lane)));
          j = w.first[pi] + (slot - w.start[pi]);
          jc = w.code[pi];
          qx = -(ox - image_shift(jc, g.Lf[0])) * sc;
          qy = -(oy - image_shift(jc >> 2, g.Lf[1])) * sc;
          qz = -(oz - image_shift(jc >> 4, g.Lf[2])) * sc;
        }
        float ax = 0, ay = 0, az = 0, bx = 0, by = 0, bz = 0, far = kFar;
        if (slot < total) {
          const Own32 e = record32<PREC>(s, MM, cur, j);
          ax = fmaf(e.ox, sc, qx);
          ay = fmaf(e.oy, sc, qy);
          az = fmaf(e.oz, sc, qz);
          bx = e.vx * kb;
          by = e.vy * kb;
          bz = e.vz * kb;
          far = 0.0f;
        }
        store_partner(w.rec, lane, ax, ay, az, bx, by, bz, far);
        w.info[lane] = make_uint2(j, jc);
        __syncwarp();
        uint32_t mask = 0;
#pragma unroll
        for (int n = 0; n < 4; ++n) {
          const uint2 b = words[2 * (8 * n + frag)];
#pragma unroll
          for (int t = 0; t < 2; ++t) {
            float d[4];
            mma_form(d, A[t], b);
#pragma unroll
            for (int e = 0; e < 4; ++e) mask = __funnelshift_l(__float_as_uint(d[e]), mask, 1);
          }
        }
        // in the own column (its first piece) only later partners than the row
        if (base == 0u) mask &= lead == 0 ? later : ~self_bits((uint32_t)lead + 1u, frag, quad);
        // survivors to the queue, one per lane and turn; 32 of them are tested at a time
        for (unsigned any; (any = __ballot_sync(kAll, mask != 0u)) != 0u;) {
          if (mask) {
            const uint32_t at = (uint32_t)__clz((int)mask);  // accumulators in order
            mask &= ~(0x80000000u >> at);
            const uint32_t row = (at & 4u) * 4u + (at & 2u) * 4u + frag;
            const uint2 ji = w.info[(at & 24u) + quad * 2u + (at & 1u)];
            const uint32_t to = queued + __popc(any & ((1u << lane) - 1u));
            w.queue[to] = make_uint2(p0 + row, ji.x);
            w.qcode[to] = ji.y;
          }
          queued += __popc(any);
          if (queued >= 32u) {
            __syncwarp();
            queued -= 32u;
            test_survivor<PREC, K>(s, w.buf, &w.count, w.queue[queued + lane], w.qcode[queued + lane]);
            __syncwarp();
            if (w.count >= (uint32_t)(kWarpBuf / 2)) flush_lanes(w.buf, &w.count, s, lane);
          }
        }
        __syncwarp();  // fragments and survivors are read before the next tile's records
      }
    }
  }
  if (kcur >= 0) finish(B.sim(kcur));
}


// --------------------------------------------------------------------------- //
// Fast particles of the speed split: one warp per fast particle p, searching cfast
// cells on each side over both populations -- every slow particle, and the fast
// particles j > p (each fast-fast pair once).  The stencil is walked by (y, z)
// columns: the lanes take one column each, trim its row of cells along x to p's
// reach (as the row search does) and read its slow and fast partner ranges -- a row
// is contiguous in the cell order, so a column costs four loads of the cell table
// whatever its length.  A warp prefix sum over the lanes' test counts then deals the
// tests of 32 columns out to the lanes, so every lane tests a pair in every
// iteration whatever the occupancies.  The pair tests are those of the other searches.
// The particles are dealt to the grid by for_dealt, a warp each: few of them go to as many
// SMs as there are (one block per 256 particles of the gas put the fast ones of 4096
// binary64 particles on 16 SMs: 18.3 -> 13.1 us), and the members of a group follow one
// another (an ensemble of 30: 103 -> 82 us; 2^24 tube 262 -> 216, 10^8 gas 1.79 -> 1.50 ms).
// fast particles of a simulation's step (fields that stay fixed during the search)
__device__ __forceinline__ uint32_t fast_count(const SimDev& s) {
  if (!sim_scheduled(s) || !s.d.grid.split) return 0u;
  const uint32_t nk = s.d.grid.nkeys;
  return __ldg(s.cell_start + 2 * nk) - __ldg(s.cell_start + nk);
}

template <int PREC>
__global__ void __launch_bounds__(kCellWarps * 32, 4) k_search_fast(Batch B) {
  __shared__ uint2 wbuf[kCellWarps][kWarpBuf];
  __shared__ uint32_t wcount[kCellWarps];
  // per column of the current batch (one per lane): its first test within the batch,
  // and up to four partner ranges (slow and fast population, each in at most two x
  // segments on a periodic x axis): first partner, length, image flags of the segment
  constexpr int kFastPieces = 4;
  __shared__ uint32_t sjb[kCellWarps][kFastPieces][32], sln[kCellWarps][kFastPieces][32];
  __shared__ uint8_t scd[kCellWarps][kFastPieces][32];
  // the batch's pieces laid end to end (column by column): first test, first partner,
  // image flags
  __shared__ uint32_t fst[kCellWarps][kFastPieces * 32], fjb[kCellWarps][kFastPieces * 32];
  __shared__ uint8_t fcd[kCellWarps][kFastPieces * 32];
  for_dealt<kCellWarps>(B, [](const SimDev& s) { return fast_count(s); },
                        [&](SimDev& s, uint32_t first, uint32_t) {
    const Grid& g = s.d.grid;
    const uint32_t* __restrict__ cs = s.cell_start;
    const uint32_t nk = g.nkeys;
    const uint32_t n = __ldg(cs + 2 * nk);  // end of the fast keys (n without absorption)
    const uint32_t nslow = __ldg(cs + nk);
    const uint32_t nfast = n - nslow;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    if (first >= nfast) return;
    uint2* buf = wbuf[warp];
    uint32_t* cnt = &wcount[warp];
    if (lane == 0) *cnt = 0;
    __syncwarp();

    const int cur = s.d.parity ^ 1;
    const int nx = g.nc[0], ny = g.nc[1], nz = g.nc[2];
    const int Cx = g.cfast[0], Cy = g.cfast[1], Cz = g.cfast[2];
    const bool px = s.bc[0] == KMC_PERIODIC, py = s.bc[1] == KMC_PERIODIC,
               pz = s.bc[2] == KMC_PERIODIC;
    const double* __restrict__ X0 = s.x[cur][0];
    const double* __restrict__ X1 = s.x[cur][1];
    const double* __restrict__ X2 = s.x[cur][2];
    const double* __restrict__ V0 = s.v[cur][0];
    const double* __restrict__ V1 = s.v[cur][1];
    const double* __restrict__ V2 = s.v[cur][2];
    const float4* __restrict__ MM = s.mir;
    const double L0 = s.box[0], L1 = s.box[1], L2 = s.box[2];
    const Guard32 q = guard_of(g);
    const float Lf0 = g.Lf[0], Lf1 = g.Lf[1], Lf2 = g.Lf[2];
    unsigned long long tests = 0;

    for (uint32_t f = first; f < nfast; f += gridDim.x * kCellWarps) {
      const uint32_t p = nslow + f;
      // the particle's cell, recomputed as the sort computed it
      const int cx = cell_coord(g, 0, X0[p]), cy = cell_coord(g, 1, X1[p]), cz = cell_coord(g, 2, X2[p]);
      double xo[3] = {0, 0, 0}, vo[3] = {0, 0, 0};
      Own32 o32 = {0, 0, 0, 0, 0, 0};
      if (PREC == KMC_FP64) {
        xo[0] = X0[p]; xo[1] = X1[p]; xo[2] = X2[p];
        vo[0] = V0[p]; vo[1] = V1[p]; vo[2] = V2[p];
        // binary32 position and velocity for the cell trimming only
        o32 = {d2f_rn(xo[0]), d2f_rn(xo[1]), d2f_rn(xo[2]), d2f_rn(vo[0]), d2f_rn(vo[1]),
               d2f_rn(vo[2])};
      } else {
        float4 a;
        float2 b;
        mirror_load(MM, p, a, b);
        o32 = {a.x, a.y, a.z, a.w, b.x, b.y};
      }
      // cell trimming: a pair (p, j) has |r| < d0 + (|v_p| + |v_j|) dt <= d0 + (|v_p| + V) dt,
      // so a stencil cell farther than that from p holds no candidate.  |v_p| from the
      // binary32 velocity times 1 + 2e-6 bounds it from above; the distance to a cell is
      // taken from its edges less eps (the binary32 error of a coordinate against a
      // cell edge), rounded down.  Squares are kept normal: the speed's by enlarging it, and
      // where the reach's is not (units of length beyond about 10^18) nothing is trimmed.
      const float sv2 = fmaf(o32.vz, o32.vz, fmaf(o32.vy, o32.vy, o32.vx * o32.vx));
      const float sp = sqrtf(fmaxf(sv2, 1e-36f)) * 1.000002f;
      const float Rp = fmaf(sp, g.row_b, g.fast_a) * 1.000001f;
      const float Rp2 = Rp * Rp * 1.000001f;
      const bool trim = Rp2 >= 1e-36f && Rp2 <= 1e36f;
      const float teps = g.row_eps;
      const int Wy = 2 * Cy + 1;
      const int ncol = Wy * (2 * Cz + 1);
      const float ivx = g.inv_wf[0], pad = g.row_pad;
      for (int c0 = 0; c0 < ncol; c0 += 32) {
        // this lane's column: its row of cells trimmed to p's reach, split at a periodic
        // x boundary, and the slow and fast partner ranges of each segment
        const int c = c0 + (int)lane;
        int np = 0;
        uint32_t tot = 0;
        if (c < ncol) {
          const int dz = c / Wy - Cz;
          const int dy = c - (dz + Cz) * Wy - Cy;
          int qy = cy + dy, qz = cz + dz;
          const int wy = qy < 0 ? -1 : (qy >= ny ? 1 : 0);
          const int wz = qz < 0 ? -1 : (qz >= nz ? 1 : 0);
          bool ok = (wy == 0 || py) && (wz == 0 || pz);
          // squared distance from p to the column (unwrapped: the image frame of p)
          float d2 = 0.f;
          if (dy != 0 && ny > 1) {
            const float e = dy > 0 ? (float)(cy + dy) * g.wf[1] - o32.oy
                                   : o32.oy - (float)(cy + dy + 1) * g.wf[1];
            const float el = fmaxf(e - teps, 0.f);
            d2 = el * el;
          }
          if (dz != 0 && nz > 1) {
            const float e = dz > 0 ? (float)(cz + dz) * g.wf[2] - o32.oz
                                   : o32.oz - (float)(cz + dz + 1) * g.wf[2];
            const float el = fmaxf(e - teps, 0.f);
            d2 = fmaf(el, el, d2);
          }
          if (trim && d2 * 0.9999995f >= Rp2) ok = false;
          if (ok) {
            qy -= wy * ny;
            qz -= wz * nz;
            const uint32_t colb = col_code(g, (uint32_t)qy, (uint32_t)qz) * (uint32_t)nx;
            // the cells along x within the reach: sqrt(Rp2 - d2) from the approximate
            // reciprocal square root (3 ulp), widened by 33 ulp and the coordinate error
            int xa = 0, xb = 0;
            if (nx > 1) {
              xa = cx - Cx;
              xb = cx + Cx;
              if (trim) {
                const float t2 = fmaxf(Rp2 - d2, 1e-30f);
                const float ex = fmaf(t2 * rsqrtf(t2), 1.000004f, pad);
                const int ta = (int)floorf((o32.ox - ex) * ivx), tb = (int)floorf((o32.ox + ex) * ivx);
                xa = max(ta, xa);
                xb = min(tb, xb);
              }
              if (!px) {
                xa = xa < 0 ? 0 : xa;
                xb = xb > nx - 1 ? nx - 1 : xb;
              }
            }
            const uint32_t code_yz = (uint32_t)((wy > 0) ? 4 : 0) | (uint32_t)((wy < 0) ? 8 : 0) |
                                     (uint32_t)((wz > 0) ? 16 : 0) | (uint32_t)((wz < 0) ? 32 : 0);
            // x segments: [xa, xb] within [0, nx), and the part past a periodic boundary
            auto segment = [&](int a0, int b0, uint32_t code) {
              const uint32_t k0 = colb + (uint32_t)a0, k1 = colb + (uint32_t)b0 + 1u;
              const uint32_t sb0 = __ldg(cs + k0), se0 = __ldg(cs + k1);
              uint32_t sb1 = __ldg(cs + nk + k0);
              const uint32_t se1 = __ldg(cs + nk + k1);
              if (sb1 <= p) sb1 = p + 1;  // fast partners j > p only
              if (se0 > sb0) {
                sjb[warp][np][lane] = sb0; sln[warp][np][lane] = se0 - sb0; scd[warp][np][lane] = (uint8_t)code;
                tot += se0 - sb0;
                ++np;
              }
              if (se1 > sb1) {
                sjb[warp][np][lane] = sb1; sln[warp][np][lane] = se1 - sb1; scd[warp][np][lane] = (uint8_t)code;
                tot += se1 - sb1;
                ++np;
              }
            };
            if (xb >= xa) {
              const int a0 = xa < 0 ? 0 : xa, b0 = xb > nx - 1 ? nx - 1 : xb;
              if (b0 >= a0) segment(a0, b0, code_yz);
              if (xa < 0) segment(xa + nx, nx - 1, code_yz | 2u);            // seen at -L
              else if (xb > nx - 1) segment(0, xb - nx, code_yz | 1u);      // seen at +L
            }
          }
        }
        // lay the batch's pieces end to end: piece base and first test of each column
        uint32_t incl = tot, pincl = (uint32_t)np;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
          const uint32_t z = __shfl_up_sync(0xFFFFFFFFu, pincl, o);
          if (lane >= (uint32_t)o) {
            incl += y;
            pincl += z;
          }
        }
        const uint32_t total = __shfl_sync(0xFFFFFFFFu, incl, 31);
        const uint32_t npw = __shfl_sync(0xFFFFFFFFu, pincl, 31);
        tests += tot;
        {
          uint32_t at = pincl - (uint32_t)np, st = incl - tot;
          for (int r = 0; r < np; ++r) {
            fst[warp][at] = st;
            fjb[warp][at] = sjb[warp][r][lane];
            fcd[warp][at] = scd[warp][r][lane];
            st += sln[warp][r][lane];
            ++at;
          }
        }
        __syncwarp();
        // walk the batch's tests 32 at a time: lane l takes test kb + l.  P is the piece
        // holding test kb; the pieces starting inside the pass (at most 31, each
        // non-empty) are among P + 1 .. P + 31 and mark their first test in one OR
        uint32_t P = 0;
        for (uint32_t kb = 0; kb < total; kb += 32) {
          const uint32_t qp = P + lane;
          const uint32_t st = qp < npw ? fst[warp][qp] : 0xFFFFFFFFu;
          const uint32_t bit = (st >= kb && st - kb < 32u) ? 1u << (st - kb) : 0u;
          const uint32_t mask = __reduce_or_sync(0xFFFFFFFFu, bit);
          const uint32_t before = __shfl_sync(0xFFFFFFFFu, st < kb ? 1u : 0u, 0);
          const uint32_t pi = P - 1u + before + __popc(mask & (0xFFFFFFFFu >> (31u - lane)));
          const uint32_t qi = kb + lane;
          if (qi < total) {
            const uint32_t j = fjb[warp][pi] + (qi - fst[warp][pi]);
            const uint32_t d = fcd[warp][pi];
            bool emit;
            if (PREC == KMC_FP64) {
              double r0 = dsub(__ldg(X0 + j), xo[0]);
              double r1 = dsub(__ldg(X1 + j), xo[1]);
              double r2 = dsub(__ldg(X2 + j), xo[2]);
              if (px) r0 = min_image(r0, L0, s.half_box[0]);
              if (py) r1 = min_image(r1, L1, s.half_box[1]);
              if (pz) r2 = min_image(r2, L2, s.half_box[2]);
              const double g0 = dsub(__ldg(V0 + j), vo[0]);
              const double g1 = dsub(__ldg(V1 + j), vo[1]);
              const double g2 = dsub(__ldg(V2 + j), vo[2]);
              const double R = dadd(dadd(dmul(r0, r0), dmul(r1, r1)), dmul(r2, r2));
              const double Bv = dadd(dadd(dmul(g0, g0), dmul(g1, g1)), dmul(g2, g2));
              emit = !(Bv >= 0x1p-900 && R > dadd(g.c0, dmul(g.c1, Bv)));
              if (emit && Bv >= 0x1p-900 &&
                  f64_cannot_approach(dadd(dadd(dmul(r0, g0), dmul(r1, g1)), dmul(r2, g2)), Bv, s.dt))
                emit = false;
            } else {
              // own coordinates moved by the image shift (j seen at x_j + w L)
              const float wxf = (float)((int)(d & 1u) - (int)((d >> 1) & 1u));
              const float wyf = (float)((int)((d >> 2) & 1u) - (int)((d >> 3) & 1u));
              const float wzf = (float)((int)((d >> 4) & 1u) - (int)((d >> 5) & 1u));
              const float sx = o32.ox - wxf * Lf0;
              const float sy = o32.oy - wyf * Lf1;
              const float sz = o32.oz - wzf * Lf2;
              float4 a;
              float2 b;
              mirror_load(MM, j, a, b);
              const float rx = a.x - sx, ry = a.y - sy, rz = a.z - sz;
              const float gx = a.w - o32.vx, gy = b.x - o32.vy, gz = b.y - o32.vz;
              const float R = fmaf(rz, rz, fmaf(ry, ry, rx * rx));
              const float Bv = fmaf(gz, gz, fmaf(gy, gy, gx * gx));
              emit = R <= fmaf(q.c1, Bv, q.c0) && full_test32(q, rx, ry, rz, gx, gy, gz, Bv);
            }
            if (emit) emit_lane(buf, cnt, s, p, j);
          }
          // the next pass starts in lane 31's piece or in the one after it
          uint32_t nextP = 0;
          if (lane == 31u) {
            const uint32_t end = pi + 1u < npw ? fst[warp][pi + 1u] : total;
            nextP = kb + 32u >= end ? pi + 1u : pi;
          }
          P = __shfl_sync(0xFFFFFFFFu, nextP, 31);
          __syncwarp();
          if (*cnt >= (uint32_t)(kWarpBuf / 2)) flush_lanes(buf, cnt, s, lane);
        }
        __syncwarp();
      }
    }
    flush_lanes(buf, cnt, s, lane);
    for (int o = 16; o > 0; o >>= 1) tests += __shfl_down_sync(0xFFFFFFFFu, tests, o);
    if (lane == 0 && tests) {
      atomicAdd(&s.d.pair_tests, tests);
      atomicAdd(&s.d.fast_tests, tests);
    }
  });
}

namespace {
// resident blocks of a kernel on the whole GPU (occupancy x SMs)
template <typename F>
int resident_blocks(F kernel, int threads, size_t smem, int num_sms) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem) != cudaSuccess ||
      per_sm < 1) {
    cudaGetLastError();
    per_sm = 2;
  }
  return per_sm * num_sms;
}

// Warps that share the partners of 32 particles in the tiled and the row search: as many as
// leave every one of them resident at once (at most eight, a block of them).  A warp with
// 32 particles for itself runs 10 to 20 us whatever the rest of the chip does, a chain of
// loads, so with fewer of them than the SMs hold the step waits for one chain; shared by 8, 8
// and 2 warps the searches of boxes of 4096 particles (binary32, binary64) and of a 50 k tube
// take 9.0, 17.0 and 12.9 us instead of 17.6, 33.0 and 17.3.  Past that the repeated set-up
// costs more than the shorter chains give: 262 k particles 38.5 us alone, 41.6 and 55.9 with
// two and four warps, the tiled search of a 2^20 binary64 tube 172 and 204 with one and four.
int shift_of(int blocks, uint32_t ptiles) {
  int shift = 0;
  while (shift < 3 && ((uint64_t)ptiles << (shift + 1)) <= (uint64_t)blocks) ++shift;
  return shift;
}

template <int PREC, int K>
void grids_of(int num_sms, uint32_t ptiles, LaunchPlan& L) {
  auto cap = [&](int blocks, int shift) {
    return (int)std::min<uint64_t>((uint64_t)blocks, (uint64_t)std::max(ptiles, 1u) << shift);
  };
  L.part_blocks = cap(resident_blocks(k_search<PREC, K>, kTile, 0, num_sms), 0);
  int blocks = resident_blocks(k_search_tiles<PREC, K, false>, kTile, 0, num_sms);
  L.tile_shift = shift_of(blocks, ptiles);
  // shared units go to the blocks one warp each: at least a block per SM
  L.tile_blocks = cap(blocks, L.tile_shift);
  if (L.tile_shift) L.tile_blocks = std::max(L.tile_blocks, num_sms);
  L.fast_blocks = std::min(resident_blocks(k_search_fast<PREC>, kCellWarps * 32, 0, num_sms),
                           (int)std::max(ptiles, (uint32_t)num_sms));
  if (PREC != KMC_GUARDED_FP32) return;
  // the row search keeps its piece lists in dynamic shared memory (above 48 KB for
  // K = 2); set before any launch or capture
  auto rows = [&](auto alone, auto shared, size_t bytes, int& grid, int& shift) {
    cudaFuncSetAttribute(alone, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    cudaFuncSetAttribute(shared, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    const int n = resident_blocks(alone, kTile, bytes, num_sms);
    shift = shift_of(n, ptiles);
    grid = cap(n, shift);
  };
  rows(k_search_rows32<K, false, false>, k_search_rows32<K, false, true>, RowLayout<K, false>::kBytes,
       L.row_blocks, L.row_shift);
  rows(k_search_rows32<K, true, false>, k_search_rows32<K, true, true>, RowLayout<K, true>::kBytes,
       L.row_blocks_px, L.row_shift_px);
}

// The searches of a step do not depend on each other (they append to one pair buffer by
// atomics), so in a captured step they become branches that join after the last: next()
// before each further search puts the capture back to where the first one started.  A step
// then waits for the longest of them instead of for their sum, and the idle ones cost nothing:
// ten binary64 steps of 4096 particles 0.96 -> 0.83 ms (17 us of tiles beside 13 of fast
// particles), four of an ensemble of 30 3.09 -> 2.73 ms, eight of 262 k particles 1.16 -> 1.10.
// Outside a capture, and after more than kMaxEnds nodes, one follows the other.
class Branches {
 public:
  explicit Branches(cudaStream_t st) : st_(st) { nfirst_ = ends(first_); }
  void next() {
    const size_t n = nfirst_ ? ends(last_ + nlast_) : 0;
    if (n == 0) return;
    nlast_ += n;
    cudaStreamUpdateCaptureDependencies(st_, first_, nullptr, nfirst_, cudaStreamSetCaptureDependencies);
  }
  void join() {  // what follows comes after the earlier branches too
    if (nlast_ == 0) return;
    cudaStreamUpdateCaptureDependencies(st_, last_, nullptr, nlast_, cudaStreamAddCaptureDependencies);
  }

 private:
  static constexpr size_t kMaxEnds = 4, kMaxSearches = 5;
  // the nodes that the next captured launch would follow (0: no capture, or too many)
  size_t ends(cudaGraphNode_t* to) const {
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    const cudaGraphNode_t* deps = nullptr;
    size_t n = 0;
    if (cudaStreamGetCaptureInfo(st_, &status, nullptr, nullptr, &deps, nullptr, &n) != cudaSuccess ||
        status != cudaStreamCaptureStatusActive || n > kMaxEnds)
      return 0;
    std::copy(deps, deps + n, to);
    return n;
  }
  cudaStream_t st_;
  cudaGraphNode_t first_[kMaxEnds], last_[kMaxEnds * kMaxSearches];
  size_t nfirst_ = 0, nlast_ = 0;
};

// Every search that a simulation of the plan may choose for a step; each runs the one its
// grid selected (the other kernels return at once).
template <int PREC, int K>
int launch_slow(const LaunchPlan& L, cudaStream_t st, Branches& b) {
  int n = 1;
  if (L.tile_shift) k_search_tiles<PREC, K, true><<<L.tile_blocks, kTile, 0, st>>>(L.b, L.tile_shift);
  else k_search_tiles<PREC, K, false><<<L.tile_blocks, kTile, 0, st>>>(L.b, 0);
  if (L.particle) {
    b.next();
    k_search<PREC, K><<<L.part_blocks, kTile, 0, st>>>(L.b);
    ++n;
  }
  auto rows = [&](auto alone, auto shared, size_t bytes, int grid, int shift) {
    b.next();
    if (shift) shared<<<grid, kTile, bytes, st>>>(L.b, shift);
    else alone<<<grid, kTile, bytes, st>>>(L.b, 0);
    ++n;
  };
  if (PREC == KMC_GUARDED_FP32 && L.bounded_x)
    rows(k_search_rows32<K, false, false>, k_search_rows32<K, false, true>, RowLayout<K, false>::kBytes,
         L.row_blocks, L.row_shift);
  if (PREC == KMC_GUARDED_FP32 && L.periodic_x)
    rows(k_search_rows32<K, true, false>, k_search_rows32<K, true, true>, RowLayout<K, true>::kBytes,
         L.row_blocks_px, L.row_shift_px);
  return n;
}
}  // namespace

void search_grids(int precision, int K, int num_sms, uint32_t ptiles, LaunchPlan& L) {
  if (precision == KMC_FP64) {
    if (K == 2) grids_of<KMC_FP64, 2>(num_sms, ptiles, L);
    else grids_of<KMC_FP64, 1>(num_sms, ptiles, L);
  } else {
    if (K == 2) grids_of<KMC_GUARDED_FP32, 2>(num_sms, ptiles, L);
    else grids_of<KMC_GUARDED_FP32, 1>(num_sms, ptiles, L);
  }
}

int launch_search(const LaunchPlan& L, int precision, int K, cudaStream_t st, cudaEvent_t* ev_slow) {
  int n = 0;
  Branches b(st);
  if (ev_slow) cudaEventRecord(ev_slow[0], st);
  if (precision == KMC_FP64) {
    n = K == 2 ? launch_slow<KMC_FP64, 2>(L, st, b) : launch_slow<KMC_FP64, 1>(L, st, b);
  } else {
    n = K == 2 ? launch_slow<KMC_GUARDED_FP32, 2>(L, st, b) : launch_slow<KMC_GUARDED_FP32, 1>(L, st, b);
  }
  if (ev_slow) cudaEventRecord(ev_slow[1], st);
  b.next();
  if (precision == KMC_FP64) k_search_fast<KMC_FP64><<<L.fast_blocks, kCellWarps * 32, 0, st>>>(L.b);
  else k_search_fast<KMC_GUARDED_FP32><<<L.fast_blocks, kCellWarps * 32, 0, st>>>(L.b);
  b.join();
  return n + 1;
}

}  // namespace kmc
