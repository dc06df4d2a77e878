// kmc_push.cu -- free streaming, boundaries, observables and the end-of-step
// bookkeeping (Sec. 2: positions updated, boundary conditions applied to particles
// that reach the walls; output at fixed intervals).
//
//   k_push      x += v dt for particles that did not collide (colliders were
//               streamed by k_collide), then the boundaries per axis:
//                 periodic   one wrap into [0, L), x == L mapped to 0;
//                 reflecting lower wall at 0; upper wall at L, or on x at the piston
//                            X = x0 - u ((step+1) dt): x -> 2X - x, v -> -v - 2u
//                            (specular reflection in the frame of the moving wall).
//               It also records the last partner and a binary32 upper bound of
//               max |v|^2 (directed rounding) for the next step's cell size.
//   k_profile   every profile_every steps: per x-bin count, sum v and sum v^2, in
//               exact fixed point (int64 digits), so the sums do not depend on the
//               order of the particles.
//   k_finalize  two warps per simulation: the next grid (kmc_grid.cuh); step record,
//               step counter and the per-step counters reset.
#include "kmc_grid.cuh"
#include "kmc_internal.cuh"

namespace kmc {

__device__ __forceinline__ void block_max_to(uint32_t* dst, float v) {
  __shared__ float wmax[kTile / 32];
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_down_sync(0xFFFFFFFFu, v, o));
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    float m = 0.0f;
    for (int w = 0; w < (int)(blockDim.x / 32); ++w) m = fmaxf(m, wmax[w]);
    atomicMax(dst, __float_as_uint(m));
  }
}

// ---- k_push ---------------------------------------------------------------- //
// The boundary fix-ups are rare (particles that crossed a wall or the periodic
// boundary in this step).  They sit in out-of-line functions so that their binary64
// operations issue only for the lanes that call them, instead of being predicated
// into every lane's instruction stream.
struct XV {
  double x, v;
};

// periodic axis: one wrap into [0, L), x == L mapped to 0
__device__ __noinline__ double wrap_periodic(double x, double L) {
  if (dbits(x) >= dbits(L)) x = dsub(x, L);
  if (lt_zero(x)) {
    x = dadd(x, L);
    if (dbits(x) == dbits(L)) x = 0.0;
  }
  return x;
}

// reflecting axis: lower wall at 0, upper wall (or piston) at X moving with u
__device__ __noinline__ XV reflect_walls(double x, double v, double X, double u) {
  if (lt_zero(x)) {
    x = -x;
    v = -v;
  }
  if (dbits(X) > 0 ? dbits(x) > dbits(X) : x > X) {
    x = dsub(dadd(X, X), x);
    v = dsub(-v, dadd(u, u));
  }
  return {x, v};
}

// Free streaming and walls of one particle (sorted position p); returns the binary32
// upper bound of its |v|^2 (0 if it left).  ABS: the simulation has absorbing walls.
template <bool ABS>
__device__ __forceinline__ float push_particle(SimDev& s, int cur, uint32_t p, double dt, double wall,
                                               bool& gone) {
  // everything is loaded before the first store (a load of the next axis cannot be moved
  // ahead of a store to this one)
  const uint32_t q = s.partner[p];
  double xs[3], vv[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    xs[a] = s.x[cur][a][p];
    vv[a] = s.v[cur][a][p];
  }
  if (q == kNone) {
#pragma unroll
    for (int a = 0; a < 3; ++a) xs[a] = dadd(xs[a], dmul(vv[a], dt));
  }
  // beyond an absorbing wall at the end of the step: the particle leaves the gas with
  // this position and velocity (tested before any other axis' boundary)
  if (ABS) {
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if (s.bc[a] == KMC_ABSORB && (lt_zero(xs[a]) || gt_bits(xs[a], s.box[a]))) gone = true;
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (ABS && (gone || s.bc[a] == KMC_ABSORB)) {
      // no wall acts (inside on this axis, or the particle has left)
    } else if (s.bc[a] == KMC_PERIODIC) {
      const double L = s.box[a];  // > 0
      if (dbits(xs[a]) >= dbits(L) || lt_zero(xs[a])) xs[a] = wrap_periodic(xs[a], L);
    } else {
      const double X = a == 0 ? wall : s.box[a];
      const double u = a == 0 ? s.piston_u : 0.0;
      if (lt_zero(xs[a]) || gt_bits(xs[a], X)) {
        const XV r = reflect_walls(xs[a], vv[a], X, u);
        xs[a] = r.x;
        vv[a] = r.v;
        s.v[cur][a][p] = r.v;
      }
    }
    s.x[cur][a][p] = xs[a];
  }
  if (ABS && gone) s.last[cur][p] = KMC_ABSORBED;
  else if (q != kNone) s.last[cur][p] = s.id[cur][q];
  return ABS && gone ? 0.0f : vmag2_up(vv[0], vv[1], vv[2]);
}

//
// What bounds it: the binary64 pipe (6 operations a particle, 173 us at 2^24 particles) and
// memory (77 bytes, 193 us).  Everything else on that pipe is kept off it: comparisons and
// conversions are on integers (an absolute value that the compiler made of a mask alone
// cost another three operations), the wall's position comes with the step.  32 registers
// (eight blocks per SM) hide one by the other: 350 -> 262 us at 2^24, where 40 registers
// take 349; 5.7 -> 4.8 us at 4096.  Each block takes every so many tiles and adds its
// maximum and counts once per simulation.
template <bool ABS>
__global__ void __launch_bounds__(kTile, 8) k_push(Batch B) {
  __shared__ uint32_t scnt[kSplitTrials];     // particles above each trial threshold
  __shared__ uint32_t sgone;                  // particles absorbed
  const uint32_t lane = threadIdx.x & 31u;
  if (threadIdx.x < kSplitTrials) scnt[threadIdx.x] = 0;
  if (ABS && threadIdx.x == 0) sgone = 0;
  float vmax = 0.0f;
  uint32_t mine = 0, left = 0;  // lane t: the warp's particles above threshold t; lane 0: gone
  const uint32_t ntiles = B.ptiles;
  for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int k = find_sim(B.ptile, B.nsims, tile);
    SimDev& s = B.sim(k);
    if (!sim_active(s)) continue;
    const int cur = s.d.parity ^ 1;
    const uint32_t p = (tile - B.tile0(B.ptile, k)) * kTile + threadIdx.x;
    // absorbing walls: particles that left earlier sit at the end of the order and stay
    // as they are (live_count is this step's sort's count of the others)
    const uint32_t n_in = ABS ? live_count(s) : s.n;
    const double dt = s.dt, wall = s.d.wall_x;
    bool gone = false;
    float vm = 0.0f;
    if (p < n_in) vm = (ABS && s.absorb) ? push_particle<true>(s, cur, p, dt, wall, gone)
                                         : push_particle<false>(s, cur, p, dt, wall, gone);
    vmax = fmaxf(vmax, vm);
    if (ABS && s.absorb) left += (uint32_t)__popc(__ballot_sync(0xFFFFFFFFu, gone));
    if (s.split_ok) {
      // particles above each trial split threshold; each particle keeps how many it
      // exceeds, which is all the next step's count needs to classify it
      const bool valid = p < n_in && !gone;
      uint32_t above = 0;
#pragma unroll
      for (int t = 1; t < kSplitTrials; ++t) {
        const bool hi = valid && vm > s.d.split_thr[t];
        above += hi ? 1u : 0u;
        const unsigned m = __ballot_sync(0xFFFFFFFFu, hi);
        if (lane == (uint32_t)t) mine += (uint32_t)__popc(m);
      }
      if (valid) s.vbucket[p] = (uint8_t)above;
    }
    const uint32_t next = tile + gridDim.x;
    if (next < ntiles && (B.nsims == 1 || find_sim(B.ptile, B.nsims, next) == k)) continue;
    // the block's last tile of the simulation: its sums to the simulation's counters
    __syncthreads();  // (the shared counters are clear)
    if (lane > 0 && lane < (uint32_t)kSplitTrials && mine) atomicAdd(&scnt[lane], mine);
    if (ABS && lane == 0 && left) atomicAdd(&sgone, left);
    block_max_to(&s.d.vmax2_acc, vmax);  // its block barrier also orders the shared counters
    if (threadIdx.x > 0 && threadIdx.x < kSplitTrials) {
      if (scnt[threadIdx.x]) atomicAdd(&s.d.split_cnt[threadIdx.x], scnt[threadIdx.x]);
      scnt[threadIdx.x] = 0;
    }
    if (ABS && threadIdx.x == 0) {
      if (sgone) atomicAdd(&s.d.n_absorbed, sgone);
      sgone = 0;
    }
    vmax = 0.0f;
    mine = left = 0;
  }
}

// The particles of a block's tiles are summed in shared memory, in 32-bit words of 16-bit
// digits (an atomic addition of 64 bits in shared memory is a compare-and-swap loop: a
// profile of 2^20 particles took 240 us, now 50), and the words flushed to the bin's
// 64-bit counters when the simulation changes or a digit could overflow: up to kProfFlush
// particles add up to less than 2^31.  A bin is kProfW words, an odd number, so that
// neighbouring bins lie in different banks: [0] the count, [1 + 6 t + c] digit c of term t
// (the three v_a, then the three v_a^2), [37] the terms out of range.
constexpr int kProfW = 39;
constexpr uint32_t kProfFlush = 1u << 15;

__device__ __forceinline__ void profile_term(int* q, double x, int& bad) {
  long long d[3];
  if (!fx_digits(x, d)) {
    ++bad;
    return;
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int m = x < 0.0 ? -1 : 1;
    const uint32_t w = (uint32_t)(d[c] < 0 ? -d[c] : d[c]);
    if (w & 0xFFFFu) atomicAdd(q + 2 * c, m * (int)(w & 0xFFFFu));
    if (w >> 16) atomicAdd(q + 2 * c + 1, m * (int)(w >> 16));
  }
}

template <bool ABS>
__global__ void __launch_bounds__(kTile) k_profile(Batch B, uint32_t ntiles) {
  extern __shared__ int acc[];
  const uint32_t per = (ntiles + gridDim.x - 1) / gridDim.x, t0 = blockIdx.x * per;
  const uint32_t t1 = t0 + per < ntiles ? t0 + per : ntiles;
  for (uint32_t tile = t0; tile < t1;) {
    // the block's tiles of one simulation, at most kProfFlush particles
    const int k = find_sim(B.prtile, B.nsims, tile);
    const uint32_t first = B.tile0(B.prtile, k);
    SimDev& s = B.sim(k);
    const uint32_t all = first + (s.n + kProfTile - 1u) / kProfTile;
    uint32_t end = t1 < all ? t1 : all;
    if (!sim_active(s) || !s.d.prof_due) {
      tile = end;
      continue;
    }
    if (end - tile > kProfFlush / kProfTile) end = tile + kProfFlush / kProfTile;
    const int nb = s.profile_bins;
    for (int i = threadIdx.x; i < nb * kProfW; i += blockDim.x) acc[i] = 0;
    __syncthreads();
    const int cur = s.d.parity ^ 1;
    const double scale = ddiv((double)nb, s.profile_range);
    const uint64_t stop = (uint64_t)(end - first) * kProfTile;
    const uint32_t pend = stop < s.n ? (uint32_t)stop : s.n;
    for (uint32_t p = (tile - first) * kProfTile + threadIdx.x; p < pend; p += blockDim.x) {
      if (ABS && s.absorb && s.last[cur][p] == KMC_ABSORBED) continue;  // out of the gas
      double x = s.x[cur][0][p];
      if (!(x >= 0.0)) continue;
      double f = dmul(x, scale);
      if (f >= (double)nb) continue;
      int* q = acc + (int)f * kProfW;
      int bad = 0;
      atomicAdd(q, 1);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const double v = s.v[cur][a][p];
        profile_term(q + 1 + 6 * a, v, bad);
        profile_term(q + 19 + 6 * a, dmul(v, v), bad);
      }
      if (bad) atomicAdd(q + 37, bad);
    }
    __syncthreads();
    long long* out = s.prof_acc + (size_t)(s.d.prof_count % s.prof_cap) * nb * kProfQ;
    for (int i = threadIdx.x; i < nb * kProfQ; i += blockDim.x) {
      const int b = i / kProfQ, c = i - b * kProfQ;
      const int* q = acc + b * kProfW;
      const long long sum = c == 0 ? q[0] : c == kProfQ - 1 ? q[37]
                                          : q[2 * c - 1] + 65536ll * q[2 * c];
      if (sum) atomicAdd((unsigned long long*)&out[i], (unsigned long long)sum);
    }
    __syncthreads();
    tile = end;
  }
}

constexpr int kFinalBlock = 256;  // two warps per simulation

// ---- end of step ------------------------------------------------------------ //
__device__ void reset_step_counters(SimDev& s) {
  s.d.n_raw = 0;
  s.d.n_edges = 0;
  for (int r = 0; r < 4; ++r) s.d.round_pairs[r] = 0;
  s.d.n_pairs = 0;
  s.d.adj_used = 0;
  for (int r = 0; r < 5; ++r) s.d.wl_len[r] = 0;
  s.d.pair_tests = 0;
  s.d.fast_tests = 0;
  s.d.n_absorbed = 0;
  s.d.vmax2_acc = 0;
}

// x % m; the 64-bit remainder (440 cycles of dependent operations) only past 2^32
__device__ __forceinline__ uint32_t mod_u32(uint64_t x, uint32_t m) {
  return (x >> 32) == 0 ? (uint32_t)x % m : (uint32_t)(x % (uint64_t)m);
}

// does the step that starts now (absolute index `step`) end with a profile?
__device__ __forceinline__ uint32_t prof_due_at(const SimDev& s, uint64_t step) {
  return (s.profile_bins > 0 && s.profile_every > 0 &&
          mod_u32(step + 1, (uint32_t)s.profile_every) == 0) ? 1u : 0u;
}

// clears the slot of the profile that the step will write (the warp's lanes together)
__device__ __forceinline__ void clear_profile(SimDev& s, uint32_t count, uint32_t lane) {
  long long* out = s.prof_acc + (size_t)(count % s.prof_cap) * s.profile_bins * kProfQ;
  for (int i = (int)lane; i < s.profile_bins * kProfQ; i += 32) out[i] = 0;
}

// Two warps per simulation: the first builds the next grid, the second keeps the books.
// Each is one chain of dependent operations, so what both need is read before the barrier
// that comes before the first store.
__global__ void __launch_bounds__(kFinalBlock) k_finalize(Batch B) {
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const int k = (int)(blockIdx.x * (kFinalBlock / 64u) + warp / 2u);
  const bool run = k < B.nsims && sim_active(B.sim(k));
  SimDev& s = B.sim(run ? k : 0);
  const uint64_t step = s.d.step;
  const float vmax2 = __uint_as_float(s.d.vmax2_acc);
  if (warp % 2u == 0u) {
    __syncthreads();
    if (run) compute_grid(s, vmax2, step + 1, s.split_ok != 0, lane);
    return;
  }
  const uint64_t hist_count = s.d.hist_count, steps_left = s.d.steps_left;
  const uint32_t hist_cap = s.hist_cap, was_due = s.d.prof_due, prof_cap = s.prof_cap;
  const uint32_t n_raw = s.d.n_raw, parity = s.d.parity;
  const uint32_t prof_count = s.d.prof_count + was_due;  // snapshots, this step's included
  const uint32_t due = prof_due_at(s, step + 1);
  kmc_step_counts rec;
  rec.step = step;
  uint32_t coll = 0;
  for (int r = 0; r < 4; ++r) {
    rec.round_pairs[r] = s.d.round_pairs[r];
    coll += rec.round_pairs[r];
  }
  rec.collisions = coll;
  rec.edges = s.d.n_edges;
  rec.survivors = n_raw;
  rec.cells = s.d.grid.nkeys;
  rec.pair_tests = s.d.pair_tests;
  rec.fast_tests = s.d.fast_tests;
  rec.absorbed = s.d.n_absorbed;
  rec.live = run ? live_count(s) - rec.absorbed : 0u;  // this step's grid, before the next one
  const uint32_t have = s.split_ok ? 1u : 0u;
  __syncthreads();
  if (!run) return;
  if (lane == 0) {
    s.hist[mod_u32(hist_count, hist_cap)] = rec;
    s.d.hist_count = hist_count + 1;
    if (was_due) {
      s.prof_step[(prof_count - 1u) % prof_cap] = step;
      s.d.prof_count = prof_count;
    }
    s.d.last_raw = n_raw;
    s.d.have_counts = have;
    s.d.parity = parity ^ 1u;
    s.d.step = step + 1;
    s.d.steps_left = steps_left - 1;
    s.d.vmax2 = vmax2;
    s.d.prof_due = due;
    reset_step_counters(s);
  }
  if (due) clear_profile(s, prof_count, lane);
}

// ---- initial grid (creation, resume, after an error is cleared) ------------ //
template <bool ABS>
__global__ void __launch_bounds__(kTile) k_vmax(Batch B) {
  int k = find_sim(B.ptile, B.nsims, blockIdx.x);
  SimDev& s = B.sim(k);
  uint32_t p = (blockIdx.x - B.tile0(B.ptile, k)) * kTile + threadIdx.x;
  float vm = 0.0f;
  if (p < s.n) {
    int par = s.d.parity;
    if (!(ABS && s.absorb && s.last[par][p] == KMC_ABSORBED))
      vm = vmag2_up(s.v[par][0][p], s.v[par][1][p], s.v[par][2][p]);
  }
  block_max_to(&s.d.vmax2_acc, vm);
}

// the trial thresholds of the speed split from the state's bound of max |v|^2
__global__ void k_init_thresholds(Batch B) {
  const uint32_t lane = threadIdx.x & 31u;
  const int nwarps = (int)(gridDim.x * blockDim.x / 32u);
  for (int k = (int)((blockIdx.x * blockDim.x + threadIdx.x) / 32u); k < B.nsims; k += nwarps) {
    SimDev& s = B.sim(k);
    const float v2 = __uint_as_float(s.d.vmax2_acc);
    if (lane == 0) s.d.vmax2 = v2;
    set_split_thresholds(s, v2, lane);
  }
}

// particles above each trial threshold, and each particle's speed class, as the push
// counts them at the end of a step: the first step can split the fast particles off
template <bool ABS>
__global__ void __launch_bounds__(kTile) k_split_count(Batch B) {
  __shared__ uint32_t scnt[kSplitTrials];
  const int k = find_sim(B.ptile, B.nsims, blockIdx.x);
  SimDev& s = B.sim(k);
  if (!s.split_ok) return;
  if (threadIdx.x < kSplitTrials) scnt[threadIdx.x] = 0;
  __syncthreads();
  const uint32_t p = (blockIdx.x - B.tile0(B.ptile, k)) * kTile + threadIdx.x;
  const int par = s.d.parity;
  const bool valid = p < s.n && !(ABS && s.absorb && s.last[par][p] == KMC_ABSORBED);
  const float vm = valid ? vmag2_up(s.v[par][0][p], s.v[par][1][p], s.v[par][2][p]) : 0.0f;
  uint32_t above = 0;
#pragma unroll
  for (int t = 1; t < kSplitTrials; ++t) {
    const bool hi = valid && vm > s.d.split_thr[t];
    above += hi ? 1u : 0u;
    const unsigned m = __ballot_sync(0xFFFFFFFFu, hi);
    if ((threadIdx.x & 31) == 0 && m) atomicAdd(&scnt[t], (uint32_t)__popc(m));
  }
  if (valid) s.vbucket[p] = (uint8_t)above;
  __syncthreads();
  if (threadIdx.x > 0 && threadIdx.x < kSplitTrials && scnt[threadIdx.x])
    atomicAdd(&s.d.split_cnt[threadIdx.x], scnt[threadIdx.x]);
}

// one warp per simulation
__global__ void k_init_grid(Batch B) {
  const uint32_t lane = threadIdx.x & 31u;
  const int nwarps = (int)(gridDim.x * blockDim.x / 32u);
  for (int k = (int)((blockIdx.x * blockDim.x + threadIdx.x) / 32u); k < B.nsims; k += nwarps) {
    SimDev& s = B.sim(k);
    if (lane == 0) s.d.have_counts = s.split_ok ? 1u : 0u;  // k_split_count's
    compute_grid(s, s.d.vmax2, s.d.step, s.split_ok != 0, lane);
    __syncwarp();
    const uint32_t due = prof_due_at(s, s.d.step);
    if (lane == 0) {
      reset_step_counters(s);
      s.d.prof_due = due;
    }
    if (due && s.prof_acc) clear_profile(s, s.d.prof_count, lane);
    __syncwarp();
  }
}

__global__ void k_zero_vmax(Batch B) {
  for (int k = threadIdx.x; k < B.nsims; k += blockDim.x) B.sim(k).d.vmax2_acc = 0;
}

int launch_init_grid(const LaunchPlan& L, cudaStream_t st) {
  k_zero_vmax<<<1, 256, 0, st>>>(L.b);
  if (L.absorb) k_vmax<true><<<L.ptiles, kTile, 0, st>>>(L.b);
  else k_vmax<false><<<L.ptiles, kTile, 0, st>>>(L.b);
  k_init_thresholds<<<(L.b.nsims + 7) / 8, 256, 0, st>>>(L.b);
  if (L.absorb) k_split_count<true><<<L.ptiles, kTile, 0, st>>>(L.b);
  else k_split_count<false><<<L.ptiles, kTile, 0, st>>>(L.b);
  k_init_grid<<<(L.b.nsims + 7) / 8, 256, 0, st>>>(L.b);
  return 5;
}

int launch_push(const LaunchPlan& L, cudaStream_t st) {
  const size_t smem = 256 * kProfW * sizeof(int);
  if (L.absorb) k_push<true><<<L.push_blocks, kTile, 0, st>>>(L.b);
  else k_push<false><<<L.push_blocks, kTile, 0, st>>>(L.b);
  if (L.profiles) {
    if (L.absorb) k_profile<true><<<L.prof_blocks, kTile, smem, st>>>(L.b, L.prtiles);
    else k_profile<false><<<L.prof_blocks, kTile, smem, st>>>(L.b, L.prtiles);
  }
  k_finalize<<<(L.b.nsims + 3) / 4, kFinalBlock, 0, st>>>(L.b);
  return L.profiles ? 3 : 2;
}

__global__ void k_add_steps(SimDev* d, uint64_t n) { d->d.steps_left += n; }
void launch_add_steps(SimDev* d, uint64_t nsteps, cudaStream_t st) {
  k_add_steps<<<1, 1, 0, st>>>(d, nsteps);
}

__global__ void k_member_states(Batch B, MemberState* out) {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < B.nsims; k += gridDim.x * blockDim.x)
    out[k] = {B.sim(k).d.step, B.sim(k).d.status};
}
void launch_member_states(const LaunchPlan& L, MemberState* out, cudaStream_t st) {
  k_member_states<<<(L.b.nsims + 255) / 256, 256, 0, st>>>(L.b, out);
}

__global__ void k_mark_refused(Batch B) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < B.nsims && sim_scheduled(B.sim(k))) B.sim(k).d.status |= ST_LAUNCH;
}
void mark_refused(const LaunchPlan& L, cudaStream_t st) {
  k_mark_refused<<<(L.b.nsims + 255) / 256, 256, 0, st>>>(L.b);
}

// ---- observables ------------------------------------------------------------ //
// The state in id order (x, y, z, vx, vy, vz as n binary64 each, then n last partners).
// Ids and positions in the cell order have nothing to do with each other, so one side of
// the copy goes to random addresses, and what counts is how many: k_state_pack writes each
// particle as one record of 64 bytes (two whole sectors, by two 32-byte stores) to its
// id's place in a scratch array, and k_state_unpack reads the records in order and writes
// the seven arrays with coalesced stores: 236 bytes of traffic per particle.  A gather of
// the seven fields (8 random bytes each, of sectors of 32 and DRAM bursts of 64) took 2.46
// ms at 2^24 and 18.6 ms at 10^8 particles; this takes 0.85 and 5.6.  The scratch is the
// state buffer that is not current with the key and rank arrays beside it, all of them
// rewritten by the next step's sort before they are read.
__device__ __forceinline__ double* state_scratch(const SimDev& s, int par) {
  return par == 0 ? reinterpret_cast<double*>(s.key) : s.x[0][0];
}

__global__ void k_state_pack(SimDev* d) {
  SimDev& s = *d;
  const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= s.n) return;
  const int par = s.d.parity;
  double* r = state_scratch(s, par) + 8 * (size_t)s.id[par][p];
  const double x = s.x[par][0][p], y = s.x[par][1][p], z = s.x[par][2][p];
  const double vx = s.v[par][0][p], vy = s.v[par][1][p], vz = s.v[par][2][p];
  const double last = __longlong_as_double((long long)s.last[par][p]);
  asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(r), "d"(x), "d"(y), "d"(z), "d"(vx)
               : "memory");
  asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(r + 4), "d"(vy), "d"(vz), "d"(last),
               "d"(0.0)
               : "memory");
}

// Few particles: the copy stays in the L2, and the random stores of the seven fields cost
// less than a second launch (4096 particles 4.7 us in two launches, 4.2 in one; 65 k 5.7 and
// 5.4, 131 k 7.2 and 7.6).
constexpr uint32_t kDirectState = 1u << 16;
__global__ void k_state_direct(SimDev* d, void* out) {
  SimDev& s = *d;
  const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x, n = s.n;
  if (p >= n) return;
  const int par = s.d.parity;
  const uint32_t id = s.id[par][p];
  double* o = (double*)out;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    o[(size_t)a * n + id] = s.x[par][a][p];
    o[(size_t)(3 + a) * n + id] = s.v[par][a][p];
  }
  ((uint32_t*)(o + (size_t)6 * n))[id] = s.last[par][p];
}
__global__ void k_state_unpack(SimDev* d, void* out) {
  SimDev& s = *d;
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t n = s.n;
  if (i >= n) return;
  const double* r = state_scratch(s, s.d.parity) + 8 * (size_t)i;
  double a[4], b[4];
  asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
               : "=d"(a[0]), "=d"(a[1]), "=d"(a[2]), "=d"(a[3]) : "l"(r) : "memory");
  asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
               : "=d"(b[0]), "=d"(b[1]), "=d"(b[2]), "=d"(b[3]) : "l"(r + 4) : "memory");
  double* o = (double*)out;
#pragma unroll
  for (int k = 0; k < 4; ++k) o[(size_t)k * n + i] = a[k];
  o[(size_t)4 * n + i] = b[0];
  o[(size_t)5 * n + i] = b[1];
  ((uint32_t*)(o + (size_t)6 * n))[i] = (uint32_t)__double_as_longlong(b[2]);
}

__global__ void k_gather_partners(SimDev* d, uint32_t* out) {
  SimDev& s = *d;
  uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= s.n) return;
  // partners refer to the buffer the last step ran on, which is the current one
  int par = s.d.parity;
  uint32_t q = s.partner[p];
  out[s.id[par][p]] = q == kNone ? kNone : s.id[par][q];
}

__global__ void k_gather_edges(SimDev* d, uint32_t cap, uint2* out, uint32_t* count) {
  SimDev& s = *d;
  int par = s.d.parity;
  uint32_t nraw = s.d.last_raw < s.edge_cap ? s.d.last_raw : s.edge_cap;
  for (uint32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < nraw; e += gridDim.x * blockDim.x) {
    uint2 sl = s.e_slot[e];
    if (sl.x == kNone) continue;
    uint2 pr = s.edge[e];
    uint32_t a = s.id[par][pr.x], b = s.id[par][pr.y];
    uint32_t pos = atomicAdd(count, 1u);
    if (pos < cap) out[pos] = a < b ? make_uint2(a, b) : make_uint2(b, a);
  }
}

__global__ void k_profile_convert(SimDev* d, uint32_t first, uint32_t count, uint32_t bins, double* out) {
  SimDev& s = *d;
  uint32_t total = count * bins * 7;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    uint32_t snap = i / (bins * 7), rem = i % (bins * 7), b = rem / 7, q = rem % 7;
    const long long* src = s.prof_acc + ((size_t)((first + snap) % s.prof_cap) * bins + b) * kProfQ;
    out[i] = profile_value(src, (int)q);
  }
}

// KMC_OBS_VMAX: max over the particles in the gas of (vx*vx + vy*vy) + vz*vz, each
// operation correctly rounded; the squares are non-negative, so their bit patterns
// order as their values and one 64-bit atomicMax per warp reduces them exactly
__global__ void k_vmax_exact(SimDev* d, unsigned long long* acc) {
  SimDev& s = *d;
  const int par = s.d.parity;
  unsigned long long m = 0ull;
  for (uint32_t p = blockIdx.x * blockDim.x + threadIdx.x; p < s.n; p += gridDim.x * blockDim.x) {
    if (s.absorb && s.last[par][p] == KMC_ABSORBED) continue;
    const double vx = s.v[par][0][p], vy = s.v[par][1][p], vz = s.v[par][2][p];
    const double q = dadd(dadd(dmul(vx, vx), dmul(vy, vy)), dmul(vz, vz));
    const unsigned long long b = (unsigned long long)__double_as_longlong(q);
    m = b > m ? b : m;
  }
  for (int off = 16; off > 0; off >>= 1) {
    const unsigned long long o = __shfl_xor_sync(0xFFFFFFFFu, m, off);
    m = o > m ? o : m;
  }
  if ((threadIdx.x & 31u) == 0 && m) atomicMax(acc, m);
}

__global__ void k_vmax_sqrt(const unsigned long long* acc, double* out) {
  out[0] = dsqrt(__longlong_as_double((long long)*acc));
}

void launch_vmax_exact(SimDev* d, unsigned long long* acc, double* out, cudaStream_t st) {
  cudaMemsetAsync(acc, 0, sizeof(unsigned long long), st);
  k_vmax_exact<<<304, 256, 0, st>>>(d, acc);
  k_vmax_sqrt<<<1, 1, 0, st>>>(acc, out);
}

// particles outside the box at creation: count them (host reports KMC_EINVAL)
// wall: where the x wall stands before the first step (+inf if it has not moved)
__global__ void k_validate(SimDev* d, uint32_t* bad, double wall) {
  SimDev& s = *d;
  uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= s.n) return;
  bool out = false;
  // a particle that already left through an absorbing wall may lie anywhere (finite)
  const bool left = s.absorb && s.last[s.d.parity][p] == KMC_ABSORBED;
  for (int a = 0; a < 3; ++a) {
    double q = s.x[s.d.parity][a][p];
    double hi = (a == 0 && s.bc[0] == KMC_REFLECT) ? s.piston_x0 : s.box[a];
    bool periodic = s.bc[a] == KMC_PERIODIC;
    if (left ? !(fabs(q) < 1e300) : (!(q >= 0.0) || (periodic ? !(q < hi) : !(q <= hi)))) out = true;
    if (!(fabs(s.v[s.d.parity][a][p]) < 1e15)) out = true;
  }
  if (s.planar && s.v[s.d.parity][2][p] != 0.0) out = true;
  if (s.mix && s.species[s.id[s.d.parity][p]] >= (uint32_t)s.mix_n) out = true;
  if (out) atomicAdd(bad, 1u);
  if (!left && gt_bits(s.x[s.d.parity][0][p], wall)) s.d.loose_from = 0;  // see watch_box
}

void launch_validate(SimDev* d, uint32_t n, uint32_t* bad, double wall, cudaStream_t st) {
  k_validate<<<(n + 255) / 256, 256, 0, st>>>(d, bad, wall);
}

void launch_gather_state(SimDev* d, uint32_t n, void* out, cudaStream_t st) {
  if (n == 0) return;
  if (n <= kDirectState) {
    k_state_direct<<<(n + 255) / 256, 256, 0, st>>>(d, out);
    return;
  }
  k_state_pack<<<(n + 255) / 256, 256, 0, st>>>(d);
  k_state_unpack<<<(n + 255) / 256, 256, 0, st>>>(d, out);
}
void launch_gather_partners(SimDev* d, uint32_t n, uint32_t* out, cudaStream_t st) {
  k_gather_partners<<<(n + 255) / 256, 256, 0, st>>>(d, out);
}
void launch_gather_edges(SimDev* d, uint32_t cap, uint2* out, uint32_t* count, cudaStream_t st) {
  k_gather_edges<<<304, 256, 0, st>>>(d, cap, out, count);
}
void launch_profile_convert(SimDev* d, uint32_t first, uint32_t count, uint32_t bins, double* out,
                            cudaStream_t st) {
  if (count == 0) return;
  k_profile_convert<<<152, 256, 0, st>>>(d, first, count, bins, out);
}

}  // namespace kmc
