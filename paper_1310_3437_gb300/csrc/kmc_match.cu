// kmc_match.cu -- exact candidate test, mutual-choice matching and the collision
// update (Sec. 2: "a closer partner replaces the one found so far"; "two particles
// only collide if they have both found each other"; positions and velocities of
// the colliding pair are then updated).
//
// All binary64 arithmetic goes through the __d*_rn intrinsics (never contracted),
// in the operation order of the definitions below, so every value is bit-identical
// to the binary64 definition evaluated on any IEEE-754 machine.
//
//   k_refine  exact test of every pair emitted by the search:
//             r = x_j - x_i (minimum image on periodic axes), v = v_j - v_i,
//             t* = -(r.v)/|v|^2, d_min^2 = |r x v|^2/|v|^2; candidate iff |v| != 0,
//             0 <= t* < dt, d_min^2 < d0^2, and the pair is not the pair that last
//             collided for both of its members.  Candidates propose themselves to both
//             members, which keep the one of least key.
//   k_settle  pairs that both members chose are matched; pairs with both members left
//             unmatched go to the next round.
//   k_rounds  the further rounds, in one launch: propose, settle.
//   k_collide isotropic centre-of-mass scatter of the matched pairs at the time of closest
//             approach.
// A domain decomposition exchanges choices between its domains inside every round, by
// particle: there k_refine hands out slots, k_alloc and k_fill build each particle's
// candidate list (only particles with candidates are touched), and kmc_domain.cu runs the
// rounds over them.
#include <algorithm>

#include "kmc_internal.cuh"
#include "kmc_rng.cuh"

namespace kmc {

// The point (u1, u2) of the unit disk from 32-bit words, u = w 2^-31 - 1 uniform in
// [-1, 1): accepted if 0 < s < 1 with s = fl(fl(u1^2) + fl(u2^2)).  Counter (id, step lo, k,
// step hi), key (seed lo, seed hi); two attempts per Philox call, both evaluated and the
// first accepted one kept, so that lanes whose first attempt fails do not split the warp.
__device__ __forceinline__ bool disk_point(uint64_t seed, uint64_t step, uint32_t id, double& u1,
                                           double& u2) {
  for (uint32_t k = 0; k < 64; ++k) {
    uint32_t c[4] = {id, (uint32_t)step, k, (uint32_t)(step >> 32)};
    philox4x32_10(c, (uint32_t)seed, (uint32_t)(seed >> 32));
    const bool oka = in_disk(c[0], c[1]), okb = in_disk(c[2], c[3]);
    if (oka || okb) {
      u1 = word_uniform(oka ? c[0] : c[2]);
      u2 = word_uniform(oka ? c[1] : c[3]);
      return true;
    }
  }
  return false;
}

// Point on the unit sphere by Marsaglia's method (Ann. Math. Stat. 43, 1972):
// n = (2 u1 sqrt(1-s), 2 u2 sqrt(1-s), 1 - 2 s).
__device__ __forceinline__ void sphere_point(double u1, double u2, double nv[3]) {
  const double s = dadd(dmul(u1, u1), dmul(u2, u2));
  const double q = dsqrt(dsub(1.0, s));
  nv[0] = dmul(dadd(u1, u1), q);
  nv[1] = dmul(dadd(u2, u2), q);
  nv[2] = dsub(1.0, dadd(s, s));
}

// Planar mode: a direction uniform on the unit circle from the same point, whose polar
// angle is uniform: the vector at twice that angle, ((u1^2 - u2^2)/s, (2 u1 u2)/s) (von
// Neumann's method, no trigonometric function).
__device__ __forceinline__ void circle_point(double u1, double u2, double nv[3]) {
  const double q1 = dmul(u1, u1), q2 = dmul(u2, u2), s = dadd(q1, q2);
  nv[0] = ddiv(dsub(q1, q2), s);
  nv[1] = ddiv(dmul(dadd(u1, u1), u2), s);
  nv[2] = 0.0;
}

// candidate pairs the search stored (a member whose buffer overflowed is not live)
__device__ __forceinline__ uint32_t raw_pairs(const SimDev& s) {
  return s.d.n_raw < s.edge_cap ? s.d.n_raw : s.edge_cap;
}

// ---- collision update ------------------------------------------------------ //
// For the pair (a, b) with a the smaller id: stream both to t*, scatter
//   g = v_a - v_b, V = (v_a + v_b) * 0.5, G = |g|,  v_a' = V + (G/2) n,  v_b' = V - (G/2) n,
// then stream the rest of the step:  x' = (x + v t*) + v' (dt - t*).
// (i the smaller id's position, j the other's.)  Everything is loaded before the first
// store: a load after one would have to wait for it (the compiler cannot know that the
// arrays do not overlap).
template <bool MIX>
__device__ __forceinline__ void collide_pair(SimDev& s, int cur, uint32_t i, uint32_t j,
                                             uint32_t ida, uint32_t idb, double t) {
  double* const px[3] = {s.x[cur][0], s.x[cur][1], s.x[cur][2]};
  double* const pv[3] = {s.v[cur][0], s.v[cur][1], s.v[cur][2]};
  const double dt = s.dt;
  double xa[3], xb[3], va[3], vb[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    va[c] = pv[c][i];
    vb[c] = pv[c][j];
    xa[c] = px[c][i];
    xb[c] = px[c][j];
  }
  // equal masses: V = (v_a + v_b)/2 and both get half the relative speed; a mixture:
  // V = (m_a v_a + m_b v_b)/M, v_a' = V + (m_b/M) G n, v_b' = V - (m_a/M) G n
  const bool mixed = MIX && s.mix;
  double ma = 1.0, mb = 1.0;
  if (mixed) {
    ma = s.sp_mass[s.species[ida]];
    mb = s.sp_mass[s.species[idb]];
  }
  double u1, u2, nv[3];
  if (!disk_point(s.seed, s.d.step, ida, u1, u2)) {
    atomicOr(&s.d.status, ST_RANDOM);
    return;
  }
  if (s.planar) circle_point(u1, u2, nv);
  else sphere_point(u1, u2, nv);
  double g[3], V[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) g[c] = dsub(va[c], vb[c]);
  double fa = 0.5, fb = 0.5;
  if (mixed) {
    const double M = dadd(ma, mb);
#pragma unroll
    for (int c = 0; c < 3; ++c) V[c] = ddiv(dadd(dmul(ma, va[c]), dmul(mb, vb[c])), M);
    fa = ddiv(mb, M);
    fb = ddiv(ma, M);
  } else {
#pragma unroll
    for (int c = 0; c < 3; ++c) V[c] = dmul(dadd(va[c], vb[c]), 0.5);
  }
  double G = dsqrt(dadd(dadd(dmul(g[0], g[0]), dmul(g[1], g[1])), dmul(g[2], g[2])));
  const double hGa = dmul(fa, G);
  const double hGb = dmul(fb, G);
  double rest = dsub(dt, t);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    double na = dadd(V[c], dmul(hGa, nv[c]));
    double nb = dsub(V[c], dmul(hGb, nv[c]));
    px[c][i] = dadd(dadd(xa[c], dmul(va[c], t)), dmul(na, rest));
    px[c][j] = dadd(dadd(xb[c], dmul(vb[c], t)), dmul(nb, rest));
    pv[c][i] = na;
    pv[c][j] = nb;
  }
}

// ---- matching by pairs ------------------------------------------------------ //
// best[round & 1][i] is the pair that particle i chose in the round: the one of least key
// (d_min^2, t*, partner id) among its pairs with both members unmatched -- a total order,
// so the choice does not depend on the order in which the pairs come.  Every pair proposes
// itself to both members (a compare-and-swap each, rarely more: a particle with candidates
// has 1.1 of them in the tubes); a pair that both members chose is matched.  A pair is
// still open after the round if neither member is matched in it, which the choices tell
// without waiting for the matches; the open pairs are the next round's list.  Against
// candidate lists per particle (built by two more launches, and two launches per round),
// exact test to last match of a step: 62 -> 27 us at 4096 particles, 403 -> 225 us at 2^24,
// 2.4 -> 1.2 ms at 10^8.
__device__ __forceinline__ bool key_less(double d2a, double ta, uint32_t ja, double d2b, double tb,
                                         uint32_t jb) {
  if (d2a < d2b) return true;
  if (d2a > d2b) return false;
  if (ta < tb) return true;
  if (ta > tb) return false;
  return ja < jb;
}

__device__ __forceinline__ uint32_t* round_best(const SimDev& s, int round) {
  return (round & 1) ? s.best : s.best_e;
}

// the other member of pair e
__device__ __forceinline__ uint32_t other_end(const SimDev& s, uint32_t e, uint32_t i) {
  const uint2 pr = __ldcg(s.edge + e);
  return pr.x == i ? pr.y : pr.x;
}

// Pair e (key d2, t; partner id) competes for particle i with the pair seen there (kNone:
// it holds the place).  The keys of the pairs that others put there are read past the L1,
// and ordered after the swap that showed the pair as their writes are before theirs: a fence
// on either side.
__device__ __forceinline__ void contest(const SimDev& s, int cur, uint32_t* best, uint32_t i, uint32_t e,
                                        double d2, double t, uint32_t partner_id, uint32_t seen) {
  while (seen != kNone) {
    __threadfence();
    if (!key_less(d2, t, partner_id, __ldcg(s.e_d2 + seen), __ldcg(s.e_t + seen),
                  s.id[cur][other_end(s, seen, i)]))
      return;
    const uint32_t old = atomicCAS(best + i, seen, e);
    if (old == seen) return;
    seen = old;
  }
}
// Pair e proposes itself to both its particles; both first swaps are in flight together.
__device__ __forceinline__ void propose(const SimDev& s, int cur, uint32_t* best, uint2 pr, uint32_t e,
                                        double d2, double t, uint32_t idi, uint32_t idj) {
  const uint32_t si = atomicCAS(best + pr.x, kNone, e), sj = atomicCAS(best + pr.y, kNone, e);
  contest(s, cur, best, pr.x, e, d2, t, idj, si);
  contest(s, cur, best, pr.y, e, d2, t, idi, sj);
}

// is particle i matched in the round whose choices are in best?
__device__ __forceinline__ bool matched_by(const SimDev& s, const uint32_t* best, uint32_t i) {
  const uint32_t e = __ldcg(best + i);
  return __ldcg(best + other_end(s, e, i)) == e;
}

// The verdict on pair e (kNone: no pair) after the proposals of a round: 2 if both members
// chose it, 1 if it is still open, 0 if a member was matched in another pair.
__device__ __forceinline__ int verdict(const SimDev& s, const uint32_t* best, uint32_t e, uint2 pr) {
  if (e == kNone) return 0;
  const uint32_t bi = __ldcg(best + pr.x), bj = __ldcg(best + pr.y);
  if (bi == e && bj == e) return 2;
  return !matched_by(s, best, pr.x) && !matched_by(s, best, pr.y) ? 1 : 0;
}

// The second half of a round for the block's turn (every thread calls it): matched pairs
// go to the list of collisions, open pairs to the next round's list with their members'
// choices cleared.  (Colliding a pair here, right after its verdict, was slower: 512 us at
// 2^24 particles where verdict and collisions apart take 300.)
__device__ __forceinline__ void settle(SimDev& s, int round, uint32_t e, uint2 pr) {
  const int v = verdict(s, round_best(s, round), e, pr);
  const uint32_t to = block_append(&s.d.n_pairs, v == 2 ? 1u : 0u, &s.d.round_pairs[round]);
  if (v == 2) {
    s.pairs[to] = e;
    s.partner[pr.x] = pr.y;
    s.partner[pr.y] = pr.x;
  }
  if (round + 1 < s.max_rounds) {
    const uint32_t at = block_append(&s.d.wl_len[round + 1], v == 1 ? 1u : 0u);
    if (v == 1) {
      uint32_t* next = round_best(s, round + 1);
      s.wl[(round + 1) & 1][at] = e;
      next[pr.x] = kNone;
      next[pr.y] = kNone;
    }
  }
}

// ---- k_refine ------------------------------------------------------------ //
// The exact test of every emitted pair, and round 0's proposals; with LISTS (a domain
// decomposition, whose rounds exchange choices between the domains) slots in the members'
// candidate lists instead.
// MIX: the plan has a mixture (per-pair contact distance, mass-weighted scatter)
template <bool MIX, bool LISTS>
__global__ void __launch_bounds__(kEdgeBlock) k_refine(Batch B, uint32_t few) {
  for_dealt(B, [](const SimDev& s) { return sim_scheduled(s) ? raw_pairs(s) : 0u; },
            [](SimDev& s, uint32_t first, uint32_t) {
    const int cur = s.d.parity ^ 1;
    const uint32_t nraw = raw_pairs(s);
    const double* const px[3] = {s.x[cur][0], s.x[cur][1], s.x[cur][2]};
    const double* const pv[3] = {s.v[cur][0], s.v[cur][1], s.v[cur][2]};
    uint32_t found = 0;
    for (uint32_t e = first; e < nraw; e += gridDim.x * kEdgeBlock) {
      uint2 pr = s.edge[e];
      uint32_t i = pr.x, j = pr.y;
      bool cand = false;
      double d2 = 0.0, t = 0.0;
      uint32_t idi = s.id[cur][i], idj = s.id[cur][j];
      const uint32_t li = s.last[cur][i], lj = s.last[cur][j];
      double r[3], v[3];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        r[a] = dsub(px[a][j], px[a][i]);
        v[a] = dsub(pv[a][j], pv[a][i]);
      }
      // contact distance: d0, or in a mixture the sum of the two effective radii (the
      // search tested against d0, at least every such sum)
      double c2 = s.d0sq;
      if (MIX && s.mix) {
        const double c = dadd(s.sp_radius[s.species[idi]], s.sp_radius[s.species[idj]]);
        c2 = dmul(c, c);
      }
      if (!(li == idj && lj == idi)) {
#pragma unroll
        for (int a = 0; a < 3; ++a)
          if (s.bc[a] == KMC_PERIODIC) r[a] = min_image(r[a], s.box[a], s.half_box[a]);
        double vv = dadd(dadd(dmul(v[0], v[0]), dmul(v[1], v[1])), dmul(v[2], v[2]));
        if (dbits(vv) != 0) {  // (a sum of squares: never -0.0)
          double rv = dadd(dadd(dmul(r[0], v[0]), dmul(r[1], v[1])), dmul(r[2], v[2]));
          t = ddiv(-rv, vv);
          double wx = dsub(dmul(r[1], v[2]), dmul(r[2], v[1]));
          double wy = dsub(dmul(r[2], v[0]), dmul(r[0], v[2]));
          double wz = dsub(dmul(r[0], v[1]), dmul(r[1], v[0]));
          d2 = ddiv(dadd(dadd(dmul(wx, wx), dmul(wy, wy)), dmul(wz, wz)), vv);
          // 0 <= t < dt and d2 < c2, on the integer pipes
          cand = !lt_zero(t) && (dbits(t) < dbits(s.dt)) &&
                 (unsigned long long)dbits(d2) < (unsigned long long)dbits(c2);
        }
      }
      if (cand) {
        s.e_d2[e] = d2;
        s.e_t[e] = t;
        if (LISTS) {
          uint32_t si = atomicAdd(&s.deg[i], 1u);
          uint32_t sj = atomicAdd(&s.deg[j], 1u);
          s.e_slot[e] = make_uint2(si, sj);
        } else {
          s.e_slot[e] = make_uint2(0u, 0u);
          __threadfence();  // the key is there before the pair can be seen
          uint32_t* best = round_best(s, 0);
          propose(s, cur, best, pr, e, d2, t, idi, idj);
        }
        ++found;
      } else {
        s.e_slot[e] = make_uint2(kNone, kNone);
      }
    }
    block_append(&s.d.n_edges, found);  // one atomic per block
  }, few);
}

// round 0's matches and open pairs
__global__ void __launch_bounds__(kEdgeBlock) k_settle(Batch B) {
  for_dealt(B, [](const SimDev& s) { return sim_scheduled(s) ? raw_pairs(s) : 0u; },
            [](SimDev& s, uint32_t first, uint32_t trips) {
    const uint32_t nraw = raw_pairs(s);
    // the block's trip count, the same for all its threads: the appends are block-wide
    uint32_t e = first;
    for (uint32_t k = 0; k < trips; ++k, e += gridDim.x * kEdgeBlock) {
      uint32_t pair = kNone;
      uint2 pr = make_uint2(0u, 0u);
      if (e < nraw && s.e_slot[e].x != kNone) {
        pair = e;
        pr = s.edge[e];
      }
      settle(s, 0, pair, pr);
    }
  });
}

// A barrier of all blocks of the launch (launched cooperatively: they all run).  The wait
// is bounded; false: it ran out, and every block that notices leaves.  The failure-path
// test's barrier never opens (closed).
constexpr int kGridWaitLimit = 1 << 20;  // spins: 0.3 s
__device__ __forceinline__ bool grid_barrier(uint32_t* ctl, bool closed) {
  __shared__ int ok;
  if (gridDim.x == 1) {
    __threadfence();
    __syncthreads();
    return true;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    ok = 1;
    volatile uint32_t* gen = ctl + 1;
    const uint32_t now = *gen;
    __threadfence();
    if (atomicAdd(ctl, 1u) == gridDim.x - 1u && !closed) {
      *(volatile uint32_t*)ctl = 0u;
      __threadfence();
      *gen = now + 1u;
    } else {
      int spins = 0;
      while (*gen == now) {
        if (++spins > kGridWaitLimit) { ok = 0; break; }
        if (spins > 16) __nanosleep(100);
      }
    }
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}

// Rounds 1 and up, all in one launch: their lists hold a few percent of round 0's pairs
// (2000 of 750 000 in the 2^24 tube), and a launch costs more than their work.  Lists and
// choices are read past the L1: other blocks wrote them in this launch.
__device__ __forceinline__ uint32_t open_pairs(const SimDev& s, int round) {
  return sim_scheduled(s) && round < s.max_rounds ? __ldcg(&s.d.wl_len[round]) : 0u;
}

__global__ void __launch_bounds__(kEdgeBlock) k_rounds(Batch B, int max_rounds, bool closed) {
  // Steps queued behind a failed one find no member that runs and do not wait again.  (Only
  // a wait that ran out changes the answer during the launch.)
  bool any = false;
  for (int k = (int)threadIdx.x; k < B.nsims; k += kEdgeBlock) any = any || sim_active(B.sim(k));
  if (!__syncthreads_or(any)) return;
  for (int round = 1; round < max_rounds; ++round) {
    for_dealt(B, [round](const SimDev& s) { return open_pairs(s, round); },
              [round](SimDev& s, uint32_t first, uint32_t) {
      const int cur = s.d.parity ^ 1;
      const uint32_t len = __ldcg(&s.d.wl_len[round]);
      const uint32_t* list = s.wl[round & 1];
      uint32_t* best = round_best(s, round);
      for (uint32_t t = first; t < len; t += gridDim.x * kEdgeBlock) {
        const uint32_t e = __ldcg(list + t);
        const uint2 pr = s.edge[e];
        const double d2 = s.e_d2[e], tt = s.e_t[e];
        propose(s, cur, best, pr, e, d2, tt, s.id[cur][pr.x], s.id[cur][pr.y]);
      }
    });
    bool in_time = grid_barrier(B.round_ctl, closed);
    if (in_time) {
      for_dealt(B, [round](const SimDev& s) { return open_pairs(s, round); },
                [round](SimDev& s, uint32_t first, uint32_t trips) {
        const uint32_t len = __ldcg(&s.d.wl_len[round]);
        const uint32_t* list = s.wl[round & 1];
        uint32_t t = first;
        for (uint32_t k = 0; k < trips; ++k, t += gridDim.x * kEdgeBlock) {
          const uint32_t e = t < len ? __ldcg(list + t) : kNone;
          settle(s, round, e, e != kNone ? s.edge[e] : make_uint2(0u, 0u));
        }
      });
      if (round + 1 == max_rounds) return;
      in_time = grid_barrier(B.round_ctl, closed);
    }
    if (!in_time) {
      for (int k = (int)threadIdx.x; k < B.nsims; k += kEdgeBlock)
        if (sim_scheduled(B.sim(k))) atomicOr(&B.sim(k).d.status, ST_ROUND_WAIT);
      return;
    }
    if (B.nsims == 1 && __ldcg(&B.sim(0).d.wl_len[round + 1]) == 0u) return;  // nothing is open
  }
}

// ---- candidate lists (domain decomposition) ---------------------------------- //

// the pair whose slot is 0 at an endpoint opens that endpoint's list
__global__ void __launch_bounds__(kEdgeBlock) k_alloc(Batch B) {
  for_dealt(B, [](const SimDev& s) { return sim_scheduled(s) ? raw_pairs(s) : 0u; },
            [](SimDev& s, uint32_t first, uint32_t trips) {
    const uint32_t nraw = raw_pairs(s);
    const uint32_t stride = gridDim.x * kEdgeBlock;
    // the block's trip count, the same for all its threads: the appends are block-wide
    uint32_t e = first;
    for (uint32_t t = 0; t < trips; ++t, e += stride) {
      uint32_t i = kNone, j = kNone, di = 0, dj = 0;
      if (e < nraw) {
        const uint2 sl = s.e_slot[e];
        if (sl.x != kNone) {
          const uint2 pr = s.edge[e];
          if (sl.x == 0) { i = pr.x; di = s.deg[i]; }
          if (sl.y == 0) { j = pr.y; dj = s.deg[j]; }
        }
      }
      const uint32_t at = block_append(&s.d.adj_used, di + dj);
      const uint32_t wa = block_append(&s.d.wl_len[0], (i != kNone ? 1u : 0u) + (j != kNone ? 1u : 0u));
      if (i != kNone) { s.off[i] = at; s.wl[0][wa] = i; }
      if (j != kNone) { s.off[j] = at + di; s.wl[0][wa + (i != kNone ? 1u : 0u)] = j; }
    }
  });
}

__global__ void __launch_bounds__(kEdgeBlock) k_fill(Batch B) {
  for_dealt(B, [](const SimDev& s) { return sim_scheduled(s) ? raw_pairs(s) : 0u; },
            [](SimDev& s, uint32_t first, uint32_t) {
    const uint32_t nraw = raw_pairs(s);
    for (uint32_t e = first; e < nraw; e += gridDim.x * kEdgeBlock) {
      uint2 sl = s.e_slot[e];
      if (sl.x == kNone) continue;
      uint2 pr = s.edge[e];
      s.adj[s.off[pr.x] + sl.x] = make_uint2(pr.y, e);
      s.adj[s.off[pr.y] + sl.y] = make_uint2(pr.x, e);
    }
  });
}

// the step's collisions: matched pairs (domains: smaller-id members with their partners)
template <bool MIX, bool LISTS>
__global__ void __launch_bounds__(kEdgeBlock) k_collide(Batch B, uint32_t few) {
  for_dealt(B, [](const SimDev& s) { return sim_scheduled(s) ? s.d.n_pairs : 0u; },
            [](SimDev& s, uint32_t first, uint32_t) {
    const int cur = s.d.parity ^ 1;
    const uint32_t total = s.d.n_pairs;
    for (uint32_t q = first; q < total; q += gridDim.x * kEdgeBlock) {
      const uint32_t at = s.pairs[q];
      const uint32_t e = LISTS ? s.medge[at] : at;
      const uint2 pr = LISTS ? make_uint2(at, s.partner[at]) : s.edge[at];
      const uint32_t idi = s.id[cur][pr.x], idj = s.id[cur][pr.y];
      const bool first_is_a = idi < idj;
      collide_pair<MIX>(s, cur, first_is_a ? pr.x : pr.y, first_is_a ? pr.y : pr.x,
                        first_is_a ? idi : idj, first_is_a ? idj : idi, s.e_t[e]);
    }
  }, few);
}

// The exact test and the collision keep 14 and more binary64 values a pair, so two to four of
// their blocks fit an SM.  Pairs that those can take in one go are dealt to that many blocks:
// dealt 32 to a block over a block per 256 particles, the 47 k collisions of a 2^20 tube ran
// in four waves of two warps per SM (28 -> 18 us, its exact test 25 -> 19).  For more pairs the
// larger grid is the better one (a 2^21 blast's exact test 61 us, 78 on the resident blocks).
void match_grids(int num_sms, LaunchPlan& L) {
  auto few = [&](auto kernel) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kEdgeBlock, 0) != cudaSuccess ||
        per_sm < 1) {
      cudaGetLastError();
      per_sm = 2;
    }
    return per_sm * num_sms;
  };
  L.refine_few = L.mix ? few(k_refine<true, false>) : few(k_refine<false, false>);
  L.collide_few = L.mix ? few(k_collide<true, false>) : few(k_collide<false, false>);
  L.round_blocks = std::min(L.round_blocks, few(k_rounds));  // the cooperative grid: all resident
}

int launch_match_lists(const LaunchPlan& L, cudaStream_t st) {
  const int nb = L.edge_blocks;
  k_refine<false, true><<<nb, kEdgeBlock, 0, st>>>(L.b, L.refine_few);  // (domains have no mixtures)
  k_alloc<<<nb, kEdgeBlock, 0, st>>>(L.b);
  k_fill<<<nb, kEdgeBlock, 0, st>>>(L.b);
  return 3;
}

int launch_collide(const LaunchPlan& L, cudaStream_t st) {
  const int nb = L.edge_blocks, few = L.collide_few;
  if (L.mix) k_collide<true, false><<<nb, kEdgeBlock, 0, st>>>(L.b, few);
  else if (L.lists) k_collide<false, true><<<nb, kEdgeBlock, 0, st>>>(L.b, few);
  else k_collide<false, false><<<nb, kEdgeBlock, 0, st>>>(L.b, few);
  return 1;
}

int launch_match(const LaunchPlan& L, int max_rounds, cudaStream_t st) {
  const int nb = L.edge_blocks;
  if (L.mix) k_refine<true, false><<<nb, kEdgeBlock, 0, st>>>(L.b, L.refine_few);
  else k_refine<false, false><<<nb, kEdgeBlock, 0, st>>>(L.b, L.refine_few);
  k_settle<<<nb, kEdgeBlock, 0, st>>>(L.b);
  int n = 2;
  if (max_rounds > 1) {
    Batch b = L.b;
    bool closed = L.round_wait_test;
    void* args[] = {&b, &max_rounds, &closed};
    // refused where fewer blocks fit than the device's attributes say (a process that has a
    // part of its SMs): without the rounds the step must not go on
    if (cudaLaunchCooperativeKernel((const void*)k_rounds, dim3(L.round_blocks), dim3(kEdgeBlock),
                                    args, 0, st) != cudaSuccess)
      return -1;
    ++n;
  }
  return n + launch_collide(L, st);
}

}  // namespace kmc
