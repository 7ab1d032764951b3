// asep_sca.cuh -- the bit-sliced two-sub-lattice SCA on units held in
// registers (kernel and launches: asep_sca.cu).
//
// A unit is 256 sites = 8 words = four groups of 32 bonds per phase.  Group g
// holds the bonds of word 2g in its even lanes and of word 2g + 1 in its odd
// lanes (bond j of a word: lanes 2j and 2j + 1).  A unit is kept as two words
// per group: e[g] = the even sites and o[g] = the odd sites, each at the lane
// of its even bond.  An even bond is then lane l of (e, o) and its flip one
// XOR of each word; the plain word layout pays shifts and masks to line up
// candidates, random planes and flips.  An odd bond joins o's lane l with e's
// next lane in bond order (0, 2, ..., 30, 1, 3, ..., 31, then the next
// group's 0): odd_sites / odd_flips move e by one bond.
#pragma once

#include <cstdint>

#include "asep_device.cuh"
#include "asep_internal.h"

namespace asep {
namespace {

constexpr uint32_t kEven = 0x55555555u;
constexpr uint32_t kOdd = 0xAAAAAAAAu;

// A unit's words in bond lanes.
struct ScaUnit {
  uint32_t e[4], o[4];
};

// Eight consecutive words (16-byte aligned) into registers.
__device__ __forceinline__ void load8(const uint32_t* p, uint32_t (&x)[8]) {
  const uint4 v0 = reinterpret_cast<const uint4*>(p)[0], v1 = reinterpret_cast<const uint4*>(p)[1];
  x[0] = v0.x; x[1] = v0.y; x[2] = v0.z; x[3] = v0.w; x[4] = v1.x; x[5] = v1.y; x[6] = v1.z; x[7] = v1.w;
}

__device__ __forceinline__ void store8(uint32_t* p, const uint32_t (&x)[8]) {
  reinterpret_cast<uint4*>(p)[0] = make_uint4(x[0], x[1], x[2], x[3]);
  reinterpret_cast<uint4*>(p)[1] = make_uint4(x[4], x[5], x[6], x[7]);
}

__device__ __forceinline__ ScaUnit to_lanes(const uint32_t (&x)[8]) {
  ScaUnit u;
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    u.e[g] = (x[2 * g] & kEven) | ((x[2 * g + 1] << 1) & kOdd);
    u.o[g] = ((x[2 * g] >> 1) & kEven) | (x[2 * g + 1] & kOdd);
  }
  return u;
}

__device__ __forceinline__ void to_words(const ScaUnit& u, uint32_t (&x)[8]) {
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    x[2 * g] = (u.e[g] & kEven) | ((u.o[g] << 1) & kOdd);
    x[2 * g + 1] = ((u.e[g] >> 1) & kEven) | (u.o[g] & kOdd);
  }
}

// Even sites at the lane of the odd bond they end (en = the next group's e).
__device__ __forceinline__ uint32_t odd_sites(uint32_t e, uint32_t en) {
  const uint32_t z = ((e >> 1) & 1u) | ((en << 1) & ~1u);  // lane 1 -> 30, next group's lane 0 -> 31
  return __funnelshift_r(e, z, 2);
}

// The flips of e's sites from the odd bonds' moves h (hp = the previous group's).
__device__ __forceinline__ uint32_t odd_flips(uint32_t h, uint32_t hp) {
  const uint32_t y = ((h << 1) & 0x80000000u) | ((hp >> 1) & 0x7FFFFFFFu);  // lane 30 -> 1, previous 31 -> 0
  return __funnelshift_l(y, h, 2);
}

// ---------------------------------------------------------------------------
// Random planes: the parts of the Philox calls that a sweep's units share
// ---------------------------------------------------------------------------

// Per sweep of a chunk: a0 (round 1 of the sweep word) and the heads of the
// plane calls and of the two lane-change calls, formed cooperatively once per
// chunk of sweeps and read by every warp as broadcasts.
constexpr uint32_t kScaHeadEntries = 160;  // heads per chunk
constexpr uint32_t kScaChunkMax = 64;      // sweeps per chunk

struct ScaHeads {
  uint32_t a0[kScaChunkMax];
  uint4 head[kScaHeadEntries];  // [sweep][calls]: planes 0 .. kmax - 1, then (lane changes) steps 0 and 1
};

__device__ __forceinline__ uint32_t sca_calls(uint32_t kmax, bool turns) { return max(1u, kmax + (turns ? 2u : 0u)); }

// Sweeps per chunk.
__device__ __forceinline__ uint32_t sca_chunk(uint32_t calls) { return min(kScaChunkMax, kScaHeadEntries / calls); }

__device__ __forceinline__ void sca_fill_heads(ScaHeads& h, uint64_t s0, uint32_t n, uint32_t kmax, uint32_t calls,
                                               uint32_t n_glob, const KeySchedule& ks) {
  for (uint32_t i = threadIdx.x; i < n * calls; i += blockDim.x) {
    const uint32_t j = i / calls, k = i - j * calls;
    const uint64_t s = s0 + j;
    const uint32_t lo = static_cast<uint32_t>(s);
    const uint4 c = k < kmax ? ctr_of(s, kTagSca, k, n_glob, 0) : ctr_of(s, kTagScaTurn, k - kmax, n_glob, 0);
    const PhiloxHead p = philox_head(lo, c.y, n_glob, ks);
    h.head[i] = make_uint4(p.c3, p.y3, p.d3, 0u);
    if (k == 0) h.a0[j] = philox_a0(lo, ks);
  }
}

__device__ __forceinline__ uint4 sca_plane(const uint4* heads, uint32_t k, const PhiloxLane& l, const KeySchedule& ks) {
  const uint4 v = heads[k];
  return philox_tail(PhiloxHead{v.x, v.y, v.z}, l, ks);
}

// ---------------------------------------------------------------------------
// Which bonds move
// ---------------------------------------------------------------------------

// All-ones where bit k (0 = most significant of 20) of a 20-bit threshold is set.
__device__ __forceinline__ uint32_t bit_mask(uint32_t t20, uint32_t k) { return 0u - ((t20 >> (19u - k)) & 1u); }

__device__ __forceinline__ uint32_t bitsel(uint32_t m, uint32_t a, uint32_t b) { return (a & m) | (b & ~m); }

// Rings without disorder whose thresholds p and q are decided by at most two
// planes (FAST = 4 p2 + q2, the thresholds' top two bits, each 1..3; 0 = any
// other thresholds): u < t is ~(u0 | u1) for t = 1, ~u0 for t = 2 and
// ~(u0 & u1) for t = 3, so whether bond lanes would swap their sites is one
// logic operation of (first sites f, planes u0, u1).
constexpr uint32_t kScaAny = 0;
constexpr uint32_t kScaHalves = 4 * 2 + 2;  // one plane

template <uint32_t T2>
__device__ __forceinline__ uint32_t below2(uint32_t u0, uint32_t u1) {
  return T2 == 1u ? ~(u0 | u1) : (T2 == 2u ? ~u0 : ~(u0 & u1));
}

// Lanes whose bond swaps (a swap of equal sites changes nothing).
template <uint32_t FAST>
__device__ __forceinline__ uint32_t swaps_fast(uint32_t f, uint32_t u0, uint32_t u1) {
  return bitsel(f, below2<(FAST >> 2)>(u0, u1), below2<(FAST & 3u)>(u0, u1));
}

// Thresholds of a ring as the plane-by-plane comparison uses them (uniform):
// t[c] of the classes c = fast right, slow right, fast left, slow left.  A
// class whose threshold is 0 or "always" needs no draw; it takes another
// class's planes, so that as few distinct ones as possible are left.
struct ScaRule {
  uint32_t p, ps, q, qs;  // 20 bits
  bool special;           // some class needs no draw
  bool by_class;          // right and left hops share their planes: the slow classes alone select
};

__device__ __forceinline__ ScaRule sca_rule(const Rates& r, bool dis) {
  const auto fixed = [](uint32_t t) { return t == 0u || t == 0xFFFFFFFFu; };
  const uint32_t p0 = r.p, s0 = dis ? r.p_slow : r.p, q0 = r.q, t0 = dis ? r.q_slow : r.q;
  ScaRule v;
  v.special = fixed(p0) || fixed(s0) || fixed(q0) || fixed(t0);
  const uint32_t p = !fixed(p0) ? p0 : (!fixed(s0) ? s0 : (!fixed(q0) ? q0 : t0));
  const uint32_t ps = !fixed(s0) ? s0 : p;
  const uint32_t q = !fixed(q0) ? q0 : (!fixed(t0) ? t0 : p);
  const uint32_t qs = !fixed(t0) ? t0 : (!fixed(q0) ? q : ps);
  v.p = p >> 12;
  v.ps = ps >> 12;
  v.q = q >> 12;
  v.qs = qs >> 12;
  v.by_class = v.p == v.q && v.ps == v.qs;
  return v;
}

constexpr uint32_t kScaBlock = 7;  // planes taken without looking for undecided lanes

// Any thresholds.  c1: slow classes of the first sites (right hops), c2: of
// the second sites (left hops); DIS = false: no classes.  The first kScaBlock
// planes decide all but a few of a warp's some 2000 candidates, so they are
// compared from the least significant side (lt = u < t and eq = u == t over the
// planes so far, no vote); the rest most significant first, until no candidate
// of the warp is undecided (some 12 planes in all).  All 32 lanes call.
// Without branches inside a plane: asking whether the thresholds' bits agree
// saves a logic operation a group there (rings of 2^17 at p = 0.8, q = 0.2 14.4
// us a sweep instead of 14.6, 201 rings of 391 units with four classes 8.74
// instead of 9.0), but where a scheduler has one warp, each branch is a wait:
// 76 rings of 32 units with classes 3.14 -> 2.66, 265 of 14 units 3.17 -> 2.86
// (both with the smaller tiles).  Two calls in flight: no gain there, 3-5 %
// slower with classes.
template <bool DIS, typename PLANE>
__device__ __forceinline__ void decide_any(const uint32_t (&f)[4], const uint32_t (&n)[4], const uint32_t (&c1)[4],
                                           const uint32_t (&c2)[4], const Rates& r, const ScaRule& rule, uint32_t kmax,
                                           PLANE plane, uint32_t (&h)[4]) {
  constexpr uint32_t kAll = 0xFFFFFFFFu;
  uint32_t eq[4], cand[4], sl[4];
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    cand[g] = f[g] ^ n[g];
    h[g] = 0u;
    sl[g] = DIS ? bitsel(f[g], c1[g], c2[g]) : 0u;
  }
  if (rule.special) {  // classes that need no draw
    const uint32_t pA = r.p == kAll ? ~0u : 0u, qA = r.q == kAll ? ~0u : 0u;
    const uint32_t pN = r.p == 0u ? ~0u : 0u, qN = r.q == 0u ? ~0u : 0u;
    const uint32_t psA = r.p_slow == kAll ? ~0u : 0u, qsA = r.q_slow == kAll ? ~0u : 0u;
    const uint32_t psN = r.p_slow == 0u ? ~0u : 0u, qsN = r.q_slow == 0u ? ~0u : 0u;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const uint32_t A = DIS ? bitsel(f[g], bitsel(sl[g], psA, pA), bitsel(sl[g], qsA, qA)) : bitsel(f[g], pA, qA);
      const uint32_t N = DIS ? bitsel(f[g], bitsel(sl[g], psN, pN), bitsel(sl[g], qsN, qN)) : bitsel(f[g], pN, qN);
      h[g] = cand[g] & A;
      cand[g] &= ~(A | N);
    }
  }
  const uint32_t kb = min(kmax, kScaBlock);
#pragma unroll
  for (int g = 0; g < 4; ++g) eq[g] = cand[g];
  // bit k of every lane's threshold: one selector tells two thresholds apart (no classes: the first sites; classes
  // that right and left hops share: the classes), or classes and first sites four
  const auto two = [&](uint32_t k, uint32_t (&t)[4]) {
    const uint32_t m1 = bit_mask(DIS ? rule.ps : rule.p, k), m0 = bit_mask(DIS ? rule.p : rule.q, k);
#pragma unroll
    for (int g = 0; g < 4; ++g) t[g] = bitsel(DIS ? sl[g] : f[g], m1, m0);
  };
  const auto four = [&](uint32_t k, uint32_t (&t)[4]) {
    const uint32_t mp = bit_mask(rule.p, k), mq = bit_mask(rule.q, k), mps = bit_mask(rule.ps, k), mqs = bit_mask(rule.qs, k);
#pragma unroll
    for (int g = 0; g < 4; ++g) t[g] = bitsel(f[g], bitsel(sl[g], mps, mp), bitsel(sl[g], mqs, mq));
  };
  const auto run = [&](auto bits) {
    uint32_t lt[4] = {0u, 0u, 0u, 0u};
    const auto up = [&](uint32_t k, const uint4 y) {
      const uint32_t u[4] = {y.x, y.y, y.z, y.w};
      uint32_t t[4];
      bits(k, t);
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        lt[g] = bitsel(t[g], lt[g] | ~u[g], lt[g] & ~u[g]);
        eq[g] &= ~(t[g] ^ u[g]);
      }
    };
#pragma unroll 1
    for (uint32_t k = kb; k-- > 0;) up(k, plane(k));
#pragma unroll
    for (int g = 0; g < 4; ++g) h[g] |= cand[g] & lt[g];
#pragma unroll 1
    for (uint32_t k = kb; k < kmax; ++k) {
      if (!__any_sync(0xffffffffu, (eq[0] | eq[1] | eq[2] | eq[3]) != 0u)) break;
      const uint4 y = plane(k);
      const uint32_t u[4] = {y.x, y.y, y.z, y.w};
      uint32_t t[4];
      bits(k, t);
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        h[g] |= eq[g] & t[g] & ~u[g];  // this bit of u is 0 where t's is 1: u < t
        eq[g] &= ~(t[g] ^ u[g]);       // equal so far
      }
    }
  };
  if (!DIS || rule.by_class) run(two);
  else run(four);
}

// In-lane bonds of one lane of the two-lane model: candidates cand, one
// threshold t for all of them.  All 32 lanes call.
template <typename PLANE>
__device__ __forceinline__ void decide_lane(const uint32_t (&cand)[4], uint32_t t, PLANE plane, uint32_t (&h)[4]) {
  const uint32_t t20 = t >> 12;
  const bool always = t == 0xFFFFFFFFu, draws = t != 0u && !always;
  uint32_t eq[4];
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    h[g] = always ? cand[g] : 0u;
    eq[g] = cand[g];
  }
  if (!draws) return;
  const uint32_t kmax = 21u - static_cast<uint32_t>(__ffs(static_cast<int>(t20)));
  for (uint32_t k = 0; k < kmax; ++k) {
    if (k > 0u && !__any_sync(0xffffffffu, (eq[0] | eq[1] | eq[2] | eq[3]) != 0u)) break;
    const uint4 y = plane(k);
    const uint32_t u[4] = {y.x, y.y, y.z, y.w};
    if ((t20 >> (19u - k)) & 1u) {
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        h[g] |= eq[g] & ~u[g];
        eq[g] &= u[g];
      }
    } else {
#pragma unroll
      for (int g = 0; g < 4; ++g) eq[g] &= ~u[g];
    }
  }
}

struct ScaCounts {
  uint32_t c[4] = {0u, 0u, 0u, 0u};  // at most 512 a sweep and unit, 128 sweeps a launch
};

// One phase of one unit of lane P (ring: P = 0), given the phase's first
// planes: updates the unit's sites, except that in the odd phase the even
// sites are left to the caller, who gets the moves h (their flips cross
// units: the last group's bond 31 ends in the next unit's site 0).  counted:
// all ones, or zero for a unit whose hops another thread counts.
template <uint32_t MODEL, bool DIS, bool PQ, bool COUNT, uint32_t FAST, uint32_t PHASE, uint32_t P>
__device__ __forceinline__ void sca_update(ScaUnit& x, uint32_t en, const ScaUnit (&Q)[(DIS && PQ) ? 2 : 1],
                                           const uint32_t (&q_odd)[4], const Rates& r, const ScaRule& rule,
                                           uint32_t kmax, const uint4* heads, const PhiloxLane& pl, const uint4 y0, const uint4 y1,
                                           const KeySchedule& ks, uint32_t counted, ScaCounts& cnt,
                                           uint32_t (&h)[4]) {
  uint32_t f[4], n[4];
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    f[g] = PHASE ? x.o[g] : x.e[g];
    n[g] = PHASE ? odd_sites(x.e[g], g < 3 ? x.e[g + 1] : en) : x.o[g];
  }
  const auto plane = [&](uint32_t k) { return k == 0u ? y0 : sca_plane(heads, k, pl, ks); };
  if (FAST != kScaAny) {
    const uint32_t u0[4] = {y0.x, y0.y, y0.z, y0.w}, u1[4] = {y1.x, y1.y, y1.z, y1.w};
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const uint32_t v = swaps_fast<FAST>(f[g], u0[g], u1[g]);
      if (PHASE == 0) {
        x.e[g] = bitsel(v, n[g], f[g]);
        x.o[g] = bitsel(v, f[g], n[g]);
      } else {
        x.o[g] = bitsel(v, n[g], f[g]);
      }
      h[g] = (f[g] ^ n[g]) & v;
    }
  } else {
    if (MODEL == kTwoLane) {
      uint32_t cand[4];
#pragma unroll
      for (int g = 0; g < 4; ++g) cand[g] = P == 0 ? f[g] & ~n[g] : n[g] & ~f[g];
      decide_lane(cand, P == 0 ? r.p : r.q, plane, h);
    } else if (DIS) {
      constexpr int kq = (DIS && PQ) ? 1 : 0;  // the classes of left hops
      decide_any<true>(f, n, PHASE ? Q[0].o : Q[0].e, PHASE ? q_odd : Q[kq].o, r, rule, kmax, plane, h);
    } else {
      decide_any<false>(f, n, q_odd, q_odd, r, rule, kmax, plane, h);
    }
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      x.o[g] ^= h[g];
      if (PHASE == 0) x.e[g] ^= h[g];
    }
  }
  if (MODEL == kTwoLane) {
#pragma unroll
    for (int g = 0; g < 4; ++g) cnt.c[P] += __popc(h[g] & counted);
  } else if (COUNT) {
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      cnt.c[0] += __popc(h[g] & f[g] & counted);
      cnt.c[1] += __popc(h[g] & ~f[g] & counted);
    }
  }
}

// The phase's planes that do not depend on the lattice: the first (and for
// the two-plane kinds the second).
template <uint32_t MODEL, uint32_t FAST>
__device__ __forceinline__ void sca_first_planes(const uint4* heads, const PhiloxLane& pl, const KeySchedule& ks,
                                                 uint4& y0, uint4& y1) {
  y0 = sca_plane(heads, 0, pl, ks);
  y1 = (FAST != kScaAny && FAST != kScaHalves) ? sca_plane(heads, 1, pl, ks) : make_uint4(0u, 0u, 0u, 0u);
}

// ---------------------------------------------------------------------------
// Lane changes of the two-lane model
// ---------------------------------------------------------------------------

// Scratch of one warp: a queue of candidate sites and the accepted moves.
constexpr uint32_t kTurnQuota = 8;  // sites a lane queues per round
struct ScaTurnScratch {
  uint16_t queue[32 * kTurnQuota];
  uint32_t flip[32][8];  // [lane][e0..e3, o0..o3]; zero between uses
};

// STEP 0 moves A -> B, STEP 1 B -> A, at turning sites (m) whose source is
// occupied and target empty, with probability omega: one draw per candidate
// site (tag SCA_TURN, call STEP, word 3 = site / 4, word site mod 4).
// Candidates are sparse (a few of a unit's 256 sites), so the warp pools
// them: each lane queues its sites, the lanes then draw 32 queued sites at a
// time, and the accepted moves go back through shared memory.  (Each lane
// walking its own eight words runs every word to the warp's largest count:
// about 21 draws a step where the pool needs 4 at density 0.05.)
// Returns the moves of counted units drawn by this lane.  All 32 lanes call.
template <uint32_t STEP>
__device__ __forceinline__ uint32_t sca_turn_pool(ScaUnit& A, ScaUnit& B, const ScaUnit& m, ScaTurnScratch& sc,
                                                  uint32_t unit, uint32_t counted, uint32_t a0, uint32_t b2,
                                                  const uint4 head, const DomainLaunch& a) {
  const uint32_t lane = threadIdx.x & 31u;
  uint32_t cand[8];
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    cand[g] = m.e[g] & (STEP == 0 ? A.e[g] & ~B.e[g] : B.e[g] & ~A.e[g]);
    cand[4 + g] = m.o[g] & (STEP == 0 ? A.o[g] & ~B.o[g] : B.o[g] & ~A.o[g]);
  }
  uint32_t left = 0, moves = 0;
#pragma unroll
  for (int w = 0; w < 8; ++w) left += __popc(cand[w]);
  while (__any_sync(0xffffffffu, left != 0u)) {
    const uint32_t mine = min(left, kTurnQuota);
    uint32_t incl = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= static_cast<uint32_t>(d)) incl += t;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    uint32_t pos = incl - mine;
#pragma unroll
    for (uint32_t w = 0; w < 8; ++w) {
      while (cand[w] && pos < incl) {
        const uint32_t b = static_cast<uint32_t>(__ffs(static_cast<int>(cand[w]))) - 1u;
        cand[w] &= cand[w] - 1u;
        sc.queue[pos++] = static_cast<uint16_t>((lane << 8) | (w << 5) | b);
      }
    }
    left -= mine;
    __syncwarp();
    for (uint32_t base = 0; base < total; base += 32) {
      const uint32_t i = base + lane;
      const uint32_t q = i < total ? sc.queue[i] : 0u;
      const uint32_t src = q >> 8, w = (q >> 5) & 7u, b = q & 31u;
      const uint32_t src_unit = __shfl_sync(0xffffffffu, unit, src);
      const uint32_t src_counted = __shfl_sync(0xffffffffu, counted & 1u, src);
      // word 2g + (b & 1) of the unit, bit 2 (b / 2) + (odd site)
      const uint32_t site = 256u * src_unit + 32u * (2u * (w & 3u) + (b & 1u)) + (b & 30u) + (w >> 2);
      const PhiloxLane pl = philox_lane(a0, b2, site >> 2);
      const uint4 r = philox_tail(PhiloxHead{head.x, head.y, head.z}, pl, a.ks);
      if (i < total && accept(pick(r, site & 3u), a.rates.omega)) {
        atomicOr(&sc.flip[src][w], 1u << b);
        moves += src_counted;
      }
    }
    __syncwarp();
  }
  uint32_t f[8];
  load8(sc.flip[lane], f);
  const uint32_t zero[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
  store8(sc.flip[lane], zero);
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    A.e[g] ^= f[g];
    B.e[g] ^= f[g];
    A.o[g] ^= f[4 + g];
    B.o[g] ^= f[4 + g];
  }
  __syncwarp();
  return moves;
}

// Crossing kind: every site is a candidate where source is occupied and target
// empty (mk: the marked sites of this direction, probability omega_slow).
// With a quarter of all sites candidates a lane takes its 64 site groups in
// turn, one call for four sites.
template <uint32_t STEP>
__device__ __forceinline__ uint32_t sca_turn_all(ScaUnit& A, ScaUnit& B, const ScaUnit& mk, uint32_t unit, bool counted,
                                                 uint32_t a0, uint32_t b2, const uint4 head, const DomainLaunch& a) {
  uint32_t moves = 0;
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    const uint32_t ce = STEP == 0 ? A.e[g] & ~B.e[g] : B.e[g] & ~A.e[g];
    const uint32_t co = STEP == 0 ? A.o[g] & ~B.o[g] : B.o[g] & ~A.o[g];
    uint32_t fe = 0u, fo = 0u;
#pragma unroll 1
    for (uint32_t i = 0; i < 16; ++i) {  // word 2g + (i & 1), sites 4 (i / 2) .. + 3
      const uint32_t b = 4u * (i >> 1) + (i & 1u);  // lanes b and b + 2 of e and o
      if (!__any_sync(0xffffffffu, ((ce | co) & (5u << b)) != 0u)) continue;
      const uint32_t n = 64u * unit + 8u * (2u * g + (i & 1u)) + (i >> 1);
      const PhiloxLane pl = philox_lane(a0, b2, n);
      const uint4 r = philox_tail(PhiloxHead{head.x, head.y, head.z}, pl, a.ks);
      const uint32_t om = a.rates.omega, os = a.rates.omega_slow;
      const uint32_t b1 = 1u << b, b3 = 4u << b;
      if ((ce & b1) && accept(r.x, (mk.e[g] & b1) ? os : om)) fe |= b1;
      if ((co & b1) && accept(r.y, (mk.o[g] & b1) ? os : om)) fo |= b1;
      if ((ce & b3) && accept(r.z, (mk.e[g] & b3) ? os : om)) fe |= b3;
      if ((co & b3) && accept(r.w, (mk.o[g] & b3) ? os : om)) fo |= b3;
    }
    if (counted) moves += __popc(fe) + __popc(fo);
    A.e[g] ^= fe;
    B.e[g] ^= fe;
    A.o[g] ^= fo;
    B.o[g] ^= fo;
  }
  return moves;
}

}  // namespace
}  // namespace asep
