// asep_domain.cuh -- the attempt and the half-domain phase of the two-phase
// Poisson-domain schedule, shared by the resident/cluster kernels
// (asep_kernels.cu) and the streamed tier (asep_stream.cu).  A CTA holds
// columns of 2D/32 (+1 mirror) rows per plane in shared memory, column g =
// super-domain g of the sweep; see asep_kernels.cu for the layout.
#pragma once

#include <cstdint>

#include "asep_device.cuh"
#include "asep_internal.h"

namespace asep {
namespace {

// K = k_lo + #{ j : tab[j] <= w } (table ascending): inversion of the
// Poisson CDF in u32 fixed point.
__device__ __forceinline__ uint32_t poisson_count(const uint32_t* tab, uint32_t n, uint32_t klo, uint32_t w) {
  uint32_t lo = 0, hi = n;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (tab[mid] <= w) lo = mid + 1;
    else hi = mid;
  }
  return klo + lo;
}

// The attempts' accesses to shared memory, by 32-bit address.  They keep their
// order among themselves; attempts_fence keeps the ordinary accesses before
// and after a phase's attempts on their sides.
// The stores of a hop are predicated explicitly: as a C++ condition they
// became a branch around them, which ended the basic block at every attempt,
// so nothing of the next Philox call could run in the shadow of an attempt's
// load, test and store.  us per sweep with the branch and without: 8 rings of
// 4096 41.0 -> 32.2, 256 rings of 2^16 with bimodal disorder 53.9 -> 44.4, 128
// pairs of lanes of 2^16 51.7 -> 47.3, 256 rings of 2^17 52.4 -> 47.0, 16
// streamed rings of 2^24 431 -> 415 (all with the shared rounds below, which
// alone gave 1 % at most).
__device__ __forceinline__ void attempts_fence() { asm volatile("" ::: "memory"); }
__device__ __forceinline__ uint32_t lds(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ void sts_if(bool p, uint32_t addr0, uint32_t v0, uint32_t addr1, uint32_t v1) {
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "setp.ne.u32 p, %4, 0;\n"
      "@p st.shared.u32 [%0], %1;\n"
      "@p st.shared.u32 [%2], %3;\n"
      "}\n" ::"r"(addr0), "r"(v0), "r"(addr1), "r"(v1), "r"(static_cast<uint32_t>(p)));
}

struct Cnt {
  uint32_t a = 0, b = 0, c = 0, d = 0;  // ring: right, left; two lanes: A hops, B hops, A->B, B->A
};

template <bool B>
struct Flag {
  static constexpr bool value = B;
};

// Plane p of the columns holds the sites' complement where this is all ones
// (see attempt).
__device__ __forceinline__ uint32_t plane_inverse(const DomainLaunch& a, uint32_t p) { return p == 0 ? a.inverse : 0u; }

struct Lane {
  uint32_t c;        // column in the CTA
  uint32_t g;        // super-domain index within the sample
  uint32_t col0;     // first column of the sample
  uint32_t c_next;   // column of super-domain g+1 (ring)
  uint32_t c_prev;   // column of super-domain g-1 (ring)
  uint32_t sample;   // sample index in the context
  uint32_t n_glob;   // global sample id (Philox counter)
  bool active;
};

// One attempt of a half-domain phase, without branches (base: 32-bit shared
// address of the lane's column in the half's first row).  The bond's two words
// are rows `row` and `row + 1` of the column (row 2D/32 is the mirror of the
// next column's row 0), both loaded unconditionally; the 64-bit flip mask
// (3 << j across the word pair) is applied under one predicate.  `valid` is
// k <= K.
//
// The hop test takes one key: bits 31 and 30 hold sites i+1 and i (the
// funnel-shifted word pair), bits 29..0 hold r >> 2.  Sites 01 (key bits 10)
// are accepted iff the key, read as signed, lies below INT_MIN + t/4
// (hop_bound: INT_MIN + t/4, INT_MIN + 2^30 for "always", INT_MIN for 0).
// Thresholds are multiples of 4096, for which r < t iff r >> 2 < t >> 2, so
// the test equals u < t of the definition; the other patterns fall outside
// the window.  Pattern 10 is brought into it by adding 2^30 to the key or,
// where every hop of a plane goes the same way, by keeping the plane's
// complement in shared memory: lane A of two lanes, and rings without left
// hops (LEFT = false), so that one compare does (plane_inverse).  us per sweep
// before and after: 8 rings of 4096 at q = 0 32.2 -> 26.5, 256 bimodal rings of
// 2^16 44.4 -> 36.4 (one class word instead of two, no selects), 128 pairs of
// lanes of 2^16 47.3 -> 41.8 (with the pooled lane changes).
//   left hops:  sites 01, bound of q_{i+1};   right hops: sites 10, p_i.
template <uint32_t MODEL, uint32_t DIS, bool COUNT, uint32_t CP, bool LEFT>
__device__ __forceinline__ void attempt(uint32_t base, const DomainLaunch& a, uint32_t PWb, uint32_t row_scale_b,
                                        uint32_t r, bool valid, Cnt& cnt) {
  const uint32_t cpb = CP ? CP * 4u : a.Cp * 4u;  // row pitch in bytes (compile-time when CP != 0)
  // row (j >> 5) of this half: (r & (D - 1) & ~31) * (4 Cp / 32)
  uint32_t p0 = base + (r & a.row_bits) * row_scale_b;
  uint32_t bR = static_cast<uint32_t>(a.rates.pb), bL = static_cast<uint32_t>(a.rates.qb);
  uint32_t laneB = 0;
  if (MODEL == kTwoLane) {
    laneB = (r >> a.logD) & 1u;  // lane A hops right only (p), lane B left only (q)
    p0 += laneB * PWb;
    bR += laneB * (bL - bR);
  }
  const uint32_t p1 = p0 + cpb;
  if (DIS == kDisBimodal || DIS == kDisBimodalPQ) {
    // the class bits select by multiplication: (slow - fast) is even
    const uint32_t dR = static_cast<uint32_t>(a.rates.pb_slow) - bR, dL = (static_cast<uint32_t>(a.rates.qb_slow) - bL) >> 1;
    const uint32_t c0 = lds(p0 + PWb);
    if (LEFT) {
      const uint32_t pc = __funnelshift_r(c0, lds(p1 + PWb), r);  // bit 0: class of site i, bit 1: of site i+1
      uint32_t qc = pc;
      if (DIS == kDisBimodalPQ)  // left hops take the class of site i+1 from the second quenched plane
        qc = __funnelshift_r(lds(p0 + 2u * PWb), lds(p1 + 2u * PWb), r);
      bR += (pc & 1u) * dR;
      bL += (qc & 2u) * dL;
    } else {
      bR += (__funnelshift_r(c0, c0, r) & 1u) * dR;
    }
  }
  const uint32_t w0 = lds(p0);
  const uint32_t w1 = lds(p1);
  const uint32_t key = __funnelshift_l(r, __funnelshift_r(w0, w1, r), 30);
  bool hop, left = false;
  if (MODEL == kTwoLane || !LEFT) {
    hop = static_cast<int32_t>(key) < static_cast<int32_t>(bR);
  } else {
    left = static_cast<int32_t>(key) < static_cast<int32_t>(bL);
    hop = static_cast<int32_t>(key + 0x40000000u) < static_cast<int32_t>(bR) || left;
  }
  hop = hop && valid;
  sts_if(hop, p0, w0 ^ __funnelshift_l(0u, 3u, r),  // 3 << (j mod 32), truncated
         p1, w1 ^ __funnelshift_l(3u, 0u, r));      // 1 when j mod 32 == 31, else 0
  if (COUNT) {  // a: all hops, b: left hops (lane B)
    cnt.a += hop;
    if (MODEL == kTwoLane) cnt.b += hop ? laneB : 0u;
    else if (LEFT) cnt.b += hop && left;
  }
}

// The draws of one domain at one sweep: call c of the attempt stream (tag DOM,
// counter (s, tag | c << 12, sample, domain)) with the rounds that lanes or
// calls share taken out (asep_device.cuh).  With a table of heads (one entry
// per call, shared by all domains of the sample and both phases) a call costs
// a lane 14 wide multiplies and one broadcast load, without one 16, instead of
// 20.
template <bool TABLE>
struct DomainStream {
  const uint4* heads;  // shared memory, entry c = call c (TABLE); else the head of every call is formed
  PhiloxLane lane;
  uint32_t h1, e1;     // without a table: round 1 of word 2 (without the call), round 2's XOR of word 2

  // table: whether the heads come from `h`; s: sweep; n: sample id; d: domain.
  __device__ __forceinline__ void open(const uint4* h, uint64_t s, uint32_t n, uint32_t d, const KeySchedule& ks) {
    const uint2 p0 = mul_wide(0xD2511F53u, static_cast<uint32_t>(s)), p1 = mul_wide(0xCD9E8D57u, n);
    heads = h;
    lane = philox_lane(p0.y ^ ks.y[0], p1.x ^ ks.x[1], d);
    h1 = p1.y ^ ks.x[0] ^ ctr_of(s, kTagDom, 0, 0, 0).y;
    e1 = p0.x ^ ks.y[1];
  }
  __device__ __forceinline__ uint4 draw(uint32_t call, const KeySchedule& ks) const {
    PhiloxHead h;
    if (TABLE) {
      const uint4 v = heads[call];
      h = PhiloxHead{v.x, v.y, v.z};
    } else {
      const uint2 q = mul_wide(0xD2511F53u, h1 ^ (call << 12));
      const uint2 r = mul_wide(0xCD9E8D57u, q.y ^ e1);
      h = PhiloxHead{r.y ^ ks.x[2], r.x, q.x ^ ks.y[2]};
    }
    return philox_tail(h, lane, ks);
  }
};

// Entry `call` of the table of sample id n at sweep s.
__device__ __forceinline__ uint4 domain_head(uint64_t s, uint32_t call, uint32_t n, const KeySchedule& ks) {
  const PhiloxHead h = philox_head(static_cast<uint32_t>(s), ctr_of(s, kTagDom, call, 0, 0).y, n, ks);
  return make_uint4(h.c3, h.y3, h.d3, 0u);
}

// Calls whose four attempts every lane of the warp makes (k + 3 <= Kmin) need
// no per-attempt count test; the remaining calls up to Kmax test k <= K.  A
// domain's attempts keep their order either way.  The fast calls are
// 1 .. (Kmin - 3) / 4.  Each iteration draws the next call's words before it
// applies the current call's four attempts (the random stream does not
// depend on the lattice), so Philox's rounds overlap the attempts' dependent
// chain; two iterations per loop trip.
template <uint32_t MODEL, uint32_t DIS, bool COUNT, uint32_t CP, bool TABLE, bool LEFT>
__device__ __forceinline__ void run_calls(uint32_t base, const uint4* heads, const DomainLaunch& a, uint32_t PWb,
                                          uint32_t row_scale_b, uint64_t s, uint32_t n_glob, uint32_t dd,
                                          const uint4 x0, uint32_t K, uint32_t Kmin, uint32_t Kmax, Cnt& cnt) {
  const auto go = [&](uint32_t r, bool valid) {
    attempt<MODEL, DIS, COUNT, CP, LEFT>(base, a, PWb, row_scale_b, r, valid, cnt);
  };
  go(x0.y, 1 <= K);
  go(x0.z, 2 <= K);
  go(x0.w, 3 <= K);
  DomainStream<TABLE> ds;
  ds.open(heads, s, n_glob, dd, a.ks);
  const uint32_t n_fast = Kmin >= 3u ? (Kmin - 3u) >> 2 : 0u;
  uint32_t call = 1;
  uint4 y = ds.draw(1, a.ks);  // call n_fast + 1's words when the fast loop ends
#pragma unroll 2
  for (; call <= n_fast;) {
    ++call;
    const uint4 yn = ds.draw(call, a.ks);  // the next call, ahead of this call's attempts
    go(y.x, true);
    go(y.y, true);
    go(y.z, true);
    go(y.w, true);
    y = yn;
  }
#pragma unroll 1
  for (; (call << 2) <= Kmax; ++call) {
    const uint32_t k = call << 2;
    uint4 yn = y;
    if (k + 4 <= Kmax) yn = ds.draw(call + 1, a.ks);  // warp-uniform
    go(y.x, k <= K);
    go(y.y, k + 1 <= K);
    go(y.z, k + 2 <= K);
    go(y.w, k + 3 <= K);
    y = yn;
  }
}

// A phase's view of its descriptor.  As a kernel parameter it lies in the
// constant bank, whose words an instruction reads as operands.  A batch's CTA
// holds it in shared memory, from where every Philox call loaded its 14 round
// keys and the rates again; pinned, these are values of registers that the
// compiler cannot load anew.  us per sweep of a batch of one context, of eight
// rings of 4096, without and with: q = 0 38.5 -> 28.4, bimodal 48.7 -> 31.6, 39
// pairs of lanes of 3840 with turning sites 54.6 -> 45.2.  Only in the class of
// up to 512 threads: at 64 registers a thread they do not fit.
template <bool PIN>
struct HotFields {
  const DomainLaunch& a;
  __device__ __forceinline__ explicit HotFields(const DomainLaunch& d) : a(d) {}
};
__device__ __forceinline__ void pin(uint32_t& v) { asm volatile("" : "+r"(v)); }
__device__ __forceinline__ void pin(int32_t& v) { asm volatile("" : "+r"(v)); }
template <>
struct HotFields<true> {
  DomainLaunch a;
  __device__ __forceinline__ explicit HotFields(const DomainLaunch& d) : a(d) {
#pragma unroll
    for (int r = 2; r < 10; ++r) {
      pin(a.ks.x[r]);
      pin(a.ks.y[r]);
    }
    pin(a.rates.pb);
    pin(a.rates.qb);
    pin(a.rates.pb_slow);
    pin(a.rates.qb_slow);
    pin(a.row_bits);
    pin(a.logD);
    pin(a.Cp);
  }
};

// One half-domain phase of one sweep.  All threads of the block must call.
//
// Lane sort: the lanes of a warp run to the largest Poisson count of the
// warp, so a warp whose domains drew similar counts wastes fewer slots.  With
// `a.lane_sort` (every warp inside one sample, and a scratch area of 5 words
// per column) each thread ranks its domain's count among the domains of the
// same shared-memory bank in its sample (columns lane, lane + 32, ...) and
// warp w runs the domains of rank w.  A domain's attempts are the same
// whichever thread runs them, and a thread stays in its own sample and bank,
// so results and bank mapping are unchanged; only the slots a warp wastes
// shrink.  G, C: the columns of the thread's sample and of the group (a
// streamed tile: both its own).  `scr` is the idle realign buffer (overwritten
// by the next realign) or the streamed tier's staged words.  The cluster tier
// passes sort = false: there other CTAs may still read that buffer remotely
// during the first phase.
//
// heads: the sample's table of heads, or nullptr.  fill: the table is formed
// here (the first phase of a sweep), in the idle buffer behind the sort's
// scratch, by the sample's threads.
template <uint32_t MODEL, uint32_t DIS, bool COUNT, uint32_t CP, uint32_t PHASE, bool TABLE, bool PIN = false>
__device__ __forceinline__ void run_phase(uint32_t* cur, uint32_t* scr, bool sort, uint4* heads, bool fill,
                                          const DomainLaunch& desc, const uint32_t* tab, uint32_t PW, uint64_t s,
                                          const Lane& ln, Cnt& cnt, uint32_t G, uint32_t C) {
  HotFields<PIN> hot(desc);
  const DomainLaunch& a = hot.a;
  const uint32_t d = 2 * ln.g + PHASE;
  uint4 x0 = make_uint4(0u, 0u, 0u, 0u);
  uint32_t K = 0;
  DomainStream<false> ds;
  if (ln.active) {
    ds.open(nullptr, s, ln.n_glob, d, a.ks);
    x0 = ds.draw(0, a.ks);
    K = poisson_count(tab, a.ptab_n, a.ptab_klo, x0.x);
  }
  if (fill && ln.c < C)
    for (uint32_t c = ln.g; c < a.heads; c += G) heads[c] = domain_head(s, c, ln.n_glob, a.ks);
  if (fill && !sort) __syncthreads();
  const uint32_t cp = CP ? CP : a.Cp;
  uint32_t col = ln.c;  // the column (domain pair) this thread runs
  uint32_t dd = d;      // its domain index in the sample
  if (sort) {
    // Only the group's own columns (c < C) take part: a persistent CTA may be
    // wider than the group, and its extra threads keep K = 0 and no column.
    const bool in_group = ln.c < C;
    uint32_t* sK = scr;
    uint32_t* sPerm = scr + cp;
    uint32_t* sX = scr + 2 * cp;
    if (in_group) {
      sK[ln.c] = K;
      sX[ln.c] = x0.y;
      sX[cp + ln.c] = x0.z;
      sX[2 * cp + ln.c] = x0.w;
    }
    __syncthreads();
    if (in_group) {
      const uint32_t lane = ln.c & 31u;
      uint32_t rank = 0;
      for (uint32_t q = ln.col0 + lane; q < ln.col0 + G; q += 32) {
        const uint32_t kq = sK[q];
        rank += (kq < K || (kq == K && q < ln.c)) ? 1u : 0u;
      }
      sPerm[ln.col0 + (rank << 5) + lane] = ln.c;
    }
    __syncthreads();
    if (in_group) {
      col = sPerm[ln.c];
      dd = 2 * (ln.g - ln.c + col) + PHASE;
      K = sK[col];
      x0.y = sX[col];
      x0.z = sX[cp + col];
      x0.w = sX[2 * cp + col];
    }
  }
  const uint32_t Kmax = __reduce_max_sync(0xffffffffu, K);
  const uint32_t Kmin = __reduce_min_sync(0xffffffffu, K);
  if (Kmax == 0u) return;  // a warp without columns
  const uint32_t base = static_cast<uint32_t>(__cvta_generic_to_shared(cur)) + (PHASE * (a.D >> 5) * cp + col) * 4u;
  const uint32_t row_scale_b = cp >> 3;  // 4 * Cp / 32
  const uint32_t PWb = PW * 4u;
  Cnt hops;
  const auto calls = [&](auto table, auto left) {
    run_calls<MODEL, DIS, COUNT, CP, decltype(table)::value, decltype(left)::value>(
        base, heads, a, PWb, row_scale_b, s, ln.n_glob, dd, x0, K, Kmin, Kmax, hops);
  };
  constexpr bool kLeft = MODEL == kRing;  // both directions on a plane are possible
  using No = Flag<false>;
  attempts_fence();
  if (TABLE && heads) {
    if (kLeft && a.left) calls(Flag<TABLE>{}, Flag<kLeft>{});
    else calls(Flag<TABLE>{}, No{});
  } else {
    if (kLeft && a.left) calls(No{}, Flag<kLeft>{});
    else calls(No{}, No{});
  }
  attempts_fence();
  cnt.a += hops.a - hops.b;
  cnt.b += hops.b;
}

}  // namespace
}  // namespace asep
