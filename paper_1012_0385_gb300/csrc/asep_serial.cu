// asep_serial.cu -- plain random-sequential update (paper sec. 2.1), exact:
// the serial schedule of the library, one CTA or one warp per sample.
//
// The attempts of a run form one sequence (sweep by sweep, each sweep's
// attempts in order).  Two attempts commute when their bonds share no site, so
// any order that keeps every pair of site-sharing attempts in sequence order
// gives the sequential lattice.  Both kernels keep a window of the earliest
// attempts not yet done, one per thread, and go in rounds:
//   refill   threads whose attempt is done take the next ones of the
//            sequence, so the window always holds every attempt before the
//            next one to be taken, except those done;
//   post     every attempt leaves the key (round << 16) | (0xFFFF - position)
//            on both its sites with an atomic max, so each site ends up
//            holding its earliest attempt of the window;
//   check    an attempt whose key survived on both its sites runs: every
//            earlier attempt that shares a site with it is done.  Attempts that
//            run in one round share no site; their flips, possibly in one word,
//            are atomic XORs of disjoint bits.
// The earliest attempt always runs, so every round makes progress.  Positions
// count from the start of a segment of at most 2^16 attempts, at whose end the
// window drains (as before records and lane changes); keys of earlier rounds
// are smaller, so the site table is cleared only when the round count wraps.
//
// How large the window should be: with n attempts in it on L sites a round runs
// n less those that wait, and a wait costs its attempt another visit (n = L/8:
// 1.27 visits an attempt, 10 rounds a sweep of 4096; n = L/4: 1.7 and 6.8).
#include <algorithm>
#include <cstdint>

#include "asep_device.cuh"
#include "asep_internal.h"
#include "asep_serial.h"

namespace asep {
namespace {

constexpr uint32_t kPerLane = 2;           // attempts a lane of the one-warp kernel holds
constexpr uint32_t kSerialWindow = 512;    // attempts in the one-CTA kernel's window, at most
// Ring entries of the one-CTA kernel.
__host__ __device__ constexpr uint32_t serial_ring(uint32_t threads) {
  return threads / 2u >= kSerialWindow ? 4u * kSerialWindow : (threads >= 128u ? 2u * threads : 256u);
}

constexpr uint32_t kSegment = 1u << 16;  // attempts between drains
constexpr uint32_t kLastRound = 0xFFFFu;

// The draws of the serial stream of one sample: call `pair` of sweep s (tag
// SER, word 3 = attempt / 2) gives attempts 2 pair and 2 pair + 1 as (bond,
// acceptance) word pairs.  What neither the sweep's low word nor the pair
// changes is kept.
struct SerialStream {
  uint32_t b2, hq, lq;  // round 2 of word 2 (XOR); round 2 of word 0: high and low product
  __device__ __forceinline__ void open(uint64_t s, uint32_t n, const KeySchedule& ks) {
    const uint2 q = mul_wide(0xD2511F53u, mul_wide(0xCD9E8D57u, n).y ^ ctr_of(s, kTagSer, 0, 0, 0).y ^ ks.x[0]);
    b2 = philox_b2(n, ks);
    hq = q.y ^ ks.y[1];
    lq = q.x ^ ks.y[2];
  }
  __device__ __forceinline__ uint4 draw(uint32_t s, uint32_t pair, const KeySchedule& ks) const {
    const uint2 p = mul_wide(0xD2511F53u, s);
    const uint2 r = mul_wide(0xCD9E8D57u, hq ^ p.x);
    return philox_tail(PhiloxHead{r.y ^ ks.x[2], r.x, lq}, philox_lane(p.y ^ ks.y[0], b2, pair), ks);
  }
};

// The lattice of one sample: planes of W words in shared or global memory, A
// and then (two lanes) B; M: quenched planes; a_s, m_s: their shared addresses.
struct SerialLattice {
  uint32_t* A;
  const uint32_t* M;
  uint32_t W, L, logL;
  uint32_t a_s, m_s;
};

// Shared memory by 32-bit address, with predicated reductions: a round is a
// chain of a few dependent steps, and branches around them cost as much again.
__device__ __forceinline__ uint32_t shared_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ uint32_t lds(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ uint2 lds2(uint32_t addr) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void red_max(uint32_t addr, uint32_t v) {
  asm volatile("red.shared.max.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void red_xor_if(bool p, uint32_t addr, uint32_t v) {
  asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %2, 0;\n@p red.shared.xor.b32 [%0], %1;\n}\n" ::"r"(addr), "r"(v),
               "r"(static_cast<uint32_t>(p))
               : "memory");
}
// Word st / 32 of the lattice (M: of the quenched planes); in global memory past
// L1, since other threads flip other bits of it.
template <bool SMEM>
__device__ __forceinline__ uint32_t word_of(const SerialLattice& lt, uint32_t st) {
  return SMEM ? lds(lt.a_s + ((st >> 3) & ~3u)) : *static_cast<const volatile uint32_t*>(lt.A + (st >> 5));
}
template <bool SMEM>
__device__ __forceinline__ uint32_t class_of(const SerialLattice& lt, uint32_t plane, uint32_t st) {
  const uint32_t w = SMEM ? lds(lt.m_s + 4u * plane * lt.W + ((st >> 3) & ~3u)) : lt.M[plane * lt.W + (st >> 5)];
  return __funnelshift_r(w, w, st) & 1u;
}
template <bool SMEM>
__device__ __forceinline__ void flip_if(bool p, const SerialLattice& lt, uint32_t st, uint32_t v) {
  if (SMEM) red_xor_if(p, lt.a_s + ((st >> 3) & ~3u), v);
  else if (p) atomicXor(lt.A + (st >> 5), v);
}

// The second site of the bond at site st (planes follow one another).
template <uint32_t MODEL>
__device__ __forceinline__ uint32_t next_site(uint32_t st, uint32_t L) {
  return MODEL == kTwoLane ? (st & ~(L - 1u)) | ((st + 1u) & (L - 1u)) : (st + 1u) & (L - 1u);
}

// Runs the attempt at bond (st, st1) with acceptance draw u; c: hop counters.
// The hop test is the domain schedule's: bits 31 and 30 of the key hold sites
// i+1 and i, the rest u >> 2, and a key below the bound (hop_bound) is a left
// hop (sites 01), plus 2^30 a right hop (sites 10).
// go: whether it runs at all (the sites are valid either way).
template <uint32_t MODEL, uint32_t DIS, bool SMEM>
__device__ __forceinline__ void serial_attempt(const SerialLattice& lt, uint32_t st, uint32_t st1, uint32_t u, bool go,
                                               const SerialLaunch& a, uint32_t (&c)[4]) {
  const uint32_t w0 = word_of<SMEM>(lt, st), w1 = word_of<SMEM>(lt, st1);
  const uint32_t key = __funnelshift_l(u, __funnelshift_r(w0, w1, st), 30);
  int32_t bR = a.rates.pb, bL = a.rates.qb;
  bool hop, second;  // second: counted as a left hop (two lanes: a hop in lane B)
  if (MODEL == kTwoLane) {
    second = st >> lt.logL;
    hop = static_cast<int32_t>(second ? key : key + 0x40000000u) < (second ? bL : bR);
  } else {
    if (DIS == kDisBimodal || DIS == kDisBimodalPQ) {  // left hops take the second plane's classes (PQ)
      bR = class_of<SMEM>(lt, 0, st) ? a.rates.pb_slow : bR;
      bL = class_of<SMEM>(lt, DIS == kDisBimodalPQ ? 1 : 0, st1) ? a.rates.qb_slow : bL;
    }
    second = static_cast<int32_t>(key) < bL;
    hop = second || static_cast<int32_t>(key + 0x40000000u) < bR;
  }
  hop = hop && go;
  flip_if<SMEM>(hop, lt, st, __funnelshift_l(0u, 3u, st));  // 3 << (st mod 32), truncated
  flip_if<SMEM>(hop && (st & 31u) == 31u, lt, st1, 1u);
  if (MODEL == kTwoLane || a.count_hops) {
    c[0] += hop && !second;
    c[1] += hop && second;
  }
}

// Lane changes at sweep s (every event touches only (A_i, B_i)), words split
// over n threads.  Crossing kind: every site, u_i (plane 0) for a particle in
// lane A, v_i (plane 1) for one in lane B.
template <uint32_t DIS>
__device__ __forceinline__ void serial_turns(const SerialLattice& lt, const SerialLaunch& a, uint64_t s,
                                             uint32_t n_glob, uint32_t tid, uint32_t n, uint32_t (&c)[4]) {
  uint32_t* A = lt.A;
  uint32_t* B = lt.A + lt.W;
  const uint32_t* M = lt.M;
  for (uint32_t w = tid; w < lt.W; w += n) {
    uint32_t e = (DIS == kDisCrossing ? ~0u : M[w]) & (A[w] ^ B[w]);
    while (e) {
      const uint32_t bit = __ffs(e) - 1;
      e &= e - 1;
      const uint32_t site = 32u * w + bit;
      const uint4 r = philox10(ctr_of(s, kTagTurn, 0, n_glob, site >> 2), a.ks);
      uint32_t thr = a.rates.omega;
      if (DIS == kDisCrossing) {
        const uint32_t marked = ((A[w] >> bit) & 1u) ? M[w] : M[lt.W + w];
        thr = ((marked >> bit) & 1u) ? a.rates.omega_slow : a.rates.omega;
      }
      if (accept(pick(r, site & 3u), thr)) {
        const bool from_a = A[w] & (1u << bit);
        c[2] += from_a;
        c[3] += !from_a;
        A[w] ^= 1u << bit;
        B[w] ^= 1u << bit;
      }
    }
  }
}

// A thread's part of a record of plane p: its words' heights from entry height
// h, profile and autocorrelation overlap.
__device__ __forceinline__ void serial_record_words(const uint32_t* pw, uint32_t w0, uint32_t w1, long long h,
                                                    const SerialLaunch& a, size_t pbase, uint64_t t, long long& s1,
                                                    unsigned long long& s2, long long& ov) {
  for (uint32_t w = w0; w < w1; ++w) {
    const uint32_t x = pw[w];
    add_word_heights(x, h, s1, s2);
    if (a.ex.profile) a.ex.profile[pbase + w] += __popc(x);
    if (a.ex.snap) {
      if (t == a.ex.t0) a.ex.snap[pbase + w] = x;
      if (t >= a.ex.t0) ov += __popc(x & a.ex.snap[pbase + w]);
    }
  }
}

// Sweeps from `it` on that run as one segment: up to the next drain.
template <uint32_t MODEL, uint32_t DIS>
__device__ __forceinline__ uint32_t segment_sweeps(const SerialLaunch& a, uint32_t it, uint64_t s0, uint32_t rec,
                                                   uint32_t n_att) {
  if (MODEL == kTwoLane && (DIS == kDisTurning || DIS == kDisCrossing)) return 1u;
  uint32_t n = min(a.n_sweeps - it, max(1u, kSegment / n_att));
  n = static_cast<uint32_t>(min(static_cast<uint64_t>(n), static_cast<uint64_t>((1ull << 32) - ((s0 + it) & 0xFFFFFFFFull))));  // SerialStream
  if (rec < a.n_times) n = static_cast<uint32_t>(min(static_cast<uint64_t>(n), a.times[rec] - (s0 + it)));
  return n;
}

// ---------------------------------------------------------------------------
// One warp per sample
// ---------------------------------------------------------------------------
//
// A window of 64, two attempts a lane.  The site table is hashed (site modulo its size): two sites that
// fall on one entry only make an attempt wait.  The draws of 64 attempts, a
// call per lane, go through a ring in shared memory.  Lattice and quenched
// planes are staged in shared memory when they fit.
// Measured against committing the conflict-free prefix of 32 attempts found
// with two match.any (whose unit the 13 warps of an SM shared at some 80 clocks
// an instruction), us per sweep: 2021 rings of 4096 157 -> 45, 512 rings of
// 2^17 1934 -> 887.  One attempt a lane 54, three or four 47.
constexpr uint32_t kHashMost = 2048, kHashLeast = 1024;  // entries of a warp's site table (a power of two)
constexpr uint32_t kWarpRing = 256;  // attempts drawn ahead: at most 63 + 64 beyond the taken ones
constexpr uint32_t serial_warp_scratch(uint32_t hash) { return 4u * hash + 8u * kWarpRing; }

template <uint32_t MODEL, uint32_t DIS, bool SMEM>
__global__ void __launch_bounds__(256) k_serial(const SerialLaunch a, uint32_t hash) {
  extern __shared__ __align__(16) uint32_t serial_smem[];
  const uint32_t lane = threadIdx.x & 31u, wib = threadIdx.x >> 5;
  const uint32_t sample = blockIdx.x * (blockDim.x >> 5) + wib;
  if (sample >= a.geo.S) return;  // whole warps leave together
  const uint32_t L = static_cast<uint32_t>(a.geo.L), W = a.geo.W;
  constexpr uint32_t NOCC = MODEL == kTwoLane ? 2u : 1u;
  constexpr uint32_t NQ = dis_planes(DIS);
  constexpr uint32_t NPL = NOCC + NQ;
  uint32_t* tab = serial_smem + wib * (serial_warp_scratch(hash) / 4u);
  uint2* ring = reinterpret_cast<uint2*>(tab + hash);
  const uint32_t tab_s = shared_addr(tab), ring_s = shared_addr(ring);
  uint32_t* gA = a.state + static_cast<size_t>(sample) * NOCC * W;
  const uint32_t* gM =
      (DIS != kDisNone) ? a.mask + static_cast<size_t>(sample / a.geo.samples_per_real) * NQ * W : nullptr;
  SerialLattice lt = {gA, gM, W, L, 31u - static_cast<uint32_t>(__clz(static_cast<int>(L))), 0u, 0u};
  if (SMEM) {
    uint32_t* mine = serial_smem + (blockDim.x >> 5) * (serial_warp_scratch(hash) / 4u) + static_cast<size_t>(wib) * NPL * W;
    for (uint32_t w = lane; w < NOCC * W; w += 32) mine[w] = gA[w];
    if (DIS != kDisNone)
      for (uint32_t w = lane; w < NQ * W; w += 32) mine[NOCC * W + w] = gM[w];
    lt.A = mine;
    lt.M = mine + NOCC * W;
    lt.a_s = shared_addr(lt.A);
    lt.m_s = shared_addr(lt.M);
  }
  for (uint32_t i = lane; i < hash; i += 32) tab[i] = 0u;
  __syncwarp();
  const uint32_t n_glob = a.geo.first_sample + sample;
  const uint32_t n_att = NOCC * L, log_att = lt.logL + NOCC - 1u;
  const uint64_t s0 = a.clock->sweep;
  uint32_t rec = a.clock->next_time;
  const uint32_t lt_mask = (1u << lane) - 1u;
  SerialStream stream;
  unsigned long long tot[4] = {0, 0, 0, 0};  // this lane's share of the sample's counters
  uint32_t round = 0;

  for (uint32_t it = 0; it < a.n_sweeps;) {
    const uint32_t n_sweeps = segment_sweeps<MODEL, DIS>(a, it, s0, rec, n_att);
    const uint32_t all = n_sweeps << log_att;  // attempts of these sweeps: at most 2^16, or one sweep's
    const uint32_t s_lo = static_cast<uint32_t>(s0 + it);
    stream.open(s0 + it, n_glob, a.ks);
    uint32_t c[4] = {0, 0, 0, 0};
    for (uint32_t q0 = 0; q0 < all; q0 += kSegment) {
      const uint32_t n = min(kSegment, all - q0);
      uint32_t taken = 0, drawn = 0;
      uint32_t st[kPerLane], u[kPerLane], order[kPerLane];
      bool pending[kPerLane];
#pragma unroll
      for (uint32_t j = 0; j < kPerLane; ++j) {
        st[j] = u[j] = order[j] = 0u;
        pending[j] = false;
      }
      for (;;) {
        while (drawn < n && drawn - taken < 32u * kPerLane) {  // the next 64 attempts' draws
          const uint32_t q = q0 + drawn + 2u * lane;
          const uint4 y = stream.draw(s_lo + (q >> log_att), (q & (n_att - 1u)) >> 1, a.ks);
          *reinterpret_cast<uint4*>(&ring[(drawn + 2u * lane) & (kWarpRing - 1u)]) =
              make_uint4(y.x & (n_att - 1u), y.y, y.z & (n_att - 1u), y.w);
          drawn += 64u;
          __syncwarp();
        }
        if (++round == kLastRound) {
          for (uint32_t i = lane; i < hash; i += 32) tab[i] = 0u;
          round = 1;
          __syncwarp();
        }
        bool idle = true;  // no attempt is left in the window
#pragma unroll
        for (uint32_t j = 0; j < kPerLane; ++j) {
          const uint32_t free = __ballot_sync(0xffffffffu, !pending[j]);
          const uint32_t pos = taken + __popc(free & lt_mask);
          idle = idle && free == 0xffffffffu && taken == n;
          const uint2 e = lds2(ring_s + 8u * (pos & (kWarpRing - 1u)));
          const bool take = !pending[j] && pos < n;
          st[j] = take ? e.x : st[j];
          u[j] = take ? e.y : u[j];
          order[j] = take ? 0xFFFFu - pos : order[j];
          pending[j] = pending[j] || take;
          taken = min(n, taken + __popc(free));
        }
        if (idle) break;
        uint32_t st1[kPerLane], t0[kPerLane], t1[kPerLane], key[kPerLane];
#pragma unroll
        for (uint32_t j = 0; j < kPerLane; ++j) {
          st1[j] = next_site<MODEL>(st[j], L);
          t0[j] = tab_s + 4u * (st[j] & (hash - 1u));
          t1[j] = tab_s + 4u * (st1[j] & (hash - 1u));
          key[j] = pending[j] ? (round << 16) | order[j] : 0u;  // 0 changes nothing
          red_max(t0[j], key[j]);
          red_max(t1[j], key[j]);
        }
        __syncwarp();
        bool go[kPerLane];
#pragma unroll
        for (uint32_t j = 0; j < kPerLane; ++j) go[j] = lds(t0[j]) == key[j] && lds(t1[j]) == key[j] && pending[j];
#pragma unroll
        for (uint32_t j = 0; j < kPerLane; ++j) {
          serial_attempt<MODEL, DIS, SMEM>(lt, st[j], st1[j], u[j], go[j], a, c);
          pending[j] = pending[j] && !go[j];
        }
        __syncwarp();
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        tot[k] += c[k];
        c[k] = 0;
      }
    }
    it += n_sweeps;
    const uint64_t s = s0 + it;  // sweeps done
    if (MODEL == kTwoLane && (DIS == kDisTurning || DIS == kDisCrossing)) {
      serial_turns<DIS>(lt, a, s - 1u, n_glob, lane, 32u, c);
#pragma unroll
      for (int k = 0; k < 4; ++k) tot[k] += c[k];
      __syncwarp();
    }
    if (rec < a.n_times && a.times[rec] == s) {
      const uint32_t chunk = (W + 31u) / 32u;
      const uint32_t w0 = min(W, lane * chunk), w1 = min(W, w0 + chunk);
      for (uint32_t p = 0; p < NOCC; ++p) {
        const uint32_t* pw = lt.A + p * W;
        long long rise = 0;
        for (uint32_t w = w0; w < w1; ++w) rise += 2 * __popc(pw[w]) - 32;
        long long h = rise;  // inclusive warp scan of the chunks
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const long long t = __shfl_up_sync(0xffffffffu, h, o);
          if (lane >= static_cast<uint32_t>(o)) h += t;
        }
        long long s1 = 0, ov = 0;
        unsigned long long s2 = 0;
        serial_record_words(pw, w0, w1, h - rise, a, (static_cast<size_t>(sample) * NOCC + p) * W, s, s1, s2, ov);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          s1 += __shfl_xor_sync(0xffffffffu, s1, o);
          ov += __shfl_xor_sync(0xffffffffu, ov, o);
        }
        unsigned __int128 s2_all = 0;
        for (int l = 0; l < 32; ++l) s2_all += __shfl_sync(0xffffffffu, s2, l);
        if (lane == 0) {
          const size_t e = (static_cast<size_t>(rec) * a.geo.S + sample) * NOCC + p;
          a.tab_sh[e] = s1;
          a.tab_sh2[2 * e] = static_cast<uint64_t>(s2_all);
          a.tab_sh2[2 * e + 1] = static_cast<uint64_t>(s2_all >> 64);
          if (a.ex.snap) a.ex.tab_ac[e] = ov;
        }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        unsigned long long v = tot[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0)
          a.ex.tab_cnt[(static_cast<size_t>(rec) * a.geo.S + sample) * 4 + k] =
              static_cast<int64_t>(a.counters[4ull * sample + k] + v);
      }
      __syncwarp();
      ++rec;
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    unsigned long long v = tot[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) a.counters[4ull * sample + k] += v;
  }
  if (SMEM) {
    __syncwarp();
    for (uint32_t w = lane; w < NOCC * W; w += 32) gA[w] = lt.A[w];
  }
}

// ---------------------------------------------------------------------------
// One CTA per sample
// ---------------------------------------------------------------------------
//
// Up to 512 threads hold the window, half as many draw ahead into a ring (the
// others of the CTA wait for the segment's end: more warps only add issue to a
// round).  One barrier a round: the site table alternates between two, so the next round's
// keys leave the ones still being checked alone.  A window thread reads its
// ring entry in the round it takes it, and the drawing warps stay within two
// windows and 64 entries of the taken count, so a ring of four windows is
// never overwritten early: what they overwrite was taken before the last
// barrier.
// Bound by the instructions of a round (some 75 a window warp, six warps a
// scheduler) and its chain of shared-memory steps: some 950 clocks.  Measured
// against rounds over a whole sweep, whose attempts were visited 2.5 times at
// two barriers a round, us per sweep of 8 rings of 4096: 14.7 -> 4.85 (a window
// of 256 6.9, of 512 in two attempts a thread 6.6).

// Sums over the block (all threads call): a signed 64-bit value and an
// unsigned 64-bit value summed exactly in 128 bits.  Results valid in thread 0.
__device__ long long block_sum_i64(long long v, long long* red) {
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) red[wid] = v;
  __syncthreads();
  long long t = 0;
  if (threadIdx.x == 0)
    for (uint32_t w = 0; w < nw; ++w) t += red[w];
  __syncthreads();
  return t;
}

__device__ unsigned __int128 block_sum_u128(unsigned long long v, unsigned long long* red) {
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  unsigned __int128 w = 0;
  for (int l = 0; l < 32; ++l) w += __shfl_sync(0xffffffffu, v, l);
  if (lane == 0) {
    red[2 * wid] = static_cast<unsigned long long>(w);
    red[2 * wid + 1] = static_cast<unsigned long long>(w >> 64);
  }
  __syncthreads();
  unsigned __int128 t = 0;
  if (threadIdx.x == 0)
    for (uint32_t k = 0; k < nw; ++k)
      t += (static_cast<unsigned __int128>(red[2 * k + 1]) << 64) | red[2 * k];
  __syncthreads();
  return t;
}

// Barrier of the whole CTA from code that differs between its warps; true when
// `v` is set in any thread.
__device__ __forceinline__ bool cta_any(bool v, uint32_t threads) {
  uint32_t r;
  asm volatile(
      "{\n"
      ".reg .pred p, q;\n"
      "setp.ne.u32 p, %1, 0;\n"
      "bar.red.or.pred q, 1, %2, p;\n"
      "selp.u32 %0, 1, 0, q;\n"
      "}\n"
      : "=r"(r)
      : "r"(static_cast<uint32_t>(v)), "r"(threads)
      : "memory");
  return r != 0u;
}

template <uint32_t MODEL, uint32_t DIS>
__global__ void __launch_bounds__(1024) k_serial_rounds(const SerialLaunch a) {
  extern __shared__ __align__(16) uint32_t serial_smem[];
  __shared__ long long s_i64[32];
  __shared__ unsigned long long s_u64[64];
  __shared__ uint32_t s_taken;
  const uint32_t sample = blockIdx.x;
  const uint32_t tid = threadIdx.x, all = blockDim.x, lane = tid & 31u;
  // window threads (a power of two), those and the drawing ones, ring entries
  const uint32_t N = min(all / 2u, kSerialWindow), T = N + max(32u, N / 2u), RING = serial_ring(all);
  const uint32_t lt_mask = (1u << lane) - 1u;
  const uint32_t L = static_cast<uint32_t>(a.geo.L), W = a.geo.W;
  constexpr uint32_t NOCC = MODEL == kTwoLane ? 2u : 1u;
  constexpr uint32_t NQ = dis_planes(DIS);
  const uint32_t n_att = NOCC * L;
  uint32_t* gA = a.state + static_cast<size_t>(sample) * NOCC * W;
  uint2* ring = reinterpret_cast<uint2*>(serial_smem);  // [RING] bond and acceptance draw
  uint32_t* tab = serial_smem + 2u * RING;              // [2][NOCC L] site keys
  uint32_t* A = tab + 2u * n_att;                       // [NOCC][W] lattice, then [NQ][W] quenched planes
  SerialLattice lt = {A, A + NOCC * W, W, L, 31u - static_cast<uint32_t>(__clz(static_cast<int>(L))), shared_addr(A),
                      shared_addr(A + NOCC * W)};
  const uint32_t ring_s = shared_addr(ring), tab_s = shared_addr(tab);
  const uint32_t log_att = lt.logL + NOCC - 1u;
  for (uint32_t w = tid; w < NOCC * W; w += all) A[w] = gA[w];
  if (DIS != kDisNone) {
    const uint32_t* gM = a.mask + static_cast<size_t>(sample / a.geo.samples_per_real) * NQ * W;
    for (uint32_t w = tid; w < NQ * W; w += all) A[NOCC * W + w] = gM[w];
  }
  for (uint32_t i = tid; i < 2u * n_att; i += all) tab[i] = 0u;
  const uint32_t n_glob = a.geo.first_sample + sample;
  const uint64_t s0 = a.clock->sweep;
  uint32_t rec = a.clock->next_time;
  SerialStream stream;
  unsigned long long tot[4] = {0, 0, 0, 0};  // this thread's share of the sample's counters
  uint32_t c[4] = {0, 0, 0, 0};
  uint32_t round = 0;

  for (uint32_t it = 0; it < a.n_sweeps;) {
    const uint32_t n_sweeps = segment_sweeps<MODEL, DIS>(a, it, s0, rec, n_att);
    const uint32_t n = n_sweeps << log_att;  // attempts of the segment (n_att <= 2^15)
    const uint32_t s_lo = static_cast<uint32_t>(s0 + it);
    stream.open(s0 + it, n_glob, a.ks);
    const auto draw = [&](uint32_t q) {      // attempts q and q + 1 (q even)
      const uint4 y = stream.draw(s_lo + (q >> log_att), (q & (n_att - 1u)) >> 1, a.ks);
      *reinterpret_cast<uint4*>(&ring[q & (RING - 1u)]) = make_uint4(y.x & (n_att - 1u), y.y, y.z & (n_att - 1u), y.w);
    };
    if (tid == 0) s_taken = 0u;
    if (tid < 2u * N && 2u * tid < n) draw(2u * tid);  // the first four windows
    __syncthreads();
    if (tid < N) {
      uint32_t st = 0, u = 0, order = 0, first = 0;
      bool pending = false;
      uint32_t free = 0xffffffffu;
      if (lane == 0) first = atomicAdd(&s_taken, 32u);
      for (;;) {
        const uint32_t pos = __shfl_sync(0xffffffffu, first, 0) + __popc(free & lt_mask);
        const uint2 e = lds2(ring_s + 8u * (pos & (RING - 1u)));
        const bool take = !pending && pos < n;
        st = take ? e.x : st;
        u = take ? e.y : u;
        order = take ? 0xFFFFu - pos : order;
        pending = pending || take;
        if (round == kLastRound) {  // the drawing warps go through the same barriers
          (void)cta_any(false, T);
          for (uint32_t i = tid; i < 2u * n_att; i += N) tab[i] = 0u;
          round = 0;
          (void)cta_any(false, T);
        }
        ++round;
        const uint32_t t_s = tab_s + (round & 1u) * (4u * n_att);
        const uint32_t st1 = next_site<MODEL>(st, L), t0 = t_s + 4u * st, t1 = t_s + 4u * st1;
        const uint32_t key = pending ? (round << 16) | order : 0u;  // 0 changes nothing
        red_max(t0, key);
        red_max(t1, key);
        if (!cta_any(pending, T)) break;
        const bool go = lds(t0) == key && lds(t1) == key && pending;
        pending = pending && !go;
        // the next refill's positions are on their way while the attempts run
        free = __ballot_sync(0xffffffffu, !pending);
        if (lane == 0) first = atomicAdd(&s_taken, __popc(free));  // beyond n once the segment runs out
        serial_attempt<MODEL, DIS, true>(lt, st, st1, u, go, a, c);
      }
    } else if (tid < T) {
      uint32_t q = 4u * N + 2u * (tid - N);  // this thread's next pair; a warp's pairs stay together
      for (;;) {
        if (round == kLastRound) {
          (void)cta_any(false, T);
          round = 0;
          (void)cta_any(false, T);
        }
        ++round;
        if (!cta_any(false, T)) break;
        const uint32_t goal = *reinterpret_cast<volatile uint32_t*>(&s_taken) + 2u * N;
        const uint32_t first = __shfl_sync(0xffffffffu, q, 0);
        const uint32_t g = __shfl_sync(0xffffffffu, goal, 0);
        if (first < g && first < n) {  // warp-uniform
          if (q < n) draw(q);
          q += 2u * (T - N);
        }
      }
    }
    __syncthreads();  // the other warps of the CTA wait here
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      tot[k] += c[k];
      c[k] = 0;
    }
    it += n_sweeps;
    const uint64_t s = s0 + it;  // sweeps done
    if (MODEL == kTwoLane && (DIS == kDisTurning || DIS == kDisCrossing)) {
      serial_turns<DIS>(lt, a, s - 1u, n_glob, tid, all, c);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        tot[k] += c[k];
        c[k] = 0;
      }
      __syncthreads();
    }
    if (rec < a.n_times && a.times[rec] == s) {
      const uint32_t chunk = (W + all - 1u) / all;
      const uint32_t w0 = min(W, tid * chunk), w1 = min(W, w0 + chunk);
      for (uint32_t p = 0; p < NOCC; ++p) {
        const uint32_t* pw = A + p * W;
        long long rise = 0;
        for (uint32_t w = w0; w < w1; ++w) rise += 2 * __popc(pw[w]) - 32;
        const long long h = block_scan_incl(rise, s_i64) - rise;
        long long s1 = 0, ov = 0;
        unsigned long long s2 = 0;
        serial_record_words(pw, w0, w1, h, a, (static_cast<size_t>(sample) * NOCC + p) * W, s, s1, s2, ov);
        const long long s1_all = block_sum_i64(s1, s_i64);
        const long long ov_all = a.ex.snap ? block_sum_i64(ov, s_i64) : 0;
        const unsigned __int128 s2_all = block_sum_u128(s2, s_u64);
        if (tid == 0) {
          const size_t e = (static_cast<size_t>(rec) * a.geo.S + sample) * NOCC + p;
          a.tab_sh[e] = s1_all;
          a.tab_sh2[2 * e] = static_cast<uint64_t>(s2_all);
          a.tab_sh2[2 * e + 1] = static_cast<uint64_t>(s2_all >> 64);
          if (a.ex.snap) a.ex.tab_ac[e] = ov_all;
        }
      }
      for (int k = 0; k < 4; ++k) {
        const long long t = block_sum_i64(static_cast<long long>(tot[k]), s_i64);
        if (tid == 0)
          a.ex.tab_cnt[(static_cast<size_t>(rec) * a.geo.S + sample) * 4 + k] =
              static_cast<int64_t>(a.counters[4ull * sample + k] + static_cast<unsigned long long>(t));
      }
      ++rec;
    }
  }
  for (int k = 0; k < 4; ++k) {
    const long long t = block_sum_i64(static_cast<long long>(tot[k]), s_i64);
    if (tid == 0) a.counters[4ull * sample + k] += static_cast<unsigned long long>(t);
  }
  __syncthreads();
  for (uint32_t w = tid; w < NOCC * W; w += all) gA[w] = A[w];
}

// Warps (samples) per CTA: up to 8, but no more than spreads the samples
// over all SMs -- each warp's attempts form one dependent chain, so a few
// samples run fastest one per SM.
uint32_t serial_warps_per_cta(uint32_t S) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                                               cudaSuccess || sms <= 0) {
    (void)cudaGetLastError();
    sms = 1;
  }
  return std::max<uint32_t>(1, std::min<uint32_t>(8, (S + sms - 1) / static_cast<uint32_t>(sms)));
}

template <uint32_t MODEL, uint32_t DIS>
cudaError_t launch_serial_t(const SerialLaunch& a, cudaStream_t st) {
  constexpr uint32_t NPL = (MODEL == kTwoLane ? 2u : 1u) + dis_planes(DIS);
  const size_t lattice = static_cast<size_t>(NPL) * a.geo.W * 4u;
  const size_t budget = 200u * 1024u;  // shared memory for the staged lattices of one block
  const uint32_t spread = serial_warps_per_cta(a.geo.S);
  // the larger table where the lattice leaves room for it (4 % faster at 1024 rings of 4096)
  const uint32_t hash = lattice + serial_warp_scratch(kHashMost) <= budget ? kHashMost : kHashLeast;
  const size_t per_sample = lattice + serial_warp_scratch(hash);
  (void)cudaGetLastError();
  const bool staged = per_sample <= budget;
  const uint32_t warps = staged ? static_cast<uint32_t>(std::min<size_t>(spread, budget / per_sample)) : spread;
  const uint32_t blocks = (a.geo.S + warps - 1) / warps;
  const size_t smem = (staged ? per_sample : serial_warp_scratch(hash)) * warps;
  const auto kernel = staged ? k_serial<MODEL, DIS, true> : k_serial<MODEL, DIS, false>;
  const cudaError_t e = allow_smem(kernel, budget);
  if (e != cudaSuccess) return e;
  kernel<<<blocks, 32 * warps, smem, st>>>(a, hash);
  return cudaGetLastError();
}

template <uint32_t MODEL, uint32_t DIS>
cudaError_t launch_serial_rounds_t(const SerialLaunch& a, cudaStream_t st) {
  const size_t smem = serial_rounds_smem_bytes(MODEL, DIS, a.geo.L);
  const uint32_t threads = serial_rounds_threads(MODEL, a.geo.L);
  if (smem == 0) return cudaErrorInvalidValue;
  (void)cudaGetLastError();
  const cudaError_t e = allow_smem(k_serial_rounds<MODEL, DIS>, kSerialRoundsSmem);
  if (e != cudaSuccess) return e;
  k_serial_rounds<MODEL, DIS><<<a.geo.S, threads, smem, st>>>(a);
  return cudaGetLastError();
}

}  // namespace

size_t serial_rounds_smem_bytes(uint32_t model, uint32_t dis, uint64_t L) {
  const uint64_t nocc = model == kTwoLane ? 2u : 1u;
  const uint64_t n_att = nocc * L;
  if (L < 64 || n_att > kSerialRoundsMaxAttempts) return 0;
  // lattice and quenched planes, two site tables, the ring
  const uint64_t words = (nocc + dis_planes(dis)) * (L / 32) + 2 * n_att +
                         2ull * serial_ring(serial_rounds_threads(model, L));
  const size_t bytes = static_cast<size_t>(4 * words);
  return bytes <= kSerialRoundsSmem ? bytes : 0;
}

uint32_t serial_rounds_threads(uint32_t model, uint64_t L) {
  const uint64_t n_att = (model == kTwoLane ? 2u : 1u) * L;
  return static_cast<uint32_t>(std::min<uint64_t>(1024, n_att));
}

cudaError_t launch_serial_plan(const SerialLaunch& a, uint32_t model, uint32_t dis, uint32_t plan, cudaStream_t st) {
  if (plan != kSerialRounds) return launch_serial(a, model, dis, st);
  if (model == kRing && dis == kDisNone) return launch_serial_rounds_t<kRing, kDisNone>(a, st);
  if (model == kRing && dis == kDisBimodal) return launch_serial_rounds_t<kRing, kDisBimodal>(a, st);
  if (model == kRing && dis == kDisBimodalPQ) return launch_serial_rounds_t<kRing, kDisBimodalPQ>(a, st);
  if (model == kTwoLane && dis == kDisNone) return launch_serial_rounds_t<kTwoLane, kDisNone>(a, st);
  if (model == kTwoLane && dis == kDisTurning) return launch_serial_rounds_t<kTwoLane, kDisTurning>(a, st);
  if (model == kTwoLane && dis == kDisCrossing) return launch_serial_rounds_t<kTwoLane, kDisCrossing>(a, st);
  return cudaErrorInvalidValue;
}

uint32_t serial_warp_plan_warps(uint32_t S) { return serial_warps_per_cta(S); }

cudaError_t launch_serial(const SerialLaunch& a, uint32_t model, uint32_t dis, cudaStream_t st) {
  if (model == kRing && dis == kDisNone) return launch_serial_t<kRing, kDisNone>(a, st);
  if (model == kRing && dis == kDisBimodal) return launch_serial_t<kRing, kDisBimodal>(a, st);
  if (model == kRing && dis == kDisBimodalPQ) return launch_serial_t<kRing, kDisBimodalPQ>(a, st);
  if (model == kTwoLane && dis == kDisNone) return launch_serial_t<kTwoLane, kDisNone>(a, st);
  if (model == kTwoLane && dis == kDisTurning) return launch_serial_t<kTwoLane, kDisTurning>(a, st);
  if (model == kTwoLane && dis == kDisCrossing) return launch_serial_t<kTwoLane, kDisCrossing>(a, st);
  return cudaErrorInvalidValue;
}

}  // namespace asep
