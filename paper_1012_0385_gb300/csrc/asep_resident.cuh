// asep_resident.cuh -- the resident tier of the two-phase Poisson-domain
// schedule: one or more whole samples in one CTA's shared memory (layout in
// asep_kernels.cu).  run_group advances one sample group for a number of
// sweeps from a given sweep index and record cursor; it is shared by the
// one-launch kernel and the persistent batch kernel (asep_kernels.cu) and by
// the balanced kernel (asep_balance.cu).  Internal linkage: every kernel file
// gets its own copy.
#pragma once

#include <cstdint>

#include "asep_device.cuh"
#include "asep_domain.cuh"
#include "asep_internal.h"

namespace asep {
namespace {

// ---------------------------------------------------------------------------
// Segmented scan (all threads of the block must call)
// ---------------------------------------------------------------------------

// Segmented scan over the columns [col0, col0 + G) of one sample.
__device__ void seg_scan(long long v, uint32_t col0, uint32_t G, long long* warp_tot, long long* arr,
                         long long& excl_in_seg, long long& seg_total) {
  const long long inc = block_scan_incl(v, warp_tot);
  arr[threadIdx.x] = inc;
  __syncthreads();
  const long long before = col0 > 0 ? arr[col0 - 1] : 0;
  excl_in_seg = inc - v - before;
  seg_total = arr[col0 + G - 1] - before;
  __syncthreads();
}

// ---------------------------------------------------------------------------
// Resident two-phase Poisson-domain kernel
// ---------------------------------------------------------------------------

// Hop counters of one lane (named fields so they stay in registers).

// How far the frame moves from offset R_old to R_new (both below 2D <= L).
__device__ __forceinline__ uint32_t frame_shift(uint32_t R_new, uint32_t R_old, uint32_t L) {
  return R_new >= R_old ? R_new - R_old : R_new + L - R_old;
}

// Rotate the planes of one column from frame offset R_old to R_new: new frame
// word f = g*R2 + r holds logical sites R_new + 32 f .. + 31, that is old
// frame words f + delta / 32 and the next: rows row0 .. R2 - 1 of one column
// and then the rows from 0 of the next, each word loaded once, eight loads in
// flight.  (One word at a time with 64-bit positions: 1.3 of 5.4 us a sweep of
// 256 rings of 2^17 outside the attempts.)
template <uint32_t NP>
__device__ __forceinline__ void realign(const uint32_t* src, uint32_t* dst, const DomainLaunch& a, const Lane& ln,
                                        uint32_t PW, uint32_t delta) {
  const uint32_t R2 = a.R2, Cp = a.Cp, G = a.G;
  const uint32_t q = delta >> 5, sh = delta & 31u, row0 = q & (R2 - 1);
  uint32_t ca = ln.g + (q >> a.logR2);
  if (ca >= G) ca -= G;
  const uint32_t cb = ca + 1 == G ? 0u : ca + 1;
  // word i of the old frame counted from (row0, ca): rows wrap once to column cb
  const uint32_t first = row0 * Cp + ln.col0 + ca, turn = R2 - row0, wrap = cb - ca - R2 * Cp;
  const auto at = [&](uint32_t i) { return first + i * Cp + (i >= turn ? wrap : 0u); };
#pragma unroll
  for (uint32_t p = 0; p < NP; ++p) {
    const uint32_t* s = src + p * PW;
    uint32_t* d = dst + p * PW + ln.c;
    uint32_t w = s[at(0)];
    uint32_t r = 0;
    for (; r + 8 <= R2; r += 8) {
      uint32_t x[8];
#pragma unroll
      for (uint32_t k = 0; k < 8; ++k) x[k] = s[at(r + k + 1)];
#pragma unroll
      for (uint32_t k = 0; k < 8; ++k) {
        d[(r + k) * Cp] = __funnelshift_r(w, x[k], sh);
        w = x[k];
      }
    }
    for (; r < R2; ++r) {
      const uint32_t x = s[at(r + 1)];
      d[r * Cp] = __funnelshift_r(w, x, sh);
      w = x;
    }
  }
}

// Mirror row: copy row 0 of the next column into row R2 of this column (all
// planes), after the even phase and before the odd phase.
template <uint32_t NP>
__device__ __forceinline__ void mirror_in(uint32_t* cur, const DomainLaunch& a, uint32_t PW, const Lane& ln) {
#pragma unroll
  for (uint32_t p = 0; p < NP; ++p) cur[p * PW + a.R2 * a.Cp + ln.c] = cur[p * PW + ln.c_next];
}

// After the odd phase: the only bit of row 0 another lane may have changed is
// bit 0 (the previous column's last odd bond); take it back from its mirror.
template <uint32_t NOCC>
__device__ __forceinline__ void mirror_out(uint32_t* cur, const DomainLaunch& a, uint32_t PW, const Lane& ln) {
#pragma unroll
  for (uint32_t p = 0; p < NOCC; ++p) {
    const uint32_t w = cur[p * PW + ln.c];
    const uint32_t m = cur[p * PW + a.R2 * a.Cp + ln.c_prev];
    cur[p * PW + ln.c] = (w & ~1u) | (m & 1u);
  }
}

// Lane changes of the two-lane model in a warp's columns: at every turning
// site (DIS = kDisTurning: the sites of the turning plane, probability omega
// both ways) or every site (DIS = kDisCrossing: A -> B with u_i, B -> A with
// v_i, the slow value at sites marked in the u and v planes) where exactly one
// lane is occupied.  Lane A's plane holds the complement.
//
// Turning sites are sparse, so the warp pools its candidates: each lane queues
// up to eight sites, the lanes draw 32 queued sites at a time and flip the two
// planes' bits atomically (a column walking its own words ran each of them to
// the warp's largest count: 7 of 47 us a sweep of 128 pairs of lanes of 2^16 at
// density 0.05).  Crossing sites are dense: a lane takes the groups of four
// sites that share a call, in each of its words.
// queue: 256 words of the warp (of the idle realign buffer).  All 32 lanes call.
constexpr uint32_t kTurnQueue = 8;  // sites a lane queues per round
template <uint32_t DIS>
__device__ __forceinline__ void turning(uint32_t* cur, uint32_t* queue, const DomainLaunch& a, uint32_t PW, uint64_t s,
                                        uint32_t R_cur, const Lane& ln, Cnt& cnt) {
  uint32_t* A = cur;
  uint32_t* B = cur + PW;
  const uint32_t* M = cur + 2 * PW;  // turning plane, or the u marks (the v marks follow)
  const uint32_t L = static_cast<uint32_t>(a.geo.L), R2 = a.R2, Cp = a.Cp;
  const uint32_t a0 = philox_a0(static_cast<uint32_t>(s), a.ks), b2 = philox_b2(ln.n_glob, a.ks);
  const PhiloxHead head = philox_head(static_cast<uint32_t>(s), ctr_of(s, kTagTurn, 0, 0, 0).y, ln.n_glob, a.ks);
  if (DIS == kDisCrossing) {
    if (!ln.active) return;
    const uint32_t sh = R_cur & 3u;  // the frame's sites 4 k - sh .. 4 k - sh + 3 share a call
    for (uint32_t r = 0; r < R2; ++r) {
      const uint32_t idx = r * Cp + ln.c;
      const uint32_t av = ~A[idx], bv = B[idx], e = av ^ bv, um = M[idx], vm = M[PW + idx];
      const uint32_t slow = (av & um) | (~av & vm);
      uint32_t f = 0u;
      uint32_t n = (R_cur >> 2) + 8u * (ln.g * R2 + r);  // site / 4 of the word's first group, modulo L / 4
      for (int b = -static_cast<int>(sh); b < 32; b += 4, ++n) {
        const uint32_t bits = b < 0 ? e << -b : e >> b, marks = b < 0 ? slow << -b : slow >> b;
        if (!(bits & 15u)) continue;
        const uint4 x = philox_tail(head, philox_lane(a0, b2, n >= L / 4u ? n - L / 4u : n), a.ks);
        const uint32_t om = a.rates.omega, os = a.rates.omega_slow;
        uint32_t g = 0u;
        if ((bits & 1u) && accept(x.x, (marks & 1u) ? os : om)) g |= 1u;
        if ((bits & 2u) && accept(x.y, (marks & 2u) ? os : om)) g |= 2u;
        if ((bits & 4u) && accept(x.z, (marks & 4u) ? os : om)) g |= 4u;
        if ((bits & 8u) && accept(x.w, (marks & 8u) ? os : om)) g |= 8u;
        f |= b < 0 ? g >> -b : g << b;
      }
      cnt.c += __popc(f & av);
      cnt.d += __popc(f & ~av);
      A[idx] ^= f;
      B[idx] ^= f;
    }
    return;
  }
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t warp_c = ln.c - lane;  // the warp's first column
  uint32_t row = 0, e = 0;              // the next row to look at, what is left of the last one
  const auto next_word = [&]() {
    while (e == 0u && row < R2) {
      const uint32_t idx = row++ * Cp + ln.c;
      e = M[idx] & ~(A[idx] ^ B[idx]);
    }
  };
  if (ln.active) next_word();
  while (__any_sync(0xffffffffu, e != 0u)) {
    uint32_t mine[kTurnQueue], n = 0;
#pragma unroll
    for (uint32_t k = 0; k < kTurnQueue; ++k) {
      if (e) {
        const uint32_t b = static_cast<uint32_t>(__ffs(static_cast<int>(e))) - 1u;
        e &= e - 1u;
        mine[k] = (lane << 16) | ((row - 1u) << 5) | b;
        ++n;
        if (e == 0u) next_word();
      }
    }
    uint32_t incl = n;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= static_cast<uint32_t>(d)) incl += t;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
#pragma unroll
    for (uint32_t k = 0; k < kTurnQueue; ++k)
      if (k < n) queue[incl - n + k] = mine[k];
    __syncwarp();
    for (uint32_t i0 = 0; i0 < total; i0 += 32) {
      const uint32_t i = i0 + lane;
      const uint32_t q = i < total ? queue[i] : 0u;
      const uint32_t src = q >> 16, rw = (q >> 5) & 0x7FFu, bit = 1u << (q & 31u);
      // columns of one warp may belong to several samples: frame, site and draw are the column's
      const uint32_t col_site = __shfl_sync(0xffffffffu, R_cur + 32u * ln.g * R2, src);
      uint32_t site = col_site + 32u * rw + (q & 31u);
      if (site >= L) site -= L;
      const uint32_t b2s = __shfl_sync(0xffffffffu, b2, src);
      const PhiloxHead hs = {__shfl_sync(0xffffffffu, head.c3, src), __shfl_sync(0xffffffffu, head.y3, src),
                             __shfl_sync(0xffffffffu, head.d3, src)};
      const uint4 x = philox_tail(hs, philox_lane(a0, b2s, site >> 2), a.ks);
      const uint32_t smp = __shfl_sync(0xffffffffu, ln.sample, src);
      if (i < total && accept(pick(x, site & 3u), a.rates.omega)) {
        const uint32_t idx = rw * Cp + warp_c + src;
        const bool from_a = (~A[idx] & bit) != 0u;
        atomicXor(&A[idx], bit);
        atomicXor(&B[idx], bit);
        if (ln.active && smp == ln.sample) {
          cnt.c += from_a;
          cnt.d += !from_a;
        } else {  // a column of another sample, or a lane without one of its own
          atomicAdd(reinterpret_cast<unsigned long long*>(a.counters + 4ull * smp + (from_a ? 2 : 3)), 1ull);
        }
      }
    }
    __syncwarp();
  }
}

// Heights of the occupancy planes (frame offset 0) into table slot `slot`.
template <uint32_t NOCC>
__device__ void record_heights(const uint32_t* cur, const DomainLaunch& a, uint32_t PW, uint32_t slot, const Lane& ln,
                               long long* warp_tot, long long* arr) {
  for (uint32_t p = 0; p < NOCC; ++p) {
    const uint32_t* pl = cur + p * PW;
    const uint32_t inv = plane_inverse(a, p);
    long long tot = 0;
    if (ln.active)
      for (uint32_t r = 0; r < a.R2; ++r) tot += 2 * __popc(pl[r * a.Cp + ln.c] ^ inv) - 32;
    long long h0, seg_unused;
    seg_scan(tot, ln.col0, a.G, warp_tot, arr, h0, seg_unused);
    long long s1 = 0;
    unsigned long long s2 = 0;
    if (ln.active) {
      long long h = h0;
      for (uint32_t r = 0; r < a.R2; ++r) add_word_heights(pl[r * a.Cp + ln.c] ^ inv, h, s1, s2);
    }
    long long e1, t1, e2, t2;
    seg_scan(s1, ln.col0, a.G, warp_tot, arr, e1, t1);
    seg_scan(static_cast<long long>(s2), ln.col0, a.G, warp_tot, arr, e2, t2);
    if (ln.active && ln.g == 0) {
      const size_t e = (static_cast<size_t>(slot) * a.geo.S + ln.sample) * NOCC + p;
      a.tab_sh[e] = t1;
      a.tab_sh2[2 * e] = static_cast<uint64_t>(t2);
      a.tab_sh2[2 * e + 1] = 0;
    }
  }
}

// Sweeps of one sample group (spc samples, one column per thread) of one
// context, for a.n_sweeps sweeps starting at the context clock.  Used by the
// one-launch-per-context kernel (group = blockIdx.x) and by the persistent
// batch kernel (group from the work queue).  All threads of the block call.
// The other observables at a sample time t (frame offset 0): cumulative hop
// counters (lane counters are flushed first), the occupancy profile, and the
// overlap with the reference lattice of the density autocorrelation.
template <uint32_t NOCC>
__device__ void record_extras(const uint32_t* cur, const DomainLaunch& a, uint32_t PW, uint32_t slot, uint64_t t,
                              const Lane& ln, long long* warp_tot, long long* arr, Cnt& cnt) {
  const Extras& ex = a.ex;
  unsigned long long* ctr = reinterpret_cast<unsigned long long*>(a.counters + 4ull * ln.sample);
  if (ln.active) {
    if (cnt.a) atomicAdd(ctr + 0, static_cast<unsigned long long>(cnt.a));
    if (cnt.b) atomicAdd(ctr + 1, static_cast<unsigned long long>(cnt.b));
    if (cnt.c) atomicAdd(ctr + 2, static_cast<unsigned long long>(cnt.c));
    if (cnt.d) atomicAdd(ctr + 3, static_cast<unsigned long long>(cnt.d));
    cnt = Cnt();
  }
  __syncthreads();  // the block's counter updates are visible below
  if (ln.active && ln.g == 0) {
    const size_t e = (static_cast<size_t>(slot) * a.geo.S + ln.sample) * 4;
    for (int k = 0; k < 4; ++k) ex.tab_cnt[e + k] = static_cast<int64_t>(atomicAdd(ctr + k, 0ull));
  }
  const uint32_t W = a.geo.W;
  for (uint32_t p = 0; p < NOCC; ++p) {
    const uint32_t* pl = cur + p * PW;
    const size_t base = (static_cast<size_t>(ln.sample) * a.geo.planes + p) * W + static_cast<size_t>(ln.g) * a.R2;
    long long ov = 0;
    if (ln.active) {
      for (uint32_t r = 0; r < a.R2; ++r) {
        const uint32_t x = pl[r * a.Cp + ln.c] ^ plane_inverse(a, p);
        if (ex.profile) ex.profile[base + r] = __ldcg(&ex.profile[base + r]) + __popc(x);
        if (ex.snap) {
          if (t == ex.t0) ex.snap[base + r] = x;
          if (t >= ex.t0) ov += __popc(x & (t == ex.t0 ? x : __ldcg(&ex.snap[base + r])));
        }
      }
    }
    if (ex.snap) {
      long long e_unused, tot;
      seg_scan(ov, ln.col0, a.G, warp_tot, arr, e_unused, tot);
      if (ln.active && ln.g == 0) ex.tab_ac[(static_cast<size_t>(slot) * a.geo.S + ln.sample) * NOCC + p] = tot;
    }
  }
}

// Global data a group reads at its start (lattice) and at records (profile,
// reference lattice) may have been written by another CTA of the same launch
// (the balanced kernel hands groups between CTAs): read them from L2
// (ld.global.cg), never from a possibly stale L1 line.
template <uint32_t MODEL, uint32_t DIS, bool COUNT, uint32_t CP, bool PIN = false>
__device__ __forceinline__ void run_group(const DomainLaunch& a, uint32_t group, unsigned char* smem_raw,
                                          uint64_t s0, uint32_t cursor, uint32_t n_sweeps) {
  constexpr uint32_t NOCC = MODEL == kTwoLane ? 2u : 1u;
  constexpr uint32_t NQ = dis_planes(DIS);
  constexpr uint32_t NP = NOCC + NQ;
  const uint32_t R2 = a.R2, Cp = a.Cp, G = a.G, W = a.geo.W;
  const uint32_t PW = (R2 + 1) * Cp;  // R2 rows + the mirror row
  const uint32_t L = static_cast<uint32_t>(a.geo.L);
  uint32_t* bufA = reinterpret_cast<uint32_t*>(smem_raw);
  uint32_t* bufB = bufA + NP * PW;
  uint32_t* tab = bufB + NP * PW;
  long long* warp_tot = reinterpret_cast<long long*>(tab + ((a.ptab_n + 1u) & ~1u));
  long long* arr = warp_tot + 32;

  Lane ln;
  ln.c = threadIdx.x;
  const bool col_ok = ln.c < a.C;
  const uint32_t s_loc = col_ok ? ln.c / G : 0u;
  ln.g = col_ok ? ln.c - s_loc * G : 0u;
  ln.col0 = s_loc * G;
  ln.c_next = ln.col0 + (ln.g + 1 == G ? 0u : ln.g + 1);
  ln.c_prev = ln.col0 + (ln.g == 0 ? G - 1 : ln.g - 1);
  ln.sample = group * a.spc + s_loc;
  ln.active = col_ok && ln.sample < a.geo.S;
  ln.n_glob = a.geo.first_sample + ln.sample;
  const uint2 key = key_of(a.seed);

  // load the Poisson table and the lattices (frame offset 0)
  for (uint32_t i = threadIdx.x; i < a.ptab_n; i += blockDim.x) tab[i] = a.ptab[i];
  const uint32_t first = group * a.spc;
  const uint32_t nloc = min(a.spc, a.geo.S - first);
  for (uint32_t p = 0; p < NP; ++p) {
    for (uint32_t idx = threadIdx.x; idx < nloc * W; idx += blockDim.x) {
      const uint32_t sl = idx / W, w = idx - sl * W;
      const uint32_t smp = first + sl;
      const uint32_t v = p < NOCC ? __ldcg(&a.state[(static_cast<size_t>(smp) * a.geo.planes + p) * W + w])
                                  : a.mask[(static_cast<size_t>(smp / a.geo.samples_per_real) * NQ + (p - NOCC)) * W + w];
      bufA[p * PW + (w & (R2 - 1)) * Cp + sl * G + (w >> a.logR2)] = v ^ plane_inverse(a, p);
    }
  }
  __syncthreads();

  uint32_t* cur = bufA;
  uint32_t* nxt = bufB;
  uint32_t R_cur = 0;
  Cnt cnt;
  uint32_t rec = cursor;

  for (uint32_t it = 0; it < n_sweeps; ++it) {
    const uint64_t s = s0 + it;
    uint32_t o = 0;
    if (ln.active) o = philox10(ctr_of(s, kTagOff, 0, ln.n_glob, 0), key).x & (2 * a.D - 1);
    if (ln.active) realign<NP>(cur, nxt, a, ln, PW, frame_shift(o, R_cur, L));
    uint32_t* t = cur;
    cur = nxt;
    nxt = t;
    R_cur = o;
    __syncthreads();
    uint4* heads =
        a.heads ? reinterpret_cast<uint4*>(nxt + (a.lane_sort ? 5u * Cp : 0u)) + s_loc * a.heads : nullptr;
    run_phase<MODEL, DIS, COUNT, CP, 0, true, PIN>(cur, nxt, a.lane_sort != 0, heads, a.heads != 0, a, tab, PW, s, ln,
                                                   cnt, a.G, a.C);
    __syncthreads();
    if (ln.active) mirror_in<NP>(cur, a, PW, ln);
    run_phase<MODEL, DIS, COUNT, CP, 1, true, PIN>(cur, nxt, a.lane_sort != 0, heads, false, a, tab, PW, s, ln, cnt,
                                                   a.G, a.C);
    __syncthreads();
    if (ln.active) mirror_out<NOCC>(cur, a, PW, ln);
    __syncthreads();
    if (MODEL == kTwoLane && (DIS == kDisTurning || DIS == kDisCrossing)) {
      if (threadIdx.x < Cp)  // whole warps
        turning<DIS>(cur, nxt + (threadIdx.x >> 5) * (32u * kTurnQueue), a, PW, s, R_cur, ln, cnt);
      __syncthreads();
    }
    if (rec < a.n_times && a.times[rec] == s + 1) {
      if (ln.active) realign<NP>(cur, nxt, a, ln, PW, frame_shift(0, R_cur, L));
      t = cur;
      cur = nxt;
      nxt = t;
      R_cur = 0;
      __syncthreads();
      record_heights<NOCC>(cur, a, PW, rec, ln, warp_tot, arr);
      record_extras<NOCC>(cur, a, PW, rec, s + 1, ln, warp_tot, arr, cnt);
      ++rec;
    }
  }

  // back to frame offset 0 and out to global memory
  if (ln.active) realign<NP>(cur, nxt, a, ln, PW, frame_shift(0, R_cur, L));
  cur = nxt;
  __syncthreads();
  for (uint32_t p = 0; p < NOCC; ++p) {
    for (uint32_t idx = threadIdx.x; idx < nloc * W; idx += blockDim.x) {
      const uint32_t sl = idx / W, w = idx - sl * W;
      a.state[(static_cast<size_t>(first + sl) * a.geo.planes + p) * W + w] =
          cur[p * PW + (w & (R2 - 1)) * Cp + sl * G + (w >> a.logR2)] ^ plane_inverse(a, p);
    }
  }
  if (ln.active) {
    unsigned long long* dst = reinterpret_cast<unsigned long long*>(a.counters + 4ull * ln.sample);
    if (cnt.a) atomicAdd(dst + 0, static_cast<unsigned long long>(cnt.a));
    if (cnt.b) atomicAdd(dst + 1, static_cast<unsigned long long>(cnt.b));
    if (cnt.c) atomicAdd(dst + 2, static_cast<unsigned long long>(cnt.c));
    if (cnt.d) atomicAdd(dst + 3, static_cast<unsigned long long>(cnt.d));
  }
  __syncthreads();  // the shared memory is reused by the next group of a persistent CTA
}

}  // namespace
}  // namespace asep
