// asep_device.cuh -- device helpers shared by the kernel files: the
// Philox4x32-10 generator (Salmon, Moraes, Dror, Shaw, SC'11) with the
// library's counter layout, and a block-wide inclusive scan.  Internal
// linkage: every kernel file gets its own copy.
#pragma once

#include <cstdint>

#include "asep_internal.h"

namespace asep {
namespace {

// ---------------------------------------------------------------------------
// Philox4x32-10 and counters
// ---------------------------------------------------------------------------

// 32 x 32 -> 64-bit product as one wide multiply; .x = low word, .y = high word.
__device__ __forceinline__ uint2 mul_wide(uint32_t a, uint32_t b) {
  unsigned long long p;
  asm("mul.wide.u32 %0, %1, %2;" : "=l"(p) : "r"(a), "r"(b));
  return make_uint2(static_cast<uint32_t>(p), static_cast<uint32_t>(p >> 32));
}

// One Philox4x32 round with round key (kx, ky).
__device__ __forceinline__ uint4 philox_round(uint4 c, uint32_t kx, uint32_t ky) {
  const uint2 p0 = mul_wide(0xD2511F53u, c.x);
  const uint2 p1 = mul_wide(0xCD9E8D57u, c.z);
  return make_uint4(p1.y ^ c.y ^ kx, p1.x, p0.y ^ c.w ^ ky, p0.x);
}

__device__ __forceinline__ uint4 philox10(uint4 c, uint2 k) {
#pragma unroll
  for (int round = 0; round < 10; ++round) {
    c = philox_round(c, k.x, k.y);
    k.x += 0x9E3779B9u;
    k.y += 0xBB67AE85u;
  }
  return c;
}

// Philox4x32-10 with the round keys precomputed (KeySchedule, filled by the
// host): in a kernel whose descriptor is a parameter the keys are read from
// the constant bank, so a call costs only the multiplies and XORs.
__device__ __forceinline__ uint4 philox10(uint4 c, const KeySchedule& ks) {
#pragma unroll
  for (int round = 0; round < 10; ++round) c = philox_round(c, ks.x[round], ks.y[round]);
  return c;
}

// Philox4x32-10 split by what varies.  A warp's calls at one sweep differ only
// in counter word 3 (domain, unit or site group) and in the call field of
// word 1, so the first three rounds need not be run per lane and call:
//   round 1: both products (of words 0 and 2) are the same for all lanes;
//   round 2: its product of word 0 depends on the call only, that of word 2
//            on word 3 only;
//   round 3: the same, the other way round.
// A call then costs a lane 7 rounds (14 wide multiplies, the unit a plain
// call saturates at 30.2 of 32 a clock and SM) and two XORs instead of 10
// rounds; the per-call part (PhiloxHead) is formed once per sweep and sample,
// the per-lane part (PhiloxLane) once per sweep, lane and counter word 3.
struct PhiloxHead {
  uint32_t c3, y3, d3;  // round 3 of one (sweep, call, sample): x ^= c3, word y, z ^= d3
};
struct PhiloxLane {
  uint32_t y2, hv, w3;  // rounds 2 and 3 of one (sweep, sample, word 3)
};

// Round 1 of counter word 0: hi(M0 x) ^ ky0, to be XORed with counter word 3.
__device__ __forceinline__ uint32_t philox_a0(uint32_t x, const KeySchedule& ks) {
  return mul_wide(0xD2511F53u, x).y ^ ks.y[0];
}

__device__ __forceinline__ PhiloxHead philox_head(uint32_t x, uint32_t y, uint32_t z, const KeySchedule& ks) {
  const uint2 q = mul_wide(0xD2511F53u, mul_wide(0xCD9E8D57u, z).y ^ y ^ ks.x[0]);  // round 2, word 0
  const uint2 r = mul_wide(0xCD9E8D57u, q.y ^ mul_wide(0xD2511F53u, x).x ^ ks.y[1]);  // round 3, word 2
  return {r.y ^ ks.x[2], r.x, q.x ^ ks.y[2]};
}

// b2 = philox_b2(z): round 2's XOR of counter word 2's low product.
__device__ __forceinline__ uint32_t philox_b2(uint32_t z, const KeySchedule& ks) {
  return mul_wide(0xCD9E8D57u, z).x ^ ks.x[1];
}

__device__ __forceinline__ PhiloxLane philox_lane(uint32_t a0, uint32_t b2, uint32_t w) {
  const uint2 t = mul_wide(0xCD9E8D57u, a0 ^ w);
  const uint2 v = mul_wide(0xD2511F53u, t.y ^ b2);
  return {t.x, v.y, v.x};
}

// Rounds 4 to 10: = philox10 of the counter the head and the lane part came from.
__device__ __forceinline__ uint4 philox_tail(const PhiloxHead& h, const PhiloxLane& l, const KeySchedule& ks) {
  uint4 c = make_uint4(h.c3 ^ l.y2, h.y3, l.hv ^ h.d3, l.w3);
#pragma unroll
  for (int round = 3; round < 10; ++round) c = philox_round(c, ks.x[round], ks.y[round]);
  return c;
}

__device__ __forceinline__ uint2 key_of(uint64_t seed) {
  return make_uint2(static_cast<uint32_t>(seed), static_cast<uint32_t>(seed >> 32));
}

__device__ __forceinline__ uint4 ctr_of(uint64_t sweep, uint32_t tag, uint32_t call, uint32_t sample, uint32_t d) {
  return make_uint4(static_cast<uint32_t>(sweep),
                    (static_cast<uint32_t>(sweep >> 32) & 0xFFu) | (tag << 8) | (call << 12), sample, d);
}

// Output word i of a Philox call.
__device__ __forceinline__ uint32_t pick(const uint4 x, uint32_t i) {
  return i == 0 ? x.x : (i == 1 ? x.y : (i == 2 ? x.z : x.w));
}

// A draw r accepts a move of threshold t (0, a multiple of 4096 or "always").
__device__ __forceinline__ bool accept(uint32_t r, uint32_t t) { return (r & kAcceptMask) < t; }

// Moves the clock n sweeps on (one thread).
__device__ __forceinline__ void advance_clock(Clock* c, const uint64_t* times, uint32_t n_times, uint32_t n) {
  const unsigned long long sweep = c->sweep + n;
  uint32_t next = c->next_time;
  while (next < n_times && times[next] <= sweep) ++next;
  c->sweep = sweep;
  c->next_time = next;
}

// ---------------------------------------------------------------------------
// Heights of a word
// ---------------------------------------------------------------------------

// Adds the heights h_i = h + sum_{j <= i} (2 n_j - 1) of the 32 sites of word x
// to s1, their squares to s2, and moves h past the word.  Four sites at a
// time: a nibble's bits are spread to bytes, summed along the bytes by one
// multiply, and the heights relative to the word's entry, biased by 64 to
// stay positive (32 .. 96), go through two byte dot products -- about 10
// instructions for four sites where 64-bit adds and a multiply a site took 40:
// 12 us less a record of 256 rings of 2^17 sites inside the resident SCA
// kernel (31 -> 19 us, records every few sweeps).
__device__ __forceinline__ void add_word_heights(uint32_t x, long long& h, long long& s1, unsigned long long& s2) {
  uint32_t t = 64u, sum = 0u, sq = 0u;  // biased height before the nibble; sums of the biased heights
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t n = (((x >> (4 * i)) & 15u) * 0x00204081u) & 0x01010101u;  // site k in byte k
    const uint32_t v = 2u * (n * 0x01010101u) + t * 0x01010101u - 0x04030201u;
    sum = __dp4a(v, 0x01010101u, sum);
    sq = __dp4a(v, v, sq);
    t = v >> 24;
  }
  const long long r1 = static_cast<long long>(sum) - 64 * 32;                       // sum of the relative heights
  const long long r2 = static_cast<long long>(sq) - 128ll * sum + 64ll * 64 * 32;  // and of their squares
  s1 += 32 * h + r1;
  s2 += static_cast<unsigned long long>(h * (32 * h + 2 * r1) + r2);
  h += static_cast<int>(t) - 64;
}

// ---------------------------------------------------------------------------
// Block scans (all threads of the block must call; blockDim.x % 32 == 0)
// ---------------------------------------------------------------------------

__device__ long long block_scan_incl(long long v, long long* warp_tot) {
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= static_cast<uint32_t>(o)) v += t;
  }
  if (lane == 31u) warp_tot[wid] = v;
  __syncthreads();
  if (wid == 0) {
    long long t = lane < nw ? warp_tot[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long u = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= static_cast<uint32_t>(o)) t += u;
    }
    if (lane < nw) warp_tot[lane] = t;
  }
  __syncthreads();
  if (wid > 0) v += warp_tot[wid - 1];
  __syncthreads();
  return v;
}

}  // namespace
}  // namespace asep
