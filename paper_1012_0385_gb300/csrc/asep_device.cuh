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
