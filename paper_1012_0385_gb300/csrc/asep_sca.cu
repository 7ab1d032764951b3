// asep_sca.cu -- the paper's own GPU schedule: the two-sub-lattice stochastic
// cellular automaton of sec. 2.1 (Fig. "parasep"), bit-sliced for sm_103a.
//
// One sweep updates every even bond (i, i+1), i = 0, 2, ..., L-2, in
// parallel, then every odd bond i = 1, 3, ..., L-1 (the last one, (L-1, 0),
// is the paper's ring-closing step; it shares no site with the other odd
// bonds, so it runs with them).  Each bond makes one attempt: 10 -> 01 with
// p_i, 01 -> 10 with q_{i+1}, accepted iff a 20-bit uniform u is below the
// threshold's top 20 bits.
//
// Bit slicing.  A group is 32 bonds of one phase: the 16 bonds of word 2g
// (lanes 0, 2, ..., 30) and the 16 of word 2g + 1 (lanes 1, 3, ..., 31).
// Bit k of every lane's u is bit `lane` of random plane k of the group; call k
// of the stream (tag SCA, ctr3 = 2 * unit + phase) gives plane k of the four
// groups of a unit (8 words).  The comparison u < t runs over all 32 lanes at
// once, and only over planes down to the lowest set bit of any threshold (p =
// 0.75, q = 0.25 need two); longer ones end when no lane is undecided
// (asep_sca.cuh).
//
// Layout.  A warp holds a tile of consecutive units of one ring in registers
// for a whole launch, in the bond-lane form of asep_sca.cuh; the lattice is in
// global memory in its plain layout (bit k of word w = site 32w + k) between
// launches.  Neighbouring units exchange the bits an odd bond joins by
// shuffles.
#include <algorithm>
#include <cstdint>

#include "asep_device.cuh"
#include "asep_internal.h"
#include "asep_sca.cuh"

namespace asep {
namespace {

// Two units a thread from here on (one-unit tiles of a launch), for the kinds
// with a fixed number of planes: the halos cost 3 % instead of 7 %, but a
// launch then has half the warps, and below some 100 tiles per SM their last
// wave costs more.  us per sweep with one and two units a thread: 256 rings of
// 2^17 (4608 tiles) 1.65 / 1.69, 400 rings of 2^18 (14000) 4.79 / 4.83, 152
// rings of 2^20 (20824) 6.96 / 6.80, 8 rings of 2^28 90.3 / 86.9.
constexpr uint64_t kScaManyTiles = 152u * 108u;

// Kinds without a fixed number of planes: a phase of a warp lasts until the
// last of its candidates is decided (some log2 of their number planes), or its
// queue of lane changes is done, so where the tiles are fewer than the
// schedulers, rings are cut into smaller ones, of four units at least, while
// no scheduler has two.  us per sweep without and with: 76 rings of 32 units with
// slow classes 3.50 -> 3.14, 113 of 19 units 3.30 -> 2.95, 191 pairs of lanes of
// 25 units with turning sites 5.29 -> 3.98; cut further, to two warps a scheduler,
// 265 rings of 14 units 3.17 -> 3.95.
constexpr uint64_t kScaFewTiles = 4u * 152u;
constexpr uint32_t kScaFewUnits = 4u;

// One launch of k_sca_tile.
struct ScaTileLaunch {
  uint32_t tiles, units;  // per ring: tiles, units per tile (the last may hold fewer)
  uint32_t n, offset;     // sweeps of this launch, and before it since the context clock
  uint32_t n_rec, rec_offset;  // sample times inside this launch (at most, if it may run at any sweep), and before
                               // it since the clock's cursor
  const uint32_t* halo_in;   // [S][tiles][first, last unit][planes][8] (one tile a ring: unused)
  uint32_t* halo_out;
  ScaPart* parts;         // [n_rec + 1][S][tiles][planes] (the last entry: the launch's hops; one tile: unused)
};

// ---------------------------------------------------------------------------
// Tiles
// ---------------------------------------------------------------------------

// A warp takes a tile of consecutive units of one ring, UPT to a thread, with
// one more unit on either side (halo), and advances it on its own for a whole
// launch of up to kScaTileSweeps sweeps: a phase carries the influence of a
// unit's unknown neighbour one site further, so after n sweeps 2 n - 1 sites
// at a halo's outer end are stale -- 255 of its 256 after 128 -- and none of
// the tile.  Nothing crosses warps inside a launch, so there are no barriers,
// and the lattice moves through memory once per launch instead of twice per
// sweep.  One tile a CTA, so that tiles spread over the SMs evenly.
// In place: a tile reads and writes only its own units of the lattice; its
// neighbours' edge units come from a buffer that the previous launch (or
// k_sca_halo, once the lattice was replaced) filled, and go to the other half of
// it.
// Bound by the integer ALU pipe (logic of Philox and of the update: 69 % busy,
// 173 of 268 instructions a unit and sweep at two planes).  Measured against
// one CTA per ring with two barriers a sweep, and against one launch per phase
// with the lattice streamed through HBM, us per sweep: 256 rings of 2^17 at
// p = 0.75, q = 0.25 (hops not counted) 1.90 -> 1.65, 128 pairs of lanes of 2^16
// with turning sites 6.35 -> 6.6 (units in registers on both sides), 201 rings
// of 391 units with independent classes 18.7 -> 9.0, 2 rings of 2^22 10.2 -> 0.55,
// 8 rings of 2^28 191 -> 87 (against the kernels with plain words).
//
// Records are taken inside the launch: a tile leaves the sums of its heights
// relative to its entry height, its height change and its hops so far, and
// k_sca_records combines the tiles of every record of the launch.  (A record
// between launches -- the launch, k_heights, the clock, the next launch --
// took some 25 us; 256 rings of 2^17 with 88 log-spaced records in 2048
// sweeps spent 2.2 of 5.6 ms there.)
//
// A ring of one tile is its own neighbour: its halos come from its own units of
// the lattice, and a record of it is whole.  It needs neither buffer, which are
// 128 B of halo a tile and plane and 40 B a record, tile and plane beside 32 B
// of lattice a unit.

// The tile's hops since the launch began.
__device__ __forceinline__ void tile_hops(const ScaCounts& cnt, ScaPart* part) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const uint32_t v = __reduce_add_sync(0xffffffffu, cnt.c[k]);
    if ((threadIdx.x & 31u) == 31u) part->hops[k] = v;
  }
}

// One record of one tile: the other observables, and its part of the height
// sums, or (one tile a ring) the record itself, in slot `slot`.
template <uint32_t NOCC, uint32_t UPT>
__device__ void tile_record(const ScaUnit (&U)[NOCC][UPT], const uint32_t (&gu)[UPT], const uint32_t (&counted)[UPT],
                            const DomainLaunch& a, uint32_t sample, uint64_t time, size_t slot, bool whole,
                            ScaPart* part, bool count, const ScaCounts& cnt) {
  const uint32_t lane = threadIdx.x & 31u;
  const Extras& ex = a.ex;
#pragma unroll
  for (uint32_t p = 0; p < NOCC; ++p) {
    int tot = 0, ov = 0;
#pragma unroll
    for (uint32_t j = 0; j < UPT; ++j) {
      if (!counted[j]) continue;
      uint32_t x[8];
      to_words(U[p][j], x);
      const size_t base = (static_cast<size_t>(sample) * NOCC + p) * a.geo.W + 8u * gu[j];
#pragma unroll
      for (int w = 0; w < 8; ++w) {
        const int ones = __popc(x[w]);
        tot += 2 * ones - 32;
        if (ex.profile) ex.profile[base + w] += ones;
        if (ex.snap) {
          if (time == ex.t0) ex.snap[base + w] = x[w];
          if (time >= ex.t0) ov += __popc(time == ex.t0 ? x[w] : x[w] & ex.snap[base + w]);
        }
      }
    }
    int incl = tot;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= static_cast<uint32_t>(d)) incl += v;
    }
    long long h = incl - tot, s1 = 0;
    unsigned long long s2 = 0;
#pragma unroll
    for (uint32_t j = 0; j < UPT; ++j) {
      if (!counted[j]) continue;
      uint32_t x[8];
      to_words(U[p][j], x);
#pragma unroll 1
      for (int w = 0; w < 8; ++w) {
        add_word_heights(x[0], h, s1, s2);
#pragma unroll
        for (int v = 0; v < 7; ++v) x[v] = x[v + 1];
      }
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      s1 += __shfl_xor_sync(0xffffffffu, s1, d);
      s2 += __shfl_xor_sync(0xffffffffu, s2, d);
      ov += __shfl_xor_sync(0xffffffffu, ov, d);
    }
    if (whole) {
      if (lane == 31u) {
        const size_t e = (slot * a.geo.S + sample) * NOCC + p;
        a.tab_sh[e] = s1;
        a.tab_sh2[2 * e] = s2;
        a.tab_sh2[2 * e + 1] = 0;
        if (ex.snap) ex.tab_ac[e] = ov;
      }
    } else if (lane == 31u) {
      part[p].tot = incl;
      part[p].ov = ov;
      part[p].s1 = s1;
      part[p].s2 = s2;
    }
  }
  if (whole) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t v = __reduce_add_sync(0xffffffffu, cnt.c[k]);  // since the launch began
      if (lane == 31u)
        ex.tab_cnt[(slot * a.geo.S + sample) * 4 + k] = static_cast<int64_t>(a.counters[4ull * sample + k] + v);
    }
  } else if (count) {
    tile_hops(cnt, part);
  }
}

template <uint32_t MODEL, bool DIS, bool COUNT, uint32_t FAST, bool PQ, uint32_t UPT>
__global__ void __launch_bounds__(32, DIS ? 20 : (MODEL == kTwoLane ? 24 : 28))
    k_sca_tile(const DomainLaunch a, const ScaTileLaunch t) {
  __shared__ __align__(16) ScaHeads heads;
  __shared__ __align__(16) unsigned char turn_raw[(MODEL == kTwoLane && DIS && !PQ) ? sizeof(ScaTurnScratch) : 16];
  constexpr uint32_t NOCC = MODEL == kTwoLane ? 2u : 1u;
  constexpr int NQ = DIS ? (PQ ? 2 : 1) : 0;
  constexpr bool TURNS = MODEL == kTwoLane && DIS;
  const uint32_t W = a.geo.W, n_units = W / 8;
  const uint32_t sample = blockIdx.x / t.tiles, n_glob = a.geo.first_sample + sample;
  const uint32_t lane = threadIdx.x;
  const uint32_t tile = blockIdx.x - sample * t.tiles;
  const uint32_t first = tile * t.units, n_own = min(t.units, n_units - first);
  const uint64_t s0 = a.clock->sweep + t.offset;
  const uint32_t kmax = a.sca_kmax, calls = sca_calls(kmax, TURNS), chunk = sca_chunk(calls);
  const uint32_t b2 = philox_b2(n_glob, a.ks);
  const ScaRule rule = sca_rule(a.rates, DIS);
  ScaTurnScratch* turn = reinterpret_cast<ScaTurnScratch*>(turn_raw);

  // local unit i = lane UPT + j: 0 and n_own + 1 are the halos
  uint32_t* state = a.state + static_cast<size_t>(sample) * NOCC * W;
  // A launch that may run at any sweep -- captured into a graph -- knows only how many sample times can fall into it.
  const uint64_t* next_time = a.times + a.clock->next_time + t.rec_offset;
  const auto more = [&](uint32_t r) { return r < t.n_rec && next_time + r < a.times + a.n_times; };
  const size_t edge0 = static_cast<size_t>(sample) * t.tiles * 2u;  // this ring's entries of the halo buffers
  uint32_t gu[UPT], counted[UPT];
  ScaUnit U[NOCC][UPT];
  ScaUnit Q[NQ == 2 ? 2 : 1];
  uint32_t q_odd[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (uint32_t j = 0; j < UPT; ++j) {
    const uint32_t i = lane * UPT + j;
    const bool own = i >= 1u && i <= n_own, used = i <= n_own + 1u;
    uint32_t g = used ? first + i + (i == 0u ? n_units : 0u) - 1u : 0u;  // modulo the ring
    if (g >= n_units) g -= n_units;
    gu[j] = g;
    counted[j] = own ? ~0u : 0u;
    // left halo: the previous tile's last unit; right halo: the next tile's first
    const uint32_t nb = i == 0u ? (tile == 0u ? t.tiles : tile) - 1u : (tile + 1u == t.tiles ? 0u : tile + 1u);
    const uint32_t* edge = t.halo_in + (edge0 + 2u * nb + (i == 0u ? 1u : 0u)) * (NOCC * 8u);
    const bool from_edges = used && !own && t.tiles > 1u;
    const uint32_t* src = from_edges ? edge : state + 8u * g;
    const uint32_t pitch = from_edges ? 8u : W;
#pragma unroll
    for (uint32_t p = 0; p < NOCC; ++p) {
      uint32_t x[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
      if (used) load8(src + p * pitch, x);
      U[p][j] = to_lanes(x);
    }
    if (DIS) {  // UPT = 1
      const uint32_t* mask = a.mask + static_cast<size_t>(sample / a.geo.samples_per_real) * NQ * W;
#pragma unroll
      for (int p = 0; p < NQ; ++p) {
        uint32_t x[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
        if (used) load8(mask + p * W + 8u * g, x);
        Q[p] = to_lanes(x);
      }
      if (MODEL == kRing) {
        constexpr int kq = NQ == 2 ? 1 : 0;
        const uint32_t nx = used ? mask[kq * W + (g + 1 == n_units ? 0u : 8u * g + 8u)] : 0u;
#pragma unroll
        for (int k = 0; k < 4; ++k) q_odd[k] = odd_sites(Q[kq].e[k], k < 3 ? Q[kq].e[k + 1] : nx);
      }
    }
  }
  if (TURNS && !PQ) {
    const uint32_t zero[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
    store8(turn->flip[lane], zero);
  }

  ScaCounts cnt;
  const size_t part_pitch = static_cast<size_t>(a.geo.S) * t.tiles * NOCC;  // entries of one record
  ScaPart* part = t.parts + (static_cast<size_t>(sample) * t.tiles + tile) * NOCC;
  uint32_t filled = 0, base = 0, recs = 0;
  for (uint32_t done = 0; done < t.n;) {
    if (done == filled) {
      base = done;
      filled = min(done + chunk, t.n);
      __syncwarp();
      sca_fill_heads(heads, s0 + base, filled - base, kmax, calls, n_glob, a.ks);
      __syncwarp();
    }
    uint32_t stop = filled;
    if (more(recs)) stop = static_cast<uint32_t>(min(static_cast<uint64_t>(stop), next_time[recs] - s0));
#pragma unroll 1
    for (; done < stop; ++done) {
      const uint32_t it = done - base;
      const uint4* hd = heads.head + it * calls;
      const uint32_t a0 = heads.a0[it];
      uint32_t h[UPT][4];
      // even phase
#pragma unroll
      for (uint32_t p = 0; p < NOCC; ++p) {
#pragma unroll
        for (uint32_t j = 0; j < UPT; ++j) {
          ScaUnit& x = U[p][j];
          uint4 y0, y1;
          const PhiloxLane pl = philox_lane(a0, b2, (2u * gu[j]) | (p << 31));
          sca_first_planes<MODEL, FAST>(hd, pl, a.ks, y0, y1);
          if (p == 0)
            sca_update<MODEL, DIS, PQ, COUNT, FAST, 0, 0>(x, 0u, Q, q_odd, a.rates, rule, kmax, hd, pl, y0, y1, a.ks,
                                                          counted[j], cnt, h[j]);
          else
            sca_update<MODEL, DIS, PQ, COUNT, FAST, 0, 1>(x, 0u, Q, q_odd, a.rates, rule, kmax, hd, pl, y0, y1, a.ks,
                                                          counted[j], cnt, h[j]);
        }
      }
      if (TURNS)
        cnt.c[2] += PQ ? sca_turn_all<0>(U[0][0], U[NOCC - 1][0], Q[0], gu[0], counted[0], a0, b2, hd[kmax], a)
                       : sca_turn_pool<0>(U[0][0], U[NOCC - 1][0], Q[0], *turn, gu[0], counted[0], a0, b2, hd[kmax], a);
      // odd phase: the last unit's next site and the first one's flip come from the neighbour lanes
#pragma unroll
      for (uint32_t p = 0; p < NOCC; ++p) {
        const uint32_t en = __shfl_down_sync(0xffffffffu, U[p][0].e[0], 1);
#pragma unroll
        for (uint32_t j = 0; j < UPT; ++j) {
          ScaUnit& x = U[p][j];
          const uint32_t ej = j + 1 < UPT ? U[p][j + 1 < UPT ? j + 1 : j].e[0] : en;
          uint4 y0, y1;
          const PhiloxLane pl = philox_lane(a0, b2, (2u * gu[j] + 1u) | (p << 31));
          sca_first_planes<MODEL, FAST>(hd, pl, a.ks, y0, y1);
          if (p == 0)
            sca_update<MODEL, DIS, PQ, COUNT, FAST, 1, 0>(x, ej, Q, q_odd, a.rates, rule, kmax, hd, pl, y0, y1, a.ks,
                                                          counted[j], cnt, h[j]);
          else
            sca_update<MODEL, DIS, PQ, COUNT, FAST, 1, 1>(x, ej, Q, q_odd, a.rates, rule, kmax, hd, pl, y0, y1, a.ks,
                                                          counted[j], cnt, h[j]);
        }
        const uint32_t hp = __shfl_up_sync(0xffffffffu, h[UPT - 1][3], 1);  // lane 0: a stale halo site either way
#pragma unroll
        for (uint32_t j = 0; j < UPT; ++j) {
          ScaUnit& x = U[p][j];
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            x.e[g] ^= odd_flips(h[j][g], g > 0 ? h[j][g > 0 ? g - 1 : 0] : (j > 0 ? h[j > 0 ? j - 1 : 0][3] : hp));
          }
        }
      }
      if (TURNS)
        cnt.c[3] += PQ ? sca_turn_all<1>(U[0][0], U[NOCC - 1][0], Q[NQ == 2 ? 1 : 0], gu[0], counted[0], a0, b2,
                                         hd[kmax + 1], a)
                       : sca_turn_pool<1>(U[0][0], U[NOCC - 1][0], Q[0], *turn, gu[0], counted[0], a0, b2,
                                          hd[kmax + 1], a);
    }
    if (more(recs) && next_time[recs] == s0 + done) {
      tile_record<NOCC, UPT>(U, gu, counted, a, sample, s0 + done, next_time + recs - a.times, t.tiles == 1u,
                             part, COUNT, cnt);
      part += part_pitch;
      ++recs;
    }
  }
  if (COUNT && t.n_rec && t.tiles > 1u) tile_hops(cnt, part + (t.n_rec - recs) * part_pitch);

#pragma unroll
  for (uint32_t j = 0; j < UPT; ++j) {
    const uint32_t i = lane * UPT + j;
    if (i < 1u || i > n_own) continue;
#pragma unroll
    for (uint32_t p = 0; p < NOCC; ++p) {
      uint32_t x[8];
      to_words(U[p][j], x);
      store8(state + p * W + 8u * gu[j], x);
      if (t.tiles == 1u) continue;
      if (i == 1u) store8(t.halo_out + ((edge0 + 2u * tile) * NOCC + p) * 8u, x);
      if (i == n_own) store8(t.halo_out + ((edge0 + 2u * tile + 1u) * NOCC + p) * 8u, x);
    }
  }
  if (COUNT) {
    constexpr int NK = TURNS ? 4 : 2;
#pragma unroll
    for (int k = 0; k < NK; ++k) {
      unsigned long long v = cnt.c[k];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0u && v) atomicAdd(reinterpret_cast<unsigned long long*>(a.counters + 4ull * sample + k), v);
    }
  }
}

// The records of one launch, a warp per record and sample: the tiles' sums
// with their entry heights H_j added back exactly (sum (H + h') = sum h' + H n,
// sum (H + h')^2 = sum h'^2 + 2 H sum h' + H^2 n), and the hop counters at the
// record: those after the launch, less the launch's hops, plus its hops so far.
// advance: sweeps that the last block to end moves the clock by (0 = none): every
// block has read it by then.  (A launch for the clock alone is 2 us of the some
// 17 of a call of one sweep of a small context.)
__device__ __forceinline__ void sca_records(const DomainLaunch& a, const ScaTileLaunch& t) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t item = static_cast<uint64_t>(blockIdx.x) * 4u + (threadIdx.x >> 5);
  const uint32_t S = a.geo.S, planes = a.geo.planes, n_units = a.geo.W / 8u;
  if (item >= static_cast<uint64_t>(t.n_rec) * S) return;  // whole warps
  const uint32_t r = static_cast<uint32_t>(item / S), sample = static_cast<uint32_t>(item - static_cast<uint64_t>(r) * S);
  const size_t slot = static_cast<size_t>(a.clock->next_time) + t.rec_offset + r;
  if (slot >= a.n_times || a.times[slot] > a.clock->sweep + t.offset + t.n) return;  // whole warps
  const ScaPart* mine = t.parts + (static_cast<size_t>(r) * S + sample) * t.tiles * planes;
  const ScaPart* after = t.parts + (static_cast<size_t>(t.n_rec) * S + sample) * t.tiles * planes;
  long long hops[4] = {0, 0, 0, 0};
  for (uint32_t p = 0; p < planes; ++p) {
    long long H = 0, s1 = 0, ov = 0;
    __int128 s2 = 0;
    for (uint32_t j0 = 0; j0 < t.tiles; j0 += 32u) {
      const uint32_t j = j0 + lane;
      const bool in = j < t.tiles;
      ScaPart q = {};
      if (in) {
        q = mine[static_cast<size_t>(j) * planes + p];
        if (p == 0 && a.count_hops) {
#pragma unroll
          for (int k = 0; k < 4; ++k)
            hops[k] += static_cast<long long>(q.hops[k]) - after[static_cast<size_t>(j) * planes].hops[k];
        }
      }
      long long incl = q.tot;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const long long v = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= static_cast<uint32_t>(d)) incl += v;
      }
      const long long h = H + incl - q.tot, n = in ? 256ll * min(t.units, n_units - j * t.units) : 0ll;
      s1 += q.s1 + h * n;
      s2 += static_cast<__int128>(q.s2) + static_cast<__int128>(2 * h) * q.s1 + static_cast<__int128>(h) * h * n;
      ov += q.ov;
      H += __shfl_sync(0xffffffffu, incl, 31);
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      s1 += __shfl_xor_sync(0xffffffffu, s1, d);
      ov += __shfl_xor_sync(0xffffffffu, ov, d);
      const unsigned long long lo = __shfl_xor_sync(0xffffffffu, static_cast<unsigned long long>(s2), d);
      const unsigned long long hi =
          __shfl_xor_sync(0xffffffffu, static_cast<unsigned long long>(static_cast<unsigned __int128>(s2) >> 64), d);
      s2 += static_cast<__int128>((static_cast<unsigned __int128>(hi) << 64) | lo);
    }
    if (lane == 0u) {
      const size_t e = (slot * S + sample) * planes + p;
      a.tab_sh[e] = s1;
      a.tab_sh2[2 * e] = static_cast<uint64_t>(static_cast<unsigned __int128>(s2));
      a.tab_sh2[2 * e + 1] = static_cast<uint64_t>(static_cast<unsigned __int128>(s2) >> 64);
      if (a.ex.snap) a.ex.tab_ac[e] = ov;
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) hops[k] += __shfl_xor_sync(0xffffffffu, hops[k], d);
    if (lane == 0u)
      a.ex.tab_cnt[(slot * S + sample) * 4 + k] =
          static_cast<int64_t>(a.counters[4ull * sample + k]) + hops[k];
  }
}

__global__ void __launch_bounds__(128) k_sca_records(const DomainLaunch a, const ScaTileLaunch t, uint32_t advance) {
  sca_records(a, t);
  if (!advance) return;
  __syncthreads();
  __threadfence();
  if (threadIdx.x == 0u && atomicInc(&a.clock->done, gridDim.x - 1u) == gridDim.x - 1u)
    advance_clock(a.clock, a.times, a.n_times, advance);
}

// The first and last unit of every tile, from the lattice: one thread per 16 bytes.
__global__ void k_sca_halo(const uint32_t* state, uint32_t* halo, uint32_t S, uint32_t planes, uint32_t W,
                           uint32_t tiles, uint32_t units) {
  const size_t total = static_cast<size_t>(S) * tiles * 2u * planes * 2u;
  const uint32_t n_units = W / 8;
  for (size_t k = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; k < total;
       k += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const uint32_t half = k & 1u;
    size_t r = k >> 1;
    const uint32_t p = static_cast<uint32_t>(r % planes);
    r /= planes;
    const uint32_t edge = static_cast<uint32_t>(r & 1u);
    r >>= 1;
    const uint32_t tile = static_cast<uint32_t>(r % tiles), sample = static_cast<uint32_t>(r / tiles);
    const uint32_t first = tile * units, u = edge ? min(first + units, n_units) - 1u : first;
    reinterpret_cast<uint4*>(halo)[k] =
        reinterpret_cast<const uint4*>(state + (static_cast<size_t>(sample) * planes + p) * W + 8u * u)[half];
  }
}

template <uint32_t MODEL, bool DIS, bool COUNT, uint32_t FAST, bool PQ = false>
cudaError_t launch_tile(const DomainLaunch& a, const ScaTileLaunch& t, uint32_t upt, cudaStream_t st) {
  if constexpr (FAST != kScaAny) {
    if (upt == 2u) {
      k_sca_tile<MODEL, DIS, COUNT, FAST, PQ, 2><<<t.tiles * a.geo.S, 32, 0, st>>>(a, t);
      return cudaGetLastError();
    }
  }
  k_sca_tile<MODEL, DIS, COUNT, FAST, PQ, 1><<<t.tiles * a.geo.S, 32, 0, st>>>(a, t);
  return cudaGetLastError();
}

// FAST of a ring without disorder (kScaAny: a rate 0, "always" or of more than two planes).
uint32_t sca_fast(uint32_t p, uint32_t q) {
  const auto two_planes = [](uint32_t t) { return t != 0u && t != 0xFFFFFFFFu && (t & 0x3FFFFFFFu) == 0u; };
  return two_planes(p) && two_planes(q) ? 4u * (p >> 30) + (q >> 30) : kScaAny;
}

template <bool COUNT>
cudaError_t launch_ring(const DomainLaunch& a, const ScaTileLaunch& t, uint32_t upt, cudaStream_t st) {
  if (a.dis == kDisBimodal) return launch_tile<kRing, true, COUNT, kScaAny>(a, t, upt, st);
  if (a.dis == kDisBimodalPQ) return launch_tile<kRing, true, COUNT, kScaAny, true>(a, t, upt, st);
  switch (sca_fast(a.rates.p, a.rates.q)) {
    case 5: return launch_tile<kRing, false, COUNT, 5>(a, t, upt, st);
    case 6: return launch_tile<kRing, false, COUNT, 6>(a, t, upt, st);
    case 7: return launch_tile<kRing, false, COUNT, 7>(a, t, upt, st);
    case 9: return launch_tile<kRing, false, COUNT, 9>(a, t, upt, st);
    case 10: return launch_tile<kRing, false, COUNT, 10>(a, t, upt, st);
    case 11: return launch_tile<kRing, false, COUNT, 11>(a, t, upt, st);
    case 13: return launch_tile<kRing, false, COUNT, 13>(a, t, upt, st);
    case 14: return launch_tile<kRing, false, COUNT, 14>(a, t, upt, st);
    case 15: return launch_tile<kRing, false, COUNT, 15>(a, t, upt, st);
    default: return launch_tile<kRing, false, COUNT, kScaAny>(a, t, upt, st);
  }
}

cudaError_t launch_tiles(const DomainLaunch& a, const ScaTileLaunch& t, uint32_t upt, cudaStream_t st) {
  (void)cudaGetLastError();
  if (a.model == kTwoLane) {  // two lanes always count hops and turns
    if (a.dis == kDisCrossing) return launch_tile<kTwoLane, true, true, kScaAny, true>(a, t, upt, st);
    return a.dis == kDisTurning ? launch_tile<kTwoLane, true, true, kScaAny>(a, t, upt, st)
                                : launch_tile<kTwoLane, false, true, kScaAny>(a, t, upt, st);
  }
  return a.count_hops ? launch_ring<true>(a, t, upt, st) : launch_ring<false>(a, t, upt, st);
}

}  // namespace

size_t sca_smem_bytes(uint32_t W, uint32_t planes, uint32_t quenched_planes) {
  return static_cast<size_t>(W) * 4u * (planes + quenched_planes) + static_cast<size_t>(planes) * (W / 8u) * 4u;
}

ScaTiles sca_tiles(uint32_t model, uint32_t dis, uint32_t p_thr, uint32_t q_thr, uint32_t W, uint32_t S) {
  const uint32_t n = W / 8u;
  const auto cut = [n](uint32_t upt, uint32_t most) {
    ScaTiles t;
    t.upt = upt;
    t.tiles = (n + most - 1u) / most;
    t.units = (n + t.tiles - 1u) / t.tiles;  // as even as the ring allows
    t.tiles = (n + t.units - 1u) / t.units;
    return t;
  };
  const ScaTiles one = cut(1, 30u);
  if (model == kRing && dis == kDisNone && sca_fast(p_thr, q_thr) != kScaAny)
    return static_cast<uint64_t>(one.tiles) * S <= kScaManyTiles ? one : cut(2, 62u);
  // kinds whose warps run to their most undecided bond (or longest queue of lane changes)
  ScaTiles best = one;
  for (uint32_t u = 29u; u >= kScaFewUnits; --u) {
    const ScaTiles t = cut(1, u);
    if (static_cast<uint64_t>(t.tiles) * S <= kScaFewTiles) best = t;
  }
  return best;
}

size_t sca_halo_words(const ScaTiles& t, uint32_t S, uint32_t planes) {
  return t.tiles == 1u ? 0u : static_cast<size_t>(2u) * S * t.tiles * 2u * planes * 8u;
}

uint32_t sca_max_records(const uint64_t* times, size_t n, uint32_t S, uint32_t tiles, uint32_t planes,
                         uint32_t* any_sweeps) {
  *any_sweeps = kScaTileSweeps;
  uint32_t most = 0;  // sample times in any kScaTileSweeps consecutive sweeps
  for (size_t i = 0, j = 0; j < n; ++j) {
    while (times[j] - times[i] >= kScaTileSweeps) ++i;
    most = std::max(most, static_cast<uint32_t>(j - i + 1));
  }
  if (tiles == 1u) return most;  // written by the tiles themselves
  // no more than 64 MB or a record's worth
  const uint64_t one = static_cast<uint64_t>(S) * tiles * planes * sizeof(ScaPart);
  const uint64_t room = std::max<uint64_t>(1u, (64ull << 20) / one);
  if (room >= most) return most;
  *any_sweeps = static_cast<uint32_t>(room);  // at most a record a sweep
  return static_cast<uint32_t>(room);
}

cudaError_t launch_sca_halo(const DomainLaunch& a, const ScaTiles& tiles, uint32_t* halo, cudaStream_t st) {
  (void)cudaGetLastError();
  const size_t n16 = sca_halo_words(tiles, a.geo.S, a.geo.planes) / 8u;
  const uint32_t blocks = static_cast<uint32_t>(std::min<size_t>((n16 + 255u) / 256u, 152u * 16u));
  k_sca_halo<<<blocks, 256, 0, st>>>(a.state, halo, a.geo.S, a.geo.planes, a.geo.W, tiles.tiles, tiles.units);
  return cudaGetLastError();
}

cudaError_t launch_sca(const DomainLaunch& a, const ScaTiles& tiles, ScaRun& run, cudaStream_t st,
                       uint32_t* launches) {
  const size_t half = sca_halo_words(tiles, a.geo.S, a.geo.planes) / 2u;
  uint32_t rec = 0;
  (void)cudaGetLastError();
  if (tiles.tiles > 1u && run.half == kScaNoHalo) {
    const cudaError_t e = launch_sca_halo(a, tiles, run.halo, st);
    if (e != cudaSuccess) return e;
    ++*launches;
  }
  uint32_t half_now = run.half == kScaNoHalo ? 0u : run.half;
  run.half = kScaNoHalo;  // until all is launched
  for (uint32_t done = 0; done < a.n_sweeps;) {
    ScaTileLaunch t;
    t.tiles = tiles.tiles;
    t.units = tiles.units;
    t.n = std::min({kScaTileSweeps, run.max_sweeps, a.n_sweeps - done});
    if (run.replayed) t.n = std::min(t.n, run.any_sweeps);
    // a launch that may run at any sweep finds its records from the clock, which then moves with every launch
    t.offset = run.replayed ? 0u : done;
    t.rec_offset = run.replayed ? 0u : rec;
    t.n_rec = run.replayed ? std::min(t.n, run.max_records) : 0u;
    while (!run.replayed && rec + t.n_rec < run.n_times && run.times[rec + t.n_rec] - run.sweep <= done + t.n) {
      if (t.n_rec == run.max_records) {  // the launch ends before the first record it has no room for
        t.n = static_cast<uint32_t>(run.times[rec + t.n_rec - 1] - run.sweep) - done;
        break;
      }
      ++t.n_rec;
    }
    t.halo_in = run.halo + half_now * half;
    t.halo_out = run.halo + (half_now ^ 1u) * half;
    t.parts = run.parts;
    cudaError_t e = launch_tiles(a, t, tiles.upt, st);
    if (e != cudaSuccess) return e;
    ++*launches;
    uint32_t advance = done + t.n < a.n_sweeps ? 0u : a.n_sweeps;
    if (run.replayed) advance = t.n;
    if (t.n_rec && tiles.tiles > 1u) {
      const uint64_t items = static_cast<uint64_t>(t.n_rec) * a.geo.S;
      k_sca_records<<<static_cast<uint32_t>((items + 3u) / 4u), 128, 0, st>>>(a, t, advance);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      ++*launches;
    } else if (advance) {
      if ((e = launch_advance(a.clock, a.times, a.n_times, advance, st)) != cudaSuccess) return e;
      ++*launches;
    }
    half_now ^= 1u;
    rec += t.n_rec;
    done += t.n;
  }
  run.half = half_now;
  return cudaSuccess;
}

}  // namespace asep
