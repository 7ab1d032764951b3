// asep_batch.cuh -- the persistent batch kernel: CTAs take (context, sample
// group) items of many contexts from a work queue and run them with the
// resident group (asep_resident.cuh).  Its two block-size classes are compiled
// in a file each (asep_batch.cu, asep_batch_wide.cu).
#pragma once

#include <cstdint>

#include "asep_device.cuh"
#include "asep_domain.cuh"
#include "asep_internal.h"
#include "asep_resident.cuh"

namespace asep {
namespace {

// Runtime dispatch of one group to the matching instantiation.
template <bool PIN>
__device__ __forceinline__ void run_group_any(const DomainLaunch& a, uint32_t group, unsigned char* smem) {
  const uint64_t s0 = a.clock->sweep;
  const uint32_t cur = a.clock->next_time, n = a.n_sweeps;
  if (a.model == kTwoLane) {
    if (a.dis == kDisTurning) run_group<kTwoLane, kDisTurning, true, 0, PIN>(a, group, smem, s0, cur, n);
    else if (a.dis == kDisCrossing) run_group<kTwoLane, kDisCrossing, true, 0, PIN>(a, group, smem, s0, cur, n);
    else run_group<kTwoLane, kDisNone, true, 0, PIN>(a, group, smem, s0, cur, n);
  } else if (a.dis == kDisBimodal) {
    if (a.count_hops) run_group<kRing, kDisBimodal, true, 0, PIN>(a, group, smem, s0, cur, n);
    else run_group<kRing, kDisBimodal, false, 0, PIN>(a, group, smem, s0, cur, n);
  } else if (a.dis == kDisBimodalPQ) {
    if (a.count_hops) run_group<kRing, kDisBimodalPQ, true, 0, PIN>(a, group, smem, s0, cur, n);
    else run_group<kRing, kDisBimodalPQ, false, 0, PIN>(a, group, smem, s0, cur, n);
  } else if (a.Cp == 256) {
    if (a.count_hops) run_group<kRing, kDisNone, true, 256, PIN>(a, group, smem, s0, cur, n);
    else run_group<kRing, kDisNone, false, 256, PIN>(a, group, smem, s0, cur, n);
  } else {
    if (a.count_hops) run_group<kRing, kDisNone, true, 0, PIN>(a, group, smem, s0, cur, n);
    else run_group<kRing, kDisNone, false, 0, PIN>(a, group, smem, s0, cur, n);
  }
}

// Persistent batch kernel: CTAs take (job, group) items until the queue is
// empty.  Items are ordered largest first by the host.  The descriptor of the
// current item is copied to shared memory once.  Two block-size classes: up
// to 512 threads (128 registers available) and up to 1024.
template <uint32_t MAXT>
__global__ void __maxnreg__(MAXT == 512 ? 104 : 64) k_batch(const DomainLaunch* jobs, const uint32_t* items, uint32_t n_items,
                                                uint32_t* queue) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint32_t item_idx;
  __shared__ DomainLaunch desc;
  for (;;) {
    if (threadIdx.x == 0) item_idx = atomicAdd(queue, 1u);
    __syncthreads();
    const uint32_t i = item_idx;
    if (i >= n_items) break;
    const uint32_t it = items[i];
    if (threadIdx.x == 0) desc = jobs[it >> kItemGroupBits];
    __syncthreads();
    run_group_any<MAXT == 512>(desc, it & (kItemMaxGroups - 1u), smem_raw);
  }
}

// One block-size class: dynamic shared memory opt-in (the kernel's static
// shared memory -- the item index and the descriptor copy -- counts against
// the same limit), launch, occupancy.
template <uint32_t MAXT>
cudaError_t batch_attr() {
  return allow_smem(k_batch<MAXT>, kSmemOptIn - sizeof(DomainLaunch) - 64);
}

template <uint32_t MAXT>
cudaError_t batch_launch(const DomainLaunch* jobs, const uint32_t* items, uint32_t n_items, uint32_t* queue,
                         uint32_t threads, uint32_t ctas, size_t smem, cudaStream_t st) {
  const cudaError_t e = batch_attr<MAXT>();
  if (e != cudaSuccess) return e;
  k_batch<MAXT><<<ctas, threads, smem, st>>>(jobs, items, n_items, queue);
  return cudaGetLastError();
}

template <uint32_t MAXT>
cudaError_t batch_occupancy(uint32_t threads, size_t smem, int* n) {
  const cudaError_t e = batch_attr<MAXT>();
  return e != cudaSuccess ? e
                          : cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k_batch<MAXT>, static_cast<int>(threads), smem);
}

template <uint32_t MAXT>
cudaError_t batch_warm(uint32_t* queue, cudaStream_t st) {
  k_batch<MAXT><<<1, 32, 0, st>>>(nullptr, nullptr, 0u, queue);
  return cudaGetLastError();
}

}  // namespace

// The class of 513 to 1024 threads (asep_batch_wide.cu).
cudaError_t batch_launch_wide(const DomainLaunch* jobs, const uint32_t* items, uint32_t n_items, uint32_t* queue,
                              uint32_t threads, uint32_t ctas, size_t smem, cudaStream_t st);
cudaError_t batch_occupancy_wide(uint32_t threads, size_t smem, int* n);
cudaError_t batch_warm_wide(uint32_t* queue, cudaStream_t st);

}  // namespace asep
