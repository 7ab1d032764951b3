// asep_batch_wide.cu -- the batch kernel for CTAs of 513 to 1024 threads.
#include "asep_batch.cuh"

namespace asep {

cudaError_t batch_launch_wide(const DomainLaunch* jobs, const uint32_t* items, uint32_t n_items, uint32_t* queue,
                              uint32_t threads, uint32_t ctas, size_t smem, cudaStream_t st) {
  return batch_launch<1024>(jobs, items, n_items, queue, threads, ctas, smem, st);
}

cudaError_t batch_occupancy_wide(uint32_t threads, size_t smem, int* n) { return batch_occupancy<1024>(threads, smem, n); }

cudaError_t batch_warm_wide(uint32_t* queue, cudaStream_t st) { return batch_warm<1024>(queue, st); }

}  // namespace asep
