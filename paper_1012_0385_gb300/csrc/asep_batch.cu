// asep_batch.cu -- launches of the persistent batch kernel (asep_batch.cuh).
#include "asep_batch.cuh"

namespace asep {

cudaError_t launch_batch(const DomainLaunch* jobs, const uint32_t* items, uint32_t n_items, uint32_t* queue,
                         uint32_t threads, uint32_t ctas, size_t smem, cudaStream_t st) {
  (void)cudaGetLastError();
  const cudaError_t e = cudaMemsetAsync(queue, 0, sizeof(uint32_t), st);
  if (e != cudaSuccess) return e;
  return threads <= 512 ? batch_launch<512>(jobs, items, n_items, queue, threads, ctas, smem, st)
                        : batch_launch_wide(jobs, items, n_items, queue, threads, ctas, smem, st);
}

// One empty launch of each batch kernel (no items, no jobs) on `st`: loads
// the kernels' code on the current device and lets the driver size their
// per-thread local memory, so later batch steps start without either.
cudaError_t warm_batch_kernels(uint32_t* queue, cudaStream_t st) {
  (void)cudaGetLastError();
  cudaError_t e;
  if ((e = cudaMemsetAsync(queue, 0, sizeof(uint32_t), st)) != cudaSuccess) return e;
  if ((e = batch_warm<512>(queue, st)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(queue, 0, sizeof(uint32_t), st)) != cudaSuccess) return e;
  if ((e = batch_warm_wide(queue, st)) != cudaSuccess) return e;
  return warm_advance_batch(st);
}

int batch_ctas_per_sm(uint32_t threads, size_t smem) {
  int n = 0;
  const cudaError_t e = threads <= 512 ? batch_occupancy<512>(threads, smem, &n) : batch_occupancy_wide(threads, smem, &n);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();  // do not leave the failure for the next launch check to find
    return 0;
  }
  return n;
}

}  // namespace asep
