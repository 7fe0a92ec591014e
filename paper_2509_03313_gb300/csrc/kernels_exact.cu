// FP64-mode kernels and the precision-independent ones (step begin, sort passes).
// Built with --fmad=false: together with the explicit _rn intrinsics in phases.cuh
// this keeps the FP64 mode's rounding identical to the FP64 reference's.
#include "kernels.cuh"

namespace chem {

__global__ void __launch_bounds__(256) k_begin(const __grid_constant__ Dev d) {
  __shared__ BeginSmem sb;
  phase_begin(d, sb);
}

__global__ void __launch_bounds__(SORT_THREADS) k_sort_pass(const __grid_constant__ Dev d, int pass) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // everything the pass starts from is read in one round: the tile, the status, the histograms
  const uint32_t tile = threadIdx.x == 0 ? atomicAdd(&d.g->tile_ctr[pass], 1u) : 0u;
  const uint32_t n = d.g->n_total;
  const uint32_t active = active_passes(d, n);
  if (!block_status_ok(d)) return;
  phase_sort_pass(d, pass, active, n, tile, *reinterpret_cast<SortSmem*>(smem_raw), blockIdx.x == 0);
}

__global__ void __launch_bounds__(256) k_set_t_end(const __grid_constant__ Dev d, const double* t_end) {
  __shared__ EndSmem sm;
  for (uint32_t b = threadIdx.x; b < d.n_trains; b += blockDim.x) d.trains[b].t_end = t_end[b];
  phase_look_ahead(d, sm);
}

cudaError_t enqueue_begin(const Dev& d, cudaStream_t s) {
  k_begin<<<1, 256, 0, s>>>(d);
  return cudaGetLastError();
}

cudaError_t enqueue_sort_pass(const Dev& d, int pass, int blocks, cudaStream_t s) {
  k_sort_pass<<<blocks, SORT_THREADS, sizeof(SortSmem), s>>>(d, pass);
  return cudaGetLastError();
}

cudaError_t sort_pass_occupancy(int* blocks_per_sm) {
  cudaError_t e = cudaFuncSetAttribute(k_sort_pass, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(sizeof(SortSmem)));
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_sort_pass, SORT_THREADS,
                                                       sizeof(SortSmem));
}

// One thread waits for a word that nothing writes (Global::never_set), polling it until
// limit_ns of the global timer have passed, then raises CHEM_ETIMEOUT: the error path of
// every bounded device wait of the library, without a fault.
__global__ void k_bounded_wait(const __grid_constant__ Dev d, unsigned long long limit_ns) {
  if (threadIdx.x != 0) return;
  unsigned long long t0, t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  const volatile uint32_t* flag = &d.g->never_set;
  for (;;) {
    if (*flag != 0u) return;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    if (t - t0 > limit_ns) {
      raise_status(d.g, CHEM_ETIMEOUT);
      return;
    }
    __nanosleep(1000);
  }
}

cudaError_t enqueue_bounded_wait(const Dev& d, double limit_s, cudaStream_t s) {
  k_bounded_wait<<<1, 32, 0, s>>>(d, static_cast<unsigned long long>(limit_s * 1e9));
  return cudaGetLastError();
}

cudaError_t enqueue_set_t_end(const Dev& d, const double* t_end_dev, cudaStream_t s) {
  k_set_t_end<<<1, 256, 0, s>>>(d, t_end_dev);
  return cudaGetLastError();
}

cudaError_t enqueue_step_f64(const Dev& d, const LaunchCfg& lc, cudaStream_t s, cudaEvent_t* ev, bool first,
                             bool last) {
  return enqueue_phases<false>(d, lc, s, ev, first, last);
}

cudaError_t enqueue_steps_f64(const Dev& d, const LaunchCfg& lc, const StepRun& r, cudaStream_t s) {
  return enqueue_steps<false>(d, lc, r, s);
}

cudaError_t step_kernel_limits_f64(int* blocks_per_sm, int* cluster_blocks) {
  return step_kernel_limits<false>(blocks_per_sm, cluster_blocks);
}

cudaError_t enqueue_check_accept_f64(const Dev& d, uint32_t n, uint32_t step, double dt, const double* d0sq,
                                     const double* d1sq, const int32_t* rxn, const uint32_t* id_lo,
                                     const uint32_t* id_hi, uint8_t* out, cudaStream_t s) {
  return enqueue_check_accept<false>(d, n, step, dt, d0sq, d1sq, rxn, id_lo, id_hi, out, s);
}

}  // namespace chem
