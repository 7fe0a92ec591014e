// Host-side entry points of the kernel translation units.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace chem {

struct Dev;

// Phase indices of chem_stats.phase_ms.
enum Phase { PH_BEGIN = 0, PH_RELEASE, PH_DIFFUSE, PH_SORT, PH_GATHER, PH_SEARCH, PH_REACT,
             PH_PERSISTENT, N_PHASES };

struct LaunchCfg {
  int stream_blocks;      // grid of the grid-stride phases (release, diffuse, gather)
  int search_blocks;      // grid of the pair search
  int sort_blocks;        // resident CTAs of a sort pass
  int persistent_blocks;  // CTAs of the persistent step kernel (resident together)
  int cluster_blocks;     // CTAs of its one-cluster form (0: not available)
  int search_tps;         // pair search: 1 one thread per home species, 0 cell tiles,
                          // 2 both launched, the step's choice runs (adaptive)
  int small;              // few species: one search kernel and one reaction kernel per step
};

// Up to n_steps steps in one launch of one cluster, or of one CTA per SM. They are the steps from
// `done` on of a group of `align` (whose ends the species' order follows; done + n_steps is
// a multiple of it), and end before a step on more than `most` species.
struct StepRun {
  bool cluster;
  int n_steps, align, done;
  uint32_t most;
};

// kernels_exact.cu (FP64 arithmetic without contraction)
cudaError_t enqueue_begin(const Dev& d, cudaStream_t s);
cudaError_t enqueue_sort_pass(const Dev& d, int pass, int blocks, cudaStream_t s);
cudaError_t sort_pass_occupancy(int* blocks_per_sm);
// One SBS step. `first`: the step begins with its own begin kernel (else the previous
// step's last kernel began it); `last`: its last kernel does not begin the next step.
cudaError_t enqueue_step_f64(const Dev& d, const LaunchCfg& lc, cudaStream_t s, cudaEvent_t* ev, bool first,
                             bool last);
cudaError_t enqueue_steps_f64(const Dev& d, const LaunchCfg& lc, const StepRun& r, cudaStream_t s);
// Sets the shared-memory limits of the precision's kernels; CTAs of the two forms above.
cudaError_t step_kernel_limits_f64(int* blocks_per_sm, int* cluster_blocks);
cudaError_t enqueue_set_t_end(const Dev& d, const double* t_end_dev, cudaStream_t s);
// one device thread waits, up to limit_s, for a word nothing writes (then CHEM_ETIMEOUT)
cudaError_t enqueue_bounded_wait(const Dev& d, double limit_s, cudaStream_t s);

// the pair acceptance test on given squared separations (diagnostic; one per precision)
cudaError_t enqueue_check_accept_f64(const Dev& d, uint32_t n, uint32_t step, double dt, const double* d0sq,
                                     const double* d1sq, const int32_t* rxn, const uint32_t* id_lo,
                                     const uint32_t* id_hi, uint8_t* out, cudaStream_t s);
cudaError_t enqueue_check_accept_f32l(const Dev& d, uint32_t n, uint32_t step, double dt, const double* d0sq,
                                      const double* d1sq, const int32_t* rxn, const uint32_t* id_lo,
                                      const uint32_t* id_hi, uint8_t* out, cudaStream_t s);

// homog.cu: homogeneous (beam-off) stage of the trains with Train::hx_sel set
cudaError_t enqueue_homogeneous(const Dev& d, int blocks, cudaStream_t s);

// state.cu: the live species of one train packed in device order. The positions' rows lie in up
// to three buffers one after the other (working memory that is idle between steps), which have
// room for `most` species like the other two arrays; rows past it are not written.
struct PackOut {
  static constexpr uint32_t SEGS = 3;
  uint32_t most;
  int32_t* type;
  uint32_t* id;
  double* xyz[SEGS];
  uint32_t rows[SEGS];
};
// counts: one word per chunk of slots and one for the total (counts[pack_counts(n)]).
uint32_t pack_counts(uint32_t n);
cudaError_t enqueue_pack_count(const Dev& d, uint32_t train, uint32_t n_slots, uint32_t n, uint32_t* counts,
                               cudaStream_t s);
// Both at once by one CTA, for at most PACK_FEW slots; the number of live species in *live.
constexpr uint32_t PACK_FEW = 4096;
cudaError_t enqueue_pack_few(const Dev& d, uint32_t train, uint32_t n_slots, uint32_t n, uint32_t* live,
                             const PackOut& out, cudaStream_t s);
cudaError_t enqueue_pack_write(const Dev& d, uint32_t train, uint32_t n_slots, uint32_t n, const uint32_t* counts,
                               const PackOut& out, cudaStream_t s);

// kernels_f32l.cu (FP32-local mode)
cudaError_t enqueue_step_f32l(const Dev& d, const LaunchCfg& lc, cudaStream_t s, cudaEvent_t* ev, bool first,
                              bool last);
cudaError_t enqueue_steps_f32l(const Dev& d, const LaunchCfg& lc, const StepRun& r, cudaStream_t s);
cudaError_t step_kernel_limits_f32l(int* blocks_per_sm, int* cluster_blocks);

}  // namespace chem
