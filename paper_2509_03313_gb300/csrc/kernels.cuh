// Kernels of one SBS step: one kernel per phase (captured into a CUDA graph of several
// steps), and a kernel that runs the same phases for several steps of every train with
// barriers in between.
#pragma once
#include <type_traits>

#include "launch.h"
#include "phases.cuh"
#include "search_cells.cuh"

namespace chem {

template <bool F32L>
__global__ void __launch_bounds__(256) k_diffuse(const __grid_constant__ Dev d) {
  __shared__ uint32_t hist[MAX_PASSES][RADIX];
  phase_diffuse<F32L>(d, hist, whole_grid());
}

template <bool F32L>
__global__ void __launch_bounds__(256) k_gather(const __grid_constant__ Dev d) {
  phase_gather<F32L>(d, whole_grid());
}

template <bool F32L>
__global__ void __launch_bounds__(256, 4) k_search(const __grid_constant__ Dev d) {
  __shared__ ScSmem<8> sm;
  phase_search_cells<F32L, 8>(d, sm);
}

constexpr int TPS_WARPS = 4;  // warps per CTA of the one-thread-per-species search

template <bool F32L, int W>
union SearchSmem {
  TpsSmem<F32L, W> tps;
  GrpSmem<W> grp;
  ScSmem<W> cells;
};

// One thread per home species, or several lanes per home when the launch has two or more lanes
// for each (the CTAs of the launch are resident together).
template <bool F32L, int W>
__device__ __forceinline__ void search_species(const Dev& d, SearchSmem<F32L, W>& sm) {
  const int lg = lanes_per_home_lg(d.g->n_total - d.g->n_dead, gridDim.x * blockDim.x);
  // warps of one CTA are a grid apart, so that few homes spread over all CTAs
  if (lg > 0) phase_search_groups<F32L, W>(d, sm.grp, lg, (threadIdx.x >> 5) * gridDim.x + blockIdx.x, gridDim.x * W);
  else phase_search_tps<F32L, W>(d, sm.tps);
}

template <bool F32L>
__global__ void __launch_bounds__(32 * TPS_WARPS, F32L ? 8 : 7) k_search_tps(const __grid_constant__ Dev d) {
  __shared__ SearchSmem<F32L, TPS_WARPS> sm;
  if (d.g->search_cells_now) return;  // this step runs the cell tiles (grid-uniform)
  search_species<F32L, TPS_WARPS>(d, sm);
}

// Either mapping in one launch, for steps of at most ONE_CTA_SPECIES species, which cost
// their launches more than their work (on 1e6 species two kernels are the faster form: the
// cell tiles want larger CTAs).
template <bool F32L>
__global__ void __launch_bounds__(32 * TPS_WARPS, F32L ? 8 : 7) k_search_any(const __grid_constant__ Dev d) {
  __shared__ SearchSmem<F32L, TPS_WARPS> sm;
  if (d.g->search_cells_now) phase_search_cells<F32L, TPS_WARPS>(d, sm.cells);
  else search_species<F32L, TPS_WARPS>(d, sm);
}

// Reaction resolution, the step's end and (begin_next) the next step's begin, one CTA.
struct alignas(16) ReactEndSmem {
  union {
    ReactAllSmem react;
    BeginSmem begin;
  };
  EndSmem end;
};
constexpr int REACT_END_THREADS = 512;
constexpr size_t REACT_END_BYTES = sizeof(ReactEndSmem) + react_all_bytes(RC_CAP);
static_assert(sizeof(ReactEndSmem) % 16 == 0, "the buffer behind it is aligned");
static_assert(REACT_END_BYTES <= 227 * 1024, "shared memory of one CTA");

template <bool F32L>
__global__ void __launch_bounds__(REACT_END_THREADS) k_react_end(const __grid_constant__ Dev d, int begin_next) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  ReactEndSmem& sm = *reinterpret_cast<ReactEndSmem*>(smem_raw);
  phase_react_all<F32L>(d, sm.react, reinterpret_cast<uint32_t*>(smem_raw + sizeof(ReactEndSmem)), RC_CAP,
                        *d.tables);
  phase_end_step(d, sm.end);
  if (begin_next) phase_begin(d, sm.begin);
}

// ---- several steps in one launch
// The steps of few species are launches and latency: seven to eleven kernels, each a chain of a
// few dependent L2 accesses. Here CTAs that are resident together run the phases of many steps
// with a barrier in between: 16 CTAs of one cluster with the hardware's cluster barrier for a
// few thousand species, or one CTA per SM with a barrier in global memory. The search gives
// every home at least two lanes; reaction resolution, the step's end and the next step's
// begin are CTA 0's. A launch ends by itself when no train has anything left to do, or before
// a step whose species (what arrives included) are more than its form is for. A step of
// 2,000 species takes 27 to 30 us (as kernels 52 to 60), of 32,000 track species 73 (105);
// at 31,000 species the sort takes 19 us, the search 13 to 35, reaction resolution 10.
constexpr int STEP_WARPS = PERSIST_THREADS / 32;
constexpr uint32_t STEP_REACT_CAP = 1024;  // accepted pairs of a step resolved in shared memory

union StepSmem {
  uint32_t hist[MAX_PASSES][RADIX];
  SortSmemP sort;
  struct { SortOneSmem one; BlockSortSmem bs; ScanSmem ss; } sort_one;
  GrpSmem<STEP_WARPS> grp;
  ScSmem<STEP_WARPS> cells;
  struct {
    PlanSmem<PLAN_TRAINS> plan;
    ReactAllSmem react;
    EndSmem end;
    alignas(16) uint32_t sbuf[react_all_bytes(STEP_REACT_CAP) / 4];
  } react;
};
static_assert(sizeof(StepSmem) <= 200 * 1024, "shared memory of one CTA");

// Barrier over all CTAs of a cooperative launch: arrivals are counted up over the whole launch
// (the last CTA to leave clears the count). The wait is bounded: past the limit CHEM_ETIMEOUT is
// raised and this CTA waits no more, so a launch always ends.
struct GridBarrier {
  uint32_t target = 0;
  bool broken = false;
  __device__ __forceinline__ void sync(const Dev& d) {
    __syncthreads();
    if (threadIdx.x == 0) {
      target += gridDim.x;
      __threadfence();
      atomicAdd(&d.g->bar_count, 1u);
      if (!broken) {
        const long long t0 = clock64();
        while (static_cast<int32_t>(ld_acquire_u32(&d.g->bar_count) - target) < 0) {
          if (clock64() - t0 > SPIN_LIMIT_CYCLES) {
            raise_status(d.g, CHEM_ETIMEOUT);
            broken = true;
            break;
          }
        }
      }
      __threadfence();
    }
    __syncthreads();
  }
  // Arrives without waiting: for a CTA that has written nothing the others read before it.
  __device__ __forceinline__ void arrive(const Dev& d) {
    if (threadIdx.x == 0) {
      target += gridDim.x;
      atomicAdd(&d.g->bar_count, 1u);
    }
  }
  __device__ __forceinline__ void leave(const Dev& d) {
    if (threadIdx.x == 0 && atomicAdd(&d.g->bar_left, 1u) + 1u == gridDim.x) {
      d.g->bar_count = 0u;
      d.g->bar_left = 0u;
    }
  }
};

// Barrier over the CTAs of one cluster (release / acquire of all memory among them). The aligned
// instructions need the warp together, which the phases' ends (work of lane or thread 0) leave open.
struct ClusterBarrier {
  __device__ __forceinline__ void sync(const Dev&) {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
  __device__ __forceinline__ void leave(const Dev&) {}
};

// Reaction resolution, the step's end and (begin_next) the next step's begin where one CTA does
// not do it (LaunchCfg::small), as one cooperative launch of a CTA per SM: matching over all
// CTAs, the serial part in CTA 0 while the last CTA plans the next step, products over the others, commit. It
// takes 30 us on 1e6 FP32-local species and 40 on 4.1e6; as four kernels (matching, serial,
// products, end and begin) with the events sorted by one CTA it took 42 and 131.
struct ReactLeadSmem {
  SerialSmem serial;
  alignas(16) uint32_t sbuf[(RC_SMEM_BYTES > 16u * EV_SMEM_CAP ? RC_SMEM_BYTES : 16u * EV_SMEM_CAP) / 4];
};
// Batches of up to so many trains plan a step ahead: the records that fit into the shared memory
// that CTA 0's part of the launch takes anyway (more would leave the products less L1). Whole sweeps
// of 5,836 steps planned / begun after the reactions: 16 trains 117 / 122 ms, 80 trains 175 / 176.
constexpr uint32_t REACT_PLAN_TRAINS =
    static_cast<uint32_t>((sizeof(ReactLeadSmem) - sizeof(PlanSmem<1>)) / sizeof(Train)) + 1u;
static_assert(sizeof(PlanSmem<REACT_PLAN_TRAINS>) <= sizeof(ReactLeadSmem), "no more than CTA 0's part");
union ReactGridSmem {
  ReactLeadSmem lead;
  struct {
    ProductsSmem products;
    Tables tb;
  } many;
  PlanSmem<REACT_PLAN_TRAINS> plan;
  BeginSmem begin;
};
static_assert(sizeof(ReactGridSmem) + sizeof(EndSmem) <= 227 * 1024, "shared memory of one CTA");

template <bool F32L>
__global__ void __launch_bounds__(REACT_THREADS, 1) k_react_grid(const __grid_constant__ Dev d, int begin_next) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ EndSmem end;
  ReactGridSmem& sm = *reinterpret_cast<ReactGridSmem*>(smem_raw);
  GridBarrier bar;
  const uint32_t block = blockIdx.x, blocks = gridDim.x;
  const bool plan = begin_next && blocks > 2u && d.n_trains <= REACT_PLAN_TRAINS;
  const bool planner = plan && block + 1u == blocks;
  if (planner) {
    bar.arrive(d);  // it matches nothing and starts at once
    stage_next(d, sm.plan);
  } else {
    phase_match_fast(d, plan ? Span{block, blocks - 1u} : whole_grid());
    bar.sync(d);
    if (block == 0u) {
      phase_react_serial(d, sm.lead.serial, sm.lead.sbuf);
    } else {  // what the products need, while the serial part runs
      clear_products(d, sm.many.products);
      const uint32_t* src = reinterpret_cast<const uint32_t*>(d.tables);
      uint32_t* dst = reinterpret_cast<uint32_t*>(&sm.many.tb);
      for (uint32_t i = threadIdx.x; i < sizeof(Tables) / 4; i += blockDim.x) dst[i] = src[i];
    }
  }
  bar.sync(d);
  if (block != 0u && !planner)
    phase_products<F32L>(d, sm.many.products, sm.many.tb, Span{block - 1u, plan ? blocks - 2u : blocks - 1u});
  bar.sync(d);
  if (planner || (!plan && block == 0u)) {
    if (!(plan && commit_next(d, sm.plan, ~0u))) {
      __syncthreads();
      phase_end_step(d, end);
      if (begin_next) phase_begin(d, sm.begin);
    }
  }
  bar.leave(d);
}

constexpr uint32_t ANY_OUTGROWN = 2u;  // Global::any_active: there is more to do, but not in this launch

// The first step is `done` steps into a group of `align`; a step of more than `most` species is
// left to the next launch (the first is taken whatever its size: the host chose it).
template <bool F32L, bool CLUSTER>
__global__ void __launch_bounds__(PERSIST_THREADS, 1) k_steps(const __grid_constant__ Dev d, int n_steps, int align,
                                                              int done, uint32_t most) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  StepSmem& sm = *reinterpret_cast<StepSmem*>(smem_raw);
  typename std::conditional<CLUSTER, ClusterBarrier, GridBarrier>::type bar;
  const Span sp = whole_grid();
  const bool lead = sp.block == 0u;
  if (lead) phase_begin(d, sm.react.plan.begin);
  bar.sync(d);
  for (int step = 0; step < n_steps; ++step) {
    // CTA 0 alone writes these between the barriers: every CTA takes the same branches
    const uint32_t any = d.g->any_active;
    const bool idle = any != 1u;
    // (the order of the species after a run is that of launches of `align` steps: one that ends
    // early re-sorts them once more, which removes the reacted and places the last products; an
    // outgrown launch has not begun this step)
    if (idle && (any == ANY_OUTGROWN || d.n_trains > 1u || (step != 0 && (done + step) % align == 0))) break;
    const bool one = d.g->n_total <= SORT_ONE_CTA;
    phase_diffuse<F32L>(d, one ? nullptr : sm.hist, sp);  // includes the release
    bar.sync(d);
    if (one) {
      if (lead) phase_sort_one(d, sm.sort_one.one, sm.sort_one.bs, sm.sort_one.ss);
      bar.sync(d);
    } else {
      const uint32_t n = d.g->n_total, active = active_passes(d, n);
      for (int p = 0; p < d.passes; ++p) {
        if (!((active >> p) & 1u) && p + 1 < d.passes) continue;  // the same for every CTA
        const uint32_t tile = threadIdx.x == 0 ? atomicAdd(&d.g->tile_ctr[p], 1u) : 0u;
        if (block_status_ok(d)) phase_sort_pass(d, p, active, n, tile, sm.sort, lead);
        bar.sync(d);
      }
    }
    phase_gather<F32L>(d, sp);
    bar.sync(d);
    if (idle) {
      if (lead) phase_end_step(d, sm.react.end);
      break;
    }
    // CTA 0 plans the next step while the others search
    const bool plan = d.n_trains <= PLAN_TRAINS && step + 1 < n_steps;
    if (plan && lead) {
      stage_next(d, sm.react.plan);
    } else if (d.g->search_cells_now) {
      phase_search_cells<F32L, STEP_WARPS>(d, sm.cells);
    } else {
      const Span others = plan ? Span{sp.block - 1u, sp.blocks - 1u} : sp;
      const int lg = lanes_per_home_lg(d.g->n_total - d.g->n_dead, others.stride());
      phase_search_groups<F32L, STEP_WARPS>(d, sm.grp, lg > 0 ? lg : 1, others.warp(), others.warps());
    }
    bar.sync(d);
    if (lead) {
      phase_react_all<F32L>(d, sm.react.react, sm.react.sbuf, STEP_REACT_CAP, plan ? sm.react.plan.begin.tb : *d.tables);
      if (!(plan && commit_next(d, sm.react.plan, most))) {
        phase_end_step(d, sm.react.end);
        const bool leave = d.g->any_active != 0u && d.g->n_ahead > most;
        __syncthreads();  // (all have read it)
        if (leave && threadIdx.x == 0) d.g->any_active = ANY_OUTGROWN;
        if (step + 1 < n_steps && !leave) phase_begin(d, sm.react.plan.begin);
      }
    }
    bar.sync(d);
  }
  bar.leave(d);
}

// One step as one kernel per phase. With ev != nullptr, CUDA events are recorded
// before and after each phase (ev[2 * phase], ev[2 * phase + 1]); a step that is not the
// first of a graph was begun by the previous step's end kernel (its time falls in the
// previous step's react phase).
template <bool F32L>
cudaError_t enqueue_phases(const Dev& d, const LaunchCfg& lc, cudaStream_t s, cudaEvent_t* ev, bool first,
                           bool last) {
  auto mark = [&](int i) { if (ev) cudaEventRecordWithFlags(ev[i], s, cudaEventRecordExternal); };
  cudaError_t e = cudaSuccess;
  mark(2 * PH_BEGIN);
  if (first) {
    e = enqueue_begin(d, s);
    if (e != cudaSuccess) return e;
  }
  mark(2 * PH_BEGIN + 1);
  mark(2 * PH_RELEASE);  // the release runs inside the diffusion kernel
  mark(2 * PH_RELEASE + 1);
  mark(2 * PH_DIFFUSE);
  k_diffuse<F32L><<<lc.stream_blocks, 256, 0, s>>>(d);
  mark(2 * PH_DIFFUSE + 1);
  mark(2 * PH_SORT);
  for (int p = 0; p < d.passes; ++p) {
    e = enqueue_sort_pass(d, p, lc.sort_blocks, s);
    if (e != cudaSuccess) return e;
  }
  mark(2 * PH_SORT + 1);
  mark(2 * PH_GATHER);
  k_gather<F32L><<<lc.stream_blocks, 256, 0, s>>>(d);
  mark(2 * PH_GATHER + 1);
  mark(2 * PH_SEARCH);
  // one mapping, or both with the one not chosen for the step returning at once
  if (lc.small) k_search_any<F32L><<<2 * lc.search_blocks, 32 * TPS_WARPS, 0, s>>>(d);
  else if (lc.search_tps != 0) k_search_tps<F32L><<<2 * lc.search_blocks, 32 * TPS_WARPS, 0, s>>>(d);
  if (!lc.small && lc.search_tps != 1) k_search<F32L><<<lc.search_blocks, 256, 0, s>>>(d);
  mark(2 * PH_SEARCH + 1);
  mark(2 * PH_REACT);
  if (lc.small) {
    k_react_end<F32L><<<1, REACT_END_THREADS, REACT_END_BYTES, s>>>(d, last ? 0 : 1);
  } else {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(lc.persistent_blocks);
    cfg.blockDim = dim3(REACT_THREADS);
    cfg.dynamicSmemBytes = sizeof(ReactGridSmem);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, k_react_grid<F32L>, d, last ? 0 : 1);
    if (e != cudaSuccess) return e;
  }
  mark(2 * PH_REACT + 1);
  return cudaGetLastError();
}

// Diagnostic: the pair search's acceptance test on given squared separations d0^2 and
// d1^2 of reaction rxn[i] for the pair (id_lo[i], id_hi[i]) at `step`, with the constants
// the begin phase derives from dt. out[i] bit 0: the tiered test of the search (FP32
// estimate, FP64 where undecided); bit 1: the FP64 test u < p itself on the same inputs
// (in FP32-local mode, on the FP32 roundings of the squared separations).
template <bool F32L>
__global__ void __launch_bounds__(256) k_check_accept(const __grid_constant__ Dev d, uint32_t n, uint32_t step,
                                                      double dt, const double* d0sq, const double* d1sq,
                                                      const int32_t* rxn, const uint32_t* id_lo,
                                                      const uint32_t* id_hi, uint8_t* out) {
  __shared__ Train tr;
  const Tables& tb = *d.tables;
  if (threadIdx.x == 0) {
    tr = d.trains[0];
    tr.step = step;
    for (int r = 0; r < tb.n_rxn; ++r) set_pair_constants(tr, tb, r, dt);
  }
  __syncthreads();
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int r = rxn[i];
    const uint32_t lo = id_lo[i], hi = id_hi[i];
    const double u = pair_uniform(lo, hi, step, tr.key0, tr.key1);
    bool tiered, exact;
    if constexpr (F32L) {
      const float a = static_cast<float>(d0sq[i]), b = static_cast<float>(d1sq[i]);
      tiered = accept_f32(a, b, r, tb, tr, lo, hi);
      exact = u < bridge_p(sqrt(static_cast<double>(a)), sqrt(static_cast<double>(b)), tb.R[r], tr.ddt[r]);
    } else {
      tiered = accept_f64(d0sq[i], d1sq[i], r, tb, tr, lo, hi);
      exact = u < bridge_p(sqrt(d0sq[i]), sqrt(d1sq[i]), tb.R[r], tr.ddt[r]);
    }
    out[i] = static_cast<uint8_t>((tiered ? 1 : 0) | (exact ? 2 : 0));
  }
}

template <bool F32L>
cudaError_t enqueue_check_accept(const Dev& d, uint32_t n, uint32_t step, double dt, const double* d0sq,
                                 const double* d1sq, const int32_t* rxn, const uint32_t* id_lo,
                                 const uint32_t* id_hi, uint8_t* out, cudaStream_t s) {
  const uint32_t blocks = n ? (n + 255u) / 256u : 1u;
  k_check_accept<F32L><<<blocks < 1024u ? blocks : 1024u, 256, 0, s>>>(d, n, step, dt, d0sq, d1sq, rxn, id_lo,
                                                                       id_hi, out);
  return cudaGetLastError();
}

// Steps in one launch (StepRun): one cluster, or one CTA per SM (cooperative).
template <bool F32L>
cudaError_t enqueue_steps(const Dev& d, const LaunchCfg& lc, const StepRun& r, cudaStream_t s) {
  const bool cluster = r.cluster;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cluster ? lc.cluster_blocks : lc.persistent_blocks);
  cfg.blockDim = dim3(PERSIST_THREADS);
  cfg.dynamicSmemBytes = sizeof(StepSmem);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  if (cluster) {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(lc.cluster_blocks);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
  } else {
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
  }
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cluster ? cudaLaunchKernelEx(&cfg, k_steps<F32L, true>, d, r.n_steps, r.align, r.done, r.most)
                 : cudaLaunchKernelEx(&cfg, k_steps<F32L, false>, d, r.n_steps, r.align, r.done, r.most);
}

// Shared-memory limits of the precision's kernels; resident CTAs per SM of the persistent form
// and the CTAs of its one-cluster form (0 when no cluster of STEP_CLUSTER or 8 fits).
template <bool F32L>
cudaError_t step_kernel_limits(int* blocks_per_sm, int* cluster_blocks) {
  cudaError_t e = cudaFuncSetAttribute(k_react_end<F32L>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(REACT_END_BYTES));
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_react_grid<F32L>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           static_cast<int>(sizeof(ReactGridSmem)));
  if (e != cudaSuccess) return e;
  const int smem = static_cast<int>(sizeof(StepSmem));
  e = cudaFuncSetAttribute(k_steps<F32L, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_steps<F32L, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_steps<F32L, true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  *cluster_blocks = 0;
  for (int c = STEP_CLUSTER; c >= 8 && *cluster_blocks == 0; c /= 2) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(c);
    cfg.blockDim = dim3(PERSIST_THREADS);
    cfg.dynamicSmemBytes = sizeof(StepSmem);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(c);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, k_steps<F32L, true>, &cfg) == cudaSuccess && clusters > 0)
      *cluster_blocks = c;
    else
      cudaGetLastError();
  }
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_steps<F32L, false>, PERSIST_THREADS,
                                                       sizeof(StepSmem));
}

}  // namespace chem
