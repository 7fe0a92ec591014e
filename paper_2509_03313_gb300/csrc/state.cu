// The live species of one train in device order, packed on the device for chem_get_state:
// count per chunk of slots, scan of the counts, then type, id and FP64 position of each live
// species at its place. (The host used to copy every slot's raw state and compact it in one
// thread: 3.6 ms for 4e5 FP32-local species, 12.6 ms for 2e6; packed, the copies into the
// caller's arrays are what is left.) Built without contraction: the FP32-local positions are
// the ones the host formed, bit for bit.
#include "launch.h"
#include "phases.cuh"

namespace chem {
namespace {

constexpr int PACK_THREADS = 256;
constexpr int PACK_ITEMS = 4;
constexpr uint32_t PACK_CHUNK = PACK_THREADS * PACK_ITEMS;

// Slot i of the train's candidates: the stepped slots, then its parked species.
struct SlotRef {
  uint32_t at;    // slot, or index into the parking buffers
  bool parked, live;
  uint32_t cell;
};
__device__ __forceinline__ SlotRef slot_ref(const Dev& d, uint32_t train, uint32_t n_slots, uint32_t n, uint32_t i) {
  SlotRef r{0u, false, false, 0u};
  if (i >= n) return r;
  if (i < n_slots) {
    r.at = i;
    r.cell = d.cell_sorted[i];
    r.live = d.dead[i] == 0 &&
             (d.n_trains == 1 || static_cast<uint32_t>(train_of_cell(d.trains, d.n_trains, r.cell)) == train);
  } else {
    r.at = d.trains[train].park_base + (i - n_slots);
    r.parked = true;
    r.cell = d.pk_cell[r.at];
    r.live = true;
  }
  return r;
}

__global__ void __launch_bounds__(PACK_THREADS) k_pack_count(const __grid_constant__ Dev d, uint32_t train,
                                                             uint32_t n_slots, uint32_t n, uint32_t* counts) {
  const uint32_t base = blockIdx.x * PACK_CHUNK;
  uint32_t live = 0;
#pragma unroll
  for (int k = 0; k < PACK_ITEMS; ++k)
    live += __popc(__ballot_sync(0xffffffffu, slot_ref(d, train, n_slots, n, base + k * PACK_THREADS + threadIdx.x).live));
  __shared__ uint32_t sum;
  if (threadIdx.x == 0) sum = 0;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) atomicAdd(&sum, live);
  __syncthreads();
  if (threadIdx.x == 0) counts[blockIdx.x] = sum;
}

// counts[0, m) to exclusive prefixes, the total in counts[m]; one CTA.
__global__ void __launch_bounds__(1024) k_pack_scan(uint32_t* counts, uint32_t m) {
  __shared__ uint32_t warp_tot[32], total_s;
  uint32_t carry = 0;
  for (uint32_t i0 = 0; i0 < m; i0 += 1024u) {
    const uint32_t i = i0 + threadIdx.x;
    uint32_t total;
    const uint32_t v = i < m ? counts[i] : 0u;
    const uint32_t ex = block_excl_scan(v, warp_tot, &total_s, total);
    if (i < m) counts[i] = carry + ex;
    carry += total;
  }
  if (threadIdx.x == 0) counts[m] = carry;
}

// Live slot r of the train to place p of the packed arrays.
template <bool F32L>
__device__ __forceinline__ void pack_one(const Dev& d, const Train& tr, const SlotRef& r, uint32_t p, const PackOut& out) {
  if (p >= out.most) return;
  uint32_t tid;
  double x, y, z;
  if (F32L) {
    const float4 v = r.parked ? d.pk4[r.at] : d.s4[r.at];
    tid = __float_as_uint(v.w);
    int ix, iy, iz;
    cell_decode(r.cell - tr.cell_base, tr.cb_ref, ix, iy, iz);  // the grid of the last step
    double y0;
    auto axis = [&](int i, float off) {
      const double q = __dadd_rn(__dsub_rn(__dmul_rn(static_cast<double>(i), tr.h_ref), tr.halfL), static_cast<double>(off));
      return wrap_box_diffused(q, tr.L, tr.halfL, y0);
    };
    x = axis(ix, v.x); y = axis(iy, v.y); z = axis(iz, v.z);
  } else if (r.parked) {
    tid = d.pk_tid[r.at]; x = d.pkx[r.at]; y = d.pky[r.at]; z = d.pkz[r.at];
  } else {
    tid = d.stid[r.at]; x = d.sx[r.at]; y = d.sy[r.at]; z = d.sz[r.at];
  }
  out.type[p] = static_cast<int32_t>(tid_type(tid));
  out.id[p] = tid_id(tid);
  uint32_t row = p, seg = 0;
  while (seg + 1 < PackOut::SEGS && row >= out.rows[seg]) row -= out.rows[seg++];
  double* to = out.xyz[seg] + 3u * static_cast<size_t>(row);
  to[0] = x; to[1] = y; to[2] = z;
}

template <bool F32L>
__global__ void __launch_bounds__(PACK_THREADS) k_pack_write(const __grid_constant__ Dev d, uint32_t train,
                                                             uint32_t n_slots, uint32_t n, const uint32_t* counts,
                                                             const __grid_constant__ PackOut out) {
  __shared__ uint32_t warp_tot[32], total_s;
  uint32_t at = counts[blockIdx.x];
  const Train& tr = d.trains[train];
  for (int k = 0; k < PACK_ITEMS; ++k) {
    const SlotRef r = slot_ref(d, train, n_slots, n, blockIdx.x * PACK_CHUNK + k * PACK_THREADS + threadIdx.x);
    uint32_t total;
    const uint32_t p = at + block_excl_scan(r.live ? 1u : 0u, warp_tot, &total_s, total);
    at += total;
    if (r.live) pack_one<F32L>(d, tr, r, p, out);
  }
}

// The same by one CTA for few slots, the number of live ones in *live: one launch and, with the
// copies that follow it, one synchronise instead of three and two. chem_get_state of 10 and 2,000
// species takes 32 and 47 us (71 and 80 as below; 48 and 62 with every slot copied to the host).
template <bool F32L>
__global__ void __launch_bounds__(1024) k_pack_few(const __grid_constant__ Dev d, uint32_t train, uint32_t n_slots,
                                                   uint32_t n, uint32_t* live, const __grid_constant__ PackOut out) {
  __shared__ uint32_t warp_tot[32], total_s;
  const Train& tr = d.trains[train];
  uint32_t at = 0;
  for (uint32_t i0 = 0; i0 < n; i0 += 1024u) {
    const SlotRef r = slot_ref(d, train, n_slots, n, i0 + threadIdx.x);
    uint32_t total;
    const uint32_t p = at + block_excl_scan(r.live ? 1u : 0u, warp_tot, &total_s, total);
    at += total;
    if (r.live) pack_one<F32L>(d, tr, r, p, out);
  }
  if (threadIdx.x == 0) *live = at;
}

}  // namespace

uint32_t pack_counts(uint32_t n) { return (n + PACK_CHUNK - 1) / PACK_CHUNK; }

cudaError_t enqueue_pack_count(const Dev& d, uint32_t train, uint32_t n_slots, uint32_t n, uint32_t* counts,
                               cudaStream_t s) {
  const uint32_t m = pack_counts(n);
  if (m) k_pack_count<<<m, PACK_THREADS, 0, s>>>(d, train, n_slots, n, counts);
  k_pack_scan<<<1, 1024, 0, s>>>(counts, m);
  return cudaGetLastError();
}

cudaError_t enqueue_pack_few(const Dev& d, uint32_t train, uint32_t n_slots, uint32_t n, uint32_t* live,
                             const PackOut& out, cudaStream_t s) {
  if (d.precision == CHEM_FP64) k_pack_few<false><<<1, 1024, 0, s>>>(d, train, n_slots, n, live, out);
  else k_pack_few<true><<<1, 1024, 0, s>>>(d, train, n_slots, n, live, out);
  return cudaGetLastError();
}

cudaError_t enqueue_pack_write(const Dev& d, uint32_t train, uint32_t n_slots, uint32_t n, const uint32_t* counts,
                               const PackOut& out, cudaStream_t s) {
  const uint32_t m = pack_counts(n);
  if (m == 0) return cudaSuccess;
  if (d.precision == CHEM_FP64) k_pack_write<false><<<m, PACK_THREADS, 0, s>>>(d, train, n_slots, n, counts, out);
  else k_pack_write<true><<<m, PACK_THREADS, 0, s>>>(d, train, n_slots, n, counts, out);
  return cudaGetLastError();
}

}  // namespace chem
