// The phases of one SBS step, as device functions usable both from one-kernel-per-phase
// launches and from the persistent batched launch. Every phase is grid-stride over its
// work and reads the device status word first: once a phase has raised an error the
// remaining phases of the step do nothing.
//
// Arithmetic that the FP64 mode shares with the FP64 reference is written with explicit
// round-to-nearest intrinsics (__dmul_rn, __dadd_rn, ...) so that no multiply-add is ever
// contracted, whatever the compilation flags: in FP64 mode the library reproduces the
// reference's positions to rounding and its decisions exactly.
#pragma once
#include <cfloat>
#include <type_traits>
#include <math_constants.h>

#include "fixed_normals.cuh"
#include "onesweep.cuh"
#include "sbs_device.cuh"

namespace chem {

constexpr double TWO_POW_M53 = 1.1102230246251565e-16;
constexpr float TWO_POW_M24F = 5.9604644775390625e-08f;

// The part of a phase's work that a CTA takes: CTA `block` of `blocks`. Warps of one CTA are
// `blocks` warps apart, so that little work spreads over all CTAs.
struct Span {
  uint32_t block, blocks;
  __device__ __forceinline__ uint32_t warp() const { return (threadIdx.x >> 5) * blocks + block; }
  __device__ __forceinline__ uint32_t warps() const { return (blockDim.x >> 5) * blocks; }
  __device__ __forceinline__ uint32_t first() const { return warp() * 32u + (threadIdx.x & 31u); }
  __device__ __forceinline__ uint32_t stride() const { return blocks * blockDim.x; }
};
__device__ __forceinline__ Span whole_grid() { return Span{blockIdx.x, gridDim.x}; }

__device__ __forceinline__ int status_of(const Dev& d) {
  return *reinterpret_cast<volatile int*>(&d.g->status);
}

// Eq. 1 applied as often as needed: x shifted by whole box lengths into [-L/2, L/2).
__device__ __forceinline__ double wrap_box(double x, double L, double halfL) {
  const double k = floor(__ddiv_rn(__dadd_rn(x, halfL), L));
  x = __dsub_rn(x, __dmul_rn(k, L));
  if (x >= halfL) x = __dsub_rn(x, L);
  if (x < -halfL) x = __dadd_rn(x, L);
  return x;
}

// A coordinate measured from the box corner folded into [0, L) (FP32-local regrid).
__device__ __forceinline__ double rebase_corner(double a, double L, double inv_L) {
  if (a >= L || a < 0.0) a -= L * floor(a * inv_L);
  if (a >= L) a -= L;
  if (a < 0.0) a += L;
  return a;
}

// Eq. 2 (minimum image) for the separation of two in-box points.
__device__ __forceinline__ double min_image(double dx, double L, double halfL) {
  if (dx >= halfL) return __dsub_rn(dx, L);
  if (dx < -halfL) return __dadd_rn(dx, L);
  return dx;
}

__device__ __forceinline__ double sq3(double x, double y, double z) {
  return __dadd_rn(__dadd_rn(__dmul_rn(x, x), __dmul_rn(y, y)), __dmul_rn(z, z));
}

// The same for the diffused position of an FP64 species, and y = x + L/2 of the result. A
// position still inside the box (0 <= y < L, compared on the bits: positive doubles order as
// integers) is its own wrap, so the division is left to the few that leave it.
__device__ __forceinline__ double wrap_box_diffused(double x, double L, double halfL, double& y) {
  y = __dadd_rn(x, halfL);
  const long long b = __double_as_longlong(y);
  if (b < 0 || b >= __double_as_longlong(L)) {
    x = wrap_box(x, L, halfL);
    y = __dadd_rn(x, halfL);
  }
  return x;
}

// y >= 0 as an exact sum of two floats, hi truncated to 24 bits (0 below 2^-60).
__device__ __forceinline__ void split_double(double y, float& hi, float& lo) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(y));
  const int e = static_cast<int>(b >> 52);  // y >= 0
  const bool tiny = e < 1023 - 60;
  hi = tiny ? 0.f : __uint_as_float((static_cast<uint32_t>(e - 896) << 23) | (static_cast<uint32_t>(b >> 29) & 0x7FFFFFu));
  lo = tiny ? 0.f : static_cast<float>(static_cast<uint32_t>(b) & 0x1FFFFFFFu) *
                        __uint_as_float(static_cast<uint32_t>(e - 896 - 52) << 23);
}

// v truncated to a float without the FP64 pipe (0 below 2^-126).
__device__ __forceinline__ float truncate_double(double v) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(v));
  const int e = static_cast<int>((b >> 52) & 0x7FFu) - 896;
  const uint32_t sign = static_cast<uint32_t>(b >> 32) & 0x80000000u;
  return e <= 0 ? 0.f : __uint_as_float(sign | (static_cast<uint32_t>(e) << 23) | (static_cast<uint32_t>(b >> 29) & 0x7FFFFFu));
}

// Three standard normals for species `id` at step `step` (FP64 mode): two Philox blocks,
// 53-bit uniforms u1 in (0,1], u2 in [0,1), Box-Muller, its functions in fixed point
// (fixed_normals.cuh).
__device__ __forceinline__ void gauss3_f64(uint32_t id, uint32_t step, uint32_t k0, uint32_t k1,
                                           double& g0, double& g1, double& g2) {
  const uint4 a = philox4x32_10(make_uint4(id, step, 0u, 0u), k0, k1);
  const uint4 b = philox4x32_10(make_uint4(id, step, 0u, 1u), k0, k1);
  const double r = fixedn::radius_fp64(u53(a.x, a.y));
  double s, c;
  fixedn::sincos_2pi(u53(a.z, a.w), s, c);
  g0 = __dmul_rn(r, c);
  g1 = __dmul_rn(r, s);
  g2 = __dmul_rn(fixedn::radius_fp64(u53(b.x, b.y)), fixedn::cos_2pi(u53(b.z, b.w)));
}

// Three standard normals (FP32-local mode): one Philox block, 24-bit uniforms.
__device__ __forceinline__ void gauss3_f32(uint32_t id, uint32_t step, uint32_t k0, uint32_t k1,
                                           float& g0, float& g1, float& g2) {
  const uint4 a = philox4x32_10(make_uint4(id, step, 0u, 0u), k0, k1);
  const float u1 = static_cast<float>((a.x >> 8) + 1u) * TWO_POW_M24F;
  const float u2 = static_cast<float>(a.y >> 8) * TWO_POW_M24F;
  const float u3 = static_cast<float>((a.z >> 8) + 1u) * TWO_POW_M24F;
  const float u4 = static_cast<float>(a.w >> 8) * TWO_POW_M24F;
  // hardware approximations (a few ulp): the FP32-local normals need no more
  const float r = sqrtf(-2.0f * __logf(u1));
  float s, c;
  __sincosf(6.2831853f * u2, &s, &c);
  g0 = r * c;
  g1 = r * s;
  g2 = sqrtf(-2.0f * __logf(u3)) * __cosf(6.2831853f * u4);
}

// Uniform in [0, 1) for the pair (id_lo, id_hi) at `step` (counter tag 2).
__device__ __forceinline__ double pair_uniform(uint32_t id_lo, uint32_t id_hi, uint32_t step,
                                               uint32_t k0, uint32_t k1) {
  const uint4 c = philox4x32_10(make_uint4(id_lo, step, id_hi, 2u), k0, k1);
  return __dmul_rn(static_cast<double>(u53(c.x, c.y)), TWO_POW_M53);
}

// Probability that the pair's relative Brownian path touched the reaction sphere during
// the step, given its start and end separations d0, d1 (p = 1 when either is inside R):
// 1 - G_abs / G_free for the angle-averaged relative motion (image solutions of r times
// the density, outside a fully absorbing sphere and free), i.e.
// (exp(-a) - exp(-b)) / (1 - exp(-b)) with a = (d0 - R)(d1 - R) / (D_AB dt) and
// b = d0 d1 / (D_AB dt), evaluated as exp(-a) expm1(-c) / expm1(-b), c = b - a =
// R (d0 + d1 - R) / (D_AB dt). Its expectation is the absorbing-sphere rate behind
// Eq. kdiff1 at any dt; for R >> sqrt(D_AB dt) it is the planar bridge exp(-a).
__device__ __forceinline__ double bridge_p(double d0, double d1, double R, double DABdt) {
  if (d1 <= R || d0 <= R) return 1.0;
  const double a = __ddiv_rn(__dmul_rn(__dsub_rn(d0, R), __dsub_rn(d1, R)), DABdt);
  const double b = __ddiv_rn(__dmul_rn(d0, d1), DABdt);
  const double c = __ddiv_rn(__dmul_rn(R, __dsub_rn(__dadd_rn(d0, d1), R)), DABdt);
  return __dmul_rn(exp(-a), __ddiv_rn(expm1(-c), expm1(-b)));
}

__device__ __forceinline__ int cell_index(double x, double halfL, double inv_h, int n) {
  int i = static_cast<int>(floor(__dmul_rn(__dadd_rn(x, halfL), inv_h)));
  return min(max(i, 0), n - 1);
}

// Cell index of an in-box coordinate y = x + L/2 (the value of cell_index) and the offset from
// the cell's corner as a float, on the FP32 pipe: FP32 places y within 2.5e-4 of a cell for
// grids up to 1024, so only coordinates closer than 1e-3 to a face repeat the FP64 test. The
// offset is within 1.5e-7 of a cell (two fused steps from the exact halves of y and h).
__device__ __forceinline__ int cell_index_split(double y, double inv_h, int n, float hf, float hlo, float inv_hf,
                                                float& off) {
  float yh, yl;
  split_double(y, yh, yl);
  const float q = yh * inv_hf;
  int i = static_cast<int>(q);
  const float fr = q - static_cast<float>(i);
  if (fr < 1e-3f || fr > 0.999f) i = static_cast<int>(floor(__dmul_rn(y, inv_h)));
  i = min(max(i, 0), n - 1);
  const float fi = static_cast<float>(-i);
  off = __fmaf_rn(fi, hf, yh) + __fmaf_rn(fi, hlo, yl);
  return i;
}

// Bits per axis of the cell index of a grid of n cells per axis: enough for the values
// 0..n, so the all-ones index (>= n) is never a cell.
__device__ __forceinline__ int axis_bits(int n) { return 32 - __clz(n); }

__device__ __forceinline__ int wrap_cell(int i, int n) {
  i %= n;
  return i < 0 ? i + n : i;
}

// Per-reaction constants of the acceptance test for a step of length dt: D_AB dt (the
// exponents' denominator) in FP64 and its reciprocal in FP32 (the first tier).
__device__ __forceinline__ void set_pair_constants(Train& tr, const Tables& tb, int r, double dt) {
  tr.ddt[r] = __dmul_rn(tb.D_AB[r], dt);
  tr.inv_ddt_f[r] = 1.0f / static_cast<float>(tr.ddt[r]);
}

// Lanes of the pair search that share a home species (phase_search_groups): 2^lg, for n species
// on `lanes` lanes as many as there are spare, up to 16 (a lane per cell of the half shell). 0:
// one thread per home species.
constexpr int GRP_MAX_LG = 4;
__device__ __forceinline__ int lanes_per_home_lg(uint32_t n, uint32_t lanes) {
  const uint32_t per = lanes / (n ? n : 1u);
  return per >= 2u ? min(GRP_MAX_LG, 31 - __clz(per)) : 0;
}

// ======================================================================== begin
constexpr int BEGIN_TRAINS = 16;  // trains whose cutoffs pass through shared memory

struct BeginSmem {
  Tables tb;                              // the reaction tables, read once per step
  uint32_t rel[MAX_TRAINS];
  double dt[MAX_TRAINS];
  unsigned long long rcmax_bits[MAX_TRAINS];
  float hf[MAX_TRAINS];                   // this step's cell side
  // between the two halves of the phase: whether the train advances, its releases (arrived,
  // re-created, unparked) and its species before them
  uint8_t act[MAX_TRAINS];
  uint32_t rel_new[MAX_TRAINS], mat[MAX_TRAINS], parked[MAX_TRAINS];
  long long live[MAX_TRAINS];
  double c[BEGIN_TRAINS];                 // cutoff factor ...
  double rc2[BEGIN_TRAINS][MAXR];         // ... and squared cutoffs of the first trains
  int cb0;                                // train 0: key bits per axis of its cells
  uint32_t base0;                         // train 0: first global cell
  uint32_t any;
};

// One CTA of at least MAX_TRAINS threads. (1) per train: release count, clock step and
// free-jump decision; (2) per (train, reaction) cutoff and bridge constants and per (train,
// type) step sigma, spread over the threads because FP64 square roots and divisions are long
// on this part; (3) per train: hash grid of the step; (4) per (train, type pair) cutoff
// tables; (5) slot offsets of the releases and the step counters. The phase is a chain of
// dependent latencies on the step's critical path, so every global load is issued at the
// start (a train's record stays in its thread's registers through (1) and (3)), later
// stages read what earlier ones wrote from shared memory, and the pending queue is only
// searched when its first arrival is due. With loads in every stage it took 8 us.
//
// The phase has two halves: begin_plan, (1) to (4), which needs nothing of the reactions of
// the step before and works on the records `trains` (the context's, or a copy of them that
// already stands at the end of that step), and begin_commit, the rest.
static __device__ void begin_plan(const Dev& d, BeginSmem& sb, Train* trains, int st) {
  const int tid = threadIdx.x, nt = blockDim.x;
  {
    const uint32_t* src = reinterpret_cast<const uint32_t*>(d.tables);
    uint32_t* dst = reinterpret_cast<uint32_t*>(&sb.tb);
    for (int i = tid; i < static_cast<int>(sizeof(Tables) / 4); i += nt) dst[i] = src[i];
  }
  if (tid == 0) sb.any = 0;
  // train `tid`
  const uint32_t b = static_cast<uint32_t>(tid);
  const bool have = b < d.n_trains;
  Train& tr = trains[have ? b : 0u];
  double t = 0, t_end = 0, t_lr = 0, horizon = 0, dt_min = 0, dt_L = 0, dt_cur = 0, next_arr = 0, L = 0, inv_L = 0;
  uint32_t p_head = 0, p_tail = 0, pend_base = 0, mat = 0, parked = 0;
  int reset = 0, tr_n_max = 0, cb_alloc = 0, n_ref = 0;
  long long live = 0;
  if (have) {
    t = tr.t; t_end = tr.t_end; t_lr = tr.t_last_release; horizon = tr.horizon;
    dt_min = tr.dt_min; dt_L = tr.dt_L; dt_cur = tr.dt_cur; next_arr = tr.next_arr;
    p_head = tr.p_head; p_tail = tr.p_tail; pend_base = tr.pend_base;
    mat = tr.mat_n;      // survivors of a homogeneous stage (already counted)
    parked = tr.park_n;  // species parked while the train was idle (counted)
    reset = tr.reset_on_release;
    L = tr.L; inv_L = tr.inv_L; tr_n_max = tr.n_max; cb_alloc = tr.cb_alloc; n_ref = tr.n_ref;
#pragma unroll
    for (int ty = 0; ty < MAXT; ++ty) live += tr.counts[ty];  // 0 past the context's types
    sb.live[b] = live;
    if (b < BEGIN_TRAINS) sb.c[b] = tr.c;
    if (b == 0) {  // the removed species' key below needs train 0's grid, idle or not
      sb.cb0 = tr.cb;
      sb.base0 = tr.cell_base;
    }
  }
  __syncthreads();
  const Tables& tb = sb.tb;
  double dt = 0.0;
  int free_jump = 0;
  if (have) {
    const bool act = (st == 0) && (t < t_end);
    uint32_t rel = 0;
    sb.rcmax_bits[b] = 0ull;
    if (act) {
      // pending arrivals are sorted; release those with arrival <= t
      uint32_t lo = p_head;
      if (next_arr <= t) {
        uint32_t hi = p_tail;
        const double* pt = d.pt + pend_base;
        while (lo < hi) {
          const uint32_t mid = (lo + hi) >> 1;
          if (pt[mid] <= t) lo = mid + 1; else hi = mid;
        }
        next_arr = (lo < p_tail) ? pt[lo] : CUDART_INF;
        tr.next_arr = next_arr;
      }
      rel = lo - p_head;
      double t_last = t_lr;
      if (rel + mat > 0) {
        t_last = t;
        tr.t_last_release = t;
        if (reset) dt_cur = dt_min;
      }
      double t_next;
      if (horizon > 0.0 && __dsub_rn(t, t_last) >= horizon && next_arr > t) {
        free_jump = 1;
        t_next = fmin(t_end, next_arr);
        dt = __dsub_rn(t_next, t);
      } else {
        dt = fmin(dt_cur, dt_L);
        if (__dsub_rn(t_end, t) <= __dmul_rn(dt, END_SLACK)) {
          dt = __dsub_rn(t_end, t);
          t_next = t_end;
        } else {
          t_next = __dadd_rn(t, dt);
        }
      }
      sb.dt[b] = dt;
      sb.rel[b] = parked + rel + mat;
      tr.dt_cur = dt_cur;
      tr.dt = dt;
      tr.t_next = t_next;
      tr.t_start = t;
      // releases: the unparked species first (they keep their ids), then the re-created
      // survivors, then the arrived species
      tr.rel_n = parked + rel + mat;
      tr.rel_park = parked;
      tr.park_n = 0;
      tr.rel_mat = mat;
      tr.mat_n = 0;
      tr.rel_p0 = p_head;
      tr.p_head = p_head + rel;
      tr.n_events_step = 0;
      atomicOr(&sb.any, 1u);
    } else {
      sb.dt[b] = 0.0;
      sb.rel[b] = 0u;
      tr.rel_n = 0;
      tr.rel_mat = 0;
      tr.rel_park = 0;
    }
    tr.active = act ? 1 : 0;
    tr.free_jump = free_jump;
    sb.act[b] = act ? 1 : 0;
    sb.rel_new[b] = rel;
    sb.mat[b] = mat;
    sb.parked[b] = parked;
  }
  __syncthreads();
  // cutoffs R + c sqrt(2 D_AB dt), bridge constants, and sigma = sqrt(2 D dt)
  const int per = MAXR + MAXT;
  for (uint32_t w = tid; w < d.n_trains * per; w += nt) {
    const uint32_t wb = w / per;
    const int q = static_cast<int>(w % per);
    const double wdt = sb.dt[wb];
    if (wdt <= 0.0) continue;  // train not advancing this step
    Train& wt = trains[wb];
    if (q < MAXR) {
      if (q >= tb.n_rxn) continue;
      const double c = wb < BEGIN_TRAINS ? sb.c[wb] : wt.c;
      const double rc = __dadd_rn(tb.R[q], __dmul_rn(c, sqrt(__dmul_rn(__dmul_rn(2.0, tb.D_AB[q]), wdt))));
      const double rc2 = __dmul_rn(rc, rc);
      atomicMax(&sb.rcmax_bits[wb], static_cast<unsigned long long>(__double_as_longlong(rc)));
      if (wb < BEGIN_TRAINS) sb.rc2[wb][q] = rc2;
      wt.rc2[q] = rc2;
      wt.rc2f[q] = static_cast<float>(rc2);
      set_pair_constants(wt, tb, q, wdt);
    } else {
      const int ty = q - MAXR;
      if (ty >= tb.n_types) continue;
      const double sig = sqrt(__dmul_rn(__dmul_rn(2.0, tb.D[ty]), wdt));
      wt.sig[ty] = sig;
      wt.sigf[ty] = static_cast<float>(sig);
    }
  }
  __syncthreads();
  if (have && dt > 0.0) {
    const int n_max = min(tr_n_max, (1 << cb_alloc) - 1);
    const double rcmax = __longlong_as_double(static_cast<long long>(sb.rcmax_bits[b]));
    // finest admissible grid: cells at least the largest cutoff (with slack), at least 3
    // per axis (no cell met twice among a cell's neighbours)
    int n_target = n_max;
    if (rcmax > 0.0) {
      const float cut = static_cast<float>(rcmax) * CELL_SLACK_F;
      const float nf1 = floorf(static_cast<float>(L) / cut);
      n_target = max(3, min(n_max, static_cast<int>(fminf(nf1, 1048576.f))));
    }
    if (n_ref == 0) {  // first step after init or reset
      n_ref = n_target;
      tr.n_ref = n_target;
      tr.h_ref = __ddiv_rn(L, static_cast<double>(n_target));
      tr.cb_ref = axis_bits(n_target);
    }
    // keep the current grid while it is valid and at most 2x too coarse; when the
    // cutoff outgrows it, move to cells 1.2x larger than needed (fewer regrids)
    int n = n_ref;
    if (!free_jump) {
      if (n > n_target) n = max(3, (5 * n_target) / 6);
      else if (2 * n < n_target) n = n_target;
    }
    double h = __ddiv_rn(L, static_cast<double>(n));
    // the search looks one cell out: a cell must cover the largest cutoff
    if (!free_jump && rcmax > 0.0 && n != n_target) {
      const double cut = rcmax * static_cast<double>(CELL_SLACK_F);
      if (h < cut) {
        n = n_target;
        h = __ddiv_rn(L, static_cast<double>(n));
      }
    }
    const double inv_h = __dmul_rn(static_cast<double>(n), inv_L);
    tr.n = n;
    tr.cb = axis_bits(n);
    tr.h = h;
    tr.inv_h = inv_h;
    tr.hf = static_cast<float>(h);
    tr.hlo = static_cast<float>(h - static_cast<double>(static_cast<float>(h)));
    tr.inv_hf = static_cast<float>(inv_h);
    sb.hf[b] = static_cast<float>(h);
    if (b == 0) sb.cb0 = axis_bits(n);
  }
  __syncthreads();
  // per type pair (the pair search's lookup tables): the squared cutoff, in FP64 and
  // FP32, and the FP32 one widened past any error of FP32 cell offsets (a few 1e-7 of a
  // cell per component), so that a pair the FP32 test rejects is outside the FP64 cutoff
  for (uint32_t w = tid; w < d.n_trains * (MAXT * MAXT); w += nt) {
    const uint32_t wb = w / (MAXT * MAXT);
    const int q = static_cast<int>(w % (MAXT * MAXT));
    if (sb.dt[wb] <= 0.0) continue;
    Train& wt = trains[wb];
    const int r = tb.pair_rxn[q / MAXT][q % MAXT];
    const double c2 = r >= 0 ? (wb < BEGIN_TRAINS ? sb.rc2[wb][r] : wt.rc2[r]) : -1.0;
    const float c2f = r >= 0 ? static_cast<float>(c2) : -1.f;
    wt.rc2_tt[q] = c2;
    wt.rc2f_tt[q] = c2f;
    const float rc = c2f >= 0.f ? sqrtf(c2f) : -1.f;
    const float rw = rc * 1.00001f + 2e-6f * sb.hf[wb];
    wt.rc2w_tt[q] = rc >= 0.f ? rw * rw * 1.00001f : -1.f;
  }
}

// Lanes that a launch of one thread per home species has at least (the per-phase form).
constexpr uint32_t SEARCH_LANES = 152u * 1024u;

// The rest of the begin: ids, slots and counters of the step (sb.live: the species per train).
static __device__ void begin_commit(const Dev& d, BeginSmem& sb, Train* trains) {
  const int tid = threadIdx.x, nt = blockDim.x;
  Global* g = d.g;
  for (int i = tid; i < MAX_PASSES * RADIX; i += nt) (&g->hist[0][0])[i] = 0u;
  uint32_t g_total = 0, g_live = 0, g_adaptive = 0, g_home = 0, g_epoch = 0, g_cells = 0;
  unsigned long long g_incut = 0, g_mark = 0;
  if (tid == 0) {  // (all in flight together)
    g_total = g->n_total; g_live = g->n_live; g_adaptive = g->search_adaptive; g_home = g->item_home;
    g_epoch = g->epoch; g_cells = g->cells_steps; g_incut = g->pairs_in_cutoff; g_mark = g->incut_mark;
  }
  const uint32_t b = static_cast<uint32_t>(tid);
  if (b < d.n_trains) {
    Train& tr = trains[b];
    const long long live = sb.live[b];
    const uint32_t rel = sb.rel_new[b], mat = sb.mat[b];
    const bool act = sb.act[b] != 0;
    // an idle train with species among the stepped slots parks them this step
    tr.park_now = (!act && d.pk_cell != nullptr && live > static_cast<long long>(sb.parked[b]) + mat) ? 1u : 0u;
    if (act) {
      const uint32_t next_id = tr.next_id;
      tr.rel_id0 = next_id;
      tr.next_id = next_id + rel + mat;
      tr.n_live_step = live + rel;
      if (static_cast<unsigned long long>(next_id) + rel + mat > tr.id_limit) raise_status(g, CHEM_ECAPACITY);
    }
  }
  if (tid == 0) {
    uint32_t off = g_total;
    const uint32_t before = off;
    unsigned long long total = off;
    for (uint32_t q = 0; q < d.n_trains; ++q) {
      trains[q].rel_off = off;
      total += sb.rel[q];
      off += sb.rel[q];
    }
    if (total > d.cap) {
      raise_status(g, CHEM_ECAPACITY);
      g->n_released = 0;
    } else {
      g->n_released = off - before;
      g->n_total = off;
    }
    for (int p = 0; p < MAX_PASSES; ++p) g->tile_ctr[p] = 0;
    g->n_cand = 0;
    g->n_conflict = 0;
    g->n_items = 0;
    g->item_ctr = 0;
    g->n_events = 0;
    g->bk_overflow = 0;
    g->n_products = 0;
    g->n_dead = 0;
    g->epoch = g_epoch + 1u;
    g->any_active = sb.any;
    // Search mapping of this step. Cell tiles amortise the neighbour-cell lookups over
    // the homes of a cell and test a pair only when the types react; one thread per
    // species has the shorter per-item latency chain. Adaptive: cell tiles when the last
    // step found more than 4 pairs inside the cutoffs per live species (1e6 track species, one
    // thread per species against tiles: 145 / 168 us at 2.9 pairs, 173 / 178 at 4.1, 240 / 213
    // at 6.8). Where the launch has several lanes for each home
    // those share the pairs of a home, and tiles only pay for a few thousand species or very
    // many pairs: at 31,000 species lanes take 43, 79 and 143 us where tiles take 95, 156
    // and 207, at 6, 16 and 25 pairs per species. Results do not depend on the mapping.
    uint32_t cells_now;
    if (g_adaptive) {
      const unsigned long long inc = g_incut - g_mark;
      const int lg = lanes_per_home_lg(g_live, SEARCH_LANES);
      const unsigned long long most = lg == 0 ? 4ull : (lg < GRP_MAX_LG ? 48ull : 3ull);
      cells_now = inc > most * static_cast<unsigned long long>(g_live) ? 1u : 0u;
    } else {
      cells_now = g_home != 0u ? 1u : 0u;
    }
    g->search_cells_now = cells_now;
    g->incut_mark = g_incut;
    if (cells_now && sb.any) g->cells_steps = g_cells + 1u;
    // removed species sort after every live one: with one train the all-ones cell index
    // of the grid's width (this step's grid, or the last one when the train is idle; no
    // cell has it, and it stays within the bits the launched passes sort), so the top
    // key bits stay zero and their radix pass is skipped; with several trains, past the
    // last train's cells
    const int kb = min(3 * sb.cb0, 8 * d.passes);
    g->sentinel_step = d.n_trains == 1 ? sb.base0 + (kb >= 32 ? 0xFFFFFFFFu : (1u << kb) - 1u) : d.sentinel;
  }
  __syncthreads();
}

static __device__ void phase_begin(const Dev& d, BeginSmem& sb) {
  begin_plan(d, sb, d.trains, status_of(d));
  __syncthreads();
  begin_commit(d, sb, d.trains);
}

// Train whose release block holds `slot` (release offsets ascend with b).
__device__ __forceinline__ int train_of_release(const Dev& d, uint32_t slot) {
  int lo = 0, hi = static_cast<int>(d.n_trains) - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (d.trains[mid].rel_off <= slot) lo = mid; else hi = mid - 1;
  }
  // skip empty blocks sharing the same offset
  while (lo > 0 && d.trains[lo].rel_n == 0) --lo;
  return lo;
}

// Warp-aggregated increment of counts[train][type].
__device__ __forceinline__ void count_add(const Dev& d, uint32_t b, uint32_t type, long long v,
                                          bool valid) {
  const uint32_t mask = __ballot_sync(0xffffffffu, valid);
  if (!valid) return;
  const uint32_t key = (b << 3) | type;
  const uint32_t peers = __match_any_sync(mask, key);
  const int lane = threadIdx.x & 31;
  if (lane == __ffs(peers) - 1)
    atomicAdd(reinterpret_cast<unsigned long long*>(&d.trains[b].counts[type]),
              static_cast<unsigned long long>(v * __popc(peers)));
}

// ======================================================================== release
// Position of a survivor of a homogeneous stage re-created with id `id`: uniform in the
// box, -L/2 + L u per axis with u from counter (id, 0, 0, 3) words (0,1) -> x, (2,3) -> y
// and counter (id, 1, 0, 3) words (0,1) -> z, then Eq. 1.
__device__ __forceinline__ void recreated_position(const Train& tr, uint32_t id, double& x, double& y,
                                                   double& z) {
  const uint4 a = philox4x32_10(make_uint4(id, 0u, 0u, 3u), tr.key0, tr.key1);
  const uint4 c = philox4x32_10(make_uint4(id, 1u, 0u, 3u), tr.key0, tr.key1);
  const double ux = __dmul_rn(static_cast<double>(u53(a.x, a.y)), TWO_POW_M53);
  const double uy = __dmul_rn(static_cast<double>(u53(a.z, a.w)), TWO_POW_M53);
  const double uz = __dmul_rn(static_cast<double>(u53(c.x, c.y)), TWO_POW_M53);
  x = wrap_box(__dadd_rn(-tr.halfL, __dmul_rn(tr.L, ux)), tr.L, tr.halfL);
  y = wrap_box(__dadd_rn(-tr.halfL, __dmul_rn(tr.L, uy)), tr.L, tr.halfL);
  z = wrap_box(__dadd_rn(-tr.halfL, __dmul_rn(tr.L, uz)), tr.L, tr.halfL);
}

// Type of the k-th re-created survivor (ascending type order).
__device__ __forceinline__ uint32_t recreated_type(const Train& tr, uint32_t k) {
  uint32_t ty = 0;
  while (ty + 1 < static_cast<uint32_t>(MAXT) && k >= tr.mat_cum[ty]) ++ty;
  return ty;
}

// ======================================================================== diffuse
// Displace every species of an active train (Sec. 2.1 SBS step) with periodic wrap
// (Eq. 1), compute its hash key, and accumulate the radix histograms of every pass.
// Species marked dead by the last step's reactions get the sentinel key. Species
// released this step (slots [n_total - n_released, n_total)) are first built from the
// pending queue (the release of Sec. 2.1) by the thread that then diffuses them.
// `hist` is the CTA's shared-memory histogram; nullptr when the sort of the step counts for
// itself.
template <bool F32L>
__device__ void phase_diffuse(const Dev& d, uint32_t (*hist)[RADIX], const Span& sp) {
  if (hist) {
    for (int i = threadIdx.x; i < MAX_PASSES * RADIX; i += blockDim.x) (&hist[0][0])[i] = 0u;
    __syncthreads();
  }
  // the trip count below must be the same for a whole warp (count_add votes)
  const bool ok = __shfl_sync(0xffffffffu, status_of(d) == 0 ? 1 : 0, 0) != 0;
  const uint32_t n_total = d.g->n_total;
  const uint32_t rel_base = n_total - d.g->n_released;
  const uint32_t stride = sp.stride(), first = sp.first();
  const uint32_t n_iter = ok ? (n_total + stride - 1) / stride : 0u;
  uint32_t n_dead_local = 0;
  // the next iteration's state of a stepped slot is loaded while this one is worked on
  // (released slots read their own sources below)
  uint32_t pf_cell = 0, pf_prev = 0, pf_tid = 0;
  bool pf_dead = false;
  float4 pf_v = make_float4(0.f, 0.f, 0.f, 0.f);
  double pf_x = 0, pf_y = 0, pf_z = 0;
  auto prefetch = [&](uint32_t s) {
    if (s < rel_base) {
      pf_cell = d.cell_sorted[s];
      pf_prev = s > 0 ? d.cell_sorted[s - 1] : 0u;
      pf_dead = d.dead[s] != 0;
      if (F32L) {
        pf_v = d.s4[s];
      } else {
        pf_x = d.sx[s]; pf_y = d.sy[s]; pf_z = d.sz[s]; pf_tid = d.stid[s];
      }
    }
  };
  if (n_iter > 0) prefetch(first);
  for (uint32_t it = 0; it < n_iter; ++it) {
    const uint32_t s = it * stride + first;
    const uint32_t c_cell = pf_cell, c_prev = pf_prev, c_tid = pf_tid;
    const bool c_dead = pf_dead;
    const float4 c_v = pf_v;
    const double c_x = pf_x, c_y = pf_y, c_z = pf_z;
    if (it + 1 < n_iter) prefetch(s + stride);
    const bool valid = s < n_total;
    const bool rel = valid && s >= rel_base;
    uint32_t rel_b = 0, rel_type = 0;
    bool rel_new = false;  // a released species not yet in the train's counts
    if (valid) {
      uint32_t key;
      uint32_t cell;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      double px = 0, py = 0, pz = 0;
      uint32_t tid = 0;
      bool dead = false;
      if (rel) {
        // release: re-created survivors of a homogeneous stage first, then the pending
        // queue; ids in that order (arrival, call order within the queue)
        rel_b = train_of_release(d, s);
        const Train& tr = d.trains[rel_b];
        const uint32_t kp = s - tr.rel_off;
        if (kp < tr.rel_park) {
          // an unparked species: its state and cell key as they were parked (the train's
          // grid has not changed since); it then takes the step like any other
          const uint32_t q = tr.park_base + kp;
          cell = d.pk_cell[q];
          if (F32L) {
            v = d.pk4[q];
            d.s4[s] = v;
          } else {
            px = d.pkx[q]; py = d.pky[q]; pz = d.pkz[q]; tid = d.pk_tid[q];
            d.sx[s] = px; d.sy[s] = py; d.sz[s] = pz; d.stid[s] = tid;
          }
          d.cell_sorted[s] = cell;
          d.dead[s] = 0;
        } else {
        const uint32_t k = kp - tr.rel_park;
        if (k < tr.rel_mat) {
          rel_type = recreated_type(tr, k);
          recreated_position(tr, tr.rel_id0 + k, px, py, pz);
        } else {
          const uint32_t p = tr.pend_base + tr.rel_p0 + (k - tr.rel_mat);
          rel_type = static_cast<uint32_t>(d.p_type[p]);
          px = d.px[p]; py = d.py[p]; pz = d.pz[p];
          rel_new = true;
        }
        tid = ((tr.rel_id0 + k) << 3) | rel_type;
        if (F32L) {
          const int n = tr.n_ref;
          const double h = tr.h_ref, inv_h = static_cast<double>(n) * tr.inv_L;
          const int ix = cell_index(px, tr.halfL, inv_h, n);
          const int iy = cell_index(py, tr.halfL, inv_h, n);
          const int iz = cell_index(pz, tr.halfL, inv_h, n);
          v = make_float4(static_cast<float>(__dsub_rn(__dadd_rn(px, tr.halfL), __dmul_rn(ix, h))),
                          static_cast<float>(__dsub_rn(__dadd_rn(py, tr.halfL), __dmul_rn(iy, h))),
                          static_cast<float>(__dsub_rn(__dadd_rn(pz, tr.halfL), __dmul_rn(iz, h))),
                          __uint_as_float(tid));
          cell = tr.cell_base + cell_encode(ix, iy, iz, tr.cb_ref);
          d.s4[s] = v;
        } else {
          cell = tr.cell_base;  // FP64 mode recomputes cells from positions
          d.sx[s] = px; d.sy[s] = py; d.sz[s] = pz; d.stid[s] = tid;
        }
        d.cell_sorted[s] = cell;
        d.dead[s] = 0;
        }  // unparked or new
      } else {
        cell = c_cell;
        // the occupancy bitmap is rebuilt by this step's gather: clear the words holding
        // the last step's cells (the first slot of each run of equal cells clears its
        // word; the last step's search has finished reading them)
        if (s == 0 || c_prev != cell) d.occ[cell >> 5] = 0u;
        dead = c_dead;
        if (dead) {
          d.dead[s] = 0;
        } else if (F32L) {
          v = c_v;
        } else {
          px = c_x; py = c_y; pz = c_z; tid = c_tid;
        }
      }
      if (dead) {
        key = d.g->sentinel_step;
        ++n_dead_local;
      } else {
        const int b = (d.n_trains == 1) ? 0 : train_of_cell(d.trains, d.n_trains, cell);
        const Train& tr = d.trains[b];
        if (!tr.active && tr.park_now) {
          // park: the species moves to its train's parking buffers and leaves the
          // stepped slots (sorted out with the removed ones)
          const uint32_t am = __activemask();
          const uint32_t peers = __match_any_sync(am, static_cast<uint32_t>(b));
          const int lane = threadIdx.x & 31, leader = __ffs(peers) - 1;
          uint32_t base = 0;
          if (lane == leader) base = atomicAdd(&d.trains[b].park_n, static_cast<uint32_t>(__popc(peers)));
          base = __shfl_sync(peers, base, leader);
          const uint32_t k = base + __popc(peers & ((1u << lane) - 1u));
          if (k < tr.park_cap) {
            const uint32_t q = tr.park_base + k;
            d.pk_cell[q] = cell;
            if (F32L) d.pk4[q] = v;
            else { d.pkx[q] = px; d.pky[q] = py; d.pkz[q] = pz; d.pk_tid[q] = tid; }
          } else {
            raise_status(d.g, CHEM_ECAPACITY);
          }
          key = d.g->sentinel_step;
          ++n_dead_local;
        } else if (!tr.active) {
          if (F32L) d.t4[s] = v;
          else { d.tx[s] = px; d.ty[s] = py; d.tz[s] = pz; d.ttid[s] = tid; }
          key = cell;
        } else if (!F32L) {
          const uint32_t ty = tid_type(tid);
          double g0, g1, g2;
          gauss3_f64(tid_id(tid), tr.step, tr.key0, tr.key1, g0, g1, g2);
          const double sig = tr.sig[ty];
          const double ex = __dmul_rn(sig, g0), ey = __dmul_rn(sig, g1), ez = __dmul_rn(sig, g2);
          double yx, yy, yz;  // from the box corner
          const double x = wrap_box_diffused(__dadd_rn(px, ex), tr.L, tr.halfL, yx);
          const double y = wrap_box_diffused(__dadd_rn(py, ey), tr.L, tr.halfL, yy);
          const double z = wrap_box_diffused(__dadd_rn(pz, ez), tr.L, tr.halfL, yz);
          d.tx[s] = x; d.ty[s] = y; d.tz[s] = z; d.ttid[s] = tid;
          d.tdx[s] = ex; d.tdy[s] = ey; d.tdz[s] = ez;
          const int n = tr.n;
          float ox, oy, oz;  // FP32 offsets from the cell's corner for the pair search's prefilter
          const int ix = cell_index_split(yx, tr.inv_h, n, tr.hf, tr.hlo, tr.inv_hf, ox);
          const int iy = cell_index_split(yy, tr.inv_h, n, tr.hf, tr.hlo, tr.inv_hf, oy);
          const int iz = cell_index_split(yz, tr.inv_h, n, tr.hf, tr.hlo, tr.inv_hf, oz);
          key = tr.cell_base + cell_encode(ix, iy, iz, tr.cb);
          d.t4[s] = make_float4(ox, oy, oz, __uint_as_float(tid));
        } else {
          const uint32_t ftid = __float_as_uint(v.w);
          const uint32_t ty = tid_type(ftid);
          float g0, g1, g2;
          gauss3_f32(tid_id(ftid), tr.step, tr.key0, tr.key1, g0, g1, g2);
          const float sig = tr.sigf[ty];
          const int nr = tr.n_ref;
          int ix, iy, iz;
          cell_decode(cell - tr.cell_base, tr.cb_ref, ix, iy, iz);
          const int n = tr.n;
          const float ex = sig * g0, ey = sig * g1, ez = sig * g2;
          d.td4[s] = make_float4(ex, ey, ez, 0.f);
          float ox, oy, oz;
          if (nr == n) {
            ox = v.x + ex; oy = v.y + ey; oz = v.z + ez;
            const float fx = floorf(ox * tr.inv_hf), fy = floorf(oy * tr.inv_hf), fz = floorf(oz * tr.inv_hf);
            ox -= fx * tr.hf; oy -= fy * tr.hf; oz -= fz * tr.hf;
            const int jx = static_cast<int>(fx), jy = static_cast<int>(fy), jz = static_cast<int>(fz);
            ix = (jx >= -1 && jx <= 1) ? step_cell(ix, jx, n) : wrap_cell(ix + jx, n);
            iy = (jy >= -1 && jy <= 1) ? step_cell(iy, jy, n) : wrap_cell(iy + jy, n);
            iz = (jz >= -1 && jz <= 1) ? step_cell(iz, jz, n) : wrap_cell(iz + jz, n);
          } else {
            // the hash grid changed this step: FP64 position from the box corner, then
            // the new cell and offset (no division)
            const double hr = tr.h_ref;
            const double ax = rebase_corner(ix * hr + static_cast<double>(v.x + ex), tr.L, tr.inv_L);
            const double ay = rebase_corner(iy * hr + static_cast<double>(v.y + ey), tr.L, tr.inv_L);
            const double az = rebase_corner(iz * hr + static_cast<double>(v.z + ez), tr.L, tr.inv_L);
            ix = min(static_cast<int>(ax * tr.inv_h), n - 1);
            iy = min(static_cast<int>(ay * tr.inv_h), n - 1);
            iz = min(static_cast<int>(az * tr.inv_h), n - 1);
            ox = static_cast<float>(ax - ix * tr.h);
            oy = static_cast<float>(ay - iy * tr.h);
            oz = static_cast<float>(az - iz * tr.h);
          }
          d.t4[s] = make_float4(ox, oy, oz, v.w);
          key = tr.cell_base + cell_encode(ix, iy, iz, tr.cb);
        }
      }
      d.keys0[s] = key;  // the first radix pass takes the slot itself as the value
      if (hist)
        for (int p = 0; p < d.passes; ++p) atomicAdd(&hist[p][(key >> (8 * p)) & 255u], 1u);
    }
    count_add(d, rel_b, rel_type, 1, rel_new);
  }
  // warp-aggregate the dead count
  for (int o = 16; o > 0; o >>= 1) n_dead_local += __shfl_xor_sync(0xffffffffu, n_dead_local, o);
  if ((threadIdx.x & 31) == 0 && n_dead_local) atomicAdd(&d.g->n_dead, n_dead_local);
  if (!hist) return;
  __syncthreads();
  if (ok) {
    for (int i = threadIdx.x; i < d.passes * RADIX; i += blockDim.x) {
      const uint32_t c = (&hist[0][0])[i];
      if (c) atomicAdd(&d.g->hist[0][0] + i, c);
    }
  }
}

// ======================================================================== sort pass
// A pass whose digit is the same for every key is the identity and is skipped; the
// ping-pong buffers of the remaining passes follow from the histograms, which every CTA
// reads identically. Bit p of the result: pass p of the n keys has something to do.
__device__ __forceinline__ uint32_t active_passes(const Dev& d, uint32_t n) {
  uint32_t h[MAX_PASSES];
#pragma unroll
  for (int p = 0; p < MAX_PASSES; ++p) h[p] = p < d.passes ? d.g->hist[p][threadIdx.x & (RADIX - 1)] : n;
  uint32_t mask = 0u;
#pragma unroll
  for (int p = 0; p < MAX_PASSES; ++p)
    if (p < d.passes && !__syncthreads_or(static_cast<int>(h[p] == n))) mask |= 1u << p;
  return mask;
}

// Status read once per CTA so that every thread takes the same branch before barriers.
__device__ __forceinline__ bool block_status_ok(const Dev& d) {
  return __syncthreads_and(threadIdx.x == 0 ? (status_of(d) == 0) : 1) != 0;
}

// One pass of the sort, `active` from active_passes. `lead` marks the CTA that records the
// buffers of the result (at the last pass). `first_tile`: thread 0's claim of a tile.
template <int NT>
__device__ void phase_sort_pass(const Dev& d, int pass, uint32_t active, uint32_t n, uint32_t first_tile,
                                SortSmemT<NT>& sm, bool lead) {
  const int before = __popc(active & ((1u << pass) - 1u));
  if (pass == d.passes - 1 && lead && threadIdx.x == 0) {
    const uint32_t all = __popc(active);
    d.g->sort_parity = all & 1u;
    d.g->sort_any = all > 0u ? 1u : 0u;
  }
  if (!((active >> pass) & 1u)) return;
  const bool odd = before & 1;
  const uint32_t* kin = odd ? d.keys1 : d.keys0;
  const uint32_t* vin = before == 0 ? nullptr : (odd ? d.vals1 : d.vals0);  // nullptr: value = index
  uint32_t* kout = odd ? d.keys0 : d.keys1;
  uint32_t* vout = odd ? d.vals0 : d.vals1;
  onesweep_pass(kin, vin, kout, vout, n, 8 * pass, d.g->hist[pass], first_tile, &d.g->tile_ctr[pass],
                d.lookback, d.g->epoch * 2 * MAX_PASSES + pass, d.g, sm);
}

// The whole sort by one CTA in shared memory, for at most SORT_ONE_CTA keys: three passes over
// the grid are three chains of look-back and barrier.
constexpr uint32_t SORT_ONE_CTA = 4096;
struct SortOneSmem {
  uint32_t k0[SORT_ONE_CTA], v0[SORT_ONE_CTA], k1[SORT_ONE_CTA], v1[SORT_ONE_CTA];
};

// ======================================================================== gather
// Reorder the diffused species into cell order, record each cell's slot range (stamped
// with this step's epoch) and drop the dead (sentinel keys sort last).
template <bool F32L>
__device__ void phase_gather(const Dev& d, const Span& sp) {
  if (status_of(d)) return;
  const uint32_t* kf = d.g->sort_parity ? d.keys1 : d.keys0;
  const uint32_t* vf = d.g->sort_any ? (d.g->sort_parity ? d.vals1 : d.vals0) : nullptr;
  const uint32_t n_total = d.g->n_total;
  const uint32_t n_live = n_total - d.g->n_dead;
  const uint32_t epoch = d.g->epoch;
  const uint32_t sentinel = d.g->sentinel_step;
  const uint32_t item_home = d.g->item_home;
  const bool items_now = item_home != 0 && d.g->search_cells_now;
  if (d.bk_cnt)  // the last step's event buckets
    for (uint32_t i = sp.first(); i < d.n_buckets; i += sp.stride()) {
      d.bk_cnt[i] = 0u;
      if (i < d.n_buckets / EV_GROUP) d.bk_group[i] = 0u;
    }
  const uint32_t stride = sp.stride();
  // GATHER_BATCH slots per thread and iteration, their loads in flight together: the
  // permutation and neighbouring keys first, then the gathered state
  for (uint32_t s0 = sp.first(); s0 < n_live; s0 += stride * GATHER_BATCH) {
    uint32_t key[GATHER_BATCH], idx[GATHER_BATCH], prv[GATHER_BATCH], nxt[GATHER_BATCH];
    bool ok[GATHER_BATCH];
#pragma unroll
    for (int g = 0; g < GATHER_BATCH; ++g) {
      const uint32_t s = s0 + static_cast<uint32_t>(g) * stride;
      ok[g] = s < n_live;
      key[g] = 0u; idx[g] = 0u; prv[g] = 0u; nxt[g] = 0u;
      if (ok[g]) {
        key[g] = kf[s];
        idx[g] = vf ? vf[s] : s;
        prv[g] = s > 0 ? kf[s - 1] : 0u;
        nxt[g] = s + 1 < n_live ? kf[s + 1] : 0u;
      }
    }
#pragma unroll
    for (int g = 0; g < GATHER_BATCH; ++g) {
      if (ok[g] && (key[g] >= sentinel || idx[g] >= n_total)) {  // only after a timed-out sort
        raise_status(d.g, CHEM_ETIMEOUT);
        ok[g] = false;
      }
    }
    if (F32L) {
      float4 a[GATHER_BATCH], b[GATHER_BATCH];
#pragma unroll
      for (int g = 0; g < GATHER_BATCH; ++g) {
        if (ok[g]) {
          a[g] = d.t4[idx[g]];
          if (d.sd4) b[g] = d.td4[idx[g]];
        }
      }
#pragma unroll
      for (int g = 0; g < GATHER_BATCH; ++g) {
        if (ok[g]) {
          const uint32_t s = s0 + static_cast<uint32_t>(g) * stride;
          d.s4[s] = a[g];
          if (d.sd4) d.sd4[s] = b[g];
        }
      }
    } else {
#pragma unroll
      for (int g = 0; g < GATHER_BATCH; ++g) {
        if (ok[g]) {
          const uint32_t s = s0 + static_cast<uint32_t>(g) * stride, i = idx[g];
          d.sx[s] = d.tx[i]; d.sy[s] = d.ty[i]; d.sz[s] = d.tz[i]; d.stid[s] = d.ttid[i];
          d.s4[s] = d.t4[i];
        }
      }
    }
#pragma unroll
    for (int g = 0; g < GATHER_BATCH; ++g) {
      if (!ok[g]) continue;
      const uint32_t s = s0 + static_cast<uint32_t>(g) * stride, k = key[g];
      d.cell_sorted[s] = k;
      int* ci = reinterpret_cast<int*>(&d.cell_info[k]);
      const bool first = (s == 0 || prv[g] != k);
      if (first) {
        ci[0] = static_cast<int>(s);
        ci[2] = static_cast<int>(epoch);
        atomicOr(&d.occ[k >> 5], 1u << (k & 31u));
      }
      if (s + 1 == n_live || nxt[g] != k) ci[1] = static_cast<int>(s + 1);
      // pair-search work item: a cell's first slot and every item_home-th slot (none when
      // the search runs one thread per species)
      if (items_now && (first || (s % item_home) == 0)) {
        const int b = (d.n_trains == 1) ? 0 : train_of_cell(d.trains, d.n_trains, k);
        if (d.trains[b].active && !d.trains[b].free_jump) {
          const uint32_t it = atomicAdd(&d.g->n_items, 1u);
          if (it < d.cap_items) d.items[it] = make_uint2(s, k);
          else raise_status(d.g, CHEM_ECAPACITY);
        }
      }
    }
  }
  if (sp.block == 0 && threadIdx.x == 0) d.g->n_live = n_live;
}

// ======================================================================== search
// For every unordered pair of live species whose types react (Table 1), separated by
// less than the reaction's cutoff under the minimum image (Eq. 2), evaluate the
// encounter probability and keep the pair if its uniform falls below it. Three mappings
// visit the same pairs: one thread per home species, several lanes per home (both below) and
// cell tiles (search_cells.cuh). With at least 3 cells per axis each unordered pair is visited
// once: the own cell's later slots and the forward half of the surrounding cells.

// Half-shell offsets: entry 0 is the own cell, 1..13 the cells one away in fwd_offset's
// order; each keeps the offsets (dz, dy, dx) that are lexicographically positive, so
// every unordered pair of cells is met once.
struct FwdOffsets {
  signed char x[N_FWD], y[N_FWD], z[N_FWD];
  int count;
};
constexpr FwdOffsets make_fwd_offsets() {
  FwdOffsets t{};
  int k = 1;
  for (int dy = -1; dy <= 1; ++dy)
    for (int dx = -1; dx <= 1; ++dx) { t.x[k] = static_cast<signed char>(dx); t.y[k] = static_cast<signed char>(dy); t.z[k] = 1; ++k; }
  for (int dx = -1; dx <= 1; ++dx) { t.x[k] = static_cast<signed char>(dx); t.y[k] = 1; t.z[k] = 0; ++k; }
  t.x[k] = 1; t.y[k] = 0; t.z[k] = 0; ++k;
  t.count = k;
  return t;
}
static_assert(make_fwd_offsets().count == N_FWD, "13 forward cells");
static __constant__ FwdOffsets c_fwd = make_fwd_offsets();

// The half-shell offsets in shared memory: looked up with a different offset number in
// each lane, the constant-memory table would serialise a warp's access per distinct
// address. Filled by every thread of the CTA (fwd_smem_fill), then a CTA barrier.
struct FwdSmem {
  float f[3][N_FWD];       // as FP32 factors of the cell side
  int8_t i[3][N_FWD + 2];  // as cell steps
};

__device__ __forceinline__ void fwd_smem_fill(FwdSmem& fo) {
  for (int k = threadIdx.x; k < N_FWD; k += blockDim.x) {
    fo.f[0][k] = c_fwd.x[k]; fo.f[1][k] = c_fwd.y[k]; fo.f[2][k] = c_fwd.z[k];
    fo.i[0][k] = c_fwd.x[k]; fo.i[1][k] = c_fwd.y[k]; fo.i[2][k] = c_fwd.z[k];
  }
}

// Half-shell offsets: 0 = own cell, 1..9 dz = +1, 10..12 (dz, dy) = (0, +1), 13 (0, 0, +1).
__device__ __forceinline__ void fwd_offset(int k, int& dx, int& dy, int& dz) {
  if (k == 0) { dx = dy = dz = 0; return; }
  if (k <= 9) { const int q = k - 1; dz = 1; dy = q / 3 - 1; dx = q % 3 - 1; return; }
  if (k <= 12) { dz = 0; dy = 1; dx = k - 11; return; }
  dz = 0; dy = 0; dx = 1;
}

// The forward cells (bits 1..13) that hold points within the squared cutoff rcmax2 of a home
// at the offset v in its cell. A cell whose nearest point is farther holds no partner and is
// not looked up (the gaps are taken 1e-5 of a cell short, which covers every rounding of the
// offsets). Per axis the gap is 0 (same layer), the distance to the lower face (offset -1) or
// to the upper face (offset +1).
__device__ __forceinline__ uint32_t cells_in_reach(const float4& v, float hf, float rcmax2) {
  rcmax2 *= 1.0001f;
  const float eps = 1e-5f * hf;
  auto gap = [&](int o, float of) {
    const float g = o > 0 ? static_cast<float>(o) * hf - of : (o < 0 ? of + static_cast<float>(-o - 1) * hf : 0.f);
    return fmaxf(g - eps, 0.f);
  };
  const float xm = gap(-1, v.x), xp = gap(1, v.x), ym = gap(-1, v.y), yp = gap(1, v.y), zp = gap(1, v.z);
  const float xm2 = xm * xm, xp2 = xp * xp, ym2 = ym * ym, yp2 = yp * yp, zp2 = zp * zp;
  uint32_t m = 0u;
#pragma unroll
  for (int k = 1; k < N_FWD; ++k) {
    int dx, dy, dz;
    fwd_offset(k, dx, dy, dz);
    const float sx = dx < 0 ? xm2 : (dx > 0 ? xp2 : 0.f);
    const float sy = dy < 0 ? ym2 : (dy > 0 ? yp2 : 0.f);
    const float sz = dz > 0 ? zp2 : 0.f;
    if ((sx + sy) + sz <= rcmax2) m |= 1u << k;
  }
  return m;
}

// FP32 separation x_j - x_i of two species held as offsets from their cells' corners,
// the neighbour's cell lying (cfx, cfy, cfz) cells away (cell side hf), and its square.
// Written with explicit roundings (no contraction left to the compiler) so that every
// kernel that forms it, both search mappings and the acceptance, gets the same bits.
__device__ __forceinline__ float sep_f32(float cfx, float cfy, float cfz, float hf, const float4& vj,
                                         const float4& vi, float& fx, float& fy, float& fz) {
  fx = __fsub_rn(__fmaf_rn(cfx, hf, vj.x), vi.x);
  fy = __fsub_rn(__fmaf_rn(cfy, hf, vj.y), vi.y);
  fz = __fsub_rn(__fmaf_rn(cfz, hf, vj.z), vi.z);
  return __fmaf_rn(fz, fz, __fmaf_rn(fy, fy, __fmul_rn(fx, fx)));
}

// Warp-reduced pair-search counters, added once per warp to the context's totals.
__device__ __forceinline__ void add_pair_counts(const Dev& d, uint32_t tested, uint32_t in_cut) {
  unsigned long long t = tested, c = in_cut;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    t += __shfl_xor_sync(0xffffffffu, t, o);
    c += __shfl_xor_sync(0xffffffffu, c, o);
  }
  if ((threadIdx.x & 31) == 0) {
    if (t) atomicAdd(&d.g->pairs_tested, t);
    if (c) atomicAdd(&d.g->pairs_in_cutoff, c);
  }
}

__device__ __forceinline__ void emit_candidate(const Dev& d, uint32_t s_lo, uint32_t s_hi, uint32_t id_lo,
                                               uint32_t id_hi, int r, int b, double d1sq) {
  const uint32_t c = atomicAdd(&d.g->n_cand, 1u);
  if (c >= d.cap_cand) { raise_status(d.g, CHEM_ECAPACITY); return; }
  atomicAdd(&d.touch[s_lo], 1u);
  atomicAdd(&d.touch[s_hi], 1u);
  Cand cd;
  cd.s_lo = s_lo; cd.s_hi = s_hi; cd.id_lo = id_lo; cd.id_hi = id_hi;
  cd.rxn_train = static_cast<uint32_t>(r) | (static_cast<uint32_t>(b) << 8);
  cd.pad = 0;
  cd.d1sq = d1sq;
  d.cand[c] = cd;
}

// Accept iff u < p with p = bridge_p evaluated in FP64 from the FP32 squared distances.
// The uniform u = (w0:w1 >> 11) 2^-53 of the pair's Philox block lies in
// [k 2^-24, (k + 1) 2^-24) with k = w0 >> 8, bounds that are exact in FP32. An FP32
// estimate of p decides whenever those bounds clear it by twice its error bound (FP32
// rounding of d0, d1, R and of the products, cancellation in d - R, the documented
// __expf error, and a few ulp for the two expm1f and their quotient, whose arguments
// suffer no cancellation since d0 + d1 - R > R); since p <= exp(-a), a uniform above the
// bound of exp(-a) alone rejects before the expm1f. Otherwise u and p are formed in FP64,
// so the outcome is always that of the FP64 test. The fast path uses no FP64
// arithmetic (a slow pipe on this part).
__device__ __forceinline__ bool accept_f32(float d0sq, float d1sq, int r, const Tables& tb, const Train& tr,
                                          uint32_t id_lo, uint32_t id_hi) {
  const float d1f = sqrtf(d1sq), d0f = sqrtf(d0sq);
  const float Rf = tb.Rf[r];
  if (d1f < Rf * 0.999f || d0f < Rf * 0.999f) return true;  // p = 1 > u
  const uint4 w = philox4x32_10(make_uint4(id_lo, tr.step, id_hi, 2u), tr.key0, tr.key1);
  if (d1f > Rf * 1.001f && d0f > Rf * 1.001f) {
    const float a = d0f - Rf, b = d1f - Rf, inv = tr.inv_ddt_f[r];
    const float x = a * b * inv;
    if (x > 60.f) {
      if ((w.x | (w.y >> 11)) != 0u) return false;  // p <= exp(-a) < 1e-26 < 2^-53 <= u
    } else {
      const float ea = __expf(-x);
      const float ulo = static_cast<float>(w.x >> 8) * 5.9604645e-8f;  // k 2^-24 <= u
      const float err = 1.2e-7f * inv * (b * (d0f + Rf) + a * (d1f + Rf)) + 1e-6f * (1.f + x) + 3e-6f;
      // p <= exp(-a): most pairs are rejected on that bound alone
      if (ulo >= ea * (1.f + 2.f * err)) return false;
      const float cb = d0f * d1f * inv, cc = Rf * (d0f + d1f - Rf) * inv;
      const float p = ea * (expm1f(-cc) / expm1f(-cb));
      const float band = 2.f * err * p;
      if (ulo >= p + band) return false;
      if (ulo + 5.9604645e-8f <= p - band) return true;               // u < (k + 1) 2^-24
    }
  }
  const double u = __dmul_rn(static_cast<double>(u53(w.x, w.y)), TWO_POW_M53);
  const double d0 = sqrt(static_cast<double>(d0sq)), d1 = sqrt(static_cast<double>(d1sq));
  return u < bridge_p(d0, d1, tb.R[r], tr.ddt[r]);
}

// The same test for FP64 squared distances: the FP32 estimate starts from their FP32
// roundings (one more rounding, covered by a doubled distance term in the error
// bound), and the exact fallback is the FP64 reference's own arithmetic.
__device__ __forceinline__ bool accept_f64(double d0sq, double d1sq, int r, const Tables& tb, const Train& tr,
                                          uint32_t id_lo, uint32_t id_hi) {
  const float d1f = sqrtf(static_cast<float>(d1sq)), d0f = sqrtf(static_cast<float>(d0sq));
  const float Rf = tb.Rf[r];
  if (d1f < Rf * 0.999f || d0f < Rf * 0.999f) return true;  // p = 1 > u
  const uint4 w = philox4x32_10(make_uint4(id_lo, tr.step, id_hi, 2u), tr.key0, tr.key1);
  if (d1f > Rf * 1.001f && d0f > Rf * 1.001f) {
    const float a = d0f - Rf, b = d1f - Rf, inv = tr.inv_ddt_f[r];
    const float x = a * b * inv;
    if (x > 60.f) {
      if ((w.x | (w.y >> 11)) != 0u) return false;
    } else {
      const float ea = __expf(-x);
      const float ulo = static_cast<float>(w.x >> 8) * 5.9604645e-8f;
      const float err = 2.4e-7f * inv * (b * (d0f + Rf) + a * (d1f + Rf)) + 1e-6f * (1.f + x) + 4e-6f;
      if (ulo >= ea * (1.f + 2.f * err)) return false;  // p <= exp(-a)
      const float cb = d0f * d1f * inv, cc = Rf * (d0f + d1f - Rf) * inv;
      const float p = ea * (expm1f(-cc) / expm1f(-cb));
      const float band = 2.f * err * p;
      if (ulo >= p + band) return false;
      if (ulo + 5.9604645e-8f <= p - band) return true;
    }
  }
  const double u = __dmul_rn(static_cast<double>(u53(w.x, w.y)), TWO_POW_M53);
  return u < bridge_p(sqrt(d0sq), sqrt(d1sq), tb.R[r], tr.ddt[r]);
}

// FP64 mode: may the pair be rejected on FP32 values alone? f2 is the squared FP32 separation
// of the species' cell offsets, (dx, dy, dz) the FP32 start separation; both distances are
// within eps of the exact ones. False: undecided (or to be accepted, which needs the exact
// separation anyway).
__device__ __forceinline__ bool surely_rejected(float d0f, float d1f, float eps, int r, const Tables& tb,
                                                const Train& tr, uint32_t id_lo, uint32_t id_hi) {
  const float Rf = tb.Rf[r];
  if (!(d1f > Rf * 1.001f + eps && d0f > Rf * 1.001f + eps)) return false;
  const uint4 w = philox4x32_10(make_uint4(id_lo, tr.step, id_hi, 2u), tr.key0, tr.key1);
  const float a = d0f - Rf, b = d1f - Rf, inv = tr.inv_ddt_f[r];
  const float x = a * b * inv;
  // accept_f64's error bound with the distances' error eps on top
  const float err = inv * (b * (eps + 2.4e-7f * (d0f + Rf)) + a * (eps + 2.4e-7f * (d1f + Rf)) + eps * eps) +
                    1e-6f * (1.f + x) + 4e-6f;
  if (x > 60.f) return err < 15.f && (w.x | (w.y >> 11)) != 0u;  // p <= exp(-x + err) < 2^-53 <= u
  if (err > 0.25f) return false;
  const float ea = __expf(-x);
  const float ulo = static_cast<float>(w.x >> 8) * 5.9604645e-8f;
  if (ulo >= ea * (1.f + 2.f * err)) return true;  // p <= exp(-a)
  // the quotient's bound below, (1 + 2 z) (1 + z)^2 <= 1 + 8 z for z = eps / R, ends at z = 0.63
  if (!(eps <= 0.25f * Rf)) return false;
  const float cb = d0f * d1f * inv, cc = Rf * (d0f + d1f - Rf) * inv;
  const float p = ea * (expm1f(-cc) / expm1f(-cb));
  // a relative error of cb or cc is at most passed on
  return ulo >= p * (1.f + 2.f * (err + 4.f * eps / Rf));
}

// FP64 mode: FP32 start separation of a pair, from its end separation f and the displacements ei, ej.
// `margin` bounds its error past that of f: the displacements are truncated to 24 bits, an error
// that grows with each of them and not with their difference (3.1e-7 of `size` in all), and the
// sums and squares are rounded (3e-7 of the result).
__device__ __forceinline__ float start_distance_f32(float fx, float fy, float fz, double eix, double eiy, double eiz,
                                                    double ejx, double ejy, double ejz, float& margin) {
  const float ix = truncate_double(eix), iy = truncate_double(eiy), iz = truncate_double(eiz);
  const float jx = truncate_double(ejx), jy = truncate_double(ejy), jz = truncate_double(ejz);
  const float rx = fx - (jx - ix), ry = fy - (jy - iy), rz = fz - (jz - iz);
  const float d0 = sqrtf(rx * rx + ry * ry + rz * rz);
  const float size = fmaxf(fmaxf(fabsf(ix) + fabsf(jx), fabsf(iy) + fabsf(jy)), fabsf(iz) + fabsf(jz));
  margin = 1e-6f * (size + d0);
  return d0;
}

// Acceptance of one queued pair (home slot si, neighbour slot j in the forward cell k of
// the home's cell) and, when accepted, its candidate record. kb = k | train << 8. All
// search mappings queue pairs that passed the FP32 cutoff test and resolve them here, one
// pair per lane. In FP64 mode that test is against a widened cutoff, the FP32 distances
// (error below eps = 2e-6 of a cell, the same margin) reject most pairs, and the rest are
// formed and tested exactly in FP64: the FP64 pipe (two lanes per clock and SM) then only
// sees the few percent that are accepted or close to a decision. The FP64 search of 1e6
// track species (mean over 1 ps to 1 us) went from 469 to 142 us with it.
template <bool F32L>
__device__ __forceinline__ void resolve_pair(const Dev& d, const Tables& tb, const FwdSmem& fo, uint32_t si,
                                             uint32_t j, uint32_t kb, const uint32_t* vf, uint32_t& n_in_cut) {
  const int k = static_cast<int>(kb & 255u), b = static_cast<int>(kb >> 8);
  const Train& tr = d.trains[b];
  const float4 hv = d.s4[si], vj = d.s4[j];
  // the walk's separation, formed the same way
  float fx, fy, fz;
  const float f2 = sep_f32(fo.f[0][k], fo.f[1][k], fo.f[2][k], tr.hf, vj, hv, fx, fy, fz);
  const uint32_t tid_i = __float_as_uint(hv.w), tid_j = __float_as_uint(vj.w);
  const uint32_t ti = tid_type(tid_i), tj = tid_type(tid_j);
  const int r = tb.pair_rxn[ti][tj];
  const uint32_t id_i = tid_id(tid_i), id_j = tid_id(tid_j);
  const bool i_lo = id_i < id_j;
  const uint32_t id_lo = i_lo ? id_i : id_j, id_hi = i_lo ? id_j : id_i;
  if constexpr (F32L) {
    if (!i_lo) { fx = -fx; fy = -fy; fz = -fz; }
    // this step's displacements, gathered into sorted order
    const float4 di = d.sd4[si], dj = d.sd4[j];
    const float4 dlo = i_lo ? di : dj, dhi = i_lo ? dj : di;
    const float r0x = fx - (dhi.x - dlo.x), r0y = fy - (dhi.y - dlo.y), r0z = fz - (dhi.z - dlo.z);
    const float d0sq = r0x * r0x + r0y * r0y + r0z * r0z;
    if (!accept_f32(d0sq, f2, r, tb, tr, id_lo, id_hi)) return;
    emit_candidate(d, i_lo ? si : j, i_lo ? j : si, id_lo, id_hi, r, b, static_cast<double>(f2));
  } else {
    const uint32_t ti_idx = vf ? vf[si] : si, tj_idx = vf ? vf[j] : j;
    const double eix = d.tdx[ti_idx], eiy = d.tdy[ti_idx], eiz = d.tdz[ti_idx];
    const double ejx = d.tdx[tj_idx], ejy = d.tdy[tj_idx], ejz = d.tdz[tj_idx];
    const float eps = 2e-6f * tr.hf;
    const float d1f = sqrtf(f2);
    const bool sure_in = d1f < sqrtf(tr.rc2f_tt[ti * MAXT + tj]) * 0.99999f - eps;
    if (sure_in) {
      ++n_in_cut;
      float margin;
      const float d0f = start_distance_f32(fx, fy, fz, eix, eiy, eiz, ejx, ejy, ejz, margin);
      if (surely_rejected(d0f, d1f, eps + margin, r, tb, tr, id_lo, id_hi)) return;
    }
    // minimum image of x_j - x_i (Eq. 2), exactly as the reference forms it up to the
    // orientation, which is negated below without rounding
    double rx1 = min_image(__dsub_rn(d.sx[j], d.sx[si]), tr.L, tr.halfL);
    double ry1 = min_image(__dsub_rn(d.sy[j], d.sy[si]), tr.L, tr.halfL);
    double rz1 = min_image(__dsub_rn(d.sz[j], d.sz[si]), tr.L, tr.halfL);
    const double d1sq = sq3(rx1, ry1, rz1);
    if (!sure_in) {
      if (!(d1sq < tr.rc2_tt[ti * MAXT + tj])) return;
      ++n_in_cut;
    }
    if (!i_lo) { rx1 = -rx1; ry1 = -ry1; rz1 = -rz1; }
    const double elx = i_lo ? eix : ejx, ely = i_lo ? eiy : ejy, elz = i_lo ? eiz : ejz;
    const double ehx = i_lo ? ejx : eix, ehy = i_lo ? ejy : eiy, ehz = i_lo ? ejz : eiz;
    const double r0x = __dsub_rn(rx1, __dsub_rn(ehx, elx));
    const double r0y = __dsub_rn(ry1, __dsub_rn(ehy, ely));
    const double r0z = __dsub_rn(rz1, __dsub_rn(ehz, elz));
    if (!accept_f64(sq3(r0x, r0y, r0z), d1sq, r, tb, tr, id_lo, id_hi)) return;
    emit_candidate(d, i_lo ? si : j, i_lo ? j : si, id_lo, id_hi, r, b, d1sq);
  }
}

// Pairs queued by one warp: home slot, neighbour slot, half-shell index | train << 8.
template <int CAP>
struct PairQueue {
  uint32_t si[CAP], j[CAP], kb[CAP];
};

// Resolves queued pairs [0, n), 32 at a time; with `all` unset a last part of fewer than 32
// is kept, moved to the front. Returns the pairs kept. Called by the whole warp.
template <bool F32L, int CAP>
__device__ __forceinline__ uint32_t resolve_queue(const Dev& d, const Tables& tb, const FwdSmem& fo,
                                                  PairQueue<CAP>& q, uint32_t n, bool all, const uint32_t* vf,
                                                  int lane, uint32_t& n_in_cut) {
  __syncwarp();
  const uint32_t full = all ? n : n & ~31u;
  for (uint32_t e = lane; e < full; e += 32) resolve_pair<F32L>(d, tb, fo, q.si[e], q.j[e], q.kb[e], vf, n_in_cut);
  __syncwarp();
  const uint32_t rest = n - full;
  if (rest != 0u && full != 0u) {
    uint32_t a = 0, b = 0, c = 0;
    if (static_cast<uint32_t>(lane) < rest) { a = q.si[full + lane]; b = q.j[full + lane]; c = q.kb[full + lane]; }
    __syncwarp();
    if (static_cast<uint32_t>(lane) < rest) { q.si[lane] = a; q.j[lane] = b; q.kb[lane] = c; }
  }
  __syncwarp();
  return rest;
}

// Neighbours whose loads one batch of the per-species walk keeps in flight together (the whole
// batch is loaded, past a range's end too).
constexpr int TPS_UNROLL = 4;
static_assert(TPS_UNROLL <= S4_SPARE, "a batch past the last range stays inside s4");
constexpr int TPS_QCAP = 32 * (TPS_UNROLL + 1);  // fewer than 32 kept pairs and one batch of a warp

// ---- one thread per home species
// Each lane takes one home species (warps take 32 consecutive sorted slots by work stealing),
// keeps the forward cells its largest cutoff can reach (a 13-bit mask from per-axis face gaps)
// and looks up the occupied ones. What bounds the walk over the neighbours found is instruction
// issue, and the homes' walks differ widely (a cell's first home has all others later, its
// last none): with a lane walking its own ranges, the longest walk of a warp took nine
// batches of TPS_UNROLL neighbours where the mean is three. The lanes' ranges are therefore
// cut into batches that go to one list per warp, and every lane takes every 32nd batch
// whosever it is (its home's offsets come from shared memory). A batch is one address and
// four loads at fixed offsets; pairs inside the cutoff go to the warp's pair queue, a whole
// batch with one vote per neighbour, three words a pair. On 1e6 FP32-local track species the
// search took 84, 87, 94, 103 us a step up to 1e-11, 1e-10, 1e-9, 1e-8 s with a walk per
// lane, and takes 64, 65, 69, 81 (with 64 registers, for 32 warps per SM, of it 3 %).
constexpr int TPS_EMIT = 8;                        // batches a lane lists at a time
constexpr int TPS_LIST = 32 * (TPS_EMIT + 1);      // fewer than 32 waiting and one round's

template <bool F32L, int W>
struct TpsSmem {
  float ct[W][MAXT * MAXT];  // per warp: squared cutoffs of one train (-1: no reaction) ...
  int ct_b[W];               // ... that train
  float4 hv[W][32];          // the homes' cell offsets and id/type bits
  uint2 list[W][TPS_LIST];   // batches: first slot; home lane | half-shell index << 5 | slots << 9
  uint16_t pl[W][32 * (N_FWD - 1)];  // (home, forward cell) pairs: home lane | half-shell index << 5
  PairQueue<TPS_QCAP> q[W];
  FwdSmem fo;                // half-shell offsets
};

template <bool F32L, int W>
__device__ void phase_search_tps(const Dev& d, TpsSmem<F32L, W>& sm) {
  constexpr uint32_t FULL = 0xffffffffu;
  if (d.g->search_cells_now) return;  // this step runs the cell tiles (grid-uniform)
  const uint32_t n_live = d.g->n_total - d.g->n_dead;
  const uint32_t epoch = d.g->epoch;
  const uint32_t* vf = d.g->sort_any ? (d.g->sort_parity ? d.vals1 : d.vals0) : nullptr;
  const Tables& tb = *d.tables;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  PairQueue<TPS_QCAP>& q = sm.q[wib];
  uint32_t qn = 0;  // queued pairs (warp-uniform)
  fwd_smem_fill(sm.fo);
  if (lane == 0) sm.ct_b[wib] = -1;
  // one status for the whole CTA (a barrier, which also publishes the offsets)
  if (!block_status_ok(d)) return;
  const FwdSmem& fo = sm.fo;
  const uint32_t lanemask_lt = (1u << lane) - 1u;
  const uint32_t n_chunks = (n_live + 31u) / 32u;
  uint32_t n_tested = 0, n_in_cut = 0;  // pair-search counters of this lane
  uint32_t c_next = 0;
  if (lane == 0) c_next = atomicAdd(&d.g->item_ctr, 1u);
  c_next = __shfl_sync(FULL, c_next, 0);
  while (c_next < n_chunks) {
    const uint32_t c = c_next;
    if (lane == 0) c_next = atomicAdd(&d.g->item_ctr, 1u);  // the next chunk, used at the end
    const uint32_t s = c * 32u + static_cast<uint32_t>(lane);
    bool home = s < n_live;
    uint32_t cell = 0;
    float4 vi = make_float4(0.f, 0.f, 0.f, 0.f);
    if (home) {
      cell = d.cell_sorted[s];
      vi = d.s4[s];  // FP64 mode tests pairs first on these FP32 cell offsets
    }
    const int b = (d.n_trains == 1 || !home) ? 0 : train_of_cell(d.trains, d.n_trains, cell);
    const Train& tr = d.trains[b];
    const uint32_t ti = tid_type(__float_as_uint(vi.w));
    home = home && tr.active && !tr.free_jump && tb.reactive_mask[ti] != 0u;
    if (!__any_sync(FULL, home)) {
      c_next = __shfl_sync(FULL, c_next, 0);
      continue;
    }
    // cutoffs from the warp's table of its train when every lane of the chunk is in one train
    // (refilled only when the train changes), else from the trains' records
    const int b0 = __shfl_sync(FULL, b, 0);
    const bool mixed = !__all_sync(FULL, b == b0);
    if (!mixed && sm.ct_b[wib] != b0) {
      const Train& t0 = d.trains[b0];
      for (int qq = lane; qq < MAXT * MAXT; qq += 32) sm.ct[wib][qq] = F32L ? t0.rc2f_tt[qq] : t0.rc2w_tt[qq];
      __syncwarp();
      if (lane == 0) sm.ct_b[wib] = b0;
    }
    __syncwarp();  // (the last chunk's homes are no longer read)
    sm.hv[wib][lane] = vi;
    __syncwarp();
    const float hf = tr.hf;
    // the lane's range: first its own cell's later slots, then one of the warp's forward cells
    uint32_t ja = 0u, ea = 0u, meta = static_cast<uint32_t>(lane), kmask = 0u;
    if (home) {
      ja = s + 1u;
      ea = static_cast<uint32_t>(d.cell_info[cell].y);
      float rcmax2 = -1.f;
#pragma unroll
      for (int t = 0; t < MAXT; ++t)
        rcmax2 = fmaxf(rcmax2, mixed ? (F32L ? tr.rc2f_tt[ti * MAXT + t] : tr.rc2w_tt[ti * MAXT + t])
                                     : sm.ct[wib][ti * MAXT + t]);
      kmask = cells_in_reach(vi, hf, rcmax2);
    }
    // the (home, forward cell) pairs within reach go to a list too: one round of lookups covers
    // what a few homes close to their cells' faces would else do in several
    uint32_t pairs, pair_at;
    {
      const uint32_t mine = __popc(kmask);
      uint32_t incl = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += y;
      }
      pairs = __shfl_sync(FULL, incl, 31);
      pair_at = incl - mine;
      while (kmask != 0u) {
        const uint32_t k = static_cast<uint32_t>(__ffs(kmask)) - 1u;
        kmask &= kmask - 1u;
        sm.pl[wib][pair_at++] = static_cast<uint16_t>(static_cast<uint32_t>(lane) | (k << 5));
      }
      __syncwarp();
    }
    uint32_t ln = 0;  // listed batches (warp-uniform)
    // batches list[at, at + n), one per lane
    auto take = [&](uint32_t at, uint32_t n) {
      uint2 e = make_uint2(0u, 0u);
      if (static_cast<uint32_t>(lane) < n) e = sm.list[wib][at + static_cast<uint32_t>(lane)];
      const uint32_t h = e.y & 31u, k = (e.y >> 5) & 15u, left = e.y >> 9;
      const float4* src = d.s4 + e.x;
      float4 vj[TPS_UNROLL];
#pragma unroll
      for (int u = 0; u < TPS_UNROLL; ++u) vj[u] = src[u];
      const float4 vh = sm.hv[wib][h];
      const float* row = &sm.ct[wib][tid_type(__float_as_uint(vh.w)) * MAXT];
      float hfh = hf;
      int bh = b0;
      if (mixed) {
        bh = __shfl_sync(FULL, b, static_cast<int>(h));
        const Train& th = d.trains[bh];
        hfh = th.hf;
        row = (F32L ? th.rc2f_tt : th.rc2w_tt) + tid_type(__float_as_uint(vh.w)) * MAXT;
      }
      const float bx = fo.f[0][k], by = fo.f[1][k], bz = fo.f[2][k];
      uint32_t bal[TPS_UNROLL], any = 0u;
#pragma unroll
      for (int u = 0; u < TPS_UNROLL; ++u) {
        float fx, fy, fz;
        const float rc2u = static_cast<uint32_t>(u) < left ? row[__float_as_uint(vj[u].w) & 7u] : -1.f;
        const bool pass = sep_f32(bx, by, bz, hfh, vj[u], vh, fx, fy, fz) < rc2u;  // -1: the types do not react
        n_tested += rc2u >= 0.f ? 1u : 0u;  // reacting type pairs only
        if constexpr (F32L) n_in_cut += pass ? 1u : 0u;
        bal[u] = __ballot_sync(FULL, pass);
        any |= bal[u];
      }
      if (any != 0u) {  // the same for every lane
#pragma unroll
        for (int u = 0; u < TPS_UNROLL; ++u) {
          if ((bal[u] >> lane) & 1u) {
            const uint32_t pos = qn + __popc(bal[u] & lanemask_lt);
            q.si[pos] = c * 32u + h;
            q.j[pos] = e.x + static_cast<uint32_t>(u);
            q.kb[pos] = k | (static_cast<uint32_t>(bh) << 8);
          }
          qn += __popc(bal[u]);
        }
        if (qn >= 32u) qn = resolve_queue<F32L>(d, tb, fo, q, qn, false, vf, lane, n_in_cut);
      }
    };
    for (uint32_t p0 = 0;; p0 += 32u) {
      // list the ranges' batches, up to TPS_EMIT of a lane at a time, and take them 32 by 32
      while (__any_sync(FULL, ja < ea)) {
        const uint32_t nb = ja < ea ? min((ea - ja + (TPS_UNROLL - 1u)) / TPS_UNROLL, static_cast<uint32_t>(TPS_EMIT)) : 0u;
        uint32_t incl = nb;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(FULL, incl, o);
          if (lane >= o) incl += y;
        }
        const uint32_t at = ln + incl - nb;
        for (uint32_t i = 0; i < nb; ++i) {
          sm.list[wib][at + i] = make_uint2(ja, meta | (min(ea - ja, static_cast<uint32_t>(TPS_UNROLL)) << 9));
          ja += TPS_UNROLL;
        }
        ln += __shfl_sync(FULL, incl, 31);
        __syncwarp();
        while (ln >= 32u) {
          ln -= 32u;
          take(ln, 32u);
        }
        __syncwarp();  // the places taken are listed anew
      }
      if (p0 >= pairs) break;
      // the next 32 pairs: the cell's bitmap word and, when it is occupied, its entry
      const uint32_t p = p0 + static_cast<uint32_t>(lane);
      meta = p < pairs ? sm.pl[wib][p] : 0u;
      const int h = static_cast<int>(meta & 31u), k = static_cast<int>(meta >> 5);
      const uint32_t hcell = __shfl_sync(FULL, cell, h);
      const Train& th = mixed ? d.trains[__shfl_sync(FULL, b, h)] : tr;
      ja = ea = 0u;
      if (p < pairs) {
        const int n = th.n;
        int ix, iy, iz;
        cell_decode(hcell - th.cell_base, th.cb, ix, iy, iz);
        const uint32_t nc = th.cell_base + cell_encode(step_cell(ix, fo.i[0][k], n), step_cell(iy, fo.i[1][k], n),
                                                       step_cell(iz, fo.i[2][k], n), th.cb);
        if ((d.occ[nc >> 5] >> (nc & 31u)) & 1u) {
          const int4 ci = d.cell_info[nc];
          if (static_cast<uint32_t>(ci.z) == epoch) {
            ja = static_cast<uint32_t>(ci.x);
            ea = static_cast<uint32_t>(ci.y);
          }
        }
      }
    }
    if (ln != 0u) take(0u, ln);
    c_next = __shfl_sync(FULL, c_next, 0);
  }
  resolve_queue<F32L>(d, tb, fo, q, qn, true, vf, lane, n_in_cut);
  add_pair_counts(d, n_tested, n_in_cut);
}

// ---- several lanes per home species
// With fewer home species than lanes on the chip, the time of a step's search is the chain
// of one home's dependent loads and its serial walk (16 to 66 us at 2,000 to 31,000 species
// with one lane per home, however few pairs there are; 10 to 29 us with several). Here 2^lg lanes share a home: each
// looks up every 2^lg-th cell of the half shell with all its loads in flight together, the
// non-empty ranges of a home are laid end to end, and its lanes take every 2^lg-th neighbour
// of that list. The same pairs are visited and queued.
constexpr int GRP_UNROLL = 4;    // neighbours a lane keeps in flight

template <int W>
struct GrpSmem {
  uint32_t rs[W][N_FWD][16];    // per home of the warp: first slot of its ranges,
  uint32_t off[W][N_FWD][16];   // their offsets in its neighbour list,
  uint8_t rk[W][N_FWD][16];     // and half-shell indices
  PairQueue<32 * (GRP_UNROLL + 1)> q[W];
  FwdSmem fo;
};

// Warp `warp` of `n_warps` (at most all of the launch) takes every n_warps-th set of homes.
template <bool F32L, int W>
__device__ void phase_search_groups(const Dev& d, GrpSmem<W>& sm, int lg, uint32_t warp, uint32_t n_warps) {
  constexpr uint32_t FULL = 0xffffffffu;
  const uint32_t n_live = d.g->n_total - d.g->n_dead;
  const uint32_t epoch = d.g->epoch;
  const uint32_t* vf = d.g->sort_any ? (d.g->sort_parity ? d.vals1 : d.vals0) : nullptr;
  const Tables& tb = *d.tables;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const uint32_t lanemask_lt = (1u << lane) - 1u;
  auto& q = sm.q[wib];
  uint32_t qn = 0, n_tested = 0, n_in_cut = 0;
  fwd_smem_fill(sm.fo);
  if (!block_status_ok(d)) return;  // (a barrier, which also publishes the offsets)
  const FwdSmem& fo = sm.fo;
  const int G = 1 << lg, g = lane & (G - 1), grp = lane >> lg;
  const uint32_t homes = 32u >> lg;
  const uint32_t n_sets = (n_live + homes - 1u) / homes;
  const uint32_t grp_mask = (lg == 5 ? FULL : (1u << G) - 1u) << (grp << lg);
  for (uint32_t c = warp; c < n_sets; c += n_warps) {
    const uint32_t s = c * homes + static_cast<uint32_t>(grp);
    bool home = s < n_live;
    uint32_t cell = 0;
    float4 vi = make_float4(0.f, 0.f, 0.f, 0.f);
    if (home) {
      cell = d.cell_sorted[s];
      vi = d.s4[s];
    }
    const int b = (d.n_trains == 1 || !home) ? 0 : train_of_cell(d.trains, d.n_trains, cell);
    const Train& tr = d.trains[b];
    const uint32_t ti = tid_type(__float_as_uint(vi.w));
    home = home && tr.active && !tr.free_jump && tb.reactive_mask[ti] != 0u;
    const float* row = F32L ? &tr.rc2f_tt[ti * MAXT] : &tr.rc2w_tt[ti * MAXT];
    float rc2[MAXT];
#pragma unroll
    for (int u = 0; u < MAXT; ++u) rc2[u] = row[u];
    const float hf = tr.hf;
    // the cells in reach (as in phase_search_tps), every G-th of them this lane's
    uint32_t kmask = 0u;
    int ix = 0, iy = 0, iz = 0;
    const int n = tr.n;
    if (home) {
      cell_decode(cell - tr.cell_base, tr.cb, ix, iy, iz);
      float rcmax2 = -1.f;
#pragma unroll
      for (int u = 0; u < MAXT; ++u) rcmax2 = fmaxf(rcmax2, rc2[u]);
      kmask = 1u | cells_in_reach(vi, hf, rcmax2);
    }
    constexpr int MAX_MINE = N_FWD / 2;  // with two lanes per home
    uint32_t nc[MAX_MINE], word[MAX_MINE];
#pragma unroll
    for (int i = 0; i < MAX_MINE; ++i) {
      const int k = g + (i << lg);
      nc[i] = 0u;
      word[i] = 0u;
      if (k < N_FWD && ((kmask >> k) & 1u)) {
        nc[i] = tr.cell_base + cell_encode(step_cell(ix, fo.i[0][k], n), step_cell(iy, fo.i[1][k], n),
                                           step_cell(iz, fo.i[2][k], n), tr.cb);
        word[i] = (d.occ[nc[i] >> 5] >> (nc[i] & 31u)) & 1u;
      }
    }
    uint32_t st[MAX_MINE], len[MAX_MINE];
#pragma unroll
    for (int i = 0; i < MAX_MINE; ++i) {
      st[i] = 0u;
      len[i] = 0u;
      if (word[i]) {
        const int4 ci = d.cell_info[nc[i]];
        if (static_cast<uint32_t>(ci.z) == epoch) {
          st[i] = (g + (i << lg)) == 0 ? s + 1u : static_cast<uint32_t>(ci.x);  // own cell: its later slots
          len[i] = static_cast<uint32_t>(ci.y) > st[i] ? static_cast<uint32_t>(ci.y) - st[i] : 0u;
        }
      }
    }
    // the home's non-empty ranges end to end (the order does not matter)
    uint32_t nr = 0, total = 0;
#pragma unroll
    for (int i = 0; i < MAX_MINE; ++i) {
      if ((i << lg) >= N_FWD) break;
      const uint32_t bal = __ballot_sync(FULL, len[i] > 0u) & grp_mask;
      uint32_t incl = len[i];
      for (int o = 1; o < G; o <<= 1) {
        const uint32_t y = __shfl_up_sync(FULL, incl, o, G);
        if (g >= o) incl += y;
      }
      if (len[i] > 0u) {
        const uint32_t at = nr + __popc(bal & lanemask_lt);
        sm.rs[wib][at][grp] = st[i];
        sm.off[wib][at][grp] = total + incl - len[i];
        sm.rk[wib][at][grp] = static_cast<uint8_t>(g + (i << lg));
      }
      nr += __popc(bal);
      total += __shfl_sync(FULL, incl, G - 1, G);
    }
    __syncwarp();
    uint32_t r = 0, f = static_cast<uint32_t>(g);  // this lane's place in the list
    while (__any_sync(FULL, f < total)) {
      uint32_t ju[GRP_UNROLL], ku[GRP_UNROLL];
      float4 vj[GRP_UNROLL];
#pragma unroll
      for (int u = 0; u < GRP_UNROLL; ++u) {
        ju[u] = 0u;
        ku[u] = 0xFFu;  // no neighbour
        if (f < total) {
          while (r + 1u < nr && sm.off[wib][r + 1u][grp] <= f) ++r;
          ju[u] = sm.rs[wib][r][grp] + (f - sm.off[wib][r][grp]);
          ku[u] = sm.rk[wib][r][grp];
        }
        f += static_cast<uint32_t>(G);
      }
#pragma unroll
      for (int u = 0; u < GRP_UNROLL; ++u) vj[u] = d.s4[ju[u]];
      uint32_t bal[GRP_UNROLL], any = 0u;
#pragma unroll
      for (int u = 0; u < GRP_UNROLL; ++u) {
        const uint32_t k = ku[u] == 0xFFu ? 0u : ku[u];
        const uint32_t tj = __float_as_uint(vj[u].w) & 7u;
        const float rc2u = ku[u] == 0xFFu ? -1.f : (F32L ? tr.rc2f_tt[ti * MAXT + tj] : tr.rc2w_tt[ti * MAXT + tj]);
        float fx, fy, fz;
        const bool pass = sep_f32(fo.f[0][k], fo.f[1][k], fo.f[2][k], hf, vj[u], vi, fx, fy, fz) < rc2u;
        n_tested += rc2u >= 0.f ? 1u : 0u;
        if constexpr (F32L) n_in_cut += pass ? 1u : 0u;
        bal[u] = __ballot_sync(FULL, pass);
        any |= bal[u];
      }
      if (any != 0u) {
#pragma unroll
        for (int u = 0; u < GRP_UNROLL; ++u) {
          if ((bal[u] >> lane) & 1u) {
            const uint32_t pos = qn + __popc(bal[u] & lanemask_lt);
            q.si[pos] = s; q.j[pos] = ju[u]; q.kb[pos] = ku[u] | (static_cast<uint32_t>(b) << 8);
          }
          qn += __popc(bal[u]);
        }
        if (qn >= 32u) qn = resolve_queue<F32L>(d, tb, fo, q, qn, false, vf, lane, n_in_cut);
      }
    }
    __syncwarp();  // the next set rewrites the ranges
  }
  resolve_queue<F32L>(d, tb, fo, q, qn, true, vf, lane, n_in_cut);
  add_pair_counts(d, n_tested, n_in_cut);
}

// ======================================================================== react
// One reaction per species (Sec. 2.4: diffusion-controlled reactions, reactants react
// on encounter):
//  1. phase_match_fast (all CTAs): an accepted pair whose two species are in no other
//     accepted pair is committed at once; the others go to a conflict list.
//  2. phase_match_rounds (one CTA): rounds of locally-dominant selection over the
//     conflict list; a pair is committed when it is the smallest (d1^2, id_lo, id_hi)
//     remaining pair of both its species. Together with 1 this equals the greedy walk
//     over all accepted pairs sorted by that key (closest first, lower ids first).
//  3. phase_react_serial runs 2 and then, in the same CTA, orders the events by
//     (train, id_lo) (a bucket or radix sort in shared memory when they fit, or in large
//     contexts the prefix over their event buckets) and forms the product-count
//     prefix in that order;
//  4. phase_products (all CTAs): product ids and positions at the diffusion-weighted
//     encounter point (Table 1 right-hand sides), tallies summed per CTA, event log;
//  5. phase_end_step (one CTA): FP64 clock, step counter, dt growth, step records.
struct MatchSmem {
  uint32_t n_alive, n_next;
  uint32_t n_won, won_base;
  uint32_t n_conflict;
};

// Events ordered in shared memory by the one-CTA react kernel (4 arrays of this size).
constexpr int EV_SMEM_CAP = 8192;

struct BlockSortSmem {
  uint32_t whist[REACT_THREADS / 32][RADIX];  // per warp: digit counts, then offsets
  uint32_t dtot[RADIX];                       // digit totals, then digit starts
  uint32_t trivial[4];                        // pass p has one digit for every key
};

struct ScanSmem {
  uint32_t carry;
  uint32_t warp_tot[REACT_THREADS / 32];
  uint32_t total;
  uint32_t first_pref[MAX_TRAINS];  // product prefix at the train's first event ...
  uint32_t first_k[MAX_TRAINS];     // ... and that event's position
  uint32_t prods_tr[MAX_TRAINS];
  uint32_t evs_tr[MAX_TRAINS];
};

struct ProductsSmem {
  int dcount[MAX_TRAINS][MAXT];
  int devents[MAX_TRAINS][MAXR];
  int dwater[MAX_TRAINS];
};

struct EndSmem {
  uint32_t any, stepped, ahead;
};

// Exclusive block-wide prefix of v (one value per thread); `total` gets the block sum.
// Warp totals are scanned once by warp 0.
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t* warp_tot, uint32_t* total_s,
                                                    uint32_t& total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_tot[w] = x;
  __syncthreads();
  if (w == 0) {
    const uint32_t t = lane < nw ? warp_tot[lane] : 0u;
    uint32_t y = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t z = __shfl_up_sync(0xffffffffu, y, o);
      if (lane >= o) y += z;
    }
    if (lane < nw) warp_tot[lane] = y - t;
    if (lane == 31) *total_s = y;
  }
  __syncthreads();
  total = *total_s;
  const uint32_t r = x - v + warp_tot[w];
  __syncthreads();
  return r;
}

__device__ __forceinline__ uint32_t event_key(const Dev& d, const Cand& cd) {
  const uint32_t b = cd.rxn_train >> 8;
  return d.train_bits ? ((b << (32 - d.train_bits)) | cd.id_lo) : cd.id_lo;
}

// Event value: candidate index (< 2^24) with the reaction's product count in bits 24-25.
constexpr uint32_t EV_CAND_MASK = 0xFFFFFFu;

// Consecutive indices from *counter for the lanes with `pred` set, one atomic per warp.
// Every lane of the warp must call it.
__device__ __forceinline__ uint32_t warp_reserve(uint32_t* counter, bool pred) {
  const uint32_t m = __ballot_sync(0xffffffffu, pred);
  const int lane = threadIdx.x & 31;
  const int leader = m ? __ffs(m) - 1 : 0;
  uint32_t base = 0;
  if (m && lane == leader) base = atomicAdd(counter, static_cast<uint32_t>(__popc(m)));
  base = __shfl_sync(0xffffffffu, base, leader);
  return base + static_cast<uint32_t>(__popc(m & ((1u << lane) - 1u)));
}

// Events of large contexts are ordered by (train, id_lo) with buckets: a train's ids up to its
// next id, in equal parts (the FP32 product is monotonic, so the buckets ascend with the ids).
// A step of 1e6 species has up to 7,000 events on 16,384 buckets; one CTA scans the counts of
// groups of buckets, and the few events of a bucket are ranked where they are written. Sorting
// them in one CTA took 10 us at 7,000 events and 90 us from 8,192 on (in global memory).
__device__ __forceinline__ uint32_t event_bucket(const Dev& d, uint32_t b, uint32_t id_lo) {
  const Train& tr = d.trains[b];
  const float per_id = static_cast<float>(tr.bk_n) / static_cast<float>(tr.next_id);
  return tr.bk_base + min(tr.bk_n - 1u, static_cast<uint32_t>(static_cast<float>(id_lo) * per_id));
}

// Record accepted pair c as event number e (reserved by the caller).
__device__ __forceinline__ void commit_event(const Dev& d, uint32_t c, const Cand& cd, uint32_t e) {
  d.dead[cd.s_lo] = 1;
  d.dead[cd.s_hi] = 1;
  const uint32_t key = event_key(d, cd), np = static_cast<uint32_t>(d.tables->n_prod[cd.rxn_train & 255u]);
  d.ev_k0[e] = key;
  d.ev_v0[e] = c | (np << 24);
  if (d.bk_cnt) {
    const uint32_t x = event_bucket(d, cd.rxn_train >> 8, cd.id_lo);
    const uint32_t at = atomicAdd(&d.bk_cnt[x], 1u | (np << 16)) & 0xFFFFu;
    atomicAdd(&d.bk_group[x / EV_GROUP], 1u | (np << 16));
    if (at < EV_SLOTS) d.bk_slot[x * EV_SLOTS + at] = (static_cast<unsigned long long>(key) << 32) | c | (np << 24);
    else d.g->bk_overflow = 1u;
  }
}

static __device__ void phase_match_fast(const Dev& d, const Span& sp) {
  const bool ok = block_status_ok(d);  // includes a barrier
  const uint32_t n_c = ok ? min(d.g->n_cand, d.cap_cand) : 0u;
  const uint32_t lane = threadIdx.x & 31u;
  for (uint32_t c0 = sp.first() - lane; c0 < n_c; c0 += sp.stride()) {  // uniform per warp
    const uint32_t c = c0 + lane;
    const bool valid = c < n_c;
    Cand cd{};
    bool lone = false;
    if (valid) {
      cd = d.cand[c];
      lone = d.touch[cd.s_lo] == 1u && d.touch[cd.s_hi] == 1u;
    }
    const uint32_t e = warp_reserve(&d.g->n_events, valid && lone);
    const uint32_t a = warp_reserve(&d.g->n_conflict, valid && !lone);
    if (valid && lone) {
      commit_event(d, c, cd, e);
      d.touch[cd.s_lo] = 0u;
      d.touch[cd.s_hi] = 0u;
    } else if (valid) {
      d.alive0[a] = c;
    }
  }
}

static __device__ void phase_match_rounds(const Dev& d, MatchSmem& sm) {
  const int tid = threadIdx.x;
  const int nt = blockDim.x;
  const bool ok = block_status_ok(d);
  unsigned long long* bd = reinterpret_cast<unsigned long long*>(d.keys0);
  unsigned long long* bp = bd + d.cap;
  const uint32_t n_c = ok ? d.g->n_conflict : 0u;
  if (tid == 0) sm.n_alive = n_c;
  // the rounds do not use the accepted-pair counts: reset them for the next step now
  for (uint32_t i = tid; i < n_c; i += nt) {
    const Cand cd = d.cand[d.alive0[i]];
    d.touch[cd.s_lo] = 0u;
    d.touch[cd.s_hi] = 0u;
  }
  __syncthreads();
  uint32_t* alive = d.alive0;
  uint32_t* nxt = d.alive1;
  for (uint32_t round = 0; sm.n_alive > 0; ++round) {
    if (round > n_c) {
      if (tid == 0) raise_status(d.g, CHEM_ESTATE);
      break;
    }
    const uint32_t na = sm.n_alive;
    for (uint32_t i = tid; i < na; i += nt) {
      const Cand cd = d.cand[alive[i]];
      bd[cd.s_lo] = ~0ull; bd[cd.s_hi] = ~0ull;
      bp[cd.s_lo] = ~0ull; bp[cd.s_hi] = ~0ull;
    }
    __syncthreads();
    for (uint32_t i = tid; i < na; i += nt) {
      const Cand cd = d.cand[alive[i]];
      const unsigned long long kd = __double_as_longlong(cd.d1sq);
      atomicMin(&bd[cd.s_lo], kd);
      atomicMin(&bd[cd.s_hi], kd);
    }
    __syncthreads();
    for (uint32_t i = tid; i < na; i += nt) {
      const Cand cd = d.cand[alive[i]];
      const unsigned long long kd = __double_as_longlong(cd.d1sq);
      const unsigned long long kp = (static_cast<unsigned long long>(cd.id_lo) << 32) | cd.id_hi;
      if (bd[cd.s_lo] == kd) atomicMin(&bp[cd.s_lo], kp);
      if (bd[cd.s_hi] == kd) atomicMin(&bp[cd.s_hi], kp);
    }
    __syncthreads();
    for (uint32_t i0 = 0; i0 < na; i0 += nt) {  // uniform trip count (warp_reserve)
      const uint32_t i = i0 + tid;
      bool win = false;
      uint32_t c = 0;
      Cand cd{};
      if (i < na) {
        c = alive[i];
        cd = d.cand[c];
        const unsigned long long kd = __double_as_longlong(cd.d1sq);
        const unsigned long long kp = (static_cast<unsigned long long>(cd.id_lo) << 32) | cd.id_hi;
        win = bd[cd.s_lo] == kd && bp[cd.s_lo] == kp && bd[cd.s_hi] == kd && bp[cd.s_hi] == kp;
      }
      const uint32_t e = warp_reserve(&d.g->n_events, win);
      if (win) commit_event(d, c, cd, e);
    }
    if (tid == 0) sm.n_next = 0;
    __syncthreads();
    for (uint32_t i0 = 0; i0 < na; i0 += nt) {
      const uint32_t i = i0 + tid;
      bool keep = false;
      uint32_t c = 0;
      if (i < na) {
        c = alive[i];
        const Cand cd = d.cand[c];
        keep = !d.dead[cd.s_lo] && !d.dead[cd.s_hi];
      }
      const uint32_t a = warp_reserve(&sm.n_next, keep);
      if (keep) nxt[a] = c;
    }
    __syncthreads();
    if (tid == 0) sm.n_alive = sm.n_next;
    uint32_t* tmp = alive; alive = nxt; nxt = tmp;
    __syncthreads();
  }
  __syncthreads();
}

// The conflict rounds of phase_match_rounds with everything in shared memory: the
// conflict pairs, a hash of their slots to local indices, and per local slot the
// smallest (d1^2) and then smallest (id_lo, id_hi) key of its remaining pairs. Returns
// false (nothing done) when the conflict list does not fit; the caller then runs the
// global-memory version. `sbuf` holds RC_SMEM_BYTES.
constexpr int RC_CAP = 1536;                 // conflict pairs
__host__ __device__ constexpr uint32_t rc_hash(uint32_t n_c) {  // hash buckets: at least two per slot
  uint32_t h = 64u;
  while (h < 4u * n_c) h <<= 1;
  return h;
}
// Bytes of sbuf for `cap` pairs (two slots each).
__host__ __device__ constexpr size_t rc_smem_bytes(uint32_t cap) {
  return static_cast<size_t>(cap) * (4 + 4 + 4 + 4 + 4 + 8 + 8) + static_cast<size_t>(rc_hash(cap)) * 8 +
         static_cast<size_t>(2 * cap) * (8 + 8 + 4);
}
constexpr size_t RC_SMEM_BYTES = rc_smem_bytes(RC_CAP);

// The rounds over the n_c accepted pairs list[0, n_c) (nullptr: pairs 0 .. n_c - 1, of which
// sm.n_conflict share a species with another), sbuf of rc_smem_bytes(n_c) or more:
// sm.n_won winners, their pairs' indices in the returned list (in sbuf).
static __device__ const uint32_t* match_rounds_in_smem(const Dev& d, MatchSmem& sm, uint32_t* sbuf, uint32_t n_c,
                                                       const uint32_t* list, const Cand* first = nullptr) {
  const int tid = threadIdx.x, nt = blockDim.x;
  const uint32_t hash = rc_hash(n_c);
  // carve the buffer (8-byte arrays first)
  unsigned long long* kd = reinterpret_cast<unsigned long long*>(sbuf);
  unsigned long long* kp = kd + n_c;
  unsigned long long* bd = kp + n_c;
  unsigned long long* bp = bd + 2 * n_c;
  uint32_t* hkey = reinterpret_cast<uint32_t*>(bp + 2 * n_c);
  uint32_t* hval = hkey + hash;
  uint32_t* lo = hval + hash;
  uint32_t* hi = lo + n_c;
  uint32_t* cix = hi + n_c;
  uint32_t* alive = cix + n_c;
  uint32_t* nxt = alive + n_c;
  uint32_t* ldead = nxt + n_c;  // per slot: its pairs, and DEAD once it reacted
  constexpr uint32_t DEAD = 0x80000000u;
  for (uint32_t i = tid; i < hash; i += nt) hkey[i] = 0xFFFFFFFFu;
  for (uint32_t i = tid; i < 2 * n_c; i += nt) ldead[i] = 0u;
  if (tid == 0) { sm.n_alive = n_c; sm.n_next = 0; sm.n_conflict = 0; }
  __syncthreads();
  // load the pairs, reset the accepted-pair counts for the next step, insert the slots
  for (uint32_t i = tid; i < n_c; i += nt) {
    const uint32_t c = list ? list[i] : i;
    const Cand cd = first && i == static_cast<uint32_t>(tid) ? *first : d.cand[c];  // (first: pair `tid`)
    d.touch[cd.s_lo] = 0u;
    d.touch[cd.s_hi] = 0u;
    cix[i] = c;
    kd[i] = static_cast<unsigned long long>(__double_as_longlong(cd.d1sq));
    kp[i] = (static_cast<unsigned long long>(cd.id_lo) << 32) | cd.id_hi;
    lo[i] = cd.s_lo;
    hi[i] = cd.s_hi;
    alive[i] = i;
  }
  __syncthreads();
  // slot -> local index: open addressing; the thread whose CAS claims a bucket numbers it
  for (uint32_t e = tid; e < 2 * n_c; e += nt) {
    const uint32_t slot = (e & 1u) ? hi[e >> 1] : lo[e >> 1];
    uint32_t h = ((slot * 2654435761u) >> 8) & (hash - 1u);
    for (uint32_t probe = 0; probe < hash; ++probe) {
      const uint32_t prev = atomicCAS(&hkey[h], 0xFFFFFFFFu, slot);
      if (prev == 0xFFFFFFFFu) { hval[h] = atomicAdd(&sm.n_next, 1u); break; }
      if (prev == slot) break;
      h = (h + 1u) & (hash - 1u);
    }
  }
  __syncthreads();
  for (uint32_t e = tid; e < 2 * n_c; e += nt) {
    const uint32_t slot = (e & 1u) ? hi[e >> 1] : lo[e >> 1];
    uint32_t h = ((slot * 2654435761u) >> 8) & (hash - 1u);
    for (uint32_t probe = 0; probe < hash && hkey[h] != slot; ++probe) h = (h + 1u) & (hash - 1u);
    if (e & 1u) hi[e >> 1] = hval[h]; else lo[e >> 1] = hval[h];
    if (!list) atomicAdd(&ldead[hval[h]], 1u);
  }
  __syncthreads();
  if (!list) {
    for (uint32_t i0 = 0; i0 < n_c; i0 += nt) {
      const uint32_t i = i0 + tid;
      const uint32_t m = __ballot_sync(0xffffffffu, i < n_c && (ldead[lo[i < n_c ? i : 0u]] > 1u || ldead[hi[i < n_c ? i : 0u]] > 1u));
      if ((tid & 31) == 0 && m) atomicAdd(&sm.n_conflict, static_cast<uint32_t>(__popc(m)));
    }
    __syncthreads();  // the winners below set DEAD
  }
  // winners are listed in shared memory (the hash values are no longer needed) and
  // recorded as events after the last round with one reservation
  uint32_t* won = hval;
  if (tid == 0) sm.n_won = 0;
  for (uint32_t a = tid; a < n_c; a += nt) {
    const uint32_t i = alive[a];
    bd[lo[i]] = ~0ull; bd[hi[i]] = ~0ull;
    bp[lo[i]] = ~0ull; bp[hi[i]] = ~0ull;
  }
  __syncthreads();
  for (uint32_t round = 0; sm.n_alive > 0; ++round) {
    if (round > n_c) {
      if (tid == 0) raise_status(d.g, CHEM_ESTATE);
      break;
    }
    const uint32_t na = sm.n_alive;
    for (uint32_t a = tid; a < na; a += nt) {
      const uint32_t i = alive[a];
      atomicMin(&bd[lo[i]], kd[i]);
      atomicMin(&bd[hi[i]], kd[i]);
    }
    __syncthreads();
    for (uint32_t a = tid; a < na; a += nt) {
      const uint32_t i = alive[a];
      if (bd[lo[i]] == kd[i]) atomicMin(&bp[lo[i]], kp[i]);
      if (bd[hi[i]] == kd[i]) atomicMin(&bp[hi[i]], kp[i]);
    }
    __syncthreads();
    for (uint32_t a0 = 0; a0 < na; a0 += nt) {  // uniform trip count (warp_reserve)
      const uint32_t a = a0 + tid;
      bool win = false;
      uint32_t i = 0;
      if (a < na) {
        i = alive[a];
        win = bd[lo[i]] == kd[i] && bp[lo[i]] == kp[i] && bd[hi[i]] == kd[i] && bp[hi[i]] == kp[i];
      }
      const uint32_t q = warp_reserve(&sm.n_won, win);
      if (win) {
        ldead[lo[i]] = DEAD;
        ldead[hi[i]] = DEAD;
        won[q] = i;
      }
    }
    if (tid == 0) sm.n_next = 0;
    __syncthreads();
    // survivors (both species still free) move to the next round with their slots'
    // minima reset; nothing reads the minima in this pass
    for (uint32_t a0 = 0; a0 < na; a0 += nt) {
      const uint32_t a = a0 + tid;
      bool keep = false;
      uint32_t i = 0;
      if (a < na) {
        i = alive[a];
        keep = ldead[lo[i]] != DEAD && ldead[hi[i]] != DEAD;
      }
      const uint32_t q = warp_reserve(&sm.n_next, keep);
      if (keep) {
        nxt[q] = i;
        bd[lo[i]] = ~0ull; bd[hi[i]] = ~0ull;
        bp[lo[i]] = ~0ull; bp[hi[i]] = ~0ull;
      }
    }
    __syncthreads();
    if (tid == 0) sm.n_alive = sm.n_next;
    uint32_t* t = alive; alive = nxt; nxt = t;
    __syncthreads();
  }
  for (uint32_t q = tid; q < sm.n_won; q += nt) won[q] = cix[won[q]];
  __syncthreads();
  return won;
}

static __device__ bool phase_match_rounds_smem(const Dev& d, MatchSmem& sm, uint32_t* sbuf) {
  const int tid = threadIdx.x, nt = blockDim.x;
  const bool ok = block_status_ok(d);
  const uint32_t n_c = ok ? d.g->n_conflict : 0u;
  if (n_c > static_cast<uint32_t>(RC_CAP)) return false;  // uniform
  const uint32_t* won = match_rounds_in_smem(d, sm, sbuf, n_c, d.alive0);
  if (tid == 0) sm.won_base = atomicAdd(&d.g->n_events, sm.n_won);
  __syncthreads();
  for (uint32_t q = tid; q < sm.n_won; q += nt) commit_event(d, won[q], d.cand[won[q]], sm.won_base + q);
  __syncthreads();
  return true;
}

// Sort of n (key, value) pairs by the whole CTA, in shared memory (keys are distinct
// here; equal keys would be ordered by value): one counting pass over 2048 buckets of
// the key range (bucket = (key - min) >> shift), then each key's rank inside its bucket
// by comparison with the bucket's other keys (buckets hold a handful of keys for the
// id-like keys sorted here). The result is in (k0, v0); (k1, v1) is scratch. Returns
// false, with nothing changed, when a bucket holds more than 64 keys (clustered keys)
// or the CTA's threads do not divide the buckets; the caller then uses block_sort_pairs.
constexpr int BUCKETS = 2048;
static __device__ bool block_bucket_sort(uint32_t* k0, uint32_t* v0, uint32_t* k1, uint32_t* v1, uint32_t n,
                                         BlockSortSmem& sm, ScanSmem& ss, bool known = false, uint32_t lowest = 0,
                                         uint32_t highest = 0) {
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, w = tid >> 5;
  if (BUCKETS % nt != 0) return false;     // whole numbers of buckets per thread in the scan below
  uint32_t* cnt = &sm.whist[0][0];         // BUCKETS counts, then exclusive starts
  uint32_t* cur = cnt + BUCKETS;           // scatter cursors, then bucket ends
  uint32_t* red = cnt + 2 * BUCKETS;       // per-warp min / max / largest bucket
  // key range (`known`: every key lies in [lowest, highest])
  uint32_t mn = lowest, mx = highest;
  for (int i = tid; i < BUCKETS; i += nt) cnt[i] = 0u;
  if (!known) {
    mn = 0xFFFFFFFFu; mx = 0u;
    for (uint32_t i = tid; i < n; i += nt) { mn = min(mn, k0[i]); mx = max(mx, k0[i]); }
    mn = __reduce_min_sync(0xffffffffu, mn);
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) { red[w] = mn; red[32 + w] = mx; }
  }
  __syncthreads();
  if (!known) {
    mn = 0xFFFFFFFFu; mx = 0u;
    for (int q = 0; q < (nt >> 5); ++q) { mn = min(mn, red[q]); mx = max(mx, red[32 + q]); }
  }
  const uint32_t range = n ? mx - mn : 0u;
  const int bits = range ? 32 - __clz(range) : 0;
  const int shift = bits > 11 ? bits - 11 : 0;
  for (uint32_t i = tid; i < n; i += nt) atomicAdd(&cnt[(k0[i] - mn) >> shift], 1u);
  __syncthreads();
  // largest bucket (clustered keys would make the in-bucket ranks quadratic)
  uint32_t big = 0u;
  for (int i = tid; i < BUCKETS; i += nt) big = max(big, cnt[i]);
  big = __reduce_max_sync(0xffffffffu, big);
  if (lane == 0) red[64 + w] = big;
  // exclusive starts: each thread scans a few consecutive buckets
  const int per = BUCKETS / nt;
  uint32_t mine = 0;
  for (int i = 0; i < per; ++i) mine += cnt[per * tid + i];
  uint32_t tot;
  uint32_t ex = block_excl_scan(mine, ss.warp_tot, &ss.total, tot);
  big = 0u;
  for (int q = 0; q < (nt >> 5); ++q) big = max(big, red[64 + q]);
  __syncthreads();               // all have read `red`, which the caller's radix sort clears next
  if (big > 64u) return false;  // uniform: every thread read the same values
  for (int i = 0; i < per; ++i) {
    const uint32_t c = cnt[per * tid + i];
    cnt[per * tid + i] = ex;
    cur[per * tid + i] = ex;
    ex += c;
  }
  __syncthreads();
  for (uint32_t i = tid; i < n; i += nt) {
    const uint32_t b = (k0[i] - mn) >> shift;
    const uint32_t p = atomicAdd(&cur[b], 1u);
    k1[p] = k0[i];
    v1[p] = v0[i];
  }
  __syncthreads();
  for (uint32_t p = tid; p < n; p += nt) {
    const uint32_t k = k1[p], v = v1[p];
    const uint32_t b = (k - mn) >> shift;
    const uint32_t lo = cnt[b], hi = cur[b];
    uint32_t r = 0;
    for (uint32_t q = lo; q < hi; ++q) r += (k1[q] < k || (k1[q] == k && v1[q] < v)) ? 1u : 0u;
    k0[lo + r] = k;
    v0[lo + r] = v;
  }
  __syncthreads();
  return true;
}

// Stable LSD radix sort of n (key, value) pairs by the whole CTA, 8-bit digits over the
// 32 key bits. Each warp owns one contiguous chunk of the input and scatters it in order
// (ranks among equal digits from match_digit8), so equal digits keep their order.
// A pass whose digit is the same for every key is skipped. The arrays may live in shared
// or global memory. Returns 0 when the result is in (k0, v0), 1 when in (k1, v1).
static __device__ int block_sort_pairs(uint32_t* k0, uint32_t* v0, uint32_t* k1, uint32_t* v1, uint32_t n,
                                BlockSortSmem& sm) {
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, w = tid >> 5, nw = nt >> 5;
  const uint32_t chunk = (n + static_cast<uint32_t>(nw) - 1u) / static_cast<uint32_t>(nw);
  const uint32_t lo = min(n, static_cast<uint32_t>(w) * chunk), hi = min(n, lo + chunk);
  const uint32_t lt = (1u << lane) - 1u;
  uint32_t *kin = k0, *vin = v0, *kout = k1, *vout = v1;
  int parity = 0;
  if (tid < 4) sm.trivial[tid] = 0u;
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 8 * pass;
    for (int i = tid; i < nw * RADIX; i += nt) (&sm.whist[0][0])[i] = 0u;
    __syncthreads();
    for (uint32_t i = lo + lane; i < hi; i += 32) atomicAdd(&sm.whist[w][(kin[i] >> shift) & 255u], 1u);
    __syncthreads();
    for (int dg = tid; dg < RADIX; dg += nt) {
      uint32_t run = 0;
      for (int q = 0; q < nw; ++q) {
        const uint32_t c = sm.whist[q][dg];
        sm.whist[q][dg] = run;
        run += c;
      }
      sm.dtot[dg] = run;
      if (run == n) sm.trivial[pass] = 1u;
    }
    __syncthreads();
    if (sm.trivial[pass]) continue;  // the same value for every thread
    if (w == 0) {
      uint32_t carry = 0;
      for (int base = 0; base < RADIX; base += 32) {
        const uint32_t v = sm.dtot[base + lane];
        uint32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
          if (lane >= o) x += y;
        }
        sm.dtot[base + lane] = carry + x - v;
        carry += __shfl_sync(0xffffffffu, x, 31);
      }
    }
    __syncthreads();
    for (uint32_t b0 = lo; b0 < hi; b0 += 32) {
      const uint32_t i = b0 + lane;
      const bool act = i < hi;
      uint32_t key = 0, val = 0, dg = RADIX;  // inactive lanes form their own group
      if (act) {
        key = kin[i];
        val = vin[i];
        dg = (key >> shift) & 255u;
      }
      const uint32_t peers = match_digit8(dg, __ballot_sync(0xffffffffu, act));
      if (act) {
        const uint32_t dst = sm.dtot[dg] + sm.whist[w][dg] + __popc(peers & lt);
        kout[dst] = key;
        vout[dst] = val;
      }
      __syncwarp();
      if (act && (peers & lt) == 0u) sm.whist[w][dg] += __popc(peers);
      __syncwarp();
    }
    __syncthreads();
    uint32_t* t = kin; kin = kout; kout = t;
    t = vin; vin = vout; vout = t;
    parity ^= 1;
  }
  return parity;
}

// See SortOneSmem. Called by one CTA, after the histogram-free diffusion. (Gathering the state in
// the same CTA, without the barrier in between, took 2 us longer than all CTAs' gather.)
static __device__ void phase_sort_one(const Dev& d, SortOneSmem& so, BlockSortSmem& bs, ScanSmem& ss) {
  const int tid = threadIdx.x, nt = blockDim.x;
  const uint32_t n = d.g->n_total, first = d.n_trains == 1 ? d.trains[0].cell_base : 0u, last = d.g->sentinel_step;
  if (!block_status_ok(d)) return;
  for (uint32_t i = tid; i < n; i += nt) { so.k0[i] = d.keys0[i]; so.v0[i] = i; }
  __syncthreads();
  const bool bucketed = block_bucket_sort(so.k0, so.v0, so.k1, so.v1, n, bs, ss, true, first, last);
  const int p = bucketed ? 0 : block_sort_pairs(so.k0, so.v0, so.k1, so.v1, n, bs);
  const uint32_t* k = p ? so.k1 : so.k0;
  const uint32_t* v = p ? so.v1 : so.v0;
  for (uint32_t i = tid; i < n; i += nt) { d.keys1[i] = k[i]; d.vals1[i] = v[i]; }
  if (tid == 0) {
    d.g->sort_parity = 1u;
    d.g->sort_any = 1u;
  }
}

// Product-count prefix over the ordered events (`order`, optionally copied to
// `order_out`), written to `pref`, plus each train's first prefix, event and product
// counts.
static __device__ void products_prefix(const Dev& d, ScanSmem& sm, const uint32_t* okeys, const uint32_t* order,
                                       uint32_t* order_out, uint32_t* pref, uint32_t E, bool ok) {
  const int tid = threadIdx.x, nt = blockDim.x;
  const int tshift = 32 - static_cast<int>(d.train_bits);
  for (uint32_t b = tid; b < d.n_trains; b += nt) {
    sm.first_pref[b] = 0; sm.first_k[b] = 0; sm.prods_tr[b] = 0; sm.evs_tr[b] = 0;
  }
  // each thread takes one contiguous segment of the ordered events: its product count,
  // one block-wide scan of the segment sums, then the per-event prefixes in the segment
  const uint32_t seg = (E + static_cast<uint32_t>(nt) - 1u) / static_cast<uint32_t>(nt);
  const uint32_t k0 = min(E, static_cast<uint32_t>(tid) * seg), k1 = min(E, k0 + seg);
  uint32_t local = 0;
  for (uint32_t k = k0; k < k1; ++k) local += order[k] >> 24;
  uint32_t total;
  uint32_t ex = block_excl_scan(local, sm.warp_tot, &sm.total, total);  // includes barriers
  // train boundaries: a train's counts are differences at its last event (events are in
  // train order)
  for (uint32_t k = k0; k < k1; ++k) {
    const uint32_t v = order[k];
    pref[k] = ex;
    if (order_out) order_out[k] = v;
    const uint32_t b = d.train_bits ? okeys[k] >> tshift : 0u;
    if (k == 0 || (d.train_bits && (okeys[k - 1] >> tshift) != b)) { sm.first_pref[b] = ex; sm.first_k[b] = k; }
    ex += v >> 24;
  }
  __syncthreads();
  for (uint32_t k = k0; k < k1; ++k) {
    const uint32_t b = d.train_bits ? okeys[k] >> tshift : 0u;
    if (k + 1 == E || (d.train_bits && (okeys[k + 1] >> tshift) != b)) {
      sm.prods_tr[b] = pref[k] + (order[k] >> 24) - sm.first_pref[b];
      sm.evs_tr[b] = k + 1 - sm.first_k[b];
    }
  }
  __syncthreads();
  for (uint32_t b = tid; b < d.n_trains; b += nt) {
    Train& tr = d.trains[b];
    tr.pref0 = sm.first_pref[b];
    tr.prods_step = sm.prods_tr[b];
    tr.n_events_step = sm.evs_tr[b];
  }
  if (tid == 0 && ok) d.g->n_products = total;
  __syncthreads();
}

struct SerialSmem {
  MatchSmem match;
  BlockSortSmem sort;
  ScanSmem scan;
  unsigned long long warp_tot64[REACT_THREADS / 32];
};

// Events and products before every group of EV_GROUP buckets (d.bk_start) and each train's, by
// one CTA. (The prefix over all buckets took 8 us at 16,384 buckets and 25 us at 65,536; the
// groups are few, and an event adds up the buckets before its own itself.)
static __device__ void bucket_prefix(const Dev& d, SerialSmem& sm) {
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, w = tid >> 5, nw = nt >> 5;
  const uint32_t n = d.n_buckets / EV_GROUP;
  unsigned long long carry = 0;  // events | products << 32
  for (uint32_t i0 = 0; i0 < n; i0 += nt) {
    const uint32_t i = i0 + tid, c = i < n ? d.bk_group[i] : 0u;
    const unsigned long long mine = static_cast<unsigned long long>(c & 0xFFFFu) | (static_cast<unsigned long long>(c >> 16) << 32);
    unsigned long long incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) sm.warp_tot64[w] = incl;
    __syncthreads();
    unsigned long long at = carry + incl - mine;
    for (int q = 0; q < nw; ++q) {
      const unsigned long long t = sm.warp_tot64[q];
      if (q < w) at += t;
      carry += t;
    }
    if (i < n) d.bk_start[i] = make_uint2(static_cast<uint32_t>(at), static_cast<uint32_t>(at >> 32));
    __syncthreads();
  }
  if (tid == 0) {
    d.bk_start[n] = make_uint2(static_cast<uint32_t>(carry), static_cast<uint32_t>(carry >> 32));
    d.g->n_products = static_cast<uint32_t>(carry >> 32);
  }
  __syncthreads();
  for (uint32_t b = tid; b < d.n_trains; b += nt) {
    Train& tr = d.trains[b];
    const uint2 lo = d.bk_start[tr.bk_base / EV_GROUP];
    const uint2 hi = d.bk_start[(b + 1u < d.n_trains ? d.trains[b + 1u].bk_base : d.n_buckets) / EV_GROUP];
    tr.pref0 = lo.y;
    tr.prods_step = hi.y - lo.y;
    tr.n_events_step = hi.x - lo.x;
  }
  __syncthreads();
}

// The one-CTA part of the react phase: conflict rounds, event order, product prefix.
// With at most EV_SMEM_CAP events the sort runs in `sbuf` (4 * EV_SMEM_CAP words of shared
// memory), otherwise in the global event buffers.
static __device__ void phase_react_serial(const Dev& d, SerialSmem& sm, uint32_t* sbuf) {
  const int tid = threadIdx.x, nt = blockDim.x;
  const uint32_t n_conflict = d.g->n_conflict;  // read before the rounds (all threads, uniform)
  const bool rounds_smem = phase_match_rounds_smem(d, sm.match, sbuf);
  if (!rounds_smem) phase_match_rounds(d, sm.match);
  const bool ok = block_status_ok(d);
  const uint32_t E = ok ? min(d.g->n_events, d.cap_cand) : 0u;
  const uint32_t* okeys;
  const uint32_t* order;
  uint32_t* order_out = nullptr;
  uint32_t* pref;
  if (tid == 0 && ok) {  // branch record (read by chem_get_stats)
    Global* g = d.g;
    if (!rounds_smem && n_conflict > 0) g->react_rounds_global += 1;
    if (n_conflict > g->max_conflict) g->max_conflict = n_conflict;
    g->pairs_accepted += min(g->n_cand, d.cap_cand);
    if (E > g->max_events) g->max_events = E;
    if (E > static_cast<uint32_t>(EV_SMEM_CAP) && (d.bk_cnt == nullptr || g->bk_overflow != 0u)) g->react_order_global += 1;
  }
  const bool buckets = d.bk_cnt != nullptr && d.g->bk_overflow == 0u;
  if (tid == 0) d.g->ev_bucketed = buckets ? 1u : 0u;
  if (buckets) {
    bucket_prefix(d, sm);
    return;
  }
  if (E <= static_cast<uint32_t>(EV_SMEM_CAP)) {
    uint32_t* k0 = sbuf;
    uint32_t* v0 = sbuf + EV_SMEM_CAP;
    uint32_t* k1 = sbuf + 2 * EV_SMEM_CAP;
    uint32_t* v1 = sbuf + 3 * EV_SMEM_CAP;
    for (uint32_t i = tid; i < E; i += nt) { k0[i] = d.ev_k0[i]; v0[i] = d.ev_v0[i]; }
    __syncthreads();
    const bool bucketed = block_bucket_sort(k0, v0, k1, v1, E, sm.sort, sm.scan);
    if (!bucketed && tid == 0 && E > 0) d.g->react_order_radix += 1;
    const int p = bucketed ? 0 : block_sort_pairs(k0, v0, k1, v1, E, sm.sort);
    okeys = p ? k1 : k0;
    order = p ? v1 : v0;
    order_out = d.ev_v0;
    pref = d.ev_k1;
    if (tid == 0) d.g->ev_parity = 0u;
  } else {
    const int p = block_sort_pairs(d.ev_k0, d.ev_v0, d.ev_k1, d.ev_v1, E, sm.sort);
    okeys = p ? d.ev_k1 : d.ev_k0;
    order = p ? d.ev_v1 : d.ev_v0;
    pref = p ? d.ev_k0 : d.ev_k1;
    if (tid == 0) d.g->ev_parity = static_cast<uint32_t>(p);
  }
  products_prefix(d, sm.scan, okeys, order, order_out, pref, E, ok);
}

// Products, tallies (summed in sm) and log record of event number k (in (train, id_lo) order):
// pair cd, first product in slot slot0 with id id0.
template <bool F32L>
__device__ __forceinline__ void write_event(const Dev& d, const Tables& tb, ProductsSmem& sm, const Cand& cd,
                                            uint32_t slot0, uint32_t id0, uint32_t k) {
  const uint32_t r = cd.rxn_train & 255u, b = cd.rxn_train >> 8;
  const uint32_t np = static_cast<uint32_t>(tb.n_prod[r]);
  Train& tr = d.trains[b];
  if (slot0 + np > d.cap) {
    raise_status(d.g, CHEM_ECAPACITY);
    return;
  }
  const uint32_t tlo = tid_type(F32L ? __float_as_uint(d.s4[cd.s_lo].w) : d.stid[cd.s_lo]);
  const uint32_t thi = tid_type(F32L ? __float_as_uint(d.s4[cd.s_hi].w) : d.stid[cd.s_hi]);
  if (F32L) {
    const float4 a = d.s4[cd.s_lo], c = d.s4[cd.s_hi];
    const uint32_t ca = d.cell_sorted[cd.s_lo], cc = d.cell_sorted[cd.s_hi];
    const int n = tr.n;
    int ax_, ay_, az_, cx_, cy_, cz_;
    cell_decode(ca - tr.cell_base, tr.cb, ax_, ay_, az_);
    cell_decode(cc - tr.cell_base, tr.cb, cx_, cy_, cz_);
    int dx = cx_ - ax_, dy = cy_ - ay_, dz = cz_ - az_;
    // the cells of a reacting pair are at most one apart per axis (n >= 3)
    dx = dx > 1 ? dx - n : (dx < -1 ? dx + n : dx);
    dy = dy > 1 ? dy - n : (dy < -1 ? dy + n : dy);
    dz = dz > 1 ? dz - n : (dz < -1 ? dz + n : dz);
    const float w = tb.Df[tlo] / (tb.Df[tlo] + tb.Df[thi]);
    const float px = a.x + w * (dx * tr.hf + (c.x - a.x));
    const float py = a.y + w * (dy * tr.hf + (c.y - a.y));
    const float pz = a.z + w * (dz * tr.hf + (c.z - a.z));
    for (uint32_t q = 0; q < np; ++q) {
      const uint32_t pt = static_cast<uint32_t>(tb.prod[r][q]);
      d.s4[slot0 + q] = make_float4(px, py, pz, __uint_as_float(((id0 + q) << 3) | pt));
      d.cell_sorted[slot0 + q] = ca;
      d.dead[slot0 + q] = 0;
    }
  } else {
    const double xa = d.sx[cd.s_lo], ya = d.sy[cd.s_lo], za = d.sz[cd.s_lo];
    const double rx = min_image(__dsub_rn(d.sx[cd.s_hi], xa), tr.L, tr.halfL);
    const double ry = min_image(__dsub_rn(d.sy[cd.s_hi], ya), tr.L, tr.halfL);
    const double rz = min_image(__dsub_rn(d.sz[cd.s_hi], za), tr.L, tr.halfL);
    const double w = tb.w_ab[r][static_cast<int>(tlo) == tb.rxn_a[r] ? 0 : 1];  // D_lo / (D_lo + D_hi)
    double from_corner;
    const double px = wrap_box_diffused(__dadd_rn(xa, __dmul_rn(w, rx)), tr.L, tr.halfL, from_corner);
    const double py = wrap_box_diffused(__dadd_rn(ya, __dmul_rn(w, ry)), tr.L, tr.halfL, from_corner);
    const double pz = wrap_box_diffused(__dadd_rn(za, __dmul_rn(w, rz)), tr.L, tr.halfL, from_corner);
    for (uint32_t q = 0; q < np; ++q) {
      const uint32_t pt = static_cast<uint32_t>(tb.prod[r][q]);
      d.sx[slot0 + q] = px; d.sy[slot0 + q] = py; d.sz[slot0 + q] = pz;
      d.stid[slot0 + q] = ((id0 + q) << 3) | pt;
      d.cell_sorted[slot0 + q] = tr.cell_base;
      d.dead[slot0 + q] = 0;
    }
  }
  atomicSub(&sm.dcount[b][tlo], 1);
  atomicSub(&sm.dcount[b][thi], 1);
  for (uint32_t q = 0; q < np; ++q) atomicAdd(&sm.dcount[b][tb.prod[r][q]], 1);
  atomicAdd(&sm.devents[b][r], 1);
  if (tb.water[r]) atomicAdd(&sm.dwater[b], tb.water[r]);
  if (d.cap_ev_log) {
    const uint32_t e = d.g->ev_log_n + k;
    if (e < d.cap_ev_log) {
      chem_event ev;
      ev.step = tr.step; ev.rxn = static_cast<int32_t>(r); ev.id_lo = cd.id_lo; ev.id_hi = cd.id_hi;
      ev.prod_id0 = id0; ev.n_prod = static_cast<int32_t>(np); ev.train = b; ev.reserved = 0;
      d.ev_log[e] = ev;
    } else {
      raise_status(d.g, CHEM_ECAPACITY);
    }
  }
}

__device__ __forceinline__ void clear_products(const Dev& d, ProductsSmem& sm) {
  for (uint32_t b = threadIdx.x; b < d.n_trains; b += blockDim.x) {
    sm.dwater[b] = 0;
    for (int q = 0; q < MAXT; ++q) sm.dcount[b][q] = 0;
    for (int q = 0; q < MAXR; ++q) sm.devents[b][q] = 0;
  }
}

// The CTA's summed tallies into the trains' records.
__device__ __forceinline__ void add_tallies(const Dev& d, const ProductsSmem& sm) {
  constexpr uint32_t per = MAXT + MAXR + 1;
  for (uint32_t w = threadIdx.x; w < d.n_trains * per; w += blockDim.x) {
    const uint32_t b = w / per;
    const int q = static_cast<int>(w % per);
    Train& tr = d.trains[b];
    const int v = q < MAXT ? sm.dcount[b][q] : (q < MAXT + MAXR ? sm.devents[b][q - MAXT] : sm.dwater[b]);
    long long* to = q < MAXT ? &tr.counts[q] : (q < MAXT + MAXR ? &tr.events[q - MAXT] : &tr.water);
    if (v) atomicAdd(reinterpret_cast<unsigned long long*>(to), static_cast<unsigned long long>(static_cast<long long>(v)));
  }
}

// sm is cleared (clear_products; a barrier follows below).
template <bool F32L>
__device__ void phase_products(const Dev& d, ProductsSmem& sm, const Tables& tb, const Span& sp) {
  const bool ok = block_status_ok(d);
  const uint32_t E = ok ? d.g->n_events : 0u;
  const uint32_t* order = d.g->ev_parity ? d.ev_v1 : d.ev_v0;
  const uint32_t* pref = d.g->ev_parity ? d.ev_k0 : d.ev_k1;
  const uint32_t n_live = d.g->n_total - d.g->n_dead;
  if (d.bk_cnt && d.g->ev_bucketed) {
    // the events as they were recorded, each ranked among the few of its bucket
    for (uint32_t e = sp.first(); e < E; e += sp.stride()) {
      const uint32_t key = d.ev_k0[e];
      const Cand cd = d.cand[d.ev_v0[e] & EV_CAND_MASK];
      const uint32_t b = cd.rxn_train >> 8, x = event_bucket(d, b, cd.id_lo), n = d.bk_cnt[x] & 0xFFFFu;
      uint2 at = d.bk_start[x / EV_GROUP];
      const uint4* before = reinterpret_cast<const uint4*>(d.bk_cnt + x / EV_GROUP * EV_GROUP);
      const uint32_t in_group = x % EV_GROUP;
#pragma unroll
      for (uint32_t i = 0; i < EV_GROUP / 4u; ++i) {
        if (4u * i >= in_group) break;
        const uint4 c = before[i];
        const uint32_t left = in_group - 4u * i;
        const uint32_t s4 = c.x + (left > 1u ? c.y : 0u) + (left > 2u ? c.z : 0u) + (left > 3u ? c.w : 0u);
        at.x += s4 & 0xFFFFu;  // (at most EV_GROUP x EV_SLOTS events: the halves do not mix)
        at.y += s4 >> 16;
      }
      for (uint32_t i = 0; i < n; ++i) {
        const unsigned long long o = d.bk_slot[x * EV_SLOTS + i];
        if (static_cast<uint32_t>(o >> 32) < key) {
          at.x += 1u;
          at.y += static_cast<uint32_t>(o) >> 24;
        }
      }
      const Train& tr = d.trains[b];
      write_event<F32L>(d, tb, sm, cd, n_live + at.y, tr.next_id + (at.y - tr.pref0), at.x);
    }
    __syncthreads();
    add_tallies(d, sm);
    return;
  }
  for (uint32_t k = sp.first(); k < E; k += sp.stride()) {
    const Cand cd = d.cand[order[k] & EV_CAND_MASK];
    const Train& tr = d.trains[cd.rxn_train >> 8];
    const uint32_t ex = pref[k];
    write_event<F32L>(d, tb, sm, cd, n_live + ex, tr.next_id + (ex - tr.pref0), k);
  }
  __syncthreads();
  add_tallies(d, sm);
}

// The whole of reaction resolution by one CTA, for steps of few accepted pairs: the rounds run
// over all of them (no fast path and no conflict list), the winners are ordered by counting
// the smaller keys, and each writes its products at once. One launch takes the place of four
// whose work is a few microseconds of dependent latencies each. More accepted pairs than
// `cap` (a crowded step) take the general phases, by this CTA alone.
struct ReactAllSmem {
  MatchSmem match;
  ProductsSmem products;
  uint32_t prods_tr[MAX_TRAINS], evs_tr[MAX_TRAINS];
  uint32_t n_prod;
};
// Bytes of sbuf for steps of up to `cap` accepted pairs (the rounds; the winners' order then
// takes the place of the pairs' keys, 20 of their 48 bytes a pair); a crowded step uses it for
// its block sort and scan.
__host__ __device__ constexpr size_t react_all_bytes(uint32_t cap) {
  const size_t a = rc_smem_bytes(cap), b = sizeof(BlockSortSmem) + sizeof(ScanSmem);
  return a > b ? a : b;
}

template <bool F32L>
__device__ void phase_react_all(const Dev& d, ReactAllSmem& sm, uint32_t* sbuf, uint32_t cap, const Tables& tb) {
  const int tid = threadIdx.x, nt = blockDim.x;
  Global* g = d.g;
  // this thread's first pair is read with the counters, before it is known to be there
  Cand mine{};
  if (static_cast<uint32_t>(tid) < d.cap_cand) mine = d.cand[tid];
  const uint32_t n_cand = g->n_cand, n_live = g->n_total - g->n_dead;
  const bool ok = block_status_ok(d);
  const uint32_t n_c = ok ? min(n_cand, d.cap_cand) : 0u;
  if (static_cast<uint32_t>(tid) < n_c) {  // what the winners' events will read
    prefetch_l1(&d.s4[mine.s_lo]);
    prefetch_l1(&d.s4[mine.s_hi]);
    prefetch_l1(&d.cell_sorted[mine.s_lo]);
    prefetch_l1(&d.cell_sorted[mine.s_hi]);
    if (!F32L) {
      prefetch_l1(&d.sx[mine.s_lo]); prefetch_l1(&d.sy[mine.s_lo]); prefetch_l1(&d.sz[mine.s_lo]);
      prefetch_l1(&d.sx[mine.s_hi]); prefetch_l1(&d.sy[mine.s_hi]); prefetch_l1(&d.sz[mine.s_hi]);
      prefetch_l1(&d.stid[mine.s_lo]); prefetch_l1(&d.stid[mine.s_hi]);
    }
  }
  if (n_c > cap) {  // uniform
    phase_match_fast(d, Span{0u, 1u});
    __syncthreads();
    const uint32_t n_conflict = g->n_conflict;
    phase_match_rounds(d, sm.match);
    const bool ok2 = block_status_ok(d);
    const uint32_t E = ok2 ? min(g->n_events, d.cap_cand) : 0u;
    BlockSortSmem& sort = *reinterpret_cast<BlockSortSmem*>(sbuf);
    ScanSmem& scan = *reinterpret_cast<ScanSmem*>(sbuf + sizeof(BlockSortSmem) / 4);
    const int p = block_sort_pairs(d.ev_k0, d.ev_v0, d.ev_k1, d.ev_v1, E, sort);
    if (tid == 0 && ok2) {  // branch record (read by chem_get_stats)
      g->ev_bucketed = 0u;
      g->ev_parity = static_cast<uint32_t>(p);
      g->react_rounds_global += n_conflict > 0u ? 1u : 0u;
      g->react_order_global += 1u;
      g->max_conflict = max(g->max_conflict, n_conflict);
      g->pairs_accepted += n_c;
      g->max_events = max(g->max_events, E);
    }
    products_prefix(d, scan, p ? d.ev_k1 : d.ev_k0, p ? d.ev_v1 : d.ev_v0, nullptr, p ? d.ev_k0 : d.ev_k1, E, ok2);
    clear_products(d, sm.products);
    phase_products<F32L>(d, sm.products, tb, Span{0u, 1u});
    for (uint32_t b = tid; b < d.n_trains; b += nt) {
      sm.prods_tr[b] = d.trains[b].prods_step;
      sm.evs_tr[b] = d.trains[b].n_events_step;
    }
    __syncthreads();
    return;
  }
  clear_products(d, sm.products);
  for (uint32_t b = tid; b < d.n_trains; b += nt) { sm.prods_tr[b] = 0u; sm.evs_tr[b] = 0u; }
  if (tid == 0) sm.n_prod = 0u;
  __syncthreads();
  uint32_t E = 0u;
  if (n_c) {
    const uint32_t* won = match_rounds_in_smem(d, sm.match, sbuf, n_c, nullptr, &mine);
    E = sm.match.n_won;
    uint32_t* key = sbuf;       // winners' (train, id_lo) keys and
    uint32_t* np = key + n_c;   // product counts | train << 8
    for (uint32_t q = tid; q < E; q += nt) {
      const Cand cd = d.cand[won[q]];
      const uint32_t b = cd.rxn_train >> 8, n = static_cast<uint32_t>(tb.n_prod[cd.rxn_train & 255u]);
      key[q] = event_key(d, cd);
      np[q] = n | (b << 8);
      atomicAdd(&sm.prods_tr[b], n);
      atomicAdd(&sm.evs_tr[b], 1u);
      atomicAdd(&sm.n_prod, n);
      d.dead[cd.s_lo] = 1;
      d.dead[cd.s_hi] = 1;
    }
    __syncthreads();
    // eight lanes count a winner's smaller keys; then the events are written by consecutive
    // threads in their order (FP64 instructions cost a warp the same for one lane as for 32)
    uint32_t* at = np + n_c;        // winner at each place of the order,
    uint32_t* pre = at + n_c;       // products before it, in all and
    uint32_t* pre_tr = pre + n_c;   // of its train
    for (uint32_t q0 = 0; q0 < E; q0 += static_cast<uint32_t>(nt) / 8u) {  // uniform (shuffles)
      const uint32_t q = q0 + static_cast<uint32_t>(tid) / 8u;
      const bool have = q < E;
      const uint32_t k = have ? key[q] : 0u, b = have ? np[q] >> 8 : 0u;
      uint32_t rank = 0, before = 0, before_tr = 0;
      for (uint32_t o = static_cast<uint32_t>(tid) & 7u; o < E; o += 8u) {
        const bool less = key[o] < k;
        const uint32_t n = less ? np[o] : 0xFFFFFF00u;
        rank += less ? 1u : 0u;
        before += n & 255u;
        before_tr += (n >> 8) == b ? (n & 255u) : 0u;
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        rank += __shfl_xor_sync(0xffffffffu, rank, o);
        before += __shfl_xor_sync(0xffffffffu, before, o);
        before_tr += __shfl_xor_sync(0xffffffffu, before_tr, o);
      }
      if (have && (tid & 7) == 0) {
        at[rank] = won[q];
        pre[rank] = before;
        pre_tr[rank] = before_tr;
      }
    }
    __syncthreads();
    for (uint32_t k = tid; k < E; k += nt) {
      const Cand cd = d.cand[at[k]];
      write_event<F32L>(d, tb, sm.products, cd, n_live + pre[k], d.trains[cd.rxn_train >> 8].next_id + pre_tr[k], k);
    }
    __syncthreads();
    add_tallies(d, sm.products);
  }
  for (uint32_t b = tid; b < d.n_trains; b += nt) {
    d.trains[b].prods_step = sm.prods_tr[b];
    d.trains[b].n_events_step = sm.evs_tr[b];
  }
  if (tid == 0 && ok) {
    g->n_events = E;
    g->n_products = sm.n_prod;
    g->pairs_accepted += n_c;
    g->max_events = max(g->max_events, E);
    if (n_c) g->max_conflict = max(g->max_conflict, sm.match.n_conflict);
  }
  __syncthreads();
}

// The end of a step and the begin of the next, most of it ahead of time: while the other CTAs
// search, one CTA takes a copy of the trains' records to the end of the step and plans the
// next one on it (stage_next), and after reaction resolution only adds what depends on it and
// writes the records back (commit_next). On the critical path the two took 6 us.
template <uint32_t TRAINS>
struct PlanSmem {
  BeginSmem begin;
  Train tr[TRAINS];
  uint32_t rel_all;  // releases of the planned step
};

template <uint32_t TRAINS>
static __device__ void stage_next(const Dev& d, PlanSmem<TRAINS>& pl) {
  const int tid = threadIdx.x, nt = blockDim.x;
  const uint32_t words = d.n_trains * static_cast<uint32_t>(sizeof(Train) / 4);
  const uint32_t* src = reinterpret_cast<const uint32_t*>(d.trains);
  uint32_t* dst = reinterpret_cast<uint32_t*>(pl.tr);
  for (uint32_t i = tid; i < words; i += nt) dst[i] = src[i];
  __syncthreads();
  if (static_cast<uint32_t>(tid) < d.n_trains) {
    Train& tr = pl.tr[tid];
    if (tr.active) {
      tr.species_steps += tr.n_live_step;
      tr.t = tr.t_next;
      tr.step += 1;
      tr.dt_cur = fmin(__dmul_rn(tr.dt_cur, tr.dt_growth), tr.dt_max);
      tr.n_ref = tr.n;
      tr.h_ref = tr.h;
      tr.cb_ref = tr.cb;
    }
  }
  __syncthreads();
  begin_plan(d, pl.begin, pl.tr, 0);
  if (tid == 0) {  // (read after a barrier, in commit_next)
    uint32_t n = 0;
    for (uint32_t b = 0; b < d.n_trains; ++b) n += pl.begin.rel[b];
    pl.rel_all = n;
  }
}

// Step record of an advancing train (before its record moves on).
__device__ __forceinline__ void log_step(const Dev& d, const Train& tr, uint32_t b, uint32_t n_events) {
  const uint32_t e = atomicAdd(&d.g->step_log_n, 1u);
  if (e >= d.cap_step_log) {
    raise_status(d.g, CHEM_ECAPACITY);
    return;
  }
  chem_step_record rec;
  rec.step = tr.step; rec.train = b; rec.t_start_s = tr.t_start; rec.dt_s = tr.dt;
  rec.n_live = tr.n_live_step; rec.n_events = n_events;
  for (int q = 0; q < 8; ++q) rec.counts[q] = q < d.tables->n_types ? tr.counts[q] : 0;
  d.step_log[e] = rec;
}

// After the step's products; false, with nothing done, when an error is raised or the planned step
// would work on more than `most` species.
template <uint32_t TRAINS>
static __device__ bool commit_next(const Dev& d, PlanSmem<TRAINS>& pl, uint32_t most) {
  const int tid = threadIdx.x, nt = blockDim.x;
  Global* g = d.g;
  uint32_t n_slots = 0;
  bool go = true;
  if (tid == 0) {
    n_slots = g->n_total - g->n_dead + g->n_products;
    go = status_of(d) == 0 && (pl.begin.any == 0u || n_slots + pl.rel_all <= most);
  }
  if (!__syncthreads_and(go ? 1 : 0)) return false;
  const uint32_t b = static_cast<uint32_t>(tid);
  bool stepped = false;
  if (b < d.n_trains && d.trains[b].active) {
    stepped = true;
    const Train& tr = d.trains[b];
    if (d.cap_step_log) log_step(d, tr, b, tr.n_events_step);
    pl.begin.live[b] += static_cast<long long>(tr.prods_step) - 2ll * static_cast<long long>(tr.n_events_step);
    pl.tr[b].next_id += tr.prods_step;
  }
  const bool any = __syncthreads_or(stepped ? 1 : 0) != 0;
  if (tid == 0) {
    if (any) g->steps_active += 1;
    g->n_total = n_slots;
    if (d.cap_ev_log) g->ev_log_n += g->n_events;
  }
  __syncthreads();
  begin_commit(d, pl.begin, pl.tr);  // (ends with a barrier)
  // everything but the tallies, which the reactions added to
  constexpr uint32_t W = sizeof(Train) / 4, T0 = offsetof(Train, water) / 4, T1 = offsetof(Train, n_ref) / 4;
  const uint32_t* src = reinterpret_cast<const uint32_t*>(pl.tr);
  uint32_t* dst = reinterpret_cast<uint32_t*>(d.trains);
  for (uint32_t i = tid; i < d.n_trains * W; i += nt) {
    const uint32_t w = i % W;
    if (w < T0 || w >= T1) dst[i] = src[i];
  }
  return true;
}

// Species that the begin of the train's next step will release.
__device__ __forceinline__ uint32_t releases_ahead(const Dev& d, const Train& tr) {
  uint32_t lo = tr.p_head, hi = tr.p_tail;
  if (tr.next_arr <= tr.t) {
    const double* pt = d.pt + tr.pend_base;
    while (lo < hi) {
      const uint32_t mid = (lo + hi) >> 1;
      if (pt[mid] <= tr.t) lo = mid + 1; else hi = mid;
    }
  }
  return tr.park_n + tr.mat_n + (lo - tr.p_head);
}

// Species the next step will work on (stepped slots and what its begin will release), for the
// choice of the launch form; between steps, one CTA.
static __device__ void phase_look_ahead(const Dev& d, EndSmem& sm) {
  __syncthreads();
  if (threadIdx.x == 0) sm.ahead = d.g->n_total;
  __syncthreads();
  for (uint32_t b = threadIdx.x; b < d.n_trains; b += blockDim.x) {
    const Train& tr = d.trains[b];
    const uint32_t more = tr.t < tr.t_end ? releases_ahead(d, tr) : 0u;
    if (more) atomicAdd(&sm.ahead, more);
  }
  __syncthreads();
  if (threadIdx.x == 0) d.g->n_ahead = sm.ahead;
}

// The end of a step; the species ahead are counted with it (phase_look_ahead).
static __device__ void phase_end_step(const Dev& d, EndSmem& sm) {
  const int tid = threadIdx.x, nt = blockDim.x;
  if (tid == 0) { sm.any = 0; sm.stepped = 0; sm.ahead = 0; }
  const bool ok = block_status_ok(d);
  for (uint32_t b = tid; b < d.n_trains; b += nt) {
    Train& tr = d.trains[b];
    if (tr.active && ok) {
      atomicOr(&sm.stepped, 1u);
      tr.next_id += tr.prods_step;
      tr.species_steps += tr.n_live_step;
      if (d.cap_step_log) log_step(d, tr, b, tr.n_events_step);
      tr.t = tr.t_next;
      tr.step += 1;
      tr.dt_cur = fmin(__dmul_rn(tr.dt_cur, tr.dt_growth), tr.dt_max);
      tr.n_ref = tr.n;
      tr.h_ref = tr.h;
      tr.cb_ref = tr.cb;
    }
    if (tr.t < tr.t_end) {
      atomicOr(&sm.any, 1u);
      const uint32_t more = releases_ahead(d, tr);
      if (more) atomicAdd(&sm.ahead, more);
    }
  }
  __syncthreads();
  if (tid == 0) {
    if (sm.stepped) d.g->steps_active += 1;
    if (ok) {
      const uint32_t n_total = d.g->n_total - d.g->n_dead + d.g->n_products;
      d.g->n_total = n_total;
      d.g->n_ahead = n_total + sm.ahead;
      if (d.cap_ev_log) d.g->ev_log_n += d.g->n_events;
    }
    d.g->any_active = sm.any;
  }
  __syncthreads();
}

}  // namespace chem
