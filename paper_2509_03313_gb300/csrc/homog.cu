// Homogeneous (beam-off) stage of a pulse train, Sec. 2.3 of arxiv 2509.03313: between
// pulses, and after the last one, the species are followed as a well-mixed system by
// the rate equations of Table 1 (Eq. 3, Eq. 4) instead of particle by particle.
//
// For every train the host selected (Train::hx_sel):
//  1. k_hx_remove marks every particle of the train removed (the next sort drops it);
//  2. k_hx_integrate, one CTA per train, takes the train's species counts n0 as
//     molecule numbers in the box volume V and integrates the reaction extents e_r
//     (events): n(e) = n0 + nu e, de_r/dt = kappa_r n_a n_b, kappa_r = k_r / (N_A V), and
//     (k_tab / 2) / (N_A V) for a self reaction whose tabulated value is 2k. This is Eq. 3
//     multiplied through by N_A V. The integrator is the extrapolated linearly implicit
//     Euler method (Deuflhard 1985; Hairer and Wanner, Solving ODEs II, Sec. IV.9) with
//     the harmonic substep sequence 1..6 (a half warp per column) and an analytic
//     Jacobian: stiff rate equations
//     (R9 at 1.1e11 L/mol/s) over 10 s take a few hundred steps;
//  3. the extents are rounded to whole events without bias, E_r = floor(e_r) +
//     [u_r < frac(e_r)], u_r from Philox4x32-10 at counter (stage, r, 0, 4); while a
//     species count would be negative, the lowest-index reaction consuming the lowest
//     negative species gives back one event; counts, event tallies and the water balance
//     take the whole events, so charge and atoms stay exactly conserved;
//  4. the survivors wait in Train::mat_n / mat_cum until the train's next step, whose
//     release re-creates them at uniform positions (phase_diffuse).
#include "launch.h"
#include "sbs_device.cuh"

namespace chem {
namespace {

constexpr double HX_N_AVOGADRO = 6.02214076e23;
constexpr double HX_TWO_POW_M53 = 1.1102230246251565e-16;
constexpr int HX_K = 6;              // extrapolation columns, substep counts 1..HX_K
constexpr double HX_RTOL = 1e-12;    // per step, relative to the extent
constexpr double HX_ATOL = 1e-8;     // per step, events
constexpr int HX_MAX_STEPS = 200000;

__device__ __forceinline__ int status_of_hx(const Dev& d) {
  return *reinterpret_cast<volatile int*>(&d.g->status);
}

// One train is integrated by one CTA of three warps: each of the six extrapolation columns
// belongs to a half warp, lane r of it to reaction r. What bounds the stage is the length
// of its dependent chain (a few hundred steps, each a factorisation and up to six
// substeps) and the FP64 pipe, which a warp's instruction occupies for 16 cycles however
// many lanes are active. Rows of the matrices therefore live in the lanes' registers and
// travel by shuffles, and the columns run side by side (two per warp, of similar length).
// Measured, 64 trains of 500 to 20,000 species over 10 s (a whole pass with its host calls):
// 64.1 -> 16.2 ms against one lane per column with its matrices in local memory, an FP64
// power for the step size and the table's divisions in one lane.
constexpr int HX_THREADS = 16 * HX_K;  // one half warp per column
static_assert(MAXR <= 16, "a half warp holds the rows of the matrix");

// Kinetics of one train in molecule numbers, and the columns' end values.
struct HxSmem {
  double n0[MAXT];
  double nu[MAXR][MAXT];      // change of species x per event of reaction r
  double nu_ab[MAXR][MAXR][2];  // [s][r]: change of r's two reactants per event of s
  double col[HX_K][MAXR];
  double e[MAXR];             // extents at the end of the integration
};

// What a lane keeps of its reaction (lanes past the reactions: kappa 0, reactants 0).
struct HxLane {
  int nr, nt, r, col;
  int a, b;
  double kappa;
};

__device__ __forceinline__ double hx_shfl(double v, int src) {
  return __shfl_sync(0xffffffffu, v, src, 16);
}

// kappa n_a and kappa n_b of this lane's reaction and its rate, at extents y (one per lane).
__device__ __forceinline__ double hx_rate(const HxLane& k, const HxSmem& sm, double y, double& na, double& nb) {
  const int x = k.r & (MAXT - 1);  // lane x also carries species x (and lane x + 8 a copy)
  double n = sm.n0[x], n2 = 0.0;
#pragma unroll
  for (int s = 0; s < MAXR; s += 2) {
    if (s < k.nr) n += sm.nu[s][x] * hx_shfl(y, s);
    if (s + 1 < k.nr) n2 += sm.nu[s + 1][x] * hx_shfl(y, s + 1);
  }
  n += n2;
  na = hx_shfl(n, k.a);
  nb = hx_shfl(n, k.b);
  return k.kappa * na * nb;
}

// One extrapolated step of length H from y0 (one extent per lane, the same in every half
// warp): column j takes j linearly implicit Euler substeps (I - hJ) d = h f(y), y += d,
// h = H / j, with the Jacobian J of y0; then lane r forms the Aitken-Neville table of
// component r, which removes the error terms in h, h^2, ... (the method's expansion is in
// powers of h). The matrix is factored once by elimination with a pivot row per column
// (largest element to 1 part in 2^16, rows stay where they are); a substep is one forward
// and one backward sweep. Returns false (for the whole CTA) when a matrix is singular or
// the result is not finite; else y1 and the scaled error estimate.
__device__ bool hx_step(const HxLane& k, HxSmem& sm, double y0, double H, double& y1, double& err) {
  const int nr = k.nr;
  const double h = H / static_cast<double>(k.col + 1);
  double na, nb;
  double f = hx_rate(k, sm, y0, na, nb);
  const double ka = k.kappa * nb, kb = k.kappa * na;
  // row r of I - hJ: d rate_r / d e_s = kappa_r (n_b nu[a][s] + n_a nu[b][s])
  double M[MAXR];
#pragma unroll
  for (int s = 0; s < MAXR; ++s) {
    M[s] = 0.0;
    if (s < nr) M[s] = (s == k.r ? 1.0 : 0.0) - h * (ka * sm.nu_ab[s][k.r][0] + kb * sm.nu_ab[s][k.r][1]);
  }
  int pos = MAXR;                // elimination order of this lane's row (MAXR: not yet)
  double inv_own = 0.0;          // 1 / pivot of this lane's row
  unsigned long long perm = 0;   // pivot lane of column c in bits 4c
  bool ok = true;
#pragma unroll
  for (int c = 0; c < MAXR; ++c) {
    if (c >= nr) break;
    const unsigned hi = static_cast<unsigned>(__double2hiint(M[c])) & 0x7FFFFFF0u;
    const bool free_row = pos == MAXR && k.r < nr;
    const unsigned key = free_row ? (hi | static_cast<unsigned>(15 - k.r)) : 0u;
    const unsigned best0 = __reduce_max_sync(0xffffffffu, (k.col & 1) ? 0u : key);
    const unsigned best1 = __reduce_max_sync(0xffffffffu, (k.col & 1) ? key : 0u);
    const unsigned best = (k.col & 1) ? best1 : best0;
    const int p = 15 - static_cast<int>(best & 15u);
    ok = ok && best >= 16u && best < 0x7FF00000u;
    perm |= static_cast<unsigned long long>(p) << (4 * c);
    const double inv = 1.0 / hx_shfl(M[c], p);
    const bool mine = k.r == p;
    if (mine) { pos = c; inv_own = inv; }
    const double l = (free_row && !mine) ? M[c] * inv : 0.0;
    if (free_row && !mine) M[c] = l;
#pragma unroll
    for (int q = c + 1; q < MAXR; ++q)
      if (q < nr) M[q] -= l * hx_shfl(M[q], p);
  }
  double y = y0;
  for (int i = 0; i <= (k.col | 1); ++i) {  // warp-uniform: as many as its longer column takes
    if (i > 0) f = hx_rate(k, sm, y, na, nb);
    double v = h * f, x = 0.0;
#pragma unroll
    for (int c = 0; c < MAXR; ++c) {
      if (c >= nr) break;
      const double xc = hx_shfl(v, static_cast<int>(perm >> (4 * c)) & 15);
      if (pos > c) v -= M[c] * xc;
    }
#pragma unroll
    for (int c = MAXR - 1; c >= 0; --c) {
      if (c >= nr) continue;
      const double xc = hx_shfl(v * inv_own, static_cast<int>(perm >> (4 * c)) & 15);
      if (pos < c) v -= M[c] * xc;
      if (k.r == c) x = xc;
    }
    if (i <= k.col) y += x;
  }
  sm.col[k.col][k.r] = y;
  ok = __syncthreads_and(ok ? 1 : 0) != 0;
  // every half warp forms the same table, so that all go on with the same values
  double prev[HX_K], cur[HX_K];
#pragma unroll
  for (int j = 1; j <= HX_K; ++j) {
    cur[0] = sm.col[j - 1][k.r];
#pragma unroll
    for (int l = 0; l + 1 < j; ++l)  // the weight is 1 / (j / (j - l - 1) - 1)
      cur[l + 1] = cur[l] + (cur[l] - prev[l]) * (static_cast<double>(j - l - 1) / static_cast<double>(l + 1));
#pragma unroll
    for (int l = 0; l < j; ++l) prev[l] = cur[l];
  }
  y1 = cur[HX_K - 1];
  const double sc = HX_ATOL + HX_RTOL * fmax(fabs(y0), fabs(y1));
  double e = k.r < nr ? fabs(y1 - cur[HX_K - 2]) / sc : 0.0;
  bool fin = k.r >= nr || isfinite(y1);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) e = fmax(e, __shfl_xor_sync(0xffffffffu, e, o, 16));
  fin = __all_sync(0xffffffffu, fin);  // (both halves hold the same components)
  err = e;
  if (k.r >= nr) y1 = 0.0;
  __syncthreads();  // the columns are rewritten by the next step
  return ok && fin;
}

// Extents after T seconds from e = 0, one per lane (identical control flow on every
// thread). Returns the accepted steps, or -1 on failure.
__device__ long long hx_integrate(const HxLane& k, HxSmem& sm, double T, double& e) {
  e = 0.0;
  if (k.nr == 0 || !(T > 0.0)) return 0;
  double t = 0.0, H = fmin(T, 1e-9);
  long long accepted = 0;
  for (int it = 0; it < HX_MAX_STEPS; ++it) {
    if (t >= T) return accepted;
    const bool last = H >= T - t;
    const double Hs = last ? T - t : H;
    double err = 0.0, y1;
    const bool ok = hx_step(k, sm, e, Hs, y1, err);
    // the step-size factor needs a few digits only: FP32 power
    const float root = (ok && err > 0.0) ? 0.9f * powf(fminf(static_cast<float>(err), 1e30f), -1.0f / HX_K) : 4.f;
    if (ok && err <= 1.0) {
      e = y1;
      t = last ? T : t + Hs;
      ++accepted;
      H = Hs * static_cast<double>(fminf(4.f, fmaxf(0.2f, root)));
    } else {
      H = Hs * static_cast<double>(ok ? fminf(0.5f, fmaxf(0.2f, root)) : 0.2f);
    }
  }
  return -1;
}

__global__ void k_hx_remove(Dev d) {
  if (status_of_hx(d)) return;
  const uint32_t n = d.g->n_total;
  for (uint32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x) {
    if (d.dead[s]) continue;
    const int b = d.n_trains == 1 ? 0 : train_of_cell(d.trains, d.n_trains, d.cell_sorted[s]);
    if (d.trains[b].hx_sel) d.dead[s] = 1;
  }
}

__global__ void __launch_bounds__(HX_THREADS) k_hx_integrate(Dev d) {
  __shared__ HxSmem sm;
  const int tid = threadIdx.x;
  const uint32_t b = blockIdx.x;
  // one answer for the CTA (another train's CTA may raise the status meanwhile)
  if (__syncthreads_or(status_of_hx(d))) return;
  Train& tr = d.trains[b];
  if (!tr.hx_sel) return;
  const Tables& tb = *d.tables;
  HxLane k;
  k.nt = tb.n_types;
  k.nr = tb.n_rxn;
  k.r = tid & 15;
  k.col = tid >> 4;
  const double NV = HX_N_AVOGADRO * (tr.L * tr.L * tr.L * 1e-24);
  for (int q = tid; q < MAXT * MAXR; q += HX_THREADS) {
    const int x = q % MAXT, r = q / MAXT;
    double v = 0.0;
    if (r < k.nr && x < k.nt) {
      if (tb.rxn_a[r] == x) v -= 1.0;
      if (tb.rxn_b[r] == x) v -= 1.0;
      for (int p = 0; p < tb.n_prod[r]; ++p) v += tb.prod[r][p] == x ? 1.0 : 0.0;
    }
    sm.nu[r][x] = v;
  }
  if (tid < MAXT) sm.n0[tid] = tid < k.nt ? static_cast<double>(tr.counts[tid]) : 0.0;
  __syncthreads();
  k.a = k.r < k.nr ? tb.rxn_a[k.r] : 0;
  k.b = k.r < k.nr ? tb.rxn_b[k.r] : 0;
  k.kappa = k.r < k.nr ? (k.a == k.b ? 0.5 * tb.k_tab[k.r] : tb.k_tab[k.r]) / NV : 0.0;
  for (int s = k.col; s < MAXR; s += HX_K) {
    sm.nu_ab[s][k.r][0] = sm.nu[s][k.a];
    sm.nu_ab[s][k.r][1] = sm.nu[s][k.b];
  }
  __syncthreads();
  double own;
  const long long steps = hx_integrate(k, sm, tr.hx_t_end - tr.t, own);
  if (tid < MAXR) sm.e[tid] = own;
  __syncthreads();
  if (tid != 0) return;  // the rounding and the train's record: one thread
  const double* e = sm.e;
  if (steps < 0) {
    raise_status(d.g, CHEM_ECAPACITY);
    d.g->err_where = 0x4858u;  // integrator step limit of the homogeneous stage
    tr.hx_sel = 0;
    return;
  }
  // whole events: unbiased rounding, then take-backs while a count is negative
  long long E[MAXR], n[MAXT];
  for (int r = 0; r < k.nr; ++r) {
    const uint4 w = philox4x32_10(make_uint4(tr.hx_stage, static_cast<uint32_t>(r), 0u, 4u), tr.key0, tr.key1);
    const double u = static_cast<double>(u53(w.x, w.y)) * HX_TWO_POW_M53;
    const double x = fmax(e[r], 0.0);
    const double fl = floor(x);
    E[r] = static_cast<long long>(fl) + (u < x - fl ? 1 : 0);
  }
  for (int x = 0; x < k.nt; ++x) {
    long long v = tr.counts[x];
    for (int r = 0; r < k.nr; ++r) v += static_cast<long long>(sm.nu[r][x]) * E[r];
    n[x] = v;
  }
  for (;;) {
    int neg = -1;
    for (int x = 0; x < k.nt && neg < 0; ++x)
      if (n[x] < 0) neg = x;
    if (neg < 0) break;
    int rr = -1;
    for (int r = 0; r < k.nr && rr < 0; ++r)
      if (sm.nu[r][neg] < 0.0 && E[r] > 0) rr = r;
    if (rr < 0) {  // cannot happen: a negative count always has a consuming event
      raise_status(d.g, CHEM_ECAPACITY);
      tr.hx_sel = 0;
      return;
    }
    E[rr] -= 1;
    for (int x = 0; x < k.nt; ++x) n[x] -= static_cast<long long>(sm.nu[rr][x]);
  }
  long long water = 0;
  uint32_t cum = 0;
  for (int r = 0; r < MAXR; ++r) {
    tr.hx_e[r] = r < k.nr ? e[r] : 0.0;
    tr.hx_E[r] = r < k.nr ? E[r] : 0;
    if (r < k.nr) {
      tr.events[r] += E[r];
      water += E[r] * tb.water[r];
    }
  }
  for (int x = 0; x < MAXT; ++x) {
    const long long v = x < k.nt ? n[x] : 0;
    tr.counts[x] = v;
    cum += static_cast<uint32_t>(v);
    tr.mat_cum[x] = cum;
  }
  tr.water += water;
  tr.mat_n = cum;
  tr.hx_steps = steps;
  tr.hx_stage += 1;
  tr.t = tr.hx_t_end;
  tr.hx_sel = 0;
}

}  // namespace

cudaError_t enqueue_homogeneous(const Dev& d, int blocks, cudaStream_t s) {
  k_hx_remove<<<blocks, 256, 0, s>>>(d);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_hx_integrate<<<static_cast<int>(d.n_trains), HX_THREADS, 0, s>>>(d);
  return cudaGetLastError();
}

}  // namespace chem
