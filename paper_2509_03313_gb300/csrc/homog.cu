// Homogeneous (beam-off) stage of a pulse train, Sec. 2.3 of arxiv 2509.03313: between
// pulses, and after the last one, the species are followed as a well-mixed system by
// the rate equations of Table 1 (Eq. 3, Eq. 4) instead of particle by particle.
//
// For every train the host selected (Train::hx_sel):
//  1. k_hx_remove marks every particle of the train removed (the next sort drops it);
//  2. k_hx_integrate, a cluster of two CTAs per train, takes the train's species counts n0 as
//     molecule numbers in the box volume V and integrates the reaction extents e_r
//     (events): n(e) = n0 + nu e, de_r/dt = kappa_r n_a n_b, kappa_r = k_r / (N_A V), and
//     (k_tab / 2) / (N_A V) for a self reaction whose tabulated value is 2k. This is Eq. 3
//     multiplied through by N_A V. The integrator is the extrapolated linearly implicit
//     Euler method (Deuflhard 1985; Hairer and Wanner, Solving ODEs II, Sec. IV.9) with
//     the harmonic substep sequence 1..6 (a warp per column) and an analytic
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

// One train is integrated by a cluster of two CTAs of three warps, one warp per extrapolation
// column. What bounds the stage is the length of its dependent chain (250 to 300 steps, each
// an inverse and up to six substeps) and the FP64 pipe, which a warp's instruction occupies
// for many cycles however many lanes are active. So the work of a column is spread over the
// lanes of its warp (lane r + 16 h: reaction r, the matrix's columns of parity h), a substep
// is one product with the inverse instead of two triangular sweeps, and no more than three
// warps lie on an SM; the columns' end values go to both CTAs through distributed shared memory.
// Measured, 64 trains of 500 to 20,000 species over 10 s (252 steps; the call): 3.1 ms, against
// 6.1 ms with a half warp per column, LU factors and one CTA per train, and the same 6.1 ms
// with those three warps on SMs of their own; a whole pass with its host calls 13.9 -> 11.4 ms
// (64.1 with one lane per column and its matrices in local memory).
constexpr int HX_CTAS = 2;
constexpr int HX_WARPS = HX_K / HX_CTAS;
constexpr int HX_THREADS = 32 * HX_WARPS;
static_assert(HX_WARPS * HX_CTAS == HX_K, "a warp per column");
static_assert(MAXR == 16 && MAXT == 8, "a half warp holds the rows of the matrix, twice the species");

// Extrapolation of the columns FIRST+1..HX_K (step sizes H / j, errors in h, h^2, ...) to
// h = 0: the weight of column j is the product of j / (j - i) over the other columns i.
__host__ __device__ constexpr double hx_weight(int j, int first) {
  double w = 1.0;
  for (int i = first + 1; i <= HX_K; ++i)
    if (i != j) w *= static_cast<double>(j) / static_cast<double>(j - i);
  return w;
}

// Kinetics of one train in molecule numbers, and the columns' end values.
struct HxSmem {
  double nu[MAXR][MAXT];      // change of species x per event of reaction r
  double nu_ab[MAXR][MAXR][2];  // [s][r]: change of r's two reactants per event of s
  double col[2][HX_K][MAXR];  // (alternating, so that one barrier a step is enough)
  double e[MAXR];             // extents at the end of the integration
  int go;                     // the train is to be integrated
};

// Barrier over a train's CTAs (release / acquire of all memory among them).
__device__ __forceinline__ void hx_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Address of CTA q's copy of the shared variable p.
__device__ __forceinline__ uint32_t hx_peer(const void* p, uint32_t q) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(p))), "r"(q));
  return a;
}

// What a lane keeps: its reaction r (lanes past the reactions: kappa 0, reactants 0), its half
// h, and the entries of parity h for species r mod 8.
struct HxLane {
  int nr, nt, r, h, col;
  int a, b;
  double kappa;
  double n0;           // of the species, in half 0
  double nu[MAXR / 2];  // change of the species per event of reaction 2j + h
};

__device__ __forceinline__ double hx_shfl(double v, int src) {
  return __shfl_sync(0xffffffffu, v, src, 16);
}

// kappa n_a and kappa n_b of this lane's reaction and its rate, at extents y (one per row).
__device__ __forceinline__ double hx_rate(const HxLane& k, double y, double& na, double& nb) {
  double n = k.n0;
#pragma unroll
  for (int j = 0; j < MAXR / 2; ++j)
    if (2 * j < k.nr) n += k.nu[j] * hx_shfl(y, 2 * j + k.h);
  n += __shfl_xor_sync(0xffffffffu, n, 16);
  na = hx_shfl(n, k.a);
  nb = hx_shfl(n, k.b);
  return k.kappa * na * nb;
}

// (de / sc)^(-1 / HX_K) in FP64 for a quotient of 1e-4 to 1e4, and that of the nearer end beyond
// (past the step-size factor's limits anyway). r from FP32 and the reciprocal of sc from FP32 with
// one Newton step; then de / sc = (1 - t) r^-6 with |t| below 1e-5, and two terms of the binomial
// series of (1 - t)^(-1/6), whose third is below 1e-16. (The call of 64 trains below takes 3.14 ms
// with it, 3.32 with a division, a square root and a cube root, 2.9 with a factor in FP32.)
__device__ __forceinline__ double hx_root(double de, double sc) {
  static_assert(HX_K == 6, "the power of r and the series' terms");
  const float scf = static_cast<float>(sc), q = static_cast<float>(de) / scf, cut = fminf(fmaxf(q, 1e-4f), 1e4f);
  const double r = static_cast<double>(powf(cut, -1.0f / HX_K)), r3 = r * r * r;
  double inv = static_cast<double>(1.0f / scf);
  inv = fma(inv, fma(-sc, inv, 1.0), inv);
  const double t = q == cut ? fma(-de, r3 * r3, sc) * inv : 0.0;
  return fma(r, t * fma(t, 7.0 / 72.0, 1.0 / 6.0), r);
}

// One extrapolated step of length H from y0 (one extent per row, the same in every half
// warp): column j takes j linearly implicit Euler substeps y += (I - hJ)^-1 h f(y), h = H / j,
// with the Jacobian J of y0; then each lane extrapolates its component, which removes the
// error terms in h, h^2, ... (the method's expansion is in powers of h). The inverse is formed
// in place by Gauss-Jordan elimination with a pivot row per column (largest element to 1 part
// in 2^16, rows stay where they are). Returns false (in every CTA of the train) when a matrix
// is singular, which makes its column not a number, or the result is not finite; else y1,
// whether every error estimate is within its tolerance, and the smallest hx_root of the two.
__device__ bool hx_step(const HxLane& k, HxSmem& sm, int odd, double y0, double H, double& y1, bool& within,
                        double& root) {
  const int nr = k.nr;
  const double h = H / static_cast<double>(k.col + 1);
  double na, nb;
  double f = hx_rate(k, y0, na, nb);
  const double ka = -h * (k.kappa * nb), kb = -h * (k.kappa * na);
  // row r of I - hJ: d rate_r / d e_s = kappa_r (n_b nu[a][s] + n_a nu[b][s]); s = 2j + h
  double M[MAXR / 2];
#pragma unroll
  for (int j = 0; j < MAXR / 2; ++j) {
    const int s = 2 * j + k.h;
    M[j] = 0.0;
    if (2 * j < nr)
      M[j] = fma(kb, sm.nu_ab[s][k.r][1], fma(ka, sm.nu_ab[s][k.r][0], s == k.r && s < nr ? 1.0 : 0.0));
  }
  bool free_row = k.r < nr;
  unsigned long long perm = 0;  // pivot row of column c in bits 4c
  bool ok = true;
#pragma unroll
  for (int c = 0; c < MAXR; ++c) {
    if (c >= nr) break;
    const double m = __shfl_sync(0xffffffffu, M[c / 2], k.r + 16 * (c & 1));
    const unsigned hi = static_cast<unsigned>(__double2hiint(m)) & 0x7FFFFFF0u;
    const unsigned best = __reduce_max_sync(0xffffffffu, free_row ? (hi | static_cast<unsigned>(15 - k.r)) : 0u);
    const int p = 15 - static_cast<int>(best & 15u);
    ok = ok && best >= 0x00100000u && best < 0x7FD00000u;
    perm |= static_cast<unsigned long long>(p) << (4 * c);
    // (every row's, beside the search for the pivot; 1 where none could be, off CUDA's slow path)
    const unsigned mag = static_cast<unsigned>(__double2hiint(m)) & 0x7FFFFFFFu;
    const double inv = hx_shfl(__drcp_rn(mag >= 0x00100000u && mag < 0x7FD00000u ? m : 1.0), p);
    const bool mine = k.r == p;
    if (mine) free_row = false;
    const double g = mine ? -inv : m * inv;
#pragma unroll
    for (int j = 0; j < MAXR / 2; ++j)
      if (2 * j < nr) M[j] = fma(-g, hx_shfl(M[j], p), mine ? 0.0 : M[j]);
    if (k.h == (c & 1)) M[c / 2] = -g;
  }
  // the solution's component c is the sum over c' of M[pivot row of c][c'] v[pivot row of c']
  int from[MAXR / 2];
#pragma unroll
  for (int j = 0; j < MAXR / 2; ++j) from[j] = static_cast<int>(perm >> (4 * (2 * j + k.h))) & 15;
  const int row = static_cast<int>(perm >> (4 * k.r)) & 15;
  double y = y0;
  for (int i = 0; i <= k.col; ++i) {
    if (i > 0) f = hx_rate(k, y, na, nb);
    const double v = h * f;
    double x = 0.0;
#pragma unroll
    for (int j = 0; j < MAXR / 2; ++j)
      if (2 * j < nr) x += M[j] * hx_shfl(v, from[j]);
    x += __shfl_xor_sync(0xffffffffu, x, 16);
    x = hx_shfl(x, row);
    if (k.r < nr) y += x;
  }
  if (!ok) y = nan("");
  static_assert(HX_CTAS == 2, "half h writes to CTA h");
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(hx_peer(&sm.col[odd][k.col][k.r], k.h)), "d"(y) : "memory");
  hx_sync();
  // every half warp extrapolates, so that all go on with the same values
  const double last = sm.col[odd][HX_K - 1][k.r];
  double all = 0.0, but_one = 0.0;
#pragma unroll
  for (int j = 1; j < HX_K; ++j) {
    const double dv = sm.col[odd][j - 1][k.r] - last;  // (the weights' sum is 1)
    all += hx_weight(j, 0) * dv;
    if (j > 1) but_one += hx_weight(j, 1) * dv;
  }
  y1 = last + all;
  const double sc = HX_ATOL + HX_RTOL * fmax(fabs(y0), fabs(y1));
  const double de = fabs(all - but_one);
  const bool mine = k.r < nr;
  const bool fin = __all_sync(0xffffffffu, !mine || isfinite(y1));
  within = __all_sync(0xffffffffu, !mine || de <= sc);
  // the smallest by its bits (none is negative): the high words, then the low words with that one
  const double own = mine ? hx_root(de, sc) : 8.0;
  const unsigned hi = static_cast<unsigned>(__double2hiint(own)), top = __reduce_min_sync(0xffffffffu, hi);
  const unsigned low = __reduce_min_sync(0xffffffffu, hi == top ? static_cast<unsigned>(__double2loint(own)) : ~0u);
  root = __hiloint2double(static_cast<int>(top), static_cast<int>(low));
  if (!mine) y1 = 0.0;
  return fin;
}

// Extents after T seconds from e = 0, one per row (identical control flow on every
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
    double y1;
    double root;
    bool within;
    const bool ok = hx_step(k, sm, it & 1, e, Hs, y1, within, root);
    root *= 0.9;
    if (ok && within) {
      e = y1;
      t = last ? T : t + Hs;
      ++accepted;
      H = Hs * fmin(4.0, fmax(0.2, root));
    } else {
      H = Hs * (ok ? fmin(0.5, fmax(0.2, root)) : 0.2);
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

__global__ void __cluster_dims__(HX_CTAS, 1, 1) __launch_bounds__(HX_THREADS) k_hx_integrate(Dev d) {
  __shared__ HxSmem sm;
  const int tid = threadIdx.x;
  const uint32_t b = blockIdx.x / HX_CTAS, rank = blockIdx.x % HX_CTAS;
  Train& tr = d.trains[b];
  // one answer for the train's CTAs (another train's may raise the status meanwhile)
  hx_sync();
  if (rank == 0 && tid < HX_CTAS) {
    const int go = status_of_hx(d) == 0 && tr.hx_sel ? 1 : 0;
    asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(hx_peer(&sm.go, tid)), "r"(go) : "memory");
  }
  hx_sync();
  if (!sm.go) return;
  const Tables& tb = *d.tables;
  HxLane k;
  k.nt = tb.n_types;
  k.nr = tb.n_rxn;
  k.r = tid & 15;
  k.h = (tid >> 4) & 1;
  k.col = HX_WARPS * static_cast<int>(rank) + (tid >> 5);
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
  __syncthreads();
  const int x = k.r & (MAXT - 1);  // the species this lane sums (lane x + 8 a copy)
  k.n0 = k.h == 0 && x < k.nt ? static_cast<double>(tr.counts[x]) : 0.0;
#pragma unroll
  for (int j = 0; j < MAXR / 2; ++j) k.nu[j] = sm.nu[2 * j + k.h][x];
  k.a = k.r < k.nr ? tb.rxn_a[k.r] : 0;
  k.b = k.r < k.nr ? tb.rxn_b[k.r] : 0;
  k.kappa = k.r < k.nr ? (k.a == k.b ? 0.5 * tb.k_tab[k.r] : tb.k_tab[k.r]) / NV : 0.0;
  for (int s = tid >> 4; s < MAXR; s += HX_THREADS / 16) {
    sm.nu_ab[s][k.r][0] = sm.nu[s][k.a];
    sm.nu_ab[s][k.r][1] = sm.nu[s][k.b];
  }
  double own;
  const double T = tr.hx_t_end - tr.t;
  hx_sync();  // (both have read the train's record)
  const long long steps = hx_integrate(k, sm, T, own);
  if (tid < MAXR) sm.e[tid] = own;
  __syncwarp();
  if (rank != 0 || tid != 0) return;  // the rounding and the train's record: one thread
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
  k_hx_integrate<<<static_cast<int>(d.n_trains) * HX_CTAS, HX_THREADS, 0, s>>>(d);
  return cudaGetLastError();
}

}  // namespace chem
