// Internal declarations shared by the planner, the kernels and the C ABI.
#pragma once

#include <cuda_runtime.h>
#include <cufft.h>

#include <cstdint>
#include <map>
#include <string>
#include <tuple>
#include <vector>

#include "../../include/fkreg.h"

namespace fk {

constexpr int kMaxD = 3;
constexpr int kMaxMono = 35;     // monomials of degree <= 4 in 3-D (s-fields of local quadratic)
constexpr int kMaxP = 10;        // unknowns of the local-quadratic system in 3-D
// Samples per sub-problem (a run of one bin's samples that one block takes in
// the spreading and the staged gathers): GeoDev::sub_max, between these.
constexpr int kSubMin = 256;
constexpr int kSubMax = 1024;
constexpr int kRadixBits = 8;
constexpr int kSortTileKeys = 4096;  // keys per radix-sort tile (one block)
// Up to 512 tiles' worth of samples the fused sort takes tiles of 1024 keys: a
// scatter is bound by the serial work of one block (16 rounds of 4096 keys), so
// a small problem is as slow as a large one unless its keys go to more blocks.
// Estimates with tiles of 4096 and of 1024 keys, us: 1-D, 10,000 samples 135 / 115,
// 520,000 samples 303 / 187; 2-D, 300,000 samples 196 / 170, 520,000 samples 224 / 212.
// At 10^6 samples a block's fixed work (per-digit counts and scans) has won: the
// 2-D step takes 677 us with 4096 keys and 692 with 1024.
constexpr int kSmallTile = 1024;
constexpr int64_t kSmallTileMaxN = 512 * kSmallTile;
constexpr int64_t kFft1dMax = 4096;  // longest 1-D transform of fft1d.cu
constexpr uint32_t kDefaultWaitLimit = 1u << 22;  // polls of a staged-window wait

// Polynomials of the spreading kernel's inner taps (phi_row), tap k at distance
// c = (w - 1)/2 - k from the centre: phi(x +- c) = E(x^2) +- x O(x^2) for
// |x| <= 1/2.  FP64 plans of an instantiated width.
constexpr int kPhiTerms = 8;
constexpr int kPhiTaps = 7;
struct PhiPoly {
  double e[kPhiTaps][kPhiTerms];
  double o[kPhiTaps][kPhiTerms];
};

// Geometry of the whole plan, passed to kernels by value.
struct GeoDev {
  int d;
  int w;            // spreading width (fine cells)
  int pad;          // ceil(w/2): tile halo on each side
  int skind;        // FKREG_SPREAD_ES / FKREG_SPREAD_GAUSS
  double beta;      // ES shape, or Gaussian exponent factor
  int64_t nf[3];    // type-1 fine grid
  int64_t L[3];     // inverse-DFT length onto the grid lattice
  int64_t M[3];     // output grid points
  int64_t K[3];     // type-1 modes (kept: |k| <= K/2 - 1)
  double P[3];      // period
  double lo[3];
  double hi[3];
  double inv_h[3];  // nf / P (double; the T-rounded copy is inv_h_t)
  float inv_h_f[3];
  int64_t tile[3];
  int64_t nbins[3];
  int kbits;        // within-bin bits of the sort key (see key_local_bits)
  int kern;         // regression kernel: FKREG_KERNEL_GAUSSIAN (NUFFT) or a compact one (direct)
  uint32_t sub_max;     // samples per sub-problem (sub_problem_size)
  uint32_t wait_limit;  // polls of a staged-window wait before it gives up (fkreg_set_wait_limit)
  int* errw;            // the plan's error word (errw[0] bits kErr*; errw[1..3] the first
                        // failed bounds check of a checked build: site, index low, high)
};

// Bits of the plan's device error word.
constexpr int kErrOutside = 1;  // a sample outside the grid box or not finite
constexpr int kErrTimeout = 2;  // a bounded device-side wait gave up
// Word errw[kStrFlag] of the direct path: the number (fkreg_plan_s::str_pass) of
// the last strengths pass in which a value was not finite.
constexpr int kStrFlag = 16;
constexpr int kTaskWord = 17;  // next group of targets of the direct at-sample pass
constexpr int kErrBounds = 4;   // a bounds check of the checked build failed (access skipped)

// Sort keys are (bin << kbits) | local, local = serpentine index of the
// centre cell of the sample's spreading window relative to its bin's first
// cell, tile_j + 1 values per axis.  kbits = 0 (bin-only keys) if the key would not
// fit 32 bits.
inline int key_local_bits(int d, const int64_t* tile, const int64_t* nbins) {
  int64_t cells = 1, bins = 1;
  for (int j = 0; j < d; ++j) {
    cells *= tile[j] + 1;
    bins *= nbins[j];
  }
  int lb = 0, bb = 0;
  while ((int64_t(1) << lb) < cells) ++lb;
  while ((int64_t(1) << bb) < bins) ++bb;
  return bb + lb <= 32 ? lb : 0;
}

// Sub-problem size of a plan for up to max_n samples in nbins bins.  Where the
// bins are fewer than two per SM they are split into about four sub-problems
// per SM, so that a small problem fills the GPU.  With 1024 and with the rule, us:
// 1-D FP64, 10,000 samples in one bin (256) 226 / 180; FP32 2-D, 30,000 samples in 63
// bins (256), estimate with ten probes 227 / 189, GCV gradient 1134 / 1004; 90,000
// samples (256) 189 / 177 and 1087 / 1059.  Every split pays for one more tile flush
// (some strengths of a 24 x 24 tile against the sub-problem's samples), so no size is
// below kSubMin, and where the bins hold many samples already the split no longer
// gains: 520,000 samples in 63 bins (864) 292 / 300 and 1458 / 1492.  More bins than
// two per SM give blocks enough by themselves.  FP64 2-D blocks are long (the FP64
// pipe) against their flush: there the split also evens out the last wave (90 bins,
// 30,000 samples 677 / 405; 520,000 samples 2660 / 2537), and so it does for the 3-D
// FP32 spreading of width 7 (the only user of sub-problems in 3-D) with few strengths:
// 300,001 samples in 336 bins, local linear (512) 932 / 888; with seventeen strengths
// the flushes cost more than that gains: 200,000 samples in 294 bins (352) 1534 / 1626.
inline uint32_t sub_problem_size(int d, int w, bool f64, int64_t nbins, int64_t max_n, int sm_count) {
  const int64_t sms = sm_count < 1 ? 1 : sm_count;
  if (d > 2 ? (f64 || w != 7) : (nbins >= 2 * sms && !f64)) return kSubMax;
  const int64_t per = (max_n / (4 * sms) + 31) / 32 * 32;
  return uint32_t(per < kSubMin ? kSubMin : (per > kSubMax ? kSubMax : per));
}

// One bandwidth, stored in the workspace (device reads it).
struct BwDev {
  double H[9];
  double sigma[3];     // sqrt(H_jj)
  double isigma[3];    // 1 / sigma
  double k0;           // K_H(0)
  int64_t K[3];        // modes this bandwidth needs
  int64_t nf[3];       // type-2 fine grid for this bandwidth
  double inv_h[3];     // nf_b / P
  int64_t phi2_off[3]; // offset (doubles) of 1/phihat tables (k >= 0) for type-2
  double Hinv[9];      // H^-1 (compact kernels)
  double kscale;       // c_d / sqrt(det H): K_H(z) = kscale k(|H^(-1/2) z|^2) (compact kernels)
  double kr2;          // R^2 of the truncated Gaussian (FKREG_KERNEL_GAUSSIAN_DIRECT), else 0
};

// Monomial exponents (degree <= 2) for device code.
struct MonoTab {
  int n;               // monomials of degree <= 2l  (s-fields)
  int nt;              // monomials of degree <= l   (t-fields)
  int toff;            // where the t-monomials start in e (0: a prefix of the s-monomials)
  int e[kMaxMono][kMaxD];
};

struct Region {
  size_t off = 0, bytes = 0;
};

}  // namespace fk

struct fkreg_plan_s {
  fkreg_opts o{};
  std::vector<double> H;        // [nbw][d][d]
  fkreg_geometry g{};
  fk::GeoDev geo{};
  fk::MonoTab mono{};
  // backward: monomials of degree <= 2l + 1 in the graded order (n), and the
  // ones that the gradients need beyond the plan's fields: s of degree 2l + 1
  // (n) and t of degree l + 1 (nt, from toff)
  fk::MonoTab mono_all{}, mono_x{};
  fk::PhiPoly poly{};           // FP64 plans
  int64_t max_n = 0;
  int d = 0, order = 0, prec = 0, ns = 0, nt = 0, p = 0;
  int nbw = 0, nrhs = 0, nrhs_real = 0, max_probes = 0;
  int smax = 0;                 // strengths of the largest pass
  int f2max = 0;                // type-2 fields of the largest pass
  int fgrid = 0;                // grid fields (ns + nrhs_real * nt)
  size_t tsize = 4;             // sizeof(T)
  std::vector<fk::BwDev> bw;    // host copy of the bandwidth table
  std::vector<double> tab;      // 1/phihat tables (type-1 per axis, then type-2)
  int64_t phi1_off[3] = {0, 0, 0};
  std::map<int64_t, int64_t> roots;  // 1-D transform lengths -> first root (complex) in root_tab
  std::vector<double> root_tab;      // roots of unity (re, im)
  int64_t nbins_total = 0;
  int64_t nsub_max = 0;
  int64_t nblk_interp = 0;      // blocks of the interpolation kernel (partials)
  int sm_count = 0;             // streaming multiprocessors of the plan's device
  int nacc = 0;                 // accumulators per (block, bandwidth)

  // workspace regions
  fk::Region r_err, r_bw, r_tab, r_roots, r_xs, r_keys0, r_vals0, r_keys1, r_vals1, r_counts,
      r_binstart, r_nsub, r_substart, r_subbin, r_subfirst, r_hist, r_hist2, r_dtot, r_scan, r_str,
      r_fine, r_spec, r_gspec, r_gfield, r_t2spec, r_t2field, r_part, r_smax, r_fftwork,
      r_fftwork_g,
      r_bV, r_bdx, r_bsc, r_gmask, r_gadj, r_gpart, r_gavec, r_gsum;
  bool backward = false;        // workspace reserved for fkreg_backward
  bool direct = false;          // compact kernel: direct sums instead of the NUFFT
  int f2bwd = 0;                // fields of the backward passes (one response + probes)
  int fxbwd = 0;                // extra moment fields of the backward (mono_x)
  size_t ws_bytes = 0;
  size_t fft_work_reserved = 0;
  size_t fft_work_reserved_g = 0;  // inverse grid transforms (their own area: they overlap)
  char* ws = nullptr;
  size_t ws_given = 0;

  // cuFFT plan cache: (kind, n0, n1, n2, batch) -> handle
  std::map<std::tuple<int, int64_t, int64_t, int64_t, int>, cufftHandle> ffts;

  // state
  int64_t n = 0;
  bool points_set = false;
  bool dens_valid = false;
  bool avec_valid = false;      // r_gavec holds the grid weights of the last smooth/df
  int perm_in_vals1 = 0;        // which ping-pong buffer holds the permutation
  std::string err;
  int device = -1;

  // profiling: own kernel launches, per-stage events
  int str_pass = 0;             // direct path: strengths passes so far
  int64_t launches = 0;
  bool timing = false;
  struct Pending {
    int stage;
    cudaEvent_t a, b;
  };
  std::vector<Pending> pending;
  std::vector<cudaEvent_t> ev_pool;
  // second stream for the grid branch of a df/smooth call, which runs beside
  // the type-2 branch (both only read the forward spectrum)
  cudaStream_t aux = nullptr;
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
  double stage_ms[FKREG_N_STAGES] = {0};
  int64_t stage_calls[FKREG_N_STAGES] = {0};
};

namespace fk {

// planner.cpp
fkreg_status compute_geometry(const fkreg_opts* o, fkreg_geometry* g, std::string* err,
                              std::vector<BwDev>* bw, std::vector<double>* tab,
                              int64_t phi1_off[3], GeoDev* geo);
double spread_phi(int kind, int w, double beta, double z);
void spread_phi_poly(int kind, int w, double beta, PhiPoly* out);
void spread_phihat(int kind, int w, double beta, int64_t nf, int64_t nk, double* out);
int nmono(int d, int deg);
void monomials(int d, int deg, int (*e)[kMaxD]);
int64_t next_fast(int64_t n);

// sort.cu
cudaError_t run_sort(fkreg_plan_s* P, int64_t n, const void* x, cudaStream_t s);

// spread.cu
cudaError_t run_spread(fkreg_plan_s* P, int s0, int ns_count, cudaStream_t s);
cudaError_t run_gather_strengths(fkreg_plan_s* P, const void* y, int first_str, int n_probes,
                                 uint64_t seed, const void* probes, int with_density,
                                 cudaStream_t s);
cudaError_t run_residual_strengths(fkreg_plan_s* P, const void* y, const void* mhat_at_x,
                                   int b, int first_str, cudaStream_t s);
cudaError_t run_logres_strengths(fkreg_plan_s* P, const void* y, const void* mhat_at_x, int b,
                                 int first_str, cudaStream_t s);

// spectral.cu
cudaError_t run_kmul_grid(fkreg_plan_s* P, int str_dens, int str_rhs, int nrhs_fields,
                          int bw_first, int bw_count, void* out_spec, cudaStream_t s);
cudaError_t run_kmul_t2(fkreg_plan_s* P, int b, const MonoTab& mono, int str_dens, int str_rhs,
                        int n_rhs_str, cudaStream_t s);
// d GCV / d log sigma from the spectra of the strengths and of the spread
// adjoints (strength slots sb ..), with run_dlogh_lattice_blocks x 3 partial sums
cudaError_t run_dlogh_spread(fkreg_plan_s* P, int b, int n_rhs_str, int sb, double* part,
                             double* dlogh, cudaStream_t s);
cudaError_t run_kmul_adj(fkreg_plan_s* P, int b, int sb, int n_classes, cudaStream_t s);
// grid-estimate backward: type-2 spectra of the adjoint functions of the
// lattice adjoint fields (their R2C spectra E [fgrid][L half]), and
// d L / d log sigma as a spectral inner product (part: FP64 partial sums of
// run_dlogh_lattice_blocks blocks x 3)
cudaError_t run_kmul_adj_lattice(fkreg_plan_s* P, int b, int nrhs, const void* E, cudaStream_t s);
int64_t run_dlogh_lattice_blocks(const fkreg_plan_s* P, int b);
cudaError_t run_dlogh_lattice(fkreg_plan_s* P, int b, int nrhs, const void* E, double* part,
                              double* dlogh, cudaStream_t s);
// backward_grid.cu: adjoint of the per-grid-point solves -> lattice adjoint
// fields qbar [fgrid][L cells] (zero where masked); and the combination of
// the gathered adjoint functions into dy [nrhs][n] and dx [n][d] (original order)
cudaError_t run_grid_adjoint(fkreg_plan_s* P, int b, int nrhs, const uint8_t* mask,
                             const void* gbar, void* qbar, cudaStream_t s);
cudaError_t run_combine_grid(fkreg_plan_s* P, int nrhs, const void* V, void* dy, void* dx,
                             cudaStream_t s);

// backward.cu
cudaError_t run_gather_fields(fkreg_plan_s* P, int b, int F, void* V, cudaStream_t s);
// Persistent interpolation kernel (FP32, width 7, 1-D / 2-D, F2 <= 64):
// launched only when it applies (*launched); vout != NULL takes the F2 fields
// (vout[f][n]), which is all that the gather-only form (gonly) does.
cudaError_t run_interp_direct(fkreg_plan_s* P, int b, int n_rhs_real, int n_probes,
                              void* mhat_at_x, cudaStream_t st, int nacc, int F2, void* vout,
                              bool gonly, bool* launched);
// Lane-per-sample kernels of interp_lane.cuh (compile-time widths, every
// dimension and order), launched only when they apply (*launched).
cudaError_t run_interp_lane_f32(fkreg_plan_s* P, int b, int n_rhs_real, int n_probes,
                                void* mhat_at_x, cudaStream_t st, int nacc, int F2, void* vout,
                                bool* launched);
cudaError_t run_interp_lane_f64(fkreg_plan_s* P, int b, int n_rhs_real, int n_probes,
                                void* mhat_at_x, cudaStream_t st, int nacc, int F2, void* vout,
                                bool* launched);
// Lane-per-sample kernel over the global field grid (FP32, width 7, 3-D
// Nadaraya-Watson or gather-only, F2 <= 64), launched only when it applies.
cudaError_t run_interp_global_lane(fkreg_plan_s* P, int b, int n_rhs_real, int n_probes,
                                   void* mhat_at_x, cudaStream_t st, int nacc, int F2,
                                   void* vout, bool* launched);
cudaError_t run_loss_scalars(fkreg_plan_s* P, int b, int n_probes, cudaStream_t s);
cudaError_t run_adjoint(fkreg_plan_s* P, int b, int n_probes, cudaStream_t s);
cudaError_t run_combine(fkreg_plan_s* P, int n_probes, void* dy, void* dx, cudaStream_t s);

// solve.cu
// avec (may be null): [bw][p][M] the solved weights a_k / tscale_k of each
// grid point (NaN where masked), kept for a variance pass on the same points
cudaError_t run_grid_solve(fkreg_plan_s* P, int bw_first, int bw_count, int nrhs_fields,
                           double* avec, const fkreg_outputs* out, void* sigma2, cudaStream_t s);
// sigma2[b][r][M] = sum_k avec[b][k] t_(r,k) from the grid t-fields alone
// (r_gfield holds nrhs_fields x p t-fields; no s-fields, no solve)
cudaError_t run_grid_apply(fkreg_plan_s* P, int b, int nrhs_fields, void* sigma2, cudaStream_t s);
// keep (may be null): also the fields themselves, [ns + (n_rhs_str + n_probes) nt][n]
cudaError_t run_interp(fkreg_plan_s* P, int b, int n_rhs_str, int n_probes, void* mhat_at_x,
                       void* keep, cudaStream_t s);
// direct path (compact kernels): grid fields of strengths [str_first, str_first + nstr)
// plus the s-fields, bandwidths [bw_first, bw_first + bw_count), into r_gfield
cudaError_t run_direct_grid(fkreg_plan_s* P, int str_first, int nstr, int bw_first,
                            int bw_count, cudaStream_t s);
// the same with a warp to each point, into the field slices from `slice` on
cudaError_t run_direct_points(fkreg_plan_s* P, int str_first, int nstr, int bw_first, int bw_count,
                              int slice, cudaStream_t s);
cudaError_t run_direct_interp(fkreg_plan_s* P, int b, int n_rhs_str, int n_probes,
                              void* mhat_at_x, cudaStream_t s);
cudaError_t run_finalize(fkreg_plan_s* P, int n_probes, const fkreg_outputs* out,
                         cudaStream_t s);
// kappa (eq. 26 normaliser) of bandwidth b for every response, and
// sigma2(g) = exp(v(g)) / kappa when sigma2 != NULL.
cudaError_t run_kappa_sigma2(fkreg_plan_s* P, int b, const void* y, const void* mhat_at_x,
                             const void* v_at_x, const void* v_grid, double* kappa, void* sigma2,
                             cudaStream_t s);

const uint32_t* perm_ptr(fkreg_plan_s* P);
int t2_record_stride(int F2, size_t tsize);
// Interleave F in-place C2R outputs (padded real rows) at src into cell records
// [cell][t2_record_stride(F, tsize)] at dst.
cudaError_t run_t2_interleave(fkreg_plan_s* P, const int64_t* dims, int F, const void* src,
                              void* dst, cudaStream_t st);

// fft1d.cu: transforms of 1-D plans in one launch; a real row of n, spectra of n/2 + 1
bool fft1d_applies(const fkreg_plan_s* P, int64_t n);
void fft1d_add_roots(fkreg_plan_s* P, int64_t n);
cudaError_t run_fft1d_r2c(fkreg_plan_s* P, int64_t n, int batch, const void* in, void* out,
                          cudaStream_t s);
// value i of row k goes to out[k * row + i * elem]
cudaError_t run_fft1d_c2r(fkreg_plan_s* P, int64_t n, int batch, const void* in, void* out,
                          int64_t row, int64_t elem, cudaStream_t s);

// fft helpers (api.cu)
fkreg_status fft_get(fkreg_plan_s* P, int kind, const int64_t* dims, int batch, cufftHandle* h);

template <typename T>
T* wsp(fkreg_plan_s* P, const Region& r) {
  return reinterpret_cast<T*>(P->ws + r.off);
}

}  // namespace fk
