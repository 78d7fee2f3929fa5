// Type-2 interpolation back to the samples, the at-sample solve, and the
// DF / GCV reductions.
//
// Every sorted sample gathers the fields of one bandwidth from that
// bandwidth's fine grid with the spreading kernel (the uniform-to-non-uniform
// NUFFT that Sec. 1.1 mentions), solves the system of eq. 3 at q = x_i, and
// contributes to
//   rss_r      = sum_i (y_ri - mhat_r(x_i))^2                 (numerator of eq. 22)
//   wSw_p      = sum_i w_pi (S w_p)_i,  ww_p = sum_i w_pi^2   (Sec. 2.1)
//   tr_exact   = K_H(0) sum_i [S(x_i)^-1]_11                  (diagonal of S_h)
// Block partials are summed in a fixed order.  (Calls of the NUFFT path still differ in
// rounding from run to run: the spreading adds its tiles with atomics, and the warps of
// interp_direct.cu claim their groups.  The direct sums repeat bit for bit, direct.cu.)
//
// Fields are stored interleaved per fine-grid cell ([cell][rec], rec >= F2 an
// odd number of 16-byte units), so a sample's fields of one cell are one
// contiguous run.
//
// The kernels:
// - interp_direct.cu: persistent, bin windows double-buffered in shared
//   memory (FP32, width 7, 1-D / 2-D, orders 0 and 1, at most 64 fields);
// - interp_global.cu: FP32 3-D Nadaraya-Watson and gather-only, lane per
//   sample over the global grid with a register epilogue;
// - interp_lane.cuh: lane per sample, every other case of a compile-time width
//   (FP32 7; FP64 7, 10, 13);
// - here: any other width.  A warp gathers one sample at a time with its lanes
//   spread over the fields, walks a group of 32 consecutive sorted samples,
//   parks each sample's field values in shared memory, and then each lane takes
//   one sample for the FP64 solve and the reductions.  Fields go in passes of
//   pass_f; pass 0 holds the s-fields.
#include <cuda_runtime.h>

#include <algorithm>

#include "device_common.cuh"
#include "gather.cuh"
#include "interp_common.cuh"
#include "internal.h"

namespace fk {

namespace {

constexpr int kI2Warps = 16;   // warps per block (upper bound)
constexpr int kMaxWRun = 32;   // widest runtime window

// Gather-only mode: the pass's field values of this lane's sample go to
// V[f][s] (sorted sample order; consecutive lanes write consecutive samples).
template <typename T>
__device__ __forceinline__ void store_fields(T* __restrict__ V, const T* my, int f_first,
                                             int fcount, bool valid, int64_t s, int64_t n) {
  if (!valid) return;
  for (int f = 0; f < fcount; ++f) V[int64_t(f_first + f) * n + s] = my[f];
}

// ---- any window width: a warp per sample, from the global field grid --------
template <typename T, int D, int NCH>
__global__ void __launch_bounds__(kI2Warps * 32)
interp_kernel(GeoDev g, MonoTab mono, const BwDev* __restrict__ bwt, int b, int order, int64_t n,
              const T* __restrict__ xs, const T* __restrict__ str, const uint32_t* __restrict__ perm,
              const T* __restrict__ fld, int rec, int F2, int pass_f, int n_rhs_real, int n_probes,
              int cplx, int n_rhs_out, T* __restrict__ mhat_at_x, int nacc, int nbw,
              double* __restrict__ part, T* __restrict__ vout) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarps = int(blockDim.x >> 5);
  const int w = g.w;
  int ncw = 1;
  for (int j = 0; j < D; ++j) ncw *= w;
  const int bstride = pass_f + 1;
  double* red_all = reinterpret_cast<double*>(smem_raw);
  double* red = red_all + warp * nacc;
  T* cellw = reinterpret_cast<T*>(red_all + nwarps * nacc) + warp * ncw;
  T* buf = reinterpret_cast<T*>(red_all + nwarps * nacc) + nwarps * ncw + warp * 32 * bstride;
  for (int a = lane; a < nacc; a += 32) red[a] = 0.0;
  __syncwarp();
  const BwDev& B = bwt[b];
  const int nf0 = int(B.nf[0]), nf1 = D > 1 ? int(B.nf[1]) : 1, nf2 = D > 2 ? int(B.nf[2]) : 1;
  const T ih0 = T(B.inv_h[0]), ih1 = T(D > 1 ? B.inv_h[1] : 1.0), ih2 = T(D > 2 ? B.inv_h[2] : 1.0);
  const T beta = T(g.beta);
  const T halfw = T(0.5) * T(w);
  GroupCtx c{mono.n, mono.nt, mono.nt, n_rhs_real + n_probes, n_rhs_real, n_probes, cplx,
             n_rhs_out, nacc, order, b};
  T tsc[kMaxP];
#pragma unroll
  for (int k = 0; k < kMaxP; ++k) tsc[k] = (k < c.p) ? T(1.0 / tscale(mono, k, B.sigma)) : T(0);
  const T k0t = T(B.k0);
  const double isg[3] = {B.isigma[0], B.isigma[1], B.isigma[2]};
  // each block walks one contiguous run of sample groups (neighbouring bins)
  const int64_t ngroups = (n + 31) / 32;
  const int64_t per_block = (ngroups + gridDim.x - 1) / gridDim.x;
  const int64_t g_begin = int64_t(blockIdx.x) * per_block;
  const int64_t g_end = min(ngroups, g_begin + per_block);
  for (int64_t grp = g_begin + warp; grp < g_end; grp += nwarps) {
    const int64_t s0 = grp * 32;
    const int cnt = int(min(int64_t(32), n - s0));
    const int64_t s = s0 + lane;
    const bool valid = lane < cnt;
    T af[kMaxP] = {T(0), T(0), T(0), T(0)};
    int q_done = 0, f_first = 0;
    for (int pass = 0; f_first < F2; ++pass) {
      const int q_in = vout ? 0
                            : (pass == 0 ? min(c.nq, (pass_f - c.ns) / c.nt)
                                         : min(c.nq - q_done, pass_f / c.nt));
      const int f_last =
          vout ? min(F2, f_first + pass_f) : (pass == 0 ? c.ns : f_first) + q_in * c.nt;
      const int fcount = f_last - f_first;
      T xn0 = xs[s0], xn1 = D > 1 ? xs[n + s0] : T(0), xn2 = D > 2 ? xs[2 * n + s0] : T(0);
      for (int j = 0; j < cnt; ++j) {
        const T x0 = xn0, x1 = xn1, x2 = xn2;
        if (j + 1 < cnt) {  // prefetch the next sample's coordinates
          xn0 = xs[s0 + j + 1];
          if (D > 1) xn1 = xs[n + s0 + j + 1];
          if (D > 2) xn2 = xs[2 * n + s0 + j + 1];
        }
        const SampleWin<T, D> sw =
            sample_window<T, D>(g, w, beta, halfw, ih0, ih1, ih2, x0, x1, x2, lane);
        T acc[NCH];
        gather_global<T, D, NCH>(fld, rec, f_first, fcount, lane, sw, w, nf0, nf1, nf2, cellw, acc);
#pragma unroll
        for (int ch = 0; ch < NCH; ++ch)
          if (lane + ch * 32 < fcount) buf[j * bstride + lane + ch * 32] = acc[ch];
        __syncwarp();
      }
      if (vout)
        store_fields<T>(vout, buf + lane * bstride, f_first, fcount, valid, s, n);
      else
        finish_pass<T, D>(c, mono, B, buf + lane * bstride, pass, q_done, q_in, lane, valid, n,
                       str + n + s, n, valid ? perm[s] : 0u, mhat_at_x, tsc, af, red, k0t, isg);
      __syncwarp();
      q_done += q_in;
      f_first = f_last;
    }
  }
  __syncthreads();
  for (int a = threadIdx.x; a < nacc; a += blockDim.x) {
    double t = 0.0;
    for (int wv = 0; wv < nwarps; ++wv) t += red_get<T>(red_all, wv * nacc + a);
    part[(int64_t(blockIdx.x) * nbw + b) * nacc + a] = t;
  }
}

// sum block partials in a fixed order: sums[b][a]; one block per output
__global__ void reduce_partials(const double* __restrict__ part, int64_t nblk, int nbw, int nacc,
                                double* __restrict__ sums) {
  __shared__ double sh[256];
  const int o = blockIdx.x;
  double t = 0.0;
  for (int64_t k = threadIdx.x; k < nblk; k += blockDim.x) t += part[k * nbw * nacc + o];
  sh[threadIdx.x] = t;
  __syncthreads();
  for (int st = blockDim.x / 2; st > 0; st >>= 1) {
    if (threadIdx.x < st) sh[threadIdx.x] += sh[threadIdx.x + st];
    __syncthreads();
  }
  if (threadIdx.x == 0) sums[o] = sh[0];
}

__global__ void finalize_kernel(const double* __restrict__ sums, int nbw, int nacc, int n_rhs_real,
                                int n_probes, int cplx, int64_t n, int use_exact,
                                double* __restrict__ rss, double* __restrict__ trace,
                                double* __restrict__ gcv) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nbw) return;
  const double* sb = sums + int64_t(b) * nacc;
  double girard = 0.0, hutch = 0.0;
  for (int p = 0; p < n_probes; ++p) {
    const double wsw = sb[n_rhs_real + p], ww = sb[n_rhs_real + n_probes + p];
    girard += wsw / ww;
    hutch += wsw;
  }
  if (n_probes > 0) {
    girard = double(n) * girard / n_probes;
    hutch = hutch / n_probes;
  } else {
    girard = hutch = __longlong_as_double(0x7ff8000000000000LL);
  }
  const double exact = sb[nacc - 1];
  if (trace) {
    trace[b * 3 + 0] = girard;
    trace[b * 3 + 1] = hutch;
    trace[b * 3 + 2] = exact;
  }
  const int mult = cplx ? 2 : 1;
  const int n_rhs = n_rhs_real / mult;
  const double tr = use_exact ? exact : girard;
  for (int r = 0; r < n_rhs; ++r) {
    double v = 0.0;
    for (int pt = 0; pt < mult; ++pt) v += sb[r * mult + pt];
    if (rss) rss[b * n_rhs + r] = v;
    if (gcv) {
      const double den = 1.0 - tr / double(n);
      gcv[b * n_rhs + r] = (v / double(n)) / (den * den);
    }
  }
}

template <typename T, int D, int NCH>
cudaError_t launch_interp_w(fkreg_plan_s* P, int b, int n_rhs_real, int n_probes, void* mhat_at_x,
                            cudaStream_t st, int nacc, int F2, T* vout = nullptr) {
  constexpr int pass_f = 32 * NCH;
  const int rec = t2_record_stride(F2, sizeof(T));
  const unsigned blocks = unsigned(P->nblk_interp);
  const size_t buf_warp = sizeof(T) * 32 * (pass_f + 1) + sizeof(double) * nacc;
  int ncw = 1;
  for (int j = 0; j < D; ++j) ncw *= P->geo.w;
  // warps per block: as many as fit (up to kI2Warps) in the shared-memory budget
  const size_t per_warp = buf_warp + sizeof(T) * ncw;
  const int nwarps = int(std::min<size_t>(kI2Warps, (200 * 1024) / per_warp));
  if (nwarps < 1) return cudaErrorInvalidConfiguration;
  const size_t smem = per_warp * nwarps;
  cudaError_t e = cudaFuncSetAttribute(interp_kernel<T, D, NCH>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  if (e != cudaSuccess) return e;
  interp_kernel<T, D, NCH><<<blocks, nwarps * 32, smem, st>>>(
      P->geo, P->mono, wsp<BwDev>(P, P->r_bw), b, P->order, P->n, wsp<T>(P, P->r_xs),
      wsp<T>(P, P->r_str), perm_ptr(P), wsp<T>(P, P->r_t2field), rec, F2, pass_f, n_rhs_real,
      n_probes, P->o.y_complex, P->nrhs, static_cast<T*>(mhat_at_x), nacc, P->nbw,
      wsp<double>(P, P->r_part), vout);
  P->launches += 1;
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_interp(fkreg_plan_s* P, int b, int n_rhs_str, int n_probes, void* mhat_at_x,
                          void* keep, bool* kept, cudaStream_t st) {
  const int n_rhs_real = n_rhs_str;
  const int nacc = n_rhs_real + 2 * n_probes + 1;
  if (nacc > kMaxAcc) return cudaErrorInvalidValue;
  const int F2 = P->ns + (n_rhs_real + n_probes) * P->nt;
  if (P->d * P->geo.w > 64 || P->geo.w > kMaxWRun) return cudaErrorInvalidValue;
  if (sizeof(T) == 4) {
    bool used = false;
    cudaError_t e =
        run_interp_direct(P, b, n_rhs_real, n_probes, mhat_at_x, st, nacc, F2, keep, false, &used);
    *kept = used && keep;
    if (used || e != cudaSuccess) return e;
    e = run_interp_global_lane(P, b, n_rhs_real, n_probes, mhat_at_x, st, nacc, F2, nullptr, &used);
    if (used || e != cudaSuccess) return e;
  }
  {
    bool used = false;
    const cudaError_t e =
        sizeof(T) == 4
            ? run_interp_lane_f32(P, b, n_rhs_real, n_probes, mhat_at_x, st, nacc, F2, nullptr, &used)
            : run_interp_lane_f64(P, b, n_rhs_real, n_probes, mhat_at_x, st, nacc, F2, nullptr, &used);
    if (used || e != cudaSuccess) return e;
  }
  // fields per pass: 64 (float) or 32 (double)
  const bool two = sizeof(T) == 4 && F2 > 32;
  if (two) {
    if (P->d == 1) return launch_interp_w<T, 1, 2>(P, b, n_rhs_real, n_probes, mhat_at_x, st, nacc, F2);
    if (P->d == 2) return launch_interp_w<T, 2, 2>(P, b, n_rhs_real, n_probes, mhat_at_x, st, nacc, F2);
    return launch_interp_w<T, 3, 2>(P, b, n_rhs_real, n_probes, mhat_at_x, st, nacc, F2);
  }
  if (P->d == 1) return launch_interp_w<T, 1, 1>(P, b, n_rhs_real, n_probes, mhat_at_x, st, nacc, F2);
  if (P->d == 2) return launch_interp_w<T, 2, 1>(P, b, n_rhs_real, n_probes, mhat_at_x, st, nacc, F2);
  return launch_interp_w<T, 3, 1>(P, b, n_rhs_real, n_probes, mhat_at_x, st, nacc, F2);
}

// Gather-only: F fields of bandwidth b's type-2 grid at every sorted sample
// into V[f][n], through the same kernels (and window staging) as above.
template <typename T>
cudaError_t launch_gather(fkreg_plan_s* P, int b, int F, T* V, cudaStream_t st) {
  if (P->n == 0) return cudaSuccess;
  if (P->d * P->geo.w > 64 || P->geo.w > kMaxWRun) return cudaErrorInvalidValue;
  if (sizeof(T) == 4) {
    bool used = false;
    cudaError_t e = run_interp_direct(P, b, 0, 0, nullptr, st, 0, F, V, true, &used);
    if (used || e != cudaSuccess) return e;
    e = run_interp_global_lane(P, b, 0, 0, nullptr, st, 0, F, V, &used);
    if (used || e != cudaSuccess) return e;
  }
  {
    bool used = false;
    const cudaError_t e = sizeof(T) == 4
                              ? run_interp_lane_f32(P, b, 0, 0, nullptr, st, 0, F, V, &used)
                              : run_interp_lane_f64(P, b, 0, 0, nullptr, st, 0, F, V, &used);
    if (used || e != cudaSuccess) return e;
  }
  if (sizeof(T) == 4 && F > 32) {
    if (P->d == 1) return launch_interp_w<T, 1, 2>(P, b, 0, 0, nullptr, st, 0, F, V);
    if (P->d == 2) return launch_interp_w<T, 2, 2>(P, b, 0, 0, nullptr, st, 0, F, V);
    return launch_interp_w<T, 3, 2>(P, b, 0, 0, nullptr, st, 0, F, V);
  }
  if (P->d == 1) return launch_interp_w<T, 1, 1>(P, b, 0, 0, nullptr, st, 0, F, V);
  if (P->d == 2) return launch_interp_w<T, 2, 1>(P, b, 0, 0, nullptr, st, 0, F, V);
  return launch_interp_w<T, 3, 1>(P, b, 0, 0, nullptr, st, 0, F, V);
}

}  // namespace

cudaError_t run_gather_fields(fkreg_plan_s* P, int b, int F, void* V, cudaStream_t st) {
  return P->prec == FKREG_F32 ? launch_gather<float>(P, b, F, static_cast<float*>(V), st)
                              : launch_gather<double>(P, b, F, static_cast<double*>(V), st);
}

cudaError_t run_interp(fkreg_plan_s* P, int b, int n_rhs_str, int n_probes, void* mhat_at_x,
                       void* keep, cudaStream_t st) {
  if (P->direct) return run_direct_interp(P, b, n_rhs_str, n_probes, mhat_at_x, st);
  bool kept = false;
  const cudaError_t e =
      P->prec == FKREG_F32
          ? launch_interp<float>(P, b, n_rhs_str, n_probes, mhat_at_x, keep, &kept, st)
          : launch_interp<double>(P, b, n_rhs_str, n_probes, mhat_at_x, keep, &kept, st);
  if (e != cudaSuccess || !keep || kept) return e;
  // kernels that don't store the fields on the way: gather them from the same grid
  return run_gather_fields(P, b, P->ns + (n_rhs_str + n_probes) * P->nt, keep, st);
}

// Sum the partials of the last interpolation passes and derive DF and GCV.
cudaError_t run_finalize(fkreg_plan_s* P, int n_probes, const fkreg_outputs* out, cudaStream_t st) {
  const int nacc = P->nrhs_real + 2 * n_probes + 1;
  double* sums = wsp<double>(P, P->r_part) + P->nblk_interp * int64_t(P->nbw) * P->nacc;
  const int64_t nblk = P->nblk_interp;
  const int tot = P->nbw * nacc;
  reduce_partials<<<tot, 256, 0, st>>>(wsp<double>(P, P->r_part), nblk, P->nbw, nacc, sums);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  finalize_kernel<<<(P->nbw + 63) / 64, 64, 0, st>>>(
      sums, P->nbw, nacc, P->nrhs_real, n_probes, P->o.y_complex, P->n,
      (P->o.flags & FKREG_GCV_EXACT_TRACE) ? 1 : 0, out ? out->rss : nullptr,
      out ? out->trace : nullptr, out ? out->gcv : nullptr);
  P->launches += 2;
  return cudaGetLastError();
}

// Field record stride (elements) of the type-2 grids for F2 fields: an odd
// number of 16-byte units (4 floats, 2 doubles), so every cell record starts
// on a 16-byte boundary for the bulk copies and neighbouring cells start on
// different shared-memory banks.
int t2_record_stride(int F2, size_t tsize) {
  const int u = int(16 / tsize);
  const int units = (F2 + u - 1) / u;
  return (units | 1) * u;
}

}  // namespace fk
