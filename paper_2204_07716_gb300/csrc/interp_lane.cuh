// Type-2 interpolation with one lane per sample (see interp.cu for the
// method): the gathers and kernels for a compile-time window width W, in the
// plan's precision.
//
// Each lane walks its own sample's w^d cells and accumulates every field of
// the pass in registers with 16-byte loads (4 floats or 2 doubles), so no
// lane of the arithmetic pipes idles however few fields there are.  Sorted
// samples share or neighbour windows, so most loads of a warp are broadcasts
// of a few addresses.  FP64 is bound by the FP64 pipe (two lanes per SM and
// clock, a warp instruction every 16 clocks): for 2-D local linear at W = 13
// the 169 x 10 multiply-adds and the 26 spreading-kernel values of a sample
// set the time, which is why fields are counted in pairs there.
//
// Two kernels: interp_lane_kernel stages a bin's window of the field grid in
// shared memory by bulk copies (2-D); interp_global_kernel reads the cells
// through the caches and serves 3-D, 1-D plans of one bin (whose whole grid
// stays in L1) and windows that do not fit.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>

#include "device_common.cuh"
#include "interp_common.cuh"
#include "internal.h"

namespace fk {

namespace {

// Fields per 16-byte unit, and the fields of one pass with NU units: any
// lane_pass<T>(NU) consecutive fields span at most NU units.
template <typename T>
__host__ __device__ constexpr int lane_unit() { return 16 / int(sizeof(T)); }

template <typename T>
struct LaneVec;
template <>
struct LaneVec<float> {
  using type = float4;
};
template <>
struct LaneVec<double> {
  using type = double2;
};

__device__ __forceinline__ void unit_fma(float (&a)[4], float w, const float4& v) {
  const float2 w2 = make_float2(w, w);
  const float2 lo = __ffma2_rn(w2, make_float2(v.x, v.y), make_float2(a[0], a[1]));
  const float2 hi = __ffma2_rn(w2, make_float2(v.z, v.w), make_float2(a[2], a[3]));
  a[0] = lo.x;
  a[1] = lo.y;
  a[2] = hi.x;
  a[3] = hi.y;
}
__device__ __forceinline__ void unit_fma(double (&a)[2], double w, const double2& v) {
  a[0] = fma(w, v.x, a[0]);
  a[1] = fma(w, v.y, a[1]);
}

// One row of W cells at `row` (cell t at row + cl[t]): acc += w0 sum_t pl[t] cell_t.
// With fewer fields than window cells the row is summed first and scaled
// once; otherwise each cell's weight is formed once.
template <typename T, int W, int NU, bool CACHED, typename Off>
__device__ __forceinline__ void lane_row(const T* row, const Off& cl, int nu, T w0,
                                         const T (&pl)[W], T (&acc)[NU][lane_unit<T>()]) {
  using V = typename LaneVec<T>::type;
  constexpr int U = lane_unit<T>();
  if constexpr (NU * U < W) {
    T rs[NU][U];
#pragma unroll
    for (int q = 0; q < NU; ++q)
#pragma unroll
      for (int c = 0; c < U; ++c) rs[q][c] = T(0);
#pragma unroll
    for (int t = 0; t < W; ++t) {
      const T* cell = row + cl(t);
#pragma unroll
      for (int q = 0; q < NU; ++q)
        if (q < nu) {
          const V* p = reinterpret_cast<const V*>(cell + U * q);
          unit_fma(rs[q], pl[t], CACHED ? __ldg(p) : *p);
        }
    }
#pragma unroll
    for (int q = 0; q < NU; ++q)
#pragma unroll
      for (int c = 0; c < U; ++c) acc[q][c] = fma(w0, rs[q][c], acc[q][c]);
  } else {
#pragma unroll
    for (int t = 0; t < W; ++t) {
      const T wgt = w0 * pl[t];
      const T* cell = row + cl(t);
#pragma unroll
      for (int q = 0; q < NU; ++q)
        if (q < nu) {
          const V* p = reinterpret_cast<const V*>(cell + U * q);
          unit_fma(acc[q], wgt, CACHED ? __ldg(p) : *p);
        }
    }
  }
}

// Window of one sample on one axis (the rounding of the bin rule): first
// cell i0 and the offset of its centre from the sample.
template <typename T>
__device__ __forceinline__ int lane_window(T x, T ih, T halfw, T& off) {
  const T u = mul_rn(x, ih);
  const T f = ceil(u - halfw);
  off = f - u;
  return int(f);
}

// Kernel values of the leading axes (all but the last), read in rolled loops.
// FP32 evaluates each where it is needed; FP64 forms a sample's values once
// (phi_row) and parks them in shared memory, [axis][W][32 lanes] per warp.
template <typename T, int D>
__host__ __device__ constexpr int lane_axes_parked() { return sizeof(T) == 8 ? D - 1 : 0; }
template <typename T, int D, int W>
__host__ __device__ constexpr size_t lane_park_bytes() {
  return sizeof(T) * 32 * W * lane_axes_parked<T, D>();
}
template <typename T, int D, int W>
struct LeadAxes {
  T* park;  // this warp's area
  int lane, skind;
  T beta;
  T off[D];
  __device__ __forceinline__ void set(const PhiTab<T>& tab, const T* o) {
#pragma unroll
    for (int j = 0; j < D; ++j) off[j] = o[j];
#pragma unroll
    for (int j = 0; j < lane_axes_parked<T, D>(); ++j) {
      T v[W];
      phi_row<W>(tab, skind, beta, o[j], v);
#pragma unroll
      for (int t = 0; t < W; ++t) park[(j * W + t) * 32 + lane] = v[t];
    }
  }
  __device__ __forceinline__ T at(int j, int t) const {  // read by the lane that wrote it
    if constexpr (sizeof(T) == 8) return park[(j * W + t) * 32 + lane];
    return phi<T>(skind, W, beta, off[j] + T(t));
  }
};

// Fields [f_first, f_last) of one sample from the global grid (periodic wrap);
// pl: the kernel values along the last axis.
template <typename T, int D, int W, int NU>
__device__ __forceinline__ void lane_cells_global(const GeoDev& g, const T* __restrict__ fld,
                                                  int rec, int ua, int nu, const int* i,
                                                  const int* nf, const LeadAxes<T, D, W>& lead,
                                                  const T (&pl)[W],
                                                  T (&acc)[NU][lane_unit<T>()]) {
  int cl[W];
#pragma unroll
  for (int t = 0; t < W; ++t) cl[t] = int(wrap_idx(i[D - 1] + t, nf[D - 1]));
  const int64_t cells = int64_t(nf[0]) * (D > 1 ? nf[1] : 1) * (D > 2 ? nf[2] : 1);
  const T* base = fld + lane_unit<T>() * ua;
#pragma unroll 1
  for (int t0 = 0; t0 < (D > 1 ? W : 1); ++t0) {
    const T w0 = D > 1 ? lead.at(0, t0) : T(1);
    const int64_t r0 = D > 1 ? wrap_idx(i[0] + t0, nf[0]) : 0;
#pragma unroll 1
    for (int t1 = 0; t1 < (D > 2 ? W : 1); ++t1) {
      const T w01 = D > 2 ? w0 * lead.at(1, t1) : w0;
      const int64_t r = D > 2 ? r0 * nf[1] + wrap_idx(i[1] + t1, nf[1]) : r0;
      const int64_t rb = D > 1 ? r * nf[D - 1] : 0;
      if (!in_range(g.errw, kSiteInterpField, rb + nf[D - 1] - 1, cells)) continue;
      lane_row<T, W, NU, true>(base + rb * rec, [&](int t) { return int64_t(cl[t]) * rec; }, nu,
                               w01, pl, acc);
    }
  }
}

template <typename T>
__device__ __forceinline__ void cp_async_elem(T* dst, const T* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_u32(dst)), "l"(src),
               "n"(sizeof(T))
               : "memory");
}

// The passes of a launch over the fields: pass 0 takes the s-fields and as
// many responses / probes as fit pass_f fields, later passes the rest; the
// gather-only form takes pass_f fields at a time.
struct LanePass {
  int q_in, f_last;
};
__device__ __forceinline__ LanePass lane_pass(const GroupCtx& c, bool gonly, int pass, int f_first,
                                              int q_done, int pass_f, int F2) {
  LanePass p;
  p.q_in = gonly ? 0
                 : (pass == 0 ? min(c.nq, (pass_f - c.ns) / c.nt) : min(c.nq - q_done, pass_f / c.nt));
  p.f_last = gonly ? min(F2, f_first + pass_f) : (pass == 0 ? c.ns : f_first) + p.q_in * c.nt;
  return p;
}

// One group of up to 32 samples, after the gather of a pass: the lane's
// fields go to V (gather-only) or to its staging row and through phase B.
template <typename T, int NU>
__device__ __forceinline__ void lane_store(const T (&acc)[NU][lane_unit<T>()], int ua, int nu,
                                           int f_first, int f_last, T* dst, int64_t stride) {
  constexpr int U = lane_unit<T>();
#pragma unroll
  for (int q = 0; q < NU; ++q)
#pragma unroll
    for (int c = 0; c < U; ++c) {
      const int f = U * (ua + q) + c;
      if (q < nu && f >= f_first && f < f_last) dst[int64_t(f - f_first) * stride] = acc[q][c];
    }
}

struct LaneArgs {
  int b, order, rec, F2, pass_f, n_rhs_real, n_probes, cplx, n_rhs_out, nacc, nbw, bstride;
  int wm0, wm1, pitch, lo_slack;  // staged windows only
};

constexpr int kLaneWarps = 8;  // warps per block (upper bound)

// ---- bin windows staged in shared memory (2-D) ------------------------------
// One block takes spreading sub-problems (samples of one bin) in turn: the
// bin's window of the field grid, [wm0][wm1][rec], comes in by bulk copies
// that complete on an mbarrier (bounded wait: if it gives up, the block raises
// the timeout bit of the error word, waits once more, bounded, for its copies
// and exits), then each warp takes groups of 32 samples.
template <typename T, int W, int NU>
__global__ void __launch_bounds__(kLaneWarps * 32)
interp_lane_kernel(GeoDev g, MonoTab mono, LaneArgs a, PhiTab<T> tab, const BwDev* __restrict__ bwt, int64_t n,
                   const T* __restrict__ xs, const T* __restrict__ str,
                   const uint32_t* __restrict__ perm, const T* __restrict__ fld,
                   T* __restrict__ mhat_at_x, double* __restrict__ part,
                   const uint32_t* __restrict__ sub_bin, const uint32_t* __restrict__ sub_first,
                   const uint32_t* __restrict__ bin_start, const uint32_t* __restrict__ sub_total,
                   T* __restrict__ vout) {
  constexpr int U = lane_unit<T>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t mbar;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarps = int(blockDim.x >> 5);
  const size_t win_bytes = (size_t(a.wm0) * a.pitch * sizeof(T) + 127) / 128 * 128;
  T* win = reinterpret_cast<T*>(smem_raw);
  double* red_all = reinterpret_cast<double*>(smem_raw + win_bytes);
  double* red = red_all + warp * a.nacc;
  T* my = reinterpret_cast<T*>(red_all + nwarps * a.nacc) + (warp * 32 + lane) * a.bstride;
  for (int k = lane; k < a.nacc; k += 32) red[k] = 0.0;
  if (threadIdx.x == 0) {
    mbar_init(&mbar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  const BwDev& B = bwt[a.b];
  const int nf[3] = {int(B.nf[0]), int(B.nf[1]), 1};
  const T ih0 = T(B.inv_h[0]), ih1 = T(B.inv_h[1]);
  const double r0 = double(B.nf[0]) / double(g.nf[0]);
  const double r1 = double(B.nf[1]) / double(g.nf[1]);
  const T beta = T(g.beta), halfw = T(0.5) * T(W);
  const GroupCtx c{mono.n, mono.nt, mono.nt, a.n_rhs_real + a.n_probes, a.n_rhs_real, a.n_probes,
                   a.cplx, a.n_rhs_out, a.nacc, a.order, a.b};
  T tsc[kMaxP];
#pragma unroll
  for (int k = 0; k < kMaxP; ++k) tsc[k] = (k < c.p) ? T(1.0 / tscale(mono, k, B.sigma)) : T(0);
  const T k0t = T(B.k0);
  const double isg[3] = {B.isigma[0], B.isigma[1], B.isigma[2]};
  LeadAxes<T, 2, W> lead{reinterpret_cast<T*>(red_all + nwarps * a.nacc) +
                             nwarps * 32 * a.bstride + warp * (lane_park_bytes<T, 2, W>() / sizeof(T)),
                         lane, g.skind, beta, {}};
  uint32_t parity = 0;
  const uint32_t nsub = *sub_total;
  bool failed = false;
  for (uint32_t k = blockIdx.x; k < nsub; k += gridDim.x) {
    const uint32_t bin = sub_bin[k];
    const uint32_t first = sub_first[k];
    const uint32_t last = min(first + g.sub_max, bin_start[bin + 1]);
    const int o0 = int(floor(double(int64_t(bin) / g.nbins[1] * g.tile[0]) * r0)) - g.pad - a.lo_slack;
    const int o1 = int(floor(double(int64_t(bin) % g.nbins[1] * g.tile[1]) * r1)) - g.pad - a.lo_slack;
    if (threadIdx.x == 0)
      issue_window_copies<T, 2>(fld, a.rec, nf[0], nf[1], o0, o1, a.wm0, a.wm1, a.pitch, win, &mbar);
    bool ok = false;
    for (uint32_t it = 0; it < g.wait_limit && !ok; ++it) ok = mbar_try_wait(&mbar, parity);
    if (__syncthreads_or(!ok)) {
      if (threadIdx.x == 0) atomicOr(g.errw, kErrTimeout);
      bool late = false;
      for (uint32_t it = 0; it < kMaxSpin && !late; ++it) late = mbar_try_wait(&mbar, parity);
      failed = true;
      break;
    }
    parity ^= 1u;
    const int ngr = int((last - first + 31) / 32);
    for (int gi = warp; gi < ngr; gi += nwarps) {
      const int64_t s = int64_t(first) + int64_t(gi) * 32 + lane;
      const bool valid = s < int64_t(last);
      const int64_t sl = valid ? s : int64_t(last) - 1;
      T off[2];
      const int i[2] = {lane_window<T>(xs[sl], ih0, halfw, off[0]),
                        lane_window<T>(xs[n + sl], ih1, halfw, off[1])};
      const int l0 = i[0] - o0, l1 = i[1] - o1;
      bool inside = l0 >= 0 && l0 + W <= a.wm0 && l1 >= 0 && l1 + W <= a.wm1;
      if constexpr (kChecked)
        if (inside) inside = in_range(g.errw, kSiteInterpWindow,
                                      int64_t(l0 + W - 1) * a.pitch + int64_t(l1 + W) * a.rec - 1,
                                      int64_t(a.wm0) * a.pitch);
      T pl[W];
      lead.set(tab, off);
      phi_row<W>(tab, g.skind, beta, off[1], pl);
      const uint32_t orig = !vout && valid ? perm[s] : 0u;
      T af[kMaxP] = {T(0), T(0), T(0), T(0)};
      int q_done = 0, f_first = 0;
      for (int pass = 0; f_first < a.F2; ++pass) {
        const LanePass ps = lane_pass(c, vout != nullptr, pass, f_first, q_done, a.pass_f, a.F2);
        const int ua = f_first / U, nu = (ps.f_last + U - 1) / U - ua;
        T acc[NU][U];
#pragma unroll
        for (int q = 0; q < NU; ++q)
#pragma unroll
          for (int cc = 0; cc < U; ++cc) acc[q][cc] = T(0);
        if (inside) {
          const T* base = win + size_t(l0) * a.pitch + l1 * a.rec + U * ua;
#pragma unroll 1
          for (int t0 = 0; t0 < W; ++t0)
            lane_row<T, W, NU, false>(base + t0 * a.pitch, [&](int t) { return t * a.rec; }, nu,
                                      lead.at(0, t0), pl, acc);
        } else if (valid) {
          lane_cells_global<T, 2, W, NU>(g, fld, a.rec, ua, nu, i, nf, lead, pl, acc);
        }
        if (vout) {
          if (valid)
            lane_store<T, NU>(acc, ua, nu, f_first, ps.f_last, vout + int64_t(f_first) * n + s, n);
        } else {
          lane_store<T, NU>(acc, ua, nu, f_first, ps.f_last, my, 1);
          finish_pass<T, 2>(c, mono, B, my, pass, q_done, ps.q_in, lane, valid, n, str + n + sl, n,
                            orig, mhat_at_x, tsc, af, red, k0t, isg);
        }
        q_done += ps.q_in;
        f_first = ps.f_last;
      }
    }
    __syncthreads();  // every read of this window is done before the next copies
  }
  if (failed) return;
  __syncthreads();
  for (int k = threadIdx.x; k < a.nacc; k += blockDim.x) {
    double t = 0.0;
    for (int wv = 0; wv < nwarps; ++wv) t += red_get<T>(red_all, wv * a.nacc + k);
    part[(int64_t(blockIdx.x) * a.nbw + a.b) * a.nacc + k] = t;
  }
}

// ---- straight from the field grid ------------------------------------------
template <typename T, int D, int W, int NU>
__global__ void __launch_bounds__(kLaneWarps * 32)
interp_global_kernel(GeoDev g, MonoTab mono, LaneArgs a, PhiTab<T> tab, const BwDev* __restrict__ bwt, int64_t n,
                     const T* __restrict__ xs, const T* __restrict__ str,
                     const uint32_t* __restrict__ perm, const T* __restrict__ fld,
                     T* __restrict__ mhat_at_x, double* __restrict__ part, T* __restrict__ vout) {
  constexpr int U = lane_unit<T>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarps = int(blockDim.x >> 5);
  double* red_all = reinterpret_cast<double*>(smem_raw);
  double* red = red_all + warp * a.nacc;
  T* my = reinterpret_cast<T*>(red_all + nwarps * a.nacc) + (warp * 32 + lane) * a.bstride;
  for (int k = lane; k < a.nacc; k += 32) red[k] = 0.0;
  __syncwarp();
  const BwDev& B = bwt[a.b];
  const int nf[3] = {int(B.nf[0]), int(B.nf[1]), int(B.nf[2])};
  T ih[D];
#pragma unroll
  for (int j = 0; j < D; ++j) ih[j] = T(B.inv_h[j]);
  const T beta = T(g.beta), halfw = T(0.5) * T(W);
  const GroupCtx c{mono.n, mono.nt, mono.nt, a.n_rhs_real + a.n_probes, a.n_rhs_real, a.n_probes,
                   a.cplx, a.n_rhs_out, a.nacc, a.order, a.b};
  T tsc[kMaxP];
#pragma unroll
  for (int k = 0; k < kMaxP; ++k) tsc[k] = (k < c.p) ? T(1.0 / tscale(mono, k, B.sigma)) : T(0);
  const T k0t = T(B.k0);
  const double isg[3] = {B.isigma[0], B.isigma[1], B.isigma[2]};
  LeadAxes<T, D, W> lead{reinterpret_cast<T*>(red_all + nwarps * a.nacc) +
                             nwarps * 32 * a.bstride + warp * (lane_park_bytes<T, D, W>() / sizeof(T)),
                         lane, g.skind, beta, {}};
  // neighbouring groups go to the warps of one block: they share cells in L1
  const int64_t ngroups = (n + 31) / 32;
  for (int64_t grp = int64_t(blockIdx.x) * nwarps + warp; grp < ngroups;
       grp += int64_t(gridDim.x) * nwarps) {
    const int64_t s = grp * 32 + lane;
    const bool valid = s < n;
    const int64_t sl = valid ? s : n - 1;
    T off[D];
    int i[D];
#pragma unroll
    for (int j = 0; j < D; ++j) i[j] = lane_window<T>(xs[int64_t(j) * n + sl], ih[j], halfw, off[j]);
    T pl[W];
    lead.set(tab, off);
    phi_row<W>(tab, g.skind, beta, off[D - 1], pl);
    const uint32_t orig = !vout && valid ? perm[s] : 0u;
    T af[kMaxP] = {T(0), T(0), T(0), T(0)};
    int q_done = 0, f_first = 0;
    for (int pass = 0; f_first < a.F2; ++pass) {
      const LanePass ps = lane_pass(c, vout != nullptr, pass, f_first, q_done, a.pass_f, a.F2);
      const int ua = f_first / U, nu = (ps.f_last + U - 1) / U - ua;
      T acc[NU][U];
#pragma unroll
      for (int q = 0; q < NU; ++q)
#pragma unroll
        for (int cc = 0; cc < U; ++cc) acc[q][cc] = T(0);
      lane_cells_global<T, D, W, NU>(g, fld, a.rec, ua, nu, i, nf, lead, pl, acc);
      if (vout) {
        if (valid)
          lane_store<T, NU>(acc, ua, nu, f_first, ps.f_last, vout + int64_t(f_first) * n + s, n);
      } else {
        lane_store<T, NU>(acc, ua, nu, f_first, ps.f_last, my, 1);
        finish_pass<T, D>(c, mono, B, my, pass, q_done, ps.q_in, lane, valid, n, str + n + sl, n,
                          orig, mhat_at_x, tsc, af, red, k0t, isg);
      }
      q_done += ps.q_in;
      f_first = ps.f_last;
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < a.nacc; k += blockDim.x) {
    double t = 0.0;
    for (int wv = 0; wv < nwarps; ++wv) t += red_get<T>(red_all, wv * a.nacc + k);
    part[(int64_t(blockIdx.x) * a.nbw + a.b) * a.nacc + k] = t;
  }
}

// ---- launches -----------------------------------------------------------------
template <typename T>
struct LaneLaunch {
  fkreg_plan_s* P;
  LaneArgs a;
  T* mhat_at_x;
  T* vout;
  cudaStream_t st;
  PhiTab<T> tab;
};

// shared memory of one warp, and warps per block that fit `budget` bytes,
// `fixed` of them taken
template <typename T, int D, int W>
size_t lane_warp_bytes(const LaneArgs& a) {
  return sizeof(double) * a.nacc + sizeof(T) * 32 * a.bstride + lane_park_bytes<T, D, W>();
}
template <typename T, int D, int W>
int lane_warps(const LaneArgs& a, size_t fixed, size_t budget) {
  const size_t per = lane_warp_bytes<T, D, W>(a);
  if (fixed >= budget) return 0;
  return int(std::min<size_t>(kLaneWarps, (budget - fixed) / per));
}

template <typename T, int W, int NU>
cudaError_t launch_lane_staged(const LaneLaunch<T>& L, bool* launched) {
  fkreg_plan_s* P = L.P;
  LaneArgs a = L.a;
  const BwDev& B = P->bw[a.b];
  a.wm0 = tma_window(P->geo, B, 0);
  a.wm1 = tma_window(P->geo, B, 1);
  if (a.wm0 > B.nf[0] || a.wm1 > B.nf[1]) return cudaSuccess;
  a.pitch = a.wm1 * a.rec + lane_unit<T>();  // rows one 16-byte unit apart in bank space
  a.lo_slack = std::max(tma_slack(P->geo, B, 0), tma_slack(P->geo, B, 1));
  const size_t win = (size_t(a.wm0) * a.pitch * sizeof(T) + 127) / 128 * 128;
  const int nw = lane_warps<T, 2, W>(a, win, 220 * 1024);
  if (nw < 4) return cudaSuccess;
  const size_t smem = win + lane_warp_bytes<T, 2, W>(a) * nw;
  auto kern = interp_lane_kernel<T, W, NU>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  if (e != cudaSuccess) return e;
  *launched = true;
  kern<<<unsigned(P->nblk_interp), nw * 32, smem, L.st>>>(
      P->geo, P->mono, a, L.tab, wsp<BwDev>(P, P->r_bw), P->n, wsp<T>(P, P->r_xs), wsp<T>(P, P->r_str),
      perm_ptr(P), wsp<T>(P, P->r_t2field), L.mhat_at_x, wsp<double>(P, P->r_part),
      wsp<uint32_t>(P, P->r_subbin), wsp<uint32_t>(P, P->r_subfirst),
      wsp<uint32_t>(P, P->r_binstart), wsp<uint32_t>(P, P->r_substart) + P->nbins_total, L.vout);
  P->launches += 1;
  return cudaGetLastError();
}

template <typename T, int D, int W, int NU>
cudaError_t launch_lane_global(const LaneLaunch<T>& L) {
  fkreg_plan_s* P = L.P;
  const int64_t ngroups = (P->n + 31) / 32;
  // small problems: one or two groups per block, so that every SM has one
  int nw = lane_warps<T, D, W>(L.a, 0, 100 * 1024);
  nw = int(std::max<int64_t>(1, std::min<int64_t>(nw, ngroups / P->sm_count)));
  const size_t smem = lane_warp_bytes<T, D, W>(L.a) * nw;
  auto kern = interp_global_kernel<T, D, W, NU>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  if (e != cudaSuccess) return e;
  kern<<<unsigned(P->nblk_interp), nw * 32, smem, L.st>>>(
      P->geo, P->mono, L.a, L.tab, wsp<BwDev>(P, P->r_bw), P->n, wsp<T>(P, P->r_xs), wsp<T>(P, P->r_str),
      perm_ptr(P), wsp<T>(P, P->r_t2field), L.mhat_at_x, wsp<double>(P, P->r_part), L.vout);
  P->launches += 1;
  return cudaGetLastError();
}

// Every field in one pass where they fit the largest instantiated number of
// units, else passes of 16 units.
template <typename T, int D, int W>
cudaError_t lane_dispatch(LaneLaunch<T> L) {
  constexpr int U = lane_unit<T>();
  const int F2 = L.a.F2;
  const int units = (F2 + U - 1) / U;
  L.a.pass_f = units <= 16 ? F2 : 16 * U - U;  // any such run of fields spans at most 16 units
  L.a.bstride = L.a.pass_f | 1;
#define FK_STAGED(NU)                                             \
  {                                                               \
    bool used = false;                                            \
    cudaError_t e = launch_lane_staged<T, W, NU>(L, &used);       \
    if (used || e != cudaSuccess) return e;                       \
  }
#define FK_LANE(NU)                              \
  if (units <= NU || NU == 16) {                 \
    if constexpr (D == 2) FK_STAGED(NU)          \
    return launch_lane_global<T, D, W, NU>(L);   \
  }
  if constexpr (D == 3) {
    FK_LANE(4)
    FK_LANE(10)
  } else if constexpr (sizeof(T) == 4) {
    FK_LANE(2)
    FK_LANE(6)
  } else {
    FK_LANE(1)
    FK_LANE(3)
    FK_LANE(5)
    FK_LANE(11)
  }
  FK_LANE(16)
#undef FK_LANE
#undef FK_STAGED
  return cudaErrorInvalidValue;
}

}  // namespace

}  // namespace fk
