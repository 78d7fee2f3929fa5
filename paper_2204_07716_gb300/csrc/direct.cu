// Direct moment sums: the sums of eq. 9 taken exactly over the samples inside
// each target's support, at the samples and at the grid points.  Serves the
// compact regression kernels (Table 1: uniform, Epanechnikov, triangle,
// biweight, triweight), whose Fourier transforms decay only algebraically, so
// that no tolerance can control a NUFFT's truncation, and the Gaussian cut at a
// Mahalanobis radius.  The samples inside a support (an ellipsoid
// |H^(-1/2) z| <= 1) are found through the bins of the sort.  The grid solve
// (solve.cu) and phase B of the at-sample pass follow as for the NUFFT path.
//
// A block takes 32 targets that lie close together (consecutive sorted
// samples, or a patch of the grid), one per lane, and its four warps share the
// candidates: the block lists the bin rows within reach of the targets' box,
// each warp takes every fourth run of 32 samples, keeps those within reach of
// the box, and when 32 are queued stages their strengths and walks them with
// broadcast loads, every lane adding each to its own fields in registers.  The
// warps' fields are added at the end.  (Before, a warp held 32 samples and tested
// every sample of the rows it staged.)  Grids too coarse for patches have a warp
// to each point (ds_patches).  Four warps to 32 targets keep
// the chains short: with one warp to 32 targets and 128 to a block the same
// instructions took four times as long, the schedulers idle nine cycles in ten
// beside the blocks of dense regions.  The grid pass sums in runs of 32
// candidates that are then added to totals, so rounding grows with the root
// of some tens, not of thousands; at the samples a warp's quarter of the
// candidates is one chain.  A form on the tensor cores (split-TF32, 32
// targets x 8 candidates a step) was tried and left out: no faster, and the
// truncating accumulators tripled the error against 64 bits.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "device_common.cuh"
#include "interp_common.cuh"
#include "internal.h"

namespace fk {

namespace {

constexpr int kDirectMaxFields = 64;
constexpr int kDsWarps = 4;              // warps per block, all on the same 32 targets
constexpr int kDsThreads = kDsWarps * 32;
constexpr int kDsRows = kDsThreads;      // bin rows listed at a time

// Record stride of a candidate's strengths, an odd number of 4-element chunks:
// the staging stores of eight candidates x four columns hit distinct banks.
template <int QC>
__host__ __device__ constexpr int ds_stride() { return 4 * (QC | 1); }

// Largest number of strength chunks (of four) that keeps F2 <= 64.
template <int D, int ORD>
__host__ __device__ constexpr int ds_max_chunks() {
  return ((kDirectMaxFields - mono_count(D, 2 * ORD)) / mono_count(D, ORD) + 3) / 4;
}

// Targets of a block of the grid pass: a patch of 4 x 8 (2-D) or 2 x 4 x 4 (3-D)
// points.
template <int D>
__device__ __forceinline__ bool ds_grid_point(const GeoDev& g, int64_t task, int lane,
                                              int64_t (&m)[3]) {
  m[0] = m[1] = m[2] = 0;
  if constexpr (D == 2) {
    const int64_t nb1 = (g.M[1] + 7) / 8;
    m[0] = task / nb1 * 4 + (lane >> 3);
    m[1] = task % nb1 * 8 + (lane & 7);
  } else {
    const int64_t nb1 = (g.M[1] + 3) / 4, nb2 = (g.M[2] + 3) / 4;
    m[2] = task % nb2 * 4 + (lane & 3);
    m[1] = task / nb2 % nb1 * 4 + ((lane >> 2) & 3);
    m[0] = task / nb2 / nb1 * 2 + (lane >> 4);
  }
  bool ok = true;
#pragma unroll
  for (int j = 0; j < D; ++j) {
    ok = ok && m[j] < g.M[j];
    m[j] = min(m[j], g.M[j] - 1);
  }
  return ok;
}

inline int64_t ds_grid_tasks(const GeoDev& g, int d) {
  if (d == 2) return (g.M[0] + 3) / 4 * ((g.M[1] + 7) / 8);
  return (g.M[0] + 1) / 2 * ((g.M[1] + 3) / 4) * ((g.M[2] + 3) / 4);
}

// Metric distance z^T H^-1 z; with a diagonal H the zero terms are left out.
template <typename T, int D>
__device__ __forceinline__ T ds_dist(const T (&hi)[D][D], bool diag, const T (&z)[D]) {
  T u2 = T(0);
  if (diag) {
#pragma unroll
    for (int a = 0; a < D; ++a) u2 += z[a] * (hi[a][a] * z[a]);
  } else {
#pragma unroll
    for (int a = 0; a < D; ++a) {
      T ra = T(0);
#pragma unroll
      for (int c = 0; c < D; ++c) ra += hi[a][c] * z[c];
      u2 += z[a] * ra;
    }
  }
  return u2;
}

// Kernel value at metric distance u2 without divergence (kern is the same for
// every lane): 0 outside the unit ball.  rc = -R^2 / 2, in FP32 times log2 e for
// the hardware's base-2 exponential.
template <typename T>
__device__ __forceinline__ T ds_kernel(int kern, T u2, T rc) {
  T w;
  if (kern == FKREG_KERNEL_GAUSSIAN_DIRECT) {
    if constexpr (sizeof(T) == 4)
      w = exp2f(rc * u2);
    else
      w = exp(rc * u2);
  } else {
    const T e = kern == FKREG_KERNEL_TRIANGLE ? T(1) - sqrt(u2) : T(1) - u2;
    w = kern == FKREG_KERNEL_UNIFORM ? T(1) : e;
    if (kern >= FKREG_KERNEL_BIWEIGHT) w *= e;
    if (kern >= FKREG_KERNEL_TRIWEIGHT) w *= e;
  }
  return u2 <= T(1) ? w : T(0);
}
static_assert(FKREG_KERNEL_UNIFORM < FKREG_KERNEL_BIWEIGHT &&
                  FKREG_KERNEL_EPANECHNIKOV < FKREG_KERNEL_BIWEIGHT &&
                  FKREG_KERNEL_TRIANGLE < FKREG_KERNEL_BIWEIGHT &&
                  FKREG_KERNEL_BIWEIGHT < FKREG_KERNEL_TRIWEIGHT,
              "the powers of ds_kernel follow the order of the kernels' codes");

template <typename T>
struct DsCoord;  // coordinates of a staged candidate, one broadcast load
template <>
struct DsCoord<float> {
  using type = float4;
};
template <>
struct DsCoord<double> {
  using type = double4;
};
struct DsArgs {
  int b, order, n_rhs_real, n_probes, cplx, n_rhs_out, nacc, nbw, bstride, str_first, nstr;
  int fields;          // fields per target (ns + nstr nt)
  int str_pass;        // the strengths' pass (see kStrFlag)
  int64_t ntask;       // groups of 32 targets
  int64_t Mtot;        // grid: points
  int slice;           // grid: field slice of the first bandwidth
};

// A target's fields.  add: one candidate of the walk, w its kernel value at this lane's target (0
// outside the support), z its offset, cv its strengths (4 QC, zero-padded).
template <typename T, int D, int ORD, int QC>
struct DsFields {
  static constexpr int NS = mono_count(D, 2 * ORD), NT = mono_count(D, ORD);
  T sf[NS];
  T tf[NT][4 * QC];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int f = 0; f < NS; ++f) sf[f] = T(0);
#pragma unroll
    for (int k = 0; k < NT; ++k)
#pragma unroll
      for (int r = 0; r < 4 * QC; ++r) tf[k][r] = T(0);
  }
  __device__ __forceinline__ void add(const DsFields& o) {
#pragma unroll
    for (int f = 0; f < NS; ++f) sf[f] += o.sf[f];
#pragma unroll
    for (int k = 0; k < NT; ++k)
#pragma unroll
      for (int r = 0; r < 4 * QC; ++r) tf[k][r] += o.tf[k][r];
  }
  __device__ __forceinline__ void add(T w, const T* z, const T* __restrict__ cv, int nstr) {
    T mo[NS];
    mono_build<T, D, 2 * ORD>(mo, z);
#pragma unroll
    for (int f = 0; f < NS; ++f) sf[f] += w * mo[f];
#pragma unroll
    for (int q = 0; q < QC; ++q)
      if (4 * q < nstr) {
        if constexpr (sizeof(T) == 4) {
          const float4 c = reinterpret_cast<const float4*>(cv)[q];
          float2 c01 = make_float2(c.x, c.y), c23 = make_float2(c.z, c.w);
          if (NT > 1) {
            const float2 w2 = make_float2(w, w);
            c01 = __fmul2_rn(w2, c01);
            c23 = __fmul2_rn(w2, c23);
          }
#pragma unroll
          for (int k = 0; k < NT; ++k) {
            const float m = NT > 1 ? mo[k] : w;
            const float2 m2 = make_float2(m, m);
            const float2 a = __ffma2_rn(c01, m2, make_float2(tf[k][4 * q], tf[k][4 * q + 1]));
            const float2 b = __ffma2_rn(c23, m2, make_float2(tf[k][4 * q + 2], tf[k][4 * q + 3]));
            tf[k][4 * q] = a.x;
            tf[k][4 * q + 1] = a.y;
            tf[k][4 * q + 2] = b.x;
            tf[k][4 * q + 3] = b.y;
          }
        } else {
          const double2 c0 = reinterpret_cast<const double2*>(cv)[2 * q];
          const double2 c1 = reinterpret_cast<const double2*>(cv)[2 * q + 1];
#pragma unroll
          for (int k = 0; k < NT; ++k) {
            const double wm = w * mo[k];
            tf[k][4 * q] += wm * c0.x;
            tf[k][4 * q + 1] += wm * c0.y;
            tf[k][4 * q + 2] += wm * c1.x;
            tf[k][4 * q + 3] += wm * c1.y;
          }
        }
      }
  }
};

// GRID: blockIdx.y is the bandwidth (a.b + y), fields go to
// field[y][fields][Mtot]; else the at-sample pass of bandwidth a.b with phase B.
template <typename T, int D, int ORD, int QC, bool GRID>
__global__ void __launch_bounds__(kDsThreads)
direct_sums_kernel(GeoDev g, MonoTab mono, DsArgs a, const BwDev* __restrict__ bwt, int64_t n,
                   const T* __restrict__ xs, const T* __restrict__ str,
                   const uint32_t* __restrict__ perm, const uint32_t* __restrict__ bin_start,
                   T* __restrict__ field, T* __restrict__ mhat_at_x, double* __restrict__ gsum,
                   uint32_t* __restrict__ task_count) {
  constexpr int NS = mono_count(D, 2 * ORD), NT = mono_count(D, ORD), RS = ds_stride<QC>();
  using C4 = typename DsCoord<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint32_t s_rbeg[kDsRows], s_rpre[kDsRows + 1], s_wsum[kDsWarps];
  __shared__ __align__(16) T s_qx[kDsWarps][64][4];  // queued candidates: coordinates, index
  __shared__ uint32_t s_qi[kDsWarps][64];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // layout: strengths [warps][32][RS], the warps' fields [warps][32][bstride],
  // the group's reduction accumulators [nacc] (RS is a multiple of 4, the rows are 128)
  T* rec = reinterpret_cast<T*>(smem_raw) + warp * 32 * RS;
  T* rows_f = reinterpret_cast<T*>(smem_raw) + kDsThreads * RS;
  T* my = rows_f + tid * a.bstride;
  double* red = reinterpret_cast<double*>(rows_f + kDsThreads * a.bstride);
  for (int k = tid; k < a.nacc; k += kDsThreads) red[k] = 0.0;
  const int bw = a.b + (GRID ? int(blockIdx.y) : 0);
  const BwDev& B = bwt[bw];
  T hi[D][D];
#pragma unroll
  for (int i = 0; i < D; ++i)
#pragma unroll
    for (int j = 0; j < D; ++j) hi[i][j] = T(B.Hinv[i * 3 + j]);
  const T ks = T(B.kscale);
  const T rc = T((sizeof(T) == 4 ? -0.5 * 1.4426950408889634 : -0.5) * B.kr2);
  const int kern = g.kern;
  const int nstr = a.nstr;
  const int64_t nbins = g.nbins[0] * g.nbins[1] * g.nbins[2];
  // some strength of this pass is not finite: it must not reach targets that
  // hold its sample outside their support through a product with zero
  const bool nonfin = g.errw[kStrFlag] == a.str_pass;
  __shared__ uint32_t s_task, s_row;
  for (int64_t task = blockIdx.x; task < a.ntask;) {
    if (!GRID && tid == 0) s_row = uint32_t(task);
    // this lane's target, the same in all four warps
    T qv[D];
    bool valid;
    int64_t s = 0, mi[3] = {0, 0, 0};
    if constexpr (GRID) {
      valid = ds_grid_point<D>(g, task, lane, mi);
#pragma unroll
      for (int j = 0; j < D; ++j)
        qv[j] = T(double(mi[j]) * (g.hi[j] - g.lo[j]) / double(g.M[j] - 1));
    } else {
      s = task * 32 + lane;
      valid = s < n;
      s = valid ? s : n - 1;
#pragma unroll
      for (int j = 0; j < D; ++j) qv[j] = xs[int64_t(j) * n + s];
    }
    DirectRows<D> rows;
    T wmn[D], wmx[D];
#pragma unroll
    for (int j = 0; j < D; ++j) {
      T mn = qv[j], mx = qv[j];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      }
      wmn[j] = mn;
      wmx[j] = mx;
      rows.mn[j] = float(mn);
      rows.mx[j] = float(mx);
    }
    rows.box(g, B);
    const bool diag = rows.diag;
    DsFields<T, D, ORD, QC> tot;
    tot.zero();
    // cnt queued candidates: strengths into shared memory (lane = candidate
    // mod 8 x column mod 4: coalesced runs, distinct banks), then the walk
    auto flush = [&](int cnt) {
      const int c8 = lane & 7, c4 = lane >> 3;
      T v[4][QC];
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const int c = 8 * h + c8;
        const int64_t i = c < cnt ? s_qi[warp][c] : 0;
#pragma unroll
        for (int k = 0; k < QC; ++k)
          v[h][k] = c < cnt && 4 * k + c4 < nstr ? str[int64_t(a.str_first + 4 * k + c4) * n + i] : T(0);
      }
#pragma unroll
      for (int h = 0; h < 4; ++h)
#pragma unroll
        for (int k = 0; k < QC; ++k) rec[(8 * h + c8) * RS + 4 * k + c4] = v[h][k];
      __syncwarp();
      // the grid pass sums in runs (see the top); at the samples the registers
      // that takes are worth more as warps in flight
      DsFields<T, D, ORD, QC> run;
      DsFields<T, D, ORD, QC>& acc = GRID ? run : tot;
      if (GRID) run.zero();
      auto weight = [&](int e, T (&z)[D]) {
        const C4 x = *reinterpret_cast<const C4*>(s_qx[warp][e]);
        const T xc[3] = {x.x, x.y, x.z};
#pragma unroll
        for (int j = 0; j < D; ++j) z[j] = xc[j] - qv[j];
        return ds_dist<T, D>(hi, diag, z);
      };
      if (sizeof(T) == 8 && !nonfin) {
        // The FP64 pipe sets the pace (a warp instruction every 16 clocks), so a
        // candidate outside every lane's support is dropped after its test: a
        // group that spans two rows of bins has most of its candidates between its
        // ends.  20,000 samples, 2-D local linear: 2370 us with every candidate
        // added, 1367 with the test (3-D 6870 -> 3284).
#pragma unroll 1
        for (int e = 0; e < cnt; ++e) {
          T z[D];
          const T u2 = weight(e, z);
          if (__any_sync(0xffffffffu, u2 <= T(1)))
            acc.add(ks * ds_kernel<T>(kern, u2, rc), z, rec + e * RS, nstr);
        }
      } else if (!nonfin) {
        // no branch inside: candidates overlap
        int e = 0;
        for (; e + 4 <= cnt; e += 4) {
          T z[4][D], w[4];
#pragma unroll
          for (int u = 0; u < 4; ++u)
            w[u] = ks * ds_kernel<T>(kern, weight(e + u, z[u]), rc);
#pragma unroll
          for (int u = 0; u < 4; ++u) acc.add(w[u], z[u], rec + (e + u) * RS, nstr);
        }
        for (; e < cnt; ++e) {
          T z[D];
          const T w = ks * ds_kernel<T>(kern, weight(e, z), rc);
          acc.add(w, z, rec + e * RS, nstr);
        }
      } else {
#pragma unroll 1
        for (int e = 0; e < cnt; ++e) {
          T z[D];
          const T u2 = weight(e, z);
          if (u2 <= T(1)) acc.add(ks * ds_kernel<T>(kern, u2, rc), z, rec + e * RS, nstr);
        }
      }
      if (GRID) tot.add(run);
      __syncwarp();
    };
    int qn = 0;  // queued candidates of this warp
    const int nr1 = rows.rows1(), nrows = rows.rows0() * nr1;
    for (int row0 = 0; row0 < nrows; row0 += kDsRows) {
      // the sample ranges of up to kDsRows bin rows, and their running count
      uint32_t beg = 0, len = 0;
      if (row0 + tid < nrows) {
        int64_t first, last;
        if (rows.row(g, (row0 + tid) / nr1, (row0 + tid) % nr1, first, last) &&
            in_range(g.errw, kSiteDirectBins, first, last + 1) &&
            in_range(g.errw, kSiteDirectBins, last, nbins)) {
          beg = bin_start[first];
          len = bin_start[last + 1] - beg;
        }
      }
      uint32_t inc = len;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
      }
      if (lane == 31) s_wsum[warp] = inc;
      __syncthreads();
      uint32_t before = 0, total = 0;
#pragma unroll
      for (int w = 0; w < kDsWarps; ++w) {
        if (w < warp) before += s_wsum[w];
        total += s_wsum[w];
      }
      s_rbeg[tid] = beg;
      s_rpre[tid] = before + inc - len;
      if (tid == 0) s_rpre[kDsRows] = total;
      __syncthreads();
      for (uint32_t base = warp * 32; base < total; base += kDsThreads) {
        const uint32_t flat = base + lane;
        bool near = flat < total;
        int lo = 0, up = kDsRows;  // last row whose first flat index is <= flat
        while (up - lo > 1) {
          const int mid = (lo + up) >> 1;
          if (s_rpre[mid] <= flat) lo = mid;
          else up = mid;
        }
        const uint32_t i = near ? s_rbeg[lo] + (flat - s_rpre[lo]) : 0;
        T x[D];
        float d2 = 0.f;
#pragma unroll
        for (int j = 0; j < D; ++j) {
          x[j] = near ? xs[int64_t(j) * n + i] : T(0);
          const float dz = float(max(max(wmn[j] - x[j], x[j] - wmx[j]), T(0)));
          near = near && dz <= rows.sg[j] * 1.001f;
          d2 = fmaf(dz * rows.isg[j], dz * rows.isg[j], d2);
        }
        if (diag) near = near && d2 <= 1.001f;
        const unsigned mask = __ballot_sync(0xffffffffu, near);
        if (near) {
          const int slot = qn + __popc(mask & ((1u << lane) - 1u));
#pragma unroll
          for (int j = 0; j < D; ++j) s_qx[warp][slot][j] = x[j];
          s_qi[warp][slot] = i;
        }
        qn += __popc(mask);
        if (qn >= 32) {
          __syncwarp();
          flush(32);
          qn -= 32;
          T mx[D];
          uint32_t mq = 0;
          if (lane < qn) {  // the overflow moves to the front of the queue
#pragma unroll
            for (int j = 0; j < D; ++j) mx[j] = s_qx[warp][32 + lane][j];
            mq = s_qi[warp][32 + lane];
          }
          if (lane < qn) {
#pragma unroll
            for (int j = 0; j < D; ++j) s_qx[warp][lane][j] = mx[j];
            s_qi[warp][lane] = mq;
          }
          __syncwarp();
        }
      }
      __syncthreads();  // every read of these ranges is done
    }
    __syncwarp();
    if (qn > 0) flush(qn);
#pragma unroll
    for (int f = 0; f < NS; ++f) my[f] = tot.sf[f];
#pragma unroll
    for (int r = 0; r < 4 * QC; ++r)
      if (r < nstr)
#pragma unroll
        for (int k = 0; k < NT; ++k) my[NS + r * NT + k] = tot.tf[k][r];
    __syncthreads();
    // the four warps' fields together: field f by warp f mod 4
    int64_t idx = mi[0];
#pragma unroll
    for (int j = 1; j < D; ++j) idx = idx * g.M[j] + mi[j];
    for (int f = warp; f < a.fields; f += kDsWarps) {
      T v = rows_f[lane * a.bstride + f];
#pragma unroll
      for (int w = 1; w < kDsWarps; ++w) v += rows_f[(w * 32 + lane) * a.bstride + f];
      if constexpr (GRID) {
        if (valid) field[(int64_t(a.slice + blockIdx.y) * a.fields + f) * a.Mtot + idx] = v;
      } else {
        rows_f[lane * a.bstride + f] = v;
      }
    }
    __syncthreads();
    if constexpr (!GRID) {
      if (warp == 0) {
        const GroupCtx c{mono.n, mono.nt, mono.nt, a.n_rhs_real + a.n_probes, a.n_rhs_real,
                         a.n_probes, a.cplx, a.n_rhs_out, a.nacc, a.order, a.b};
        T tsc[kMaxP], af[kMaxP] = {T(0), T(0), T(0), T(0)};
#pragma unroll
        for (int k = 0; k < kMaxP; ++k)
          tsc[k] = (k < c.p) ? T(1.0 / tscale(mono, k, B.sigma)) : T(0);
        const double isg[3] = {B.isigma[0], B.isigma[1], B.isigma[2]};
        finish_pass<T, D, ORD>(c, mono, B, my, 0, 0, c.nq, lane, valid, n, str + n + s, n,
                               valid ? perm[s] : 0u, mhat_at_x, tsc, af, red, T(B.k0), isg);
      }
      // the groups of a dense region cost tens of times those of a sparse one: the
      // resident blocks take them from a counter (dealt out in turn, half the
      // SMs idled through the second half of the pass).  Which block takes a group
      // differs from run to run, so each group leaves its own row of sums
      // (ds_rows_kernel adds them in a fixed order)
      if (tid == 0) s_task = gridDim.x + atomicAdd(task_count, 1u);
      const uint32_t row = s_row;
      __syncthreads();  // also: the rows are rewritten by the next task
      for (int k = tid; k < a.nacc; k += kDsThreads) {
        gsum[int64_t(row) * a.nacc + k] = red_get<T>(red, k);
        red[k] = 0.0;
      }
      task = s_task;
    } else {
      break;  // one block per patch
    }
  }
}

// The rows of partial sums that the reduction reads, from the groups' sums: row r
// adds groups r, r + rows, ... in turn, whichever block took them, so the scalars of
// a call repeat bit for bit.
__global__ void ds_rows_kernel(const double* __restrict__ gsum, int64_t ntask, int nacc, int nbw,
                               int b, int64_t rows, double* __restrict__ part) {
  const int64_t id = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (id >= rows * nacc) return;
  const int64_t r = id / nacc;
  const int k = int(id - r * nacc);
  double t = 0.0;
  for (int64_t i = r; i < ntask; i += rows) t += gsum[i * nacc + k];
  part[(r * nbw + b) * nacc + k] = t;
}

template <typename T, int D, int ORD, int QC, bool GRID>
cudaError_t launch_ds(fkreg_plan_s* P, DsArgs a, int bw_count, void* mhat_at_x, cudaStream_t st) {
  a.bstride = a.fields | 1;
  a.str_pass = P->str_pass;
  const size_t smem = sizeof(T) * kDsThreads * (ds_stride<QC>() + a.bstride) + sizeof(double) * a.nacc;
  auto kern = direct_sums_kernel<T, D, ORD, QC, GRID>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  if (e != cudaSuccess) return e;
  uint32_t* task_count = wsp<uint32_t>(P, P->r_err) + kTaskWord;
  int64_t blocks = a.ntask;
  if (!GRID) {
    // one wave of resident blocks, each striding over the tasks
    int per_sm = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kDsThreads, smem)) !=
        cudaSuccess)
      return e;
    blocks = std::min<int64_t>(int64_t(std::max(per_sm, 1)) * P->sm_count,
                               std::min<int64_t>(P->nblk_interp, a.ntask));
    if ((e = cudaMemsetAsync(task_count, 0, sizeof(uint32_t), st)) != cudaSuccess) return e;
  }
  kern<<<dim3(unsigned(blocks), unsigned(bw_count)), kDsThreads, smem, st>>>(
      P->geo, P->mono, a, wsp<BwDev>(P, P->r_bw), P->n, wsp<T>(P, P->r_xs), wsp<T>(P, P->r_str),
      perm_ptr(P), wsp<uint32_t>(P, P->r_binstart), wsp<T>(P, P->r_gfield),
      static_cast<T*>(mhat_at_x), wsp<double>(P, P->r_gsum), task_count);
  P->launches += 1;
  if ((e = cudaGetLastError()) != cudaSuccess || GRID) return e;
  const int64_t cells = P->nblk_interp * a.nacc;
  ds_rows_kernel<<<unsigned((cells + 255) / 256), 256, 0, st>>>(
      wsp<double>(P, P->r_gsum), a.ntask, a.nacc, a.nbw, a.b, P->nblk_interp,
      wsp<double>(P, P->r_part));
  P->launches += 1;
  return cudaGetLastError();
}

// Chunks of four strengths, in the sizes that occur: one response, the default
// ten probes beside it, 32 probes, and as many as F2 <= 64 holds.  The largest
// Nadaraya-Watson size holds 64 sums a lane (255 registers) and takes twice the time
// of size 3 with five to twelve strengths: FP64 at 15,000 3-D samples 2905 us against
// 7950, FP32 on 28^3 points 265 us against 515.
template <typename T, int D, int ORD, bool GRID>
cudaError_t dispatch_ds(fkreg_plan_s* P, const DsArgs& a, int bw_count, void* mhat_at_x,
                        cudaStream_t st) {
  constexpr int QM = ds_max_chunks<D, ORD>();
  const int qc = (a.nstr + 3) / 4;
  if (qc <= 1) return launch_ds<T, D, ORD, 1, GRID>(P, a, bw_count, mhat_at_x, st);
  if constexpr (QM > (!GRID && sizeof(T) == 4 ? 3 : 9))
    if (qc <= 3) return launch_ds<T, D, ORD, 3, GRID>(P, a, bw_count, mhat_at_x, st);
  if constexpr (!GRID && QM > 9)
    if (qc <= 9) return launch_ds<T, D, ORD, 9, GRID>(P, a, bw_count, mhat_at_x, st);
  return launch_ds<T, D, ORD, QM, GRID>(P, a, bw_count, mhat_at_x, st);
}

template <typename T, bool GRID>
cudaError_t run_ds(fkreg_plan_s* P, const DsArgs& a, int bw_count, void* mhat_at_x,
                   cudaStream_t st) {
#define FK_DS(DD, OO)                                                        \
  if constexpr (!GRID || DD > 1) /* 1-D grids have a warp to each point */   \
    if (P->d == DD && P->order == OO)                                        \
      return dispatch_ds<T, DD, OO, GRID>(P, a, bw_count, mhat_at_x, st);
  FK_DS(1, 0) FK_DS(1, 1) FK_DS(1, 2) FK_DS(2, 0) FK_DS(2, 1) FK_DS(2, 2) FK_DS(3, 0) FK_DS(3, 1)
#undef FK_DS
  return cudaErrorInvalidValue;
}

}  // namespace

// Patches of 32 points, or a warp to each point (direct_points.cu)?  A patch walks
// every sample within reach of its box, so its work per point grows by `reach`, the
// box of support and patch against the support's; a warp per point adds only the
// samples inside, in 32 lanes, and pays a fixed part of some hundred samples.  A
// patch is also one block with a long chain: few of them leave SMs idle.  On a
// GB300, over 660 random calls (1-D to 3-D, orders 0 to 2, 1 to 12 responses, 3000 to
// 10^6 samples), us with patches and with points:
//   FP32 2-D: 338^2 points, reach 1.2, 400 samples inside 220 / 610; 181^2, 1.6, 2200:
//   397 / 473; 82 x 43, 2.8, 4700: 562 / 164; 16^2, 5.0, 530: 119 / 51;
//   FP32 3-D: 53^3, 2.1, 67: 312 / 2488; 13^3, 3.3, 8500: 1655 / 343;
//   FP64 2-D: 186^2, 2.5, 12: 190 / 524; 262^2, 3.4, 73: 1968 / 1417; 100^2, 3.5, 500:
//   2610 / 614; FP64 3-D: 38^3, 2.3, 24: 762 / 3271; 18^3, 5.0, 3200: 21678 / 2518;
//   1-D, where 32 points are a long box: 0.7 to 1.7 times in FP32 at reach below 2.1, 18
//   times at 117; 1.5 to 72 times in FP64.
// The rule loses 2 % on average against the better of the two, 1.6 times at most.
static bool ds_patches(const fkreg_plan_s* P, int b) {
  if (P->d == 1) return false;
  const GeoDev& g = P->geo;
  const BwDev& B = P->bw[b];
  const int64_t patch[3] = {P->d == 2 ? 4 : 2, P->d == 2 ? 8 : 4, 4};
  double reach = 1.0, inside = double(P->n) * (P->d == 2 ? M_PI : 4.0 / 3.0 * M_PI);
  for (int j = 0; j < P->d; ++j) {
    const double w = g.hi[j] - g.lo[j];
    reach *= 1.0 + w * double(std::min(patch[j], g.M[j]) - 1) / double(g.M[j] - 1) / (2.0 * B.sigma[j]);
    inside *= B.sigma[j] / w;
  }
  inside = std::min(inside, double(P->n));
  const double idle = std::max(1.0, 4.0 * P->sm_count / double(ds_grid_tasks(g, P->d)));
  return P->prec == FKREG_F32
             ? 0.35 * reach * inside * idle < inside + 400.0
             : reach * inside * idle < inside + 200.0;
}

cudaError_t run_direct_grid(fkreg_plan_s* P, int str_first, int nstr, int bw_first,
                            int bw_count, cudaStream_t st) {
  DsArgs a{};
  a.b = bw_first;
  a.order = P->order;
  a.str_first = str_first;
  a.nstr = nstr;
  a.fields = P->ns + nstr * P->nt;
  a.ntask = ds_grid_tasks(P->geo, P->d);
  a.Mtot = P->geo.M[0] * P->geo.M[1] * P->geo.M[2];
  if (a.fields > kDirectMaxFields) return cudaErrorInvalidValue;
  if (a.Mtot * bw_count == 0) return cudaSuccess;
  for (int i = 0; i < bw_count;) {  // runs of bandwidths that take the same kernel
    const bool patches = ds_patches(P, bw_first + i);
    int k = i + 1;
    while (k < bw_count && ds_patches(P, bw_first + k) == patches) ++k;
    a.b = bw_first + i;
    a.slice = i;
    const cudaError_t e =
        !patches ? run_direct_points(P, str_first, nstr, a.b, k - i, i, st)
                 : (P->prec == FKREG_F32 ? run_ds<float, true>(P, a, k - i, nullptr, st)
                                         : run_ds<double, true>(P, a, k - i, nullptr, st));
    if (e != cudaSuccess) return e;
    i = k;
  }
  return cudaSuccess;
}

cudaError_t run_direct_interp(fkreg_plan_s* P, int b, int n_rhs_str, int n_probes,
                              void* mhat_at_x, cudaStream_t st) {
  if (P->n == 0) return cudaSuccess;
  DsArgs a{};
  a.b = b;
  a.order = P->order;
  a.n_rhs_real = n_rhs_str;
  a.n_probes = n_probes;
  a.cplx = P->o.y_complex;
  a.n_rhs_out = P->nrhs;
  a.nacc = n_rhs_str + 2 * n_probes + 1;
  a.nbw = P->nbw;
  a.str_first = 1;
  a.nstr = n_rhs_str + n_probes;
  a.fields = P->ns + a.nstr * P->nt;
  a.ntask = (P->n + 31) / 32;
  if (a.fields > kDirectMaxFields || a.nacc > kMaxAcc) return cudaErrorInvalidValue;
  return P->prec == FKREG_F32 ? run_ds<float, false>(P, a, 1, mhat_at_x, st)
                              : run_ds<double, false>(P, a, 1, mhat_at_x, st);
}

}  // namespace fk
