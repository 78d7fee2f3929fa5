// Direct moment sums at the grid points, a warp to each point: the lanes stride over
// the candidates, the ones inside the support are queued and added 32 at a time, so
// that no lane works on a sample outside.  For 1-D grids and those whose points lie
// far apart for their supports (ds_patches in direct.cu, with both sides' times).
// Bound by the candidates' tests and the reduction of every field over the warp, some
// hundred samples' worth a point: 101 x 101 points, 1900 samples inside, FP64 1.4 ms.
#include <cuda_runtime.h>

#include "device_common.cuh"
#include "internal.h"

namespace fk {

namespace {

constexpr int kDirectMaxFields = 64;

// Radial profile k(|u|^2) of the regression kernels (unit ball;
// normalisation in BwDev::kscale): uniform, Epanechnikov, triangle,
// biweight, triweight, and the Gaussian cut at Mahalanobis radius R
// (u = z / R in the bandwidth's metric, k = exp(-R^2 |u|^2 / 2), r2 = R^2).
template <typename T>
__device__ __forceinline__ T compact_k(int kern, T u2, T r2) {
  if (!(u2 <= T(1))) return T(0);
  const T e = T(1) - u2;
  switch (kern) {
    case FKREG_KERNEL_UNIFORM: return T(1);
    case FKREG_KERNEL_EPANECHNIKOV: return e;
    case FKREG_KERNEL_TRIANGLE: return T(1) - sqrt(u2);
    case FKREG_KERNEL_BIWEIGHT: return e * e;
    case FKREG_KERNEL_GAUSSIAN_DIRECT: return exp(T(-0.5) * r2 * u2);
    default: return e * e * e;
  }
}

// Shared memory of one warp's candidate queue in direct_warp_sums: 64
// entries of (z[0..D), weight) in T, then 64 sample indices.
template <typename T, int D>
__host__ __device__ constexpr int direct_queue_bytes() {
  return 64 * (D + 1) * int(sizeof(T)) + 64 * 4;
}

// Warp-cooperative moment sums of one evaluation point q (coordinates
// relative to lo) over the binned samples inside its kernel support: the
// lanes stride over the sample ranges of the support's bins (bins adjacent
// along the last axis are one contiguous range of the sort) and test each
// candidate; the ones inside the support are compacted into a per-warp queue
// in shared memory (qmem, direct_queue_bytes), and each time 32 are queued
// every lane adds one of them to all fields in registers, so that the
// monomial and strength work runs on full warps.  The fields are reduced
// across the warp at the end: field f is returned to lane f mod 32 (out0 for
// f < 32, out1 above): [0, NS) the s-fields, NS + r NT + k the t-fields of
// strength str_first + r.  NS and NT are the monomial counts of degrees 2*ORD
// and ORD; FMAX >= NS + nstr NT bounds the fields.  Sums are in the plan
// precision T.
template <typename T, int D, int ORD, int FMAX>
__device__ __forceinline__ void direct_warp_sums(const GeoDev& g, const BwDev& B, int64_t n,
                                                 const T* __restrict__ xs,
                                                 const T* __restrict__ str, int str_first,
                                                 int nstr, const uint32_t* __restrict__ bin_start,
                                                 const double* q, int lane, unsigned char* qmem,
                                                 T& out0, T& out1) {
  constexpr int NS = mono_count(D, 2 * ORD), NT = mono_count(D, ORD);
  constexpr int QMAX = (FMAX - NS) / NT;
  static_assert(QMAX >= 1 && FMAX <= 64, "field bucket");
  T* qv = reinterpret_cast<T*>(qmem);                                   // [D + 1][64]
  uint32_t* qi = reinterpret_cast<uint32_t*>(qmem + 64 * (D + 1) * sizeof(T));  // [64]
  DirectRows<D> rows;
#pragma unroll
  for (int j = 0; j < D; ++j) rows.mn[j] = rows.mx[j] = float(q[j]);
  rows.box(g, B);
  T qt[D], hi[D][D];
#pragma unroll
  for (int a = 0; a < D; ++a) {
    qt[a] = T(q[a]);
#pragma unroll
    for (int c = 0; c < D; ++c) hi[a][c] = T(B.Hinv[a * 3 + c]);
  }
  const T ks = T(B.kscale), kr2 = T(B.kr2);
  const int kern = g.kern;
  T acc[FMAX];
#pragma unroll
  for (int f = 0; f < FMAX; ++f) acc[f] = T(0);
  // one queued candidate per lane (lane < cnt) into every field
  auto consume = [&](int cnt) {
    if (lane < cnt) {
      T z[D];
#pragma unroll
      for (int j = 0; j < D; ++j) z[j] = qv[j * 64 + lane];
      const T wgt = qv[D * 64 + lane];
      const int64_t i = qi[lane];
      T mo[NS];
      mono_build<T, D, 2 * ORD>(mo, z);
#pragma unroll
      for (int f = 0; f < NS; ++f) acc[f] += wgt * mo[f];
#pragma unroll
      for (int r = 0; r < QMAX; ++r)
        if (r < nstr) {
          const T cw = wgt * str[int64_t(str_first + r) * n + i];
#pragma unroll
          for (int k = 0; k < NT; ++k) acc[NS + r * NT + k] += cw * mo[k];
        }
    }
  };
  int qn = 0;  // queued candidates (warp-uniform)
  const unsigned below = (1u << lane) - 1u;
  const int o0 = rows.rows0(), o1 = rows.rows1();
  for (int r0 = 0; r0 < o0; ++r0)
    for (int r1 = 0; r1 < o1; ++r1) {
      int64_t first, last;  // bins [first, last] are adjacent in sorted order
      if (!rows.row(g, r0, r1, first, last)) continue;
      if (!in_range(g.errw, kSiteDirectBins, first, last + 1) ||
          !in_range(g.errw, kSiteDirectBins, last, g.nbins[0] * g.nbins[1] * g.nbins[2]))
        continue;
      const uint32_t i1 = bin_start[last + 1];
      for (uint32_t base = bin_start[first]; base < i1; base += 32) {
        const uint32_t i = base + uint32_t(lane);
        T z[D];
        bool in = false;
        T wgt = T(0);
        if (i < i1) {
#pragma unroll
          for (int j = 0; j < D; ++j) z[j] = xs[int64_t(j) * n + i] - qt[j];
          T u2 = T(0);
#pragma unroll
          for (int a = 0; a < D; ++a) {
            T ra = T(0);
#pragma unroll
            for (int c = 0; c < D; ++c) ra += hi[a][c] * z[c];
            u2 += z[a] * ra;
          }
          in = u2 <= T(1);
          if (in) wgt = ks * compact_k<T>(kern, u2, kr2);
        }
        const unsigned m = __ballot_sync(0xffffffffu, in);
        if (in) {
          const int slot = qn + __popc(m & below);
#pragma unroll
          for (int j = 0; j < D; ++j) qv[j * 64 + slot] = z[j];
          qv[D * 64 + slot] = wgt;
          qi[slot] = i;
        }
        qn += __popc(m);
        if (qn >= 32) {
          __syncwarp();
          consume(32);
          __syncwarp();
          if (lane < qn - 32) {  // move the overflow to the front of the queue
#pragma unroll
            for (int j = 0; j <= D; ++j) qv[j * 64 + lane] = qv[j * 64 + 32 + lane];
            qi[lane] = qi[32 + lane];
          }
          qn -= 32;
          __syncwarp();
        }
      }
    }
  __syncwarp();
  consume(qn);
  __syncwarp();
  out0 = T(0);
  out1 = T(0);
  const int nf = NS + nstr * NT;
#pragma unroll
  for (int f = 0; f < FMAX; ++f) {
    if (f < nf) {
      T v = acc[f];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == (f & 31)) {
        if (f < 32)
          out0 = v;
        else
          out1 = v;
      }
    }
  }
}

// warp per (grid point m, bandwidth bw_first + bb), eight per block:
// fields [bb][fgrid][Mtot]
template <typename T, int D, int ORD, int FMAX>
__global__ void __launch_bounds__(256)
direct_grid_kernel(GeoDev g, const BwDev* __restrict__ bwt, int bw_first, int bw_count,
                   int64_t Mtot, int64_t n, const T* __restrict__ xs, const T* __restrict__ str,
                   int str_first, int nstr, const uint32_t* __restrict__ bin_start, int fgrid,
                   T* __restrict__ field) {
  constexpr int QB = direct_queue_bytes<T, D>();
  __shared__ __align__(16) unsigned char qsm[8 * QB];
  const int lane = threadIdx.x & 31;
  const int64_t gid = int64_t(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (gid >= Mtot * bw_count) return;
  const int64_t m = gid % Mtot;
  const int bb = int(gid / Mtot);
  const BwDev& B = bwt[bw_first + bb];
  double q[3] = {0.0, 0.0, 0.0};
  int64_t rem = m;
  for (int a = D - 1; a >= 0; --a) {
    const int64_t idx = rem % g.M[a];
    rem /= g.M[a];
    q[a] = double(idx) * (g.hi[a] - g.lo[a]) / double(g.M[a] - 1);
  }
  T o0, o1;
  direct_warp_sums<T, D, ORD, FMAX>(g, B, n, xs, str, str_first, nstr, bin_start, q, lane,
                                    qsm + (threadIdx.x >> 5) * QB, o0, o1);
  T* fb = field + int64_t(bb) * fgrid * Mtot + m;
  if (lane < fgrid) fb[int64_t(lane) * Mtot] = o0;
  if (lane + 32 < fgrid) fb[int64_t(lane + 32) * Mtot] = o1;
}

template <typename T, int D, int ORD, int FMAX>
cudaError_t launch_direct_grid(fkreg_plan_s* P, int str_first, int nstr, int bw_first,
                               int bw_count, int slice, int64_t Mtot, int fgrid, cudaStream_t st) {
  constexpr int NS = mono_count(D, 2 * ORD), NT = mono_count(D, ORD);
  if constexpr (FMAX < kDirectMaxFields) {
    if (fgrid > FMAX)
      return launch_direct_grid<T, D, ORD, FMAX == 16 ? 40 : 64>(P, str_first, nstr, bw_first,
                                                                           bw_count, slice, Mtot, fgrid, st);
  }
  if constexpr ((FMAX - NS) / NT < 1) {
    return cudaErrorInvalidValue;
  } else {
    const unsigned blocks = unsigned((Mtot * bw_count + 7) / 8);
    direct_grid_kernel<T, D, ORD, FMAX><<<blocks, 256, 0, st>>>(
        P->geo, wsp<BwDev>(P, P->r_bw), bw_first, bw_count, Mtot, P->n, wsp<T>(P, P->r_xs),
        wsp<T>(P, P->r_str), str_first, nstr, wsp<uint32_t>(P, P->r_binstart), fgrid,
        wsp<T>(P, P->r_gfield) + int64_t(slice) * fgrid * Mtot);
    return cudaSuccess;
  }
}

template <typename T>
cudaError_t dispatch_direct_grid(fkreg_plan_s* P, int str_first, int nstr, int bw_first,
                                 int bw_count, int slice, int64_t Mtot, int fgrid, cudaStream_t st) {
#define FK_DG(DD, OO)                                                                         \
  if (P->d == DD && P->order == OO)                                                           \
    return launch_direct_grid<T, DD, OO, 16>(P, str_first, nstr, bw_first, bw_count, slice,  \
                                             Mtot, fgrid, st);
  FK_DG(1, 0) FK_DG(1, 1) FK_DG(1, 2) FK_DG(2, 0) FK_DG(2, 1) FK_DG(2, 2) FK_DG(3, 0) FK_DG(3, 1)
#undef FK_DG
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t run_direct_points(fkreg_plan_s* P, int str_first, int nstr, int bw_first, int bw_count,
                              int slice, cudaStream_t st) {
  const int64_t Mtot = P->geo.M[0] * P->geo.M[1] * P->geo.M[2];
  const int fgrid = P->ns + nstr * P->nt;
  if (fgrid > kDirectMaxFields) return cudaErrorInvalidValue;
  if (Mtot * bw_count == 0) return cudaSuccess;
  const cudaError_t e =
      P->prec == FKREG_F32
          ? dispatch_direct_grid<float>(P, str_first, nstr, bw_first, bw_count, slice, Mtot, fgrid, st)
          : dispatch_direct_grid<double>(P, str_first, nstr, bw_first, bw_count, slice, Mtot, fgrid, st);
  if (e != cudaSuccess) return e;
  P->launches += 1;
  return cudaGetLastError();
}

}  // namespace fk
