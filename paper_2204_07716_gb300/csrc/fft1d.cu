// Fourier transforms of 1-D plans up to 4096 points: one block per transform,
// mixed radix (4, 2, 3, 5, 7) Stockham passes in shared memory with a table of
// the roots of unity that the plan computes once in FP64.
//
// A 1-D problem's transforms are a few hundred points in a handful of fields.
// cuFFT took 9 to 24 us a call for them (FP64, 126 to 256 points, with a
// separate pre-processing kernel for some lengths) and 0.3 ms of host time for
// each plan, of which a bandwidth selection over ten candidates makes 25.  Here a
// transform is one launch of a few microseconds, bound by the latency of its
// log n passes, no library plan is made, and the type-2 fields go straight
// into their cell records.  Longer 1-D transforms and all 2-D and 3-D ones stay
// with cuFFT.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "internal.h"

namespace fk {

namespace {

constexpr int kMaxStages = 12;

struct Fft1dArgs {
  int n, stages;
  int radix[kMaxStages];
};

template <typename T>
struct Cplx;
template <>
struct Cplx<float> {
  using type = float2;
};
template <>
struct Cplx<double> {
  using type = double2;
};

template <typename C>
__device__ __forceinline__ C cadd(C a, C b) { return C{a.x + b.x, a.y + b.y}; }
template <typename C>
__device__ __forceinline__ C csub(C a, C b) { return C{a.x - b.x, a.y - b.y}; }
// a * w, or a * conj(w) for the inverse transform
template <bool INV, typename C>
__device__ __forceinline__ C ctw(C a, C w) {
  const auto wy = INV ? -w.y : w.y;
  return C{a.x * w.x - a.y * wy, a.x * wy + a.y * w.x};
}
// a * (-i), or a * i for the inverse transform
template <bool INV, typename C>
__device__ __forceinline__ C crot(C a) { return INV ? C{-a.y, a.x} : C{a.y, -a.x}; }

// One pass of radix R over the n points of `a` into `b`: l is the product of
// the radices done, m = n / (l R).  Element q + l (p + m k) is input k of the
// butterfly (p, q); output j goes, times w^(p j l), to q + l (R p + j).
template <int R, bool INV, typename C>
__device__ __forceinline__ void pass(const C* a, C* b, const C* tw, int n, int l) {
  const int m = n / (l * R);
  for (int idx = threadIdx.x; idx < n / R; idx += blockDim.x) {
    const int p = idx / l, q = idx - p * l;
    C x[R], y[R];
#pragma unroll
    for (int k = 0; k < R; ++k) x[k] = a[q + l * (p + m * k)];
    if constexpr (R == 2) {
      y[0] = cadd(x[0], x[1]);
      y[1] = csub(x[0], x[1]);
    } else if constexpr (R == 4) {
      const C s0 = cadd(x[0], x[2]), s1 = csub(x[0], x[2]);
      const C s2 = cadd(x[1], x[3]), s3 = crot<INV>(csub(x[1], x[3]));
      y[0] = cadd(s0, s2);
      y[1] = cadd(s1, s3);
      y[2] = csub(s0, s2);
      y[3] = csub(s1, s3);
    } else {
      // odd: with s_k = x_k + x_(R-k), d_k = x_k - x_(R-k) and w_R^k = c_k + i e_k,
      // outputs j and R - j are a_j +- i b_j, a_j = x_0 + sum c_(jk) s_k,
      // b_j = sum e_(jk) d_k
      constexpr int H = (R - 1) / 2;
      C w[R], s[H], e[H];
#pragma unroll
      for (int k = 1; k < R; ++k) {
        w[k] = tw[k * (n / R)];
        if (INV) w[k].y = -w[k].y;
      }
      y[0] = x[0];
#pragma unroll
      for (int k = 1; k <= H; ++k) {
        s[k - 1] = cadd(x[k], x[R - k]);
        e[k - 1] = csub(x[k], x[R - k]);
        y[0] = cadd(y[0], s[k - 1]);
      }
#pragma unroll
      for (int j = 1; j <= H; ++j) {
        C a = x[0], c{0, 0};
#pragma unroll
        for (int k = 1; k <= H; ++k) {
          const C v = w[(j * k) % R];
          a.x += v.x * s[k - 1].x;
          a.y += v.x * s[k - 1].y;
          c.x += v.y * e[k - 1].x;
          c.y += v.y * e[k - 1].y;
        }
        y[j] = C{a.x - c.y, a.y + c.x};
        y[R - j] = C{a.x + c.y, a.y - c.x};
      }
    }
    b[q + l * (R * p)] = y[0];
#pragma unroll
    for (int j = 1; j < R; ++j)
      b[q + l * (R * p + j)] = p == 0 ? y[j] : ctw<INV>(y[j], tw[p * j * l]);
  }
}

template <bool INV, typename C>
__device__ __forceinline__ const C* fft_shared(C* a, C* b, const C* tw, const Fft1dArgs& f) {
  int l = 1;
  for (int s = 0; s < f.stages; ++s) {
    __syncthreads();
    switch (f.radix[s]) {
      case 2: pass<2, INV>(a, b, tw, f.n, l); break;
      case 3: pass<3, INV>(a, b, tw, f.n, l); break;
      case 4: pass<4, INV>(a, b, tw, f.n, l); break;
      case 5: pass<5, INV>(a, b, tw, f.n, l); break;
      default: pass<7, INV>(a, b, tw, f.n, l); break;
    }
    l *= f.radix[s];
    C* t = a;
    a = b;
    b = t;
  }
  __syncthreads();
  return a;
}

// Block k: row k of in [batch][n] (real) -> out [batch][n/2 + 1].
template <typename T>
__global__ void __launch_bounds__(256)
fft1d_r2c_kernel(Fft1dArgs f, const typename Cplx<T>::type* __restrict__ tw,
                 const T* __restrict__ in, typename Cplx<T>::type* __restrict__ out) {
  using C = typename Cplx<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* a = reinterpret_cast<C*>(smem_raw);
  const T* row = in + int64_t(blockIdx.x) * f.n;
  for (int i = threadIdx.x; i < f.n; i += blockDim.x) {
    a[i] = C{row[i], T(0)};
    a[2 * f.n + i] = tw[i];
  }
  const C* r = fft_shared<false>(a, a + f.n, a + 2 * f.n, f);
  const int half = f.n / 2 + 1;
  C* o = out + int64_t(blockIdx.x) * half;
  for (int i = threadIdx.x; i < half; i += blockDim.x) o[i] = r[i];
}

// Block k: row k of in [batch][n/2 + 1] (Hermitian) -> n reals, value i at
// out[k * row + i * elem].
template <typename T>
__global__ void __launch_bounds__(256)
fft1d_c2r_kernel(Fft1dArgs f, const typename Cplx<T>::type* __restrict__ tw,
                 const typename Cplx<T>::type* __restrict__ in, T* __restrict__ out, int64_t row,
                 int64_t elem) {
  using C = typename Cplx<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* a = reinterpret_cast<C*>(smem_raw);
  const int half = f.n / 2 + 1;
  const C* h = in + int64_t(blockIdx.x) * half;
  for (int i = threadIdx.x; i < half; i += blockDim.x) {
    const C v = h[i];
    a[i] = v;
    if (i > 0 && f.n - i >= half) a[f.n - i] = C{v.x, -v.y};
  }
  for (int i = threadIdx.x; i < f.n; i += blockDim.x) a[2 * f.n + i] = tw[i];
  const C* r = fft_shared<true>(a, a + f.n, a + 2 * f.n, f);
  T* o = out + int64_t(blockIdx.x) * row;
  for (int i = threadIdx.x; i < f.n; i += blockDim.x) o[i * elem] = r[i].x;
}

Fft1dArgs make_args(int64_t n) {
  Fft1dArgs f{};
  f.n = int(n);
  for (int r : {4, 2, 3, 5, 7})
    while (n % r == 0) {
      f.radix[f.stages++] = r;
      n /= r;
    }
  return f;
}

template <typename T>
cudaError_t launch(fkreg_plan_s* P, bool inverse, int64_t n, int batch, const void* in, void* out,
                   int64_t row, int64_t elem, cudaStream_t st) {
  using C = typename Cplx<T>::type;
  const Fft1dArgs f = make_args(n);
  const C* tw = reinterpret_cast<const C*>(P->ws + P->r_roots.off) + P->roots.at(n);
  const size_t smem = 3 * size_t(n) * sizeof(C);  // points twice, roots
  const unsigned threads = unsigned(std::min<int64_t>(256, std::max<int64_t>(32, (n / 4 + 31) / 32 * 32)));
  cudaError_t e;
  if (inverse) {
    auto kern = fft1d_c2r_kernel<T>;
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem))) !=
        cudaSuccess)
      return e;
    kern<<<unsigned(batch), threads, smem, st>>>(f, tw, static_cast<const C*>(in),
                                                 static_cast<T*>(out), row, elem);
  } else {
    auto kern = fft1d_r2c_kernel<T>;
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem))) !=
        cudaSuccess)
      return e;
    kern<<<unsigned(batch), threads, smem, st>>>(f, tw, static_cast<const T*>(in),
                                                 static_cast<C*>(out));
  }
  P->launches += 1;
  return cudaGetLastError();
}

}  // namespace

// Lengths this file transforms: 7-smooth (every length of the planner is), two
// copies of the points and their roots in a block's shared memory (196 KB for 4096
// points in FP64).  Past that one block is no longer quicker than cuFFT's many.
bool fft1d_applies(const fkreg_plan_s* P, int64_t n) {
  if (P->d != 1 || n < 2 || n > kFft1dMax) return false;
  for (int r : {2, 3, 5, 7})
    while (n % r == 0) n /= r;
  return n == 1;
}

// Appends exp(-2 pi i t / n), t = 0 .. n-1, to the plan's root tables (once per
// length), in FP64: fkreg_set_workspace uploads them in the plan's precision.
void fft1d_add_roots(fkreg_plan_s* P, int64_t n) {
  if (P->roots.count(n)) return;
  P->roots[n] = int64_t(P->root_tab.size() / 2);
  for (int64_t t = 0; t < n; ++t) {
    const double x = 2.0 * M_PI * double(t) / double(n);
    P->root_tab.push_back(std::cos(x));
    P->root_tab.push_back(-std::sin(x));
  }
}

cudaError_t run_fft1d_r2c(fkreg_plan_s* P, int64_t n, int batch, const void* in, void* out,
                          cudaStream_t st) {
  return P->prec == FKREG_F32 ? launch<float>(P, false, n, batch, in, out, 0, 0, st)
                              : launch<double>(P, false, n, batch, in, out, 0, 0, st);
}

cudaError_t run_fft1d_c2r(fkreg_plan_s* P, int64_t n, int batch, const void* in, void* out,
                          int64_t row, int64_t elem, cudaStream_t st) {
  return P->prec == FKREG_F32 ? launch<float>(P, true, n, batch, in, out, row, elem, st)
                              : launch<double>(P, true, n, batch, in, out, row, elem, st);
}

}  // namespace fk
