// FP64 vector kernels for norms, the Krylov outer loop and precision
// conversion.  Reductions use a fixed grid (kRedBlocks partials) and a
// fixed-order final sum, so results do not depend on scheduling.
#include <algorithm>

#include "cmg_common.cuh"

namespace cmg {

namespace {

constexpr int kRedThreads = 256;

__device__ __forceinline__ double block_sum(double v, double* sh) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += sh[w];
  return s;
}

__global__ void __launch_bounds__(kRedThreads) sumsq_kernel(const double* __restrict__ a, size_t n,
                                                            double* __restrict__ partial, int accumulate,
                                                            double w2) {
  __shared__ double sh[32];
  double s = 0.0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const double v = a[i];
    s = fma(v, v, s);
  }
  s = block_sum(s, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = accumulate ? partial[blockIdx.x] + w2 * s : w2 * s;
}

// wy2 ||y||^2 + ||u||^2 + ||p||^2, 16 bytes per load (one launch; a launch per
// block with 304 CTAs took 3.3 ms at n = 1023, N = 256 for 0.6 ms of bytes).
__global__ void __launch_bounds__(kRedThreads) sumsq3_kernel(const double* __restrict__ y, const double* __restrict__ u,
                                                             const double* __restrict__ p, size_t ny, size_t nu,
                                                             double wy2, double* __restrict__ partial) {
  pdl_enter();
  __shared__ double sh[32];
  const size_t t0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (size_t)gridDim.x * blockDim.x;
  double sy = 0.0, sp = 0.0;
#pragma unroll 4
  for (size_t i = t0; i < ny / 2; i += stride) {
    const double2 a = reinterpret_cast<const double2*>(y)[i], b = reinterpret_cast<const double2*>(p)[i];
    sy = fma(a.x, a.x, fma(a.y, a.y, sy));
    sp = fma(b.x, b.x, fma(b.y, b.y, sp));
  }
  if (t0 == 0 && (ny & 1)) {
    sy = fma(y[ny - 1], y[ny - 1], sy);
    sp = fma(p[ny - 1], p[ny - 1], sp);
  }
  for (size_t i = t0; i < nu; i += stride) sp = fma(u[i], u[i], sp);
  const double s = block_sum(fma(wy2, sy, sp), sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

__global__ void finish_sum_kernel(const double* __restrict__ partial, int count, double* __restrict__ out) {
  __shared__ double sh[32];
  double s = 0.0;
  for (int i = threadIdx.x; i < count; i += blockDim.x) s += partial[i];
  s = block_sum(s, sh);
  if (threadIdx.x == 0) *out = s;
}

// Dots of C basis vectors with w, 16 bytes per load; n even, all vectors
// 16-byte aligned.  Bound by the FP64 pipe from C = 2 on (one FMA per element
// and vector at two lanes per clock and SM); C known at compile time and two
// elements per load keep 9 loads in flight at C = 8 (8.4 M elements, 5 vectors
// on average: 140 us with single elements and predicated vectors).
constexpr int kDotGroup = 8;
template <int C>
__global__ void __launch_bounds__(kRedThreads) mdot_kernel(const double* __restrict__ V, size_t stride,
                                                           const double* __restrict__ w, size_t n,
                                                           double* __restrict__ partial) {
  __shared__ double sh[32];
  double acc[C];
#pragma unroll
  for (int k = 0; k < C; ++k) acc[k] = 0.0;
  const double2* w2 = reinterpret_cast<const double2*>(w);
#pragma unroll(C > 4 ? 1 : 2)
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n / 2; i += (size_t)gridDim.x * blockDim.x) {
    const double2 wi = w2[i];
    double2 v[C];
#pragma unroll
    for (int k = 0; k < C; ++k) v[k] = reinterpret_cast<const double2*>(V + (size_t)k * stride)[i];
#pragma unroll
    for (int k = 0; k < C; ++k) acc[k] = fma(v[k].y, wi.y, fma(v[k].x, wi.x, acc[k]));
  }
#pragma unroll
  for (int k = 0; k < C; ++k) {
    const double s = block_sum(acc[k], sh);
    if (threadIdx.x == 0) partial[(size_t)k * gridDim.x + blockIdx.x] = s;
  }
}

__global__ void mdot_finish_kernel(const double* __restrict__ partial, int count, double* __restrict__ out) {
  __shared__ double sh[32];
  double s = 0.0;
  for (int i = threadIdx.x; i < count; i += blockDim.x) s += partial[(size_t)blockIdx.x * count + i];
  s = block_sum(s, sh);
  if (threadIdx.x == 0) out[blockIdx.x] = s;
}

// w += sign * sum_{k < C} coef[k] V_k, and the partial sums of ||w||^2 where
// partial is given (a pass over w less).  Bound by the FP64 pipe as the dots;
// C at compile time keeps all of a pair's loads in flight (a loop over the
// vectors, unrolled by four, took 116 us for 7 vectors of 8.4 M).
constexpr int kAxpyGroup = 16;
template <int C>
__global__ void __launch_bounds__(kRedThreads) maxpy_kernel(const double* __restrict__ V, size_t stride,
                                                            const double* __restrict__ coef, double sign,
                                                            double* __restrict__ w, size_t n,
                                                            double* __restrict__ partial) {
  __shared__ double sh[32];
  double c[C], sq = 0.0;
#pragma unroll
  for (int k = 0; k < C; ++k) c[k] = sign * coef[k];
#pragma unroll(C > 4 ? 1 : 2)
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n / 2; i += (size_t)gridDim.x * blockDim.x) {
    double2 acc = reinterpret_cast<const double2*>(w)[i], v[C];
#pragma unroll
    for (int k = 0; k < C; ++k) v[k] = reinterpret_cast<const double2*>(V + (size_t)k * stride)[i];
#pragma unroll
    for (int k = 0; k < C; ++k) {
      acc.x = fma(c[k], v[k].x, acc.x);
      acc.y = fma(c[k], v[k].y, acc.y);
    }
    reinterpret_cast<double2*>(w)[i] = acc;
    if (partial) sq = fma(acc.x, acc.x, fma(acc.y, acc.y, sq));
  }
  if (partial) {
    sq = block_sum(sq, sh);
    if (threadIdx.x == 0) partial[blockIdx.x] = sq;
  }
}

__global__ void scale_by_kernel(const double* __restrict__ x, const double* __restrict__ den,
                                double* __restrict__ y, size_t n) {
  const double s = 1.0 / sqrt(*den);
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    y[i] = x[i] * s;
}

template <typename Tx, typename Ty>
__global__ void axpy_kernel(double a, const Tx* __restrict__ x, Ty* __restrict__ y, size_t n) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    y[i] = (Ty)((double)y[i] + a * (double)x[i]);
}

template <typename Tx, typename Ty>
__global__ void scale_cast_kernel(double a, const Tx* __restrict__ x, Ty* __restrict__ y, size_t n) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    y[i] = (Ty)(a * (double)x[i]);
}

__global__ void rhs_kernel(int n, int N, double h, const double* __restrict__ yd, const double* __restrict__ fsrc,
                           double* __restrict__ fy, double* __restrict__ fu, double* __restrict__ fp) {
  const size_t total = (size_t)n * n * N;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    const size_t node = i / N;
    fy[i] = h * h / N * yd[node];
    fp[i] = fsrc ? h * h * fsrc[node] : 0.0;
    if (i % N == 0) fu[node] = 0.0;
  }
}

inline unsigned stream_blocks(size_t n) {
  const size_t b = (n + kRedThreads - 1) / kRedThreads;
  return (unsigned)(b < 152 * 16 ? (b == 0 ? 1 : b) : 152 * 16);
}

}  // namespace

cudaError_t launch_sumsq(const double* a, size_t n, double* partial, int accumulate, double w2, cudaStream_t s) {
  sumsq_kernel<<<kRedBlocks, kRedThreads, 0, s>>>(a, n, partial, accumulate, w2);
  count_launches(1);
  return cudaGetLastError();
}

int launch_sumsq3(const double* y, const double* u, const double* p, size_t ny, size_t nu, double wy2,
                  double* partial, cudaStream_t s) {
  const size_t want = (std::max(ny / 2, nu) + kRedThreads - 1) / kRedThreads;
  const int grid = (int)std::min<size_t>(std::max<size_t>(want, 1), 2 * kRedBlocks);
  if (launch_k(sumsq3_kernel, dim3((unsigned)grid), dim3(kRedThreads), 0, s, y, u, p, ny, nu, wy2, partial) != cudaSuccess)
    return -1;
  count_launches(1);
  return grid;
}

cudaError_t launch_finish_sum(const double* partial, int count, double* out, cudaStream_t s) {
  finish_sum_kernel<<<1, kRedThreads, 0, s>>>(partial, count, out);
  count_launches(1);
  return cudaGetLastError();
}

namespace {
bool pairs(const void* a, const void* b, size_t stride, size_t n) {
  return n % 2 == 0 && stride % 2 == 0 &&
         ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b)) & 15) == 0;
}
template <int C>
void dots(int c, const double* V, size_t stride, const double* w, size_t n, double* partial, cudaStream_t s) {
  if constexpr (C > 1) {
    if (c < C) return dots<C - 1>(c, V, stride, w, n, partial, s);
  }
  mdot_kernel<C><<<kRedBlocks, kRedThreads, 0, s>>>(V, stride, w, n, partial);
}
template <int C>
void axpys(int c, const double* V, size_t stride, const double* coef, double sign, double* w, size_t n,
           double* partial, cudaStream_t s) {
  if constexpr (C > 1) {
    if (c < C) return axpys<C - 1>(c, V, stride, coef, sign, w, n, partial, s);
  }
  maxpy_kernel<C><<<kAxpyBlocks, kRedThreads, 0, s>>>(V, stride, coef, sign, w, n, partial);
}
}  // namespace

cudaError_t launch_mdot(const double* V, size_t stride, int nv, const double* w, size_t n, double* partial,
                        double* out, cudaStream_t s) {
  if (nv < 1 || !pairs(V, w, stride, n)) return cudaErrorInvalidValue;
  // groups of equal size, so that none reads w for a vector or two
  const int groups = (nv + kDotGroup - 1) / kDotGroup, per = (nv + groups - 1) / groups;
  for (int g = 0; g < nv; g += per)
    dots<kDotGroup>(std::min(per, nv - g), V + (size_t)g * stride, stride, w, n, partial + (size_t)g * kRedBlocks, s);
  mdot_finish_kernel<<<nv, kRedThreads, 0, s>>>(partial, kRedBlocks, out);
  count_launches((nv + per - 1) / per + 1);
  return cudaGetLastError();
}

cudaError_t launch_maxpy(const double* V, size_t stride, int nv, const double* coef, double sign, double* w,
                         size_t n, cudaStream_t s, double* partial) {
  if (nv < 1 || nv > 128 || !pairs(V, w, stride, n)) return cudaErrorInvalidValue;
  const int groups = (nv + kAxpyGroup - 1) / kAxpyGroup, per = (nv + groups - 1) / groups;
  for (int g = 0; g < nv; g += per)
    axpys<kAxpyGroup>(std::min(per, nv - g), V + (size_t)g * stride, stride, coef + g, sign, w, n,
                      g + per >= nv ? partial : nullptr, s);
  count_launches((nv + per - 1) / per);
  return cudaGetLastError();
}

cudaError_t launch_scale_by(const double* x, const double* den, double* y, size_t n, cudaStream_t s) {
  scale_by_kernel<<<stream_blocks(n), kRedThreads, 0, s>>>(x, den, y, n);
  count_launches(1);
  return cudaGetLastError();
}

template <typename Tx, typename Ty>
cudaError_t launch_axpy(double a, const Tx* x, Ty* y, size_t n, cudaStream_t s) {
  axpy_kernel<Tx, Ty><<<stream_blocks(n), kRedThreads, 0, s>>>(a, x, y, n);
  count_launches(1);
  return cudaGetLastError();
}

namespace {
template <typename Tx, typename Ty>
__global__ void cast_rows_kernel(double a, const Tx* __restrict__ src, int lds, Ty* __restrict__ dst, int ldd,
                                 size_t rows, int N) {
  const size_t total = rows * (size_t)ldd, stride = (size_t)gridDim.x * blockDim.x;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += stride) {
    const size_t r = i / ldd;
    const int j = (int)(i - r * ldd);
    dst[i] = j < N ? (Ty)((decltype(Tx() + Ty()))a * src[r * lds + j]) : Ty(0);
  }
}
}  // namespace

template <typename Tx, typename Ty>
cudaError_t launch_cast_rows(double a, const Tx* src, int lds, Ty* dst, int ldd, size_t rows, int N, cudaStream_t s) {
  size_t blocks = (rows * (size_t)ldd + 255) / 256;
  if (blocks > 152 * 32) blocks = 152 * 32;
  cast_rows_kernel<<<(unsigned)blocks, 256, 0, s>>>(a, src, lds, dst, ldd, rows, N);
  count_launches(1);
  return cudaGetLastError();
}
template cudaError_t launch_cast_rows<double, float>(double, const double*, int, float*, int, size_t, int, cudaStream_t);
template cudaError_t launch_cast_rows<float, double>(double, const float*, int, double*, int, size_t, int, cudaStream_t);
template cudaError_t launch_cast_rows<float, float>(double, const float*, int, float*, int, size_t, int, cudaStream_t);

template <typename Tx, typename Ty>
cudaError_t launch_scale_cast(double a, const Tx* x, Ty* y, size_t n, cudaStream_t s) {
  scale_cast_kernel<Tx, Ty><<<stream_blocks(n), kRedThreads, 0, s>>>(a, x, y, n);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_rhs(int n, int N, double h, const double* yd, const double* fsrc, double* fy, double* fu,
                       double* fp, cudaStream_t s) {
  rhs_kernel<<<stream_blocks((size_t)n * n * N), kRedThreads, 0, s>>>(n, N, h, yd, fsrc, fy, fu, fp);
  count_launches(1);
  return cudaGetLastError();
}

template cudaError_t launch_axpy<double, double>(double, const double*, double*, size_t, cudaStream_t);
template cudaError_t launch_axpy<float, double>(double, const float*, double*, size_t, cudaStream_t);
template cudaError_t launch_scale_cast<double, float>(double, const double*, float*, size_t, cudaStream_t);
template cudaError_t launch_scale_cast<float, double>(double, const float*, double*, size_t, cudaStream_t);
template cudaError_t launch_scale_cast<double, double>(double, const double*, double*, size_t, cudaStream_t);

}  // namespace cmg
