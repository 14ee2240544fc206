// Node-sample kernels of the collective multigrid cycle:
//   residual r = f - S x (Eq. (2) blocks), red-black collective Gauss-Seidel
//   half-sweep (reduced node systems Eq. (12) solved by Eq. (13)), damped
//   collective Jacobi update (Eq. (11)), restriction P^T and prolongation P
//   (Algorithm 1).
//
// One kernel per step; the per-node work is in cmg_items.cuh.
// Layout: node arrays [n*n][ld] with the sample index fastest.  The lpn
// lanes of a node group read that node's samples as contiguous V-element
// vectors (coalesced 128-bit loads); neighbour rows are re-read from L2 by
// the CTAs of adjacent rows, which run close together in launch order.
// The sum over samples in the control row (u) is a shuffle reduction over
// the node group, carried in the cycle's precision (FP32 or FP64).
#include <cstdlib>

#include "cmg_items.cuh"

namespace cmg {

namespace {

// On grids whose vectors exceed L2 the launches of a cycle alternate in the
// direction in which their CTAs walk the grid (colour 0, residual,
// prolongation, recursion forwards; colour 1 and the restriction backwards):
// what the preceding launch touched last is read first, from L2, where a
// fixed order always finds it just evicted.  V(2,2) cycle, forwards -> turned:
// n = 511, N = 27 859 -> 815 us, n = 255, N = 100 633 -> 605, n = 1023, N = 256
// 13.37 -> 13.25 ms; within L2 (n = 255, N = 64: 100 MB) it costs 1 %.
__device__ __forceinline__ unsigned turned_block(int backwards) {
  return backwards ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
}
// y, p, f_y, f_p and two faces of an n x n grid against the 126 MB L2.
bool exceeds_l2(int n, int N, size_t elem) { return (size_t)n * n * N * 6 * elem > (size_t)126 << 20; }

template <typename T, int V, int SPL>
__global__ void __launch_bounds__(kBlock) residual_kernel(LevelView<T> L, Vec3c<T> x, Vec3c<T> f, Vec3<T> r,
                                                          int lpn, T wy) {
  pdl_enter();
  const long node = ((long)blockIdx.x * blockDim.x + threadIdx.x) / lpn;
  residual_item<T, V, SPL, false>(L, x, f, r, node, threadIdx.x & (lpn - 1), lpn, wy);
}

// r = f - S x at the colour-0 nodes only (the g-th node of colour 0).
template <typename T, int V, int SPL>
__global__ void __launch_bounds__(kBlock) residual_c0_kernel(LevelView<T> L, Vec3c<T> x, Vec3c<T> f, Vec3<T> r,
                                                             int lpn) {
  pdl_enter();
  const long g = ((long)blockIdx.x * blockDim.x + threadIdx.x) / lpn;
  long node = (long)L.n * L.n;   // out of range: the item does nothing but its shuffles
  if (g < colour_count(L.n, 0)) {
    int iy, ix;
    colour_node(g, L.n, 0, iy, ix);
    node = (long)iy * L.n + ix;
  }
  residual_item<T, V, SPL, false>(L, x, f, r, node, threadIdx.x & (lpn - 1), lpn, T(1));
}

// The widest FP32 variants (16 samples per lane) at more CTAs per SM than
// their registers would allow: more warps in flight to cover the load latency
// (a few spilled registers cost less).
template <typename T, int V, int SPL>
constexpr int wide_ctas(int k) { return (sizeof(T) == 4 && V * SPL == 16) ? k : 1; }
// The half-sweep on single samples too: 78 registers otherwise (three CTAs
// per SM, n = 511, N = 125: 448 against 362 us), none spilled at 64.
template <typename T, int V, int SPL>
constexpr int half_ctas() {
  return sizeof(T) == 4 && V == 1 && SPL > 1 ? (SPL == 8 ? 3 : 4) : wide_ctas<T, V, SPL>(3);
}

template <typename T, int V, int SPL>
__global__ void __launch_bounds__(kBlock, half_ctas<T, V, SPL>())
    rbgs_half_kernel(LevelView<T> L, Vec3<T> x, Vec3c<T> f, int colour, int lpn, int turned) {
  pdl_enter();
  const long g = ((long)turned_block(turned) * blockDim.x + threadIdx.x) / lpn;
  rbgs_item<T, V, SPL, false>(L, x, f, colour, g, threadIdx.x & (lpn - 1), lpn);
}

// Colour-0 half-sweep from a zero iterate (see rbgs_item, ZG).
template <typename T, int V, int SPL>
__global__ void __launch_bounds__(kBlock, wide_ctas<T, V, SPL>(3))
    rbgs_zero_kernel(LevelView<T> L, Vec3<T> x, Vec3c<T> f, int lpn) {
  pdl_enter();
  const long g = ((long)blockIdx.x * blockDim.x + threadIdx.x) / lpn;
  rbgs_item<T, V, SPL, false, false, true>(L, x, f, 0, g, threadIdx.x & (lpn - 1), lpn);
}

// Colour-0 half-sweep that reads its neighbours as x + P e (prolongation of
// the coarse correction e fused in; see rbgs_item).
template <typename T, int V, int SPL>
__global__ void __launch_bounds__(kBlock) rbgs_prolong_kernel(LevelView<T> L, Vec3<T> x, Vec3c<T> f, Vec3c<T> e,
                                                              int nc, int lpn) {
  pdl_enter();
  const long g = ((long)blockIdx.x * blockDim.x + threadIdx.x) / lpn;
  rbgs_item<T, V, SPL, false, true>(L, x, f, 0, g, threadIdx.x & (lpn - 1), lpn, e, nc);
}

template <typename T, int V, int SPL>
__global__ void __launch_bounds__(kBlock) jacobi_update_kernel(LevelView<T> L, Vec3<T> x, Vec3c<T> r,
                                                               double theta, int lpn) {
  pdl_enter();
  const long node = ((long)blockIdx.x * blockDim.x + threadIdx.x) / lpn;
  jacobi_item<T, V, SPL, false>(L, x, r, theta, node, threadIdx.x & (lpn - 1), lpn);
}

template <typename T, int V, int SPL>
__global__ void __launch_bounds__(kBlock) restrict_kernel(int nf, int N, Vec3c<T> r, Vec3<T> cv, Vec3<T> zx,
                                                          int lpn, int colour0, int turned) {
  pdl_enter();
  const long node = ((long)turned_block(turned) * blockDim.x + threadIdx.x) / lpn;
  restrict_item<T, V, SPL, false>(nf, N, r, cv, zx, node, threadIdx.x & (lpn - 1), lpn, colour0 != 0);
}

// The restriction, and the coarse grid's zero-guess half-sweep at its colour-0
// nodes (see rbgs_item, ZG) by the lanes that hold their right sides: a launch
// and a pass over the right sides fewer per grid and cycle.
template <typename T, int V, int SPL>
__global__ void __launch_bounds__(kBlock) restrict_zero_kernel(int nf, LevelView<T> L, Vec3c<T> r, Vec3<T> cv,
                                                               Vec3<T> x, int lpn, int colour0, int turned) {
  pdl_enter();
  const long node = ((long)turned_block(turned) * blockDim.x + threadIdx.x) / lpn;
  const int lane = threadIdx.x & (lpn - 1);
  restrict_item<T, V, SPL, false>(nf, L.ld, r, cv, Vec3<T>{nullptr, nullptr, nullptr}, node, lane, lpn, colour0 != 0);
  __syncwarp();   // the control right side was written by the node's first lane
  const int J = (int)(node / L.n), I = (int)(node - (long)J * L.n);
  rbgs_node<T, V, SPL, false, false, true>(L, cview(x), x, cview(cv), node < (long)L.n * L.n && ((J + I) & 1) == 0, J, I,
                                           lane, lpn, Vec3c<T>{nullptr, nullptr, nullptr}, 0);
}

template <typename T, int V, int SPL>
__global__ void __launch_bounds__(kBlock) prolong_add_kernel(int nf, int N, Vec3c<T> e, Vec3<T> x, int lpn,
                                                             CtlBox ctl) {
  pdl_enter();
  const long node = ((long)blockIdx.x * blockDim.x + threadIdx.x) / lpn;
  prolong_item<T, V, SPL, false>(nf, N, e, x, node, threadIdx.x & (lpn - 1), lpn, ctl);
}

// One pass of FP64 refinement: r32 = s (f - S x) and per-CTA partial sums
// of ||W r32||^2 (squares in FP32, CTA sum in FP64).
template <int V, int SPL>
__global__ void __launch_bounds__(kBlock) residual_cast_kernel(LevelView<double> L, Vec3c<double> x,
                                                              Vec3c<double> f, Vec3<float> r, int lpn, double s,
                                                              const double* __restrict__ sdev, float wy2,
                                                              double* __restrict__ partial,
                                                              const double* __restrict__ gate) {
  pdl_enter();
  __shared__ double sh[kBlock / 32];
  if (gate && *gate == 0.0) return;   // refinement anchor not due (residual replacement)
  const long node = ((long)blockIdx.x * blockDim.x + threadIdx.x) / lpn;
  const double sc = sdev ? *sdev : s;
  double v = (double)residual_cast_item<V, SPL>(L, x, f, r, node, threadIdx.x & (lpn - 1), lpn, sc, wy2);
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kBlock / 32; ++w) t += sh[w];
    partial[blockIdx.x] = t;
  }
}

// FP32 refinement between FP64 anchors (residual replacement): the scaled
// residual r (the cycle's right side) is updated in place, r <- r - S e (A e
// from neighbour differences, see recur_item), the
// running correction d += e, and per-CTA partial sums of ||W r||^2 are
// written (squares in FP32, CTA sum in FP64).  Each lane reads its own f
// entries before writing r at the same place, so the update in place is safe.
template <int V, int SPL>
__global__ void __launch_bounds__(kBlock, wide_ctas<float, V, SPL>(3)) recur_kernel(LevelView<float> L, Vec3c<float> e, Vec3<float> r,
                                                       Vec3<float> d, int lpn, float wy2,
                                                       double* __restrict__ partial) {
  pdl_enter();
  __shared__ double sh[kBlock / 32];
  const long node = ((long)blockIdx.x * blockDim.x + threadIdx.x) / lpn;
  const int lane = threadIdx.x & (lpn - 1);
  const float sq = recur_item<V, SPL>(L, e, r, d, node, lane, lpn, wy2);
  double v = (double)sq;
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kBlock / 32; ++w) t += sh[w];
    partial[blockIdx.x] = t;
  }
}

// Anchor of residual replacement: x += a d (a = *adev) and d = 0, when
// *gate is nonzero.  The y and p blocks move as pairs (16-byte FP64 and
// 8-byte FP32 vectors; the blocks start 16-byte aligned), one odd tail
// element and the u block singly.
__global__ void fold_kernel(const double* __restrict__ adev, const double* __restrict__ gate, Vec3<float> d,
                            Vec3<double> x, size_t ny, size_t nu) {
  pdl_enter();
  if (*gate == 0.0) return;
  const double a = *adev;
  const size_t np = ny / 2;
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  const size_t t0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (size_t i = t0; i < 2 * np; i += stride) {
    const bool isp = i >= np;
    const size_t k = isp ? i - np : i;
    double2* xv = reinterpret_cast<double2*>(isp ? x.p : x.y) + k;
    float2* dv = reinterpret_cast<float2*>(isp ? d.p : d.y) + k;
    double2 xx = *xv;
    const float2 dd = *dv;
    xx.x = fma(a, (double)dd.x, xx.x);
    xx.y = fma(a, (double)dd.y, xx.y);
    *xv = xx;
    *dv = make_float2(0.f, 0.f);
  }
  for (size_t i = t0; i < nu; i += stride) {
    x.u[i] = fma(a, (double)d.u[i], x.u[i]);
    d.u[i] = 0.f;
  }
  if (t0 == 0 && (ny & 1)) {
    const size_t k = ny - 1;
    x.y[k] = fma(a, (double)d.y[k], x.y[k]);
    d.y[k] = 0.f;
    x.p[k] = fma(a, (double)d.p[k], x.p[k]);
    d.p[k] = 0.f;
  }
}

// The same where d's rows are padded (ld > N, a multiple of 4): a thread takes
// four samples of d at a time.
__global__ void fold_rows_kernel(const double* __restrict__ adev, const double* __restrict__ gate, Vec3<float> d,
                                 Vec3<double> x, size_t nodes, int N, int ld) {
  pdl_enter();
  if (*gate == 0.0) return;
  const double a = *adev;
  const size_t per = (size_t)ld / 4, total = nodes * per;
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  const size_t t0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (size_t i = t0; i < 2 * total; i += stride) {
    const bool isp = i >= total;
    const size_t c = isp ? i - total : i, node = c / per;
    const int j = (int)(c - node * per) * 4;
    float4* dv = reinterpret_cast<float4*>((isp ? d.p : d.y) + node * ld + j);
    const float4 dd = *dv;
    const float e[4] = {dd.x, dd.y, dd.z, dd.w};
    double* xv = (isp ? x.p : x.y) + node * N + j;
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (j + k < N) xv[k] = fma(a, (double)e[k], xv[k]);
    *dv = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  for (size_t i = t0; i < nodes; i += stride) {
    x.u[i] = fma(a, (double)d.u[i], x.u[i]);
    d.u[i] = 0.f;
  }
}

// (y, u, p) = 0 for an FP32 level vector (a kernel, so that it can be a
// programmatic dependent of the kernels around it).
__global__ void zero3_kernel(Vec3<float> v, size_t ny, size_t nu) {
  pdl_enter();
  const size_t total = 2 * ny + nu;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    if (i < ny) v.y[i] = 0.f;
    else if (i < ny + nu) v.u[i - ny] = 0.f;
    else v.p[i - ny - nu] = 0.f;
  }
}

// x += a * e for the three blocks (FP64 iterate, FP32 correction); a read
// from adev when given.
__global__ void axpy3_kernel(double a0, const double* __restrict__ adev, Vec3c<float> e, Vec3<double> x, size_t ny,
                             size_t nu) {
  pdl_enter();
  const double a = adev ? *adev : a0;
  const size_t total = 2 * ny + nu;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    if (i < ny) x.y[i] = fma(a, (double)e.y[i], x.y[i]);
    else if (i < ny + nu) x.u[i - ny] = fma(a, (double)e.u[i - ny], x.u[i - ny]);
    else x.p[i - ny - nu] = fma(a, (double)e.p[i - ny - nu], x.p[i - ny - nu]);
  }
}

// Whole CTAs of kBlock threads (the kernels that sum over their CTA).
inline unsigned grid_for(long groups, int lpn) {
  const long threads = groups * lpn;
  return (unsigned)((threads + kBlock - 1) / kBlock);
}

}  // namespace

bool pdl_enabled() {
  static const bool on = [] {
    const char* e = std::getenv("CMG_PDL");
    return !(e && e[0] == '0');
  }();
  return on;
}

SampleMap choose_map(int N, int elem_bytes, long items, int spl_target) {
  SampleMap m;
  if ((spl_target & kTuneWide) && elem_bytes == 4 && wide_supported(N)) {
    m.V = 2;
    m.spl = 1;
    m.lpn = 1;
    while (m.lpn < N / 2) m.lpn <<= 1;
    return m;
  }
  const int vmax = 16 / elem_bytes;     // 2 for double, 4 for float
  m.V = (N % vmax == 0) ? vmax : 1;
  const int chunks = (N + m.V - 1) / m.V;
  // Chunks per lane by what the launch has to offer (kMinLanes*): 16 samples
  // per lane only where that still leaves a dozen waves of CTAs, 8 from a few CTAs per
  // SM on; and at least two (four) lanes per node, else a warp's 16-byte loads fall
  // apart into single sectors.  FP64 takes two chunks at most: with four, the
  // registers leave the FP64 pipe too few warps (n = 255, N = 64: 96 against 81
  // us per half-sweep).  FP32 half-sweeps, 4 -> 2 chunks: n = 255, N = 64 20.8 -> 18.9 us,
  // n = 511, N = 16 50.9 -> 25.9 us; 1 -> 2: n = 127, N = 64 7.2 -> 5.5 us.
  // Rows of a few single samples have no 16-byte loads to keep whole: up to four in a lane
  // (FP32 sweep at n = 1023, two -> four: N = 3 64 -> 53 us, one: 107; N = 9 247 -> 172), in
  // FP64 where that leaves fewer lanes idle (N = 5 266 -> 227, N = 9 541 -> 439, but N = 7 270 -> 302).
  int target = 1;
  if (items > 0) {
    const long lanes = items * chunks;
    const auto slots = [chunks](int t) {   // lanes times the chunks that any of them takes
      int l = 1;
      while (l < (chunks + t - 1) / t && l < 32) l <<= 1;
      return l * ((chunks + l - 1) / l);
    };
    if (lanes >= 2 * kMinLanes2 && chunks >= (m.V == 1 ? 2 : 3)) target = 2;
    if (m.V == 1) {
      if (lanes >= 4 * kMinLanes1 && chunks >= 2 && (chunks >= 16 || elem_bytes == 4 || slots(4) < slots(2))) target = 4;
    } else if (elem_bytes == 4 && lanes >= 4 * kMinLanes4 && chunks >= 16) {
      target = 4;
    }
  }
  if ((spl_target & 15) > 0) target = spl_target & 15;   // the staged and wide flags are not part of it
  const int want = (chunks + target - 1) / target;   // lanes needed at `target` chunks each
  int lpn = 1;
  while (lpn < want && lpn < 32) lpn <<= 1;
  m.lpn = lpn;
  int spl = (chunks + lpn - 1) / lpn;
  int p2 = 1;
  while (p2 < spl) p2 <<= 1;
  m.spl = p2;
  return m;
}



// Target of a residual over `nodes` nodes: the grid's (cmg_set_tuning,
// cmg_autotune); without one in FP64, four chunks per lane (all of them where
// there are fewer) where two 256-thread CTAs per SM remain, else choose_map's
// rule: here they hide the loads better than twice the warps (n = 255, N = 64:
// 141 against 186 us; n = 1023, N = 3 119 against 165, N = 6 215 against 292).
static int residual_target(int N, int elem_bytes, long nodes, int spl_target) {
  if (elem_bytes == 4 || (spl_target & 15) > 0) return spl_target;
  const long chunks = N % 2 == 0 ? N / 2 : N;
  return chunks >= 2 && nodes * chunks >= 4 * 2L * 152 * 256 ? 4 : 0;
}

// Map of the prolongation-fused half-sweep: 16 samples per lane take 128
// registers there (the coarse loads), so eight unless the target asks for more.
static SampleMap prolong_map(int N, int elem_bytes, long groups, int spl_target) {
  const SampleMap m = choose_map(N, elem_bytes, groups, spl_target);
  return m.V * m.spl > 8 && (spl_target & 15) == 0 ? choose_map(N, elem_bytes, groups, spl_target | 2) : m;
}

int size_rule_target(int n, int N, int elem_bytes) {
  const auto same = [](const SampleMap& a, const SampleMap& b) { return a.lpn == b.lpn && a.V == b.V && a.spl == b.spl; };
  const long c0 = colour_count(n, 0), c1 = colour_count(n, 1), all = (long)n * n;
  for (int t : {1, 2, 4}) {
    const auto residual = [&](long items) {
      return same(choose_map(N, elem_bytes, items, residual_target(N, elem_bytes, items, 0)),
                  choose_map(N, elem_bytes, items, t));
    };
    if (same(choose_map(N, elem_bytes, c0, 0), choose_map(N, elem_bytes, c0, t)) &&
        same(choose_map(N, elem_bytes, c1, 0), choose_map(N, elem_bytes, c1, t)) &&
        same(prolong_map(N, elem_bytes, c0, 0), prolong_map(N, elem_bytes, c0, t)) && residual(c0) &&
        (elem_bytes == 4 || residual(all)))
      return t;
  }
  return 0;
}

template <typename T>
cudaError_t launch_residual(const LevelView<T>& L, Vec3c<T> x, Vec3c<T> f, Vec3<T> r, cudaStream_t st, double wy) {
  const long nodes = (long)L.n * L.n;
  const SampleMap m = choose_map(L.N, sizeof(T), nodes, residual_target(L.N, sizeof(T), nodes, L.spl_target));
  const long threads = ((long)L.n * L.n) * m.lpn;
  cudaError_t e_ = cudaSuccess;
  CMG_DISPATCH(T, m, (e_ = launch_k(residual_kernel<T, V, SPL>, ctas_for(threads), block_for(threads), 0, st, L, x, f, r, m.lpn, (T)wy)));
  count_launches(1);
  return e_ != cudaSuccess ? e_ : cudaGetLastError();
}

template <typename T>
cudaError_t launch_residual_c0(const LevelView<T>& L, Vec3c<T> x, Vec3c<T> f, Vec3<T> r, cudaStream_t st) {
  const long groups = colour_count(L.n, 0);
  const SampleMap m = choose_map(L.N, sizeof(T), groups, residual_target(L.N, sizeof(T), groups, L.spl_target));
  const long threads = (groups) * m.lpn;
  cudaError_t e_ = cudaSuccess;
  CMG_DISPATCH(T, m, (e_ = launch_k(residual_c0_kernel<T, V, SPL>, ctas_for(threads), block_for(threads), 0, st, L, x, f, r, m.lpn)));
  count_launches(1);
  return e_ != cudaSuccess ? e_ : cudaGetLastError();
}

template <typename T>
cudaError_t launch_rbgs_half(const LevelView<T>& L, Vec3<T> x, Vec3c<T> f, int colour, cudaStream_t st) {
  const SampleMap m = choose_map(L.N, sizeof(T), colour_count(L.n, colour), L.spl_target);
  if constexpr (sizeof(T) == 4) {
    if (L.spl_target & kTuneStaged) {
      const cudaError_t e = launch_rbgs_half_staged(L, x, f, colour, m, st);
      if (e != cudaErrorNotSupported) return e;
    }
    if (L.spl_target & kTuneTma) {
      const cudaError_t e = launch_rbgs_half_tma(L, x, f, colour, m, st);
      if (e != cudaErrorNotSupported) return e;
    }
  }
  const long threads = (colour_count(L.n, colour)) * m.lpn;
  cudaError_t e_ = cudaSuccess;
  CMG_DISPATCH(T, m, (e_ = launch_k(rbgs_half_kernel<T, V, SPL>, ctas_for(threads), block_for(threads), 0, st, L, x, f, colour, m.lpn,
                                   colour && exceeds_l2(L.n, L.N, sizeof(T)) ? 1 : 0)));
  count_launches(1);
  return e_ != cudaSuccess ? e_ : cudaGetLastError();
}

template <typename T>
cudaError_t launch_rbgs_zero(const LevelView<T>& L, Vec3<T> x, Vec3c<T> f, cudaStream_t st) {
  const long groups = colour_count(L.n, 0);
  const SampleMap m = choose_map(L.N, sizeof(T), groups, L.spl_target);
  const long threads = (groups) * m.lpn;
  cudaError_t e_ = cudaSuccess;
  CMG_DISPATCH(T, m, (e_ = launch_k(rbgs_zero_kernel<T, V, SPL>, ctas_for(threads), block_for(threads), 0, st, L, x, f, m.lpn)));
  count_launches(1);
  return e_ != cudaSuccess ? e_ : cudaGetLastError();
}

template <typename T>
cudaError_t launch_rbgs_prolong(const LevelView<T>& L, Vec3<T> x, Vec3c<T> f, Vec3c<T> e, int nc, cudaStream_t st) {
  const long groups = colour_count(L.n, 0);
  const SampleMap m = prolong_map(L.N, sizeof(T), groups, L.spl_target);
  const long threads = (groups) * m.lpn;
  cudaError_t e_ = cudaSuccess;
  CMG_DISPATCH(T, m, (e_ = launch_k(rbgs_prolong_kernel<T, V, SPL>, ctas_for(threads), block_for(threads), 0, st, L, x, f, e, nc, m.lpn)));
  count_launches(1);
  return e_ != cudaSuccess ? e_ : cudaGetLastError();
}

template <typename T>
cudaError_t launch_jacobi_update(const LevelView<T>& L, Vec3<T> x, Vec3c<T> r, double theta, cudaStream_t st) {
  const SampleMap m = choose_map(L.N, sizeof(T), (long)L.n * L.n, L.spl_target);
  const long threads = ((long)L.n * L.n) * m.lpn;
  cudaError_t e_ = cudaSuccess;
  CMG_DISPATCH(T, m, (e_ = launch_k(jacobi_update_kernel<T, V, SPL>, ctas_for(threads), block_for(threads), 0, st, L, x, r, theta, m.lpn)));
  count_launches(1);
  return e_ != cudaSuccess ? e_ : cudaGetLastError();
}

template <typename T>
cudaError_t launch_restrict(int nf, int N, Vec3c<T> r, Vec3<T> c, cudaStream_t st, Vec3<T> zx, int colour0) {
  const int nc = (nf - 1) / 2;
  const SampleMap m = choose_map(N, sizeof(T), (long)nc * nc);
  const long threads = ((long)nc * nc) * m.lpn;
  cudaError_t e_ = cudaSuccess;
  CMG_DISPATCH(T, m, (e_ = launch_k(restrict_kernel<T, V, SPL>, ctas_for(threads), block_for(threads), 0, st, nf, N, r, c, zx, m.lpn, colour0,
                                   exceeds_l2(nf, N, sizeof(T)) ? 1 : 0)));
  count_launches(1);
  return e_ != cudaSuccess ? e_ : cudaGetLastError();
}

template <typename T>
cudaError_t launch_restrict_zero(int nf, const LevelView<T>& L, Vec3c<T> r, Vec3<T> c, Vec3<T> x, cudaStream_t st,
                                 int colour0) {
  // the half-sweep's own map: the samples are summed in the order of launch_rbgs_zero
  const SampleMap m = choose_map(L.N, sizeof(T), colour_count(L.n, 0), L.spl_target);
  const long threads = (long)L.n * L.n * m.lpn;
  cudaError_t e_ = cudaSuccess;
  CMG_DISPATCH(T, m, (e_ = launch_k(restrict_zero_kernel<T, V, SPL>, ctas_for(threads), block_for(threads), 0, st, nf, L, r, c, x,
                                   m.lpn, colour0, exceeds_l2(nf, L.N, sizeof(T)) ? 1 : 0)));
  count_launches(1);
  return e_ != cudaSuccess ? e_ : cudaGetLastError();
}

template <typename T>
cudaError_t launch_prolong_add(int nf, int N, Vec3c<T> e, Vec3<T> x, cudaStream_t st, CtlBox ctl) {
  const SampleMap m = choose_map(N, sizeof(T), (long)nf * nf);
  const long threads = ((long)nf * nf) * m.lpn;
  cudaError_t e_ = cudaSuccess;
  CMG_DISPATCH(T, m, (e_ = launch_k(prolong_add_kernel<T, V, SPL>, ctas_for(threads), block_for(threads), 0, st, nf, N, e, x, m.lpn, ctl)));
  count_launches(1);
  return e_ != cudaSuccess ? e_ : cudaGetLastError();
}

int launch_residual_cast(const LevelView<double>& L, Vec3c<double> x, Vec3c<double> f, Vec3<float> r, double s,
                         const double* sdev, double wy, double* partial, int max_partials, cudaStream_t st,
                         const double* gate) {
  const SampleMap m = choose_map(L.N, 8, (long)L.n * L.n, residual_target(L.N, 8, (long)L.n * L.n, 0));
  const unsigned grid = grid_for((long)L.n * L.n, m.lpn);
  if ((int)grid > max_partials) return -1;
  const float wy2 = (float)(wy * wy);
  using T = double;
  auto go = [&]() -> cudaError_t {
    cudaError_t e_ = cudaSuccess;
    CMG_DISPATCH(T, m, (e_ = launch_k(residual_cast_kernel<V, SPL>, grid, kBlock, 0, st, L, x, f, r, m.lpn, s, sdev,
                                                   wy2, partial, gate)));
    return e_ != cudaSuccess ? e_ : cudaGetLastError();
  };
  if (go() != cudaSuccess) return -1;
  count_launches(1);
  return (int)grid;
}

int launch_recur(const LevelView<float>& L, Vec3c<float> e, Vec3<float> r, Vec3<float> d, double wy, double* partial,
                 int max_partials, cudaStream_t st) {
  const SampleMap m = choose_map(L.N, 4, (long)L.n * L.n, L.spl_target);
  const unsigned grid = grid_for((long)L.n * L.n, m.lpn);
  if ((int)grid > max_partials) return -1;
  const float wy2 = (float)(wy * wy);
  using T = float;
  auto go = [&]() -> cudaError_t {
    cudaError_t e_ = cudaSuccess;
    CMG_DISPATCH(T, m, (e_ = launch_k(recur_kernel<V, SPL>, grid, kBlock, 0, st, L, e, r, d, m.lpn, wy2, partial)));
    return e_ != cudaSuccess ? e_ : cudaGetLastError();
  };
  if (go() != cudaSuccess) return -1;
  count_launches(1);
  return (int)grid;
}

cudaError_t launch_fold(const double* adev, const double* gate, Vec3<float> d, Vec3<double> x, size_t nodes, int N,
                        int ld, cudaStream_t st) {
  const size_t ny = nodes * N, total = ny + nodes;
  size_t blocks = (total + kBlock - 1) / kBlock;
  if (blocks > 152 * 16) blocks = 152 * 16;
  const cudaError_t e_ =
      ld == N ? launch_k(fold_kernel, dim3((unsigned)blocks), dim3(kBlock), 0, st, adev, gate, d, x, ny, nodes)
              : launch_k(fold_rows_kernel, dim3((unsigned)blocks), dim3(kBlock), 0, st, adev, gate, d, x, nodes, N, ld);
  if (e_ != cudaSuccess) return e_;
  count_launches(1);
  return e_ != cudaSuccess ? e_ : cudaGetLastError();
}

cudaError_t launch_zero3(Vec3<float> v, size_t ny, size_t nu, cudaStream_t st) {
  const size_t total = 2 * ny + nu;
  size_t blocks = (total + kBlock - 1) / kBlock;
  if (blocks > 152 * 8) blocks = 152 * 8;
  const cudaError_t e_ = launch_k(zero3_kernel, dim3((unsigned)blocks), dim3(kBlock), 0, st, v, ny, nu);
  count_launches(1);
  return e_;
}

cudaError_t launch_axpy3(double a, const double* adev, Vec3c<float> e, Vec3<double> x, size_t ny, size_t nu,
                         cudaStream_t st) {
  const size_t total = 2 * ny + nu;
  size_t blocks = (total + kBlock - 1) / kBlock;
  if (blocks > 152 * 16) blocks = 152 * 16;
  const cudaError_t e_ = launch_k(axpy3_kernel, dim3((unsigned)blocks), dim3(kBlock), 0, st, a, adev, e, x, ny, nu);
  if (e_ != cudaSuccess) return e_;
  count_launches(1);
  return e_ != cudaSuccess ? e_ : cudaGetLastError();
}

#define CMG_INST(T)                                                                                   \
  template cudaError_t launch_residual<T>(const LevelView<T>&, Vec3c<T>, Vec3c<T>, Vec3<T>, cudaStream_t, double); \
  template cudaError_t launch_rbgs_half<T>(const LevelView<T>&, Vec3<T>, Vec3c<T>, int, cudaStream_t);    \
  template cudaError_t launch_rbgs_zero<T>(const LevelView<T>&, Vec3<T>, Vec3c<T>, cudaStream_t);         \
  template cudaError_t launch_jacobi_update<T>(const LevelView<T>&, Vec3<T>, Vec3c<T>, double, cudaStream_t); \
  template cudaError_t launch_restrict<T>(int, int, Vec3c<T>, Vec3<T>, cudaStream_t, Vec3<T>, int);         \
  template cudaError_t launch_residual_c0<T>(const LevelView<T>&, Vec3c<T>, Vec3c<T>, Vec3<T>, cudaStream_t);       \
  template cudaError_t launch_rbgs_prolong<T>(const LevelView<T>&, Vec3<T>, Vec3c<T>, Vec3c<T>, int, cudaStream_t);                     \
  template cudaError_t launch_restrict_zero<T>(int, const LevelView<T>&, Vec3c<T>, Vec3<T>, Vec3<T>, cudaStream_t, int);             \
  template cudaError_t launch_prolong_add<T>(int, int, Vec3c<T>, Vec3<T>, cudaStream_t, CtlBox);

CMG_INST(double)
CMG_INST(float)

}  // namespace cmg
