// Layer kernels of the warm-start network besides the convolutions, the head
// (cmg_nn_conv.cu) and the GEMM: 2x2 average pooling, nearest upsampling with the
// additive skip, the one-pass gradient of a layer's activation (resampling,
// skip, ReLU and head gradients with the bias sums), the sums of the weight
// gradient's slices, the masked MSE loss, AdamW, BF16 casts, and the
// conversions between solver grids (n x n, FP64) and the network's S x S BF16
// images.  Also the same layers one at a time (im2col and col2im, transposes,
// flip3x3, ReLU / pooling / upsampling gradients, add, outer, column and slice
// sums): entry points of the C ABI that the network itself does not use; the
// gradients are tested against the chain they make.
//
// Activations are NHWC BF16 ([B][H][W][C], C a multiple of 8 so a 16-byte
// chunk holds 8 channels of one pixel); convolution weights are
// [Cout][9 Cin] BF16 with column t*Cin + c for tap t = 3 dy + dx.
#include <cuda_bf16.h>
#include <stdint.h>

#include "cmg_common.cuh"

using bf16 = __nv_bfloat16;

namespace cmg {
namespace {

constexpr int kT = 256;

inline unsigned blocks(long n) {
  long b = (n + kT - 1) / kT;
  if (b > 152L * 32) b = 152L * 32;
  return (unsigned)(b < 1 ? 1 : b);
}

#define GRID_STRIDE(i, n) for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < (n); i += (long)gridDim.x * blockDim.x)

// col[p][t*C + c] = X[b][y+dy-1][x+dx-1][c] (zero outside); one 16-byte chunk per thread.
__global__ void im2col_kernel(const bf16* __restrict__ X, bf16* __restrict__ col, int B, int H, int W, int C) {
  const int c8 = C / 8;
  const long total = (long)B * H * W * 9 * c8;
  GRID_STRIDE(i, total) {
    const int ch = (int)(i % c8);
    long r = i / c8;
    const int t = (int)(r % 9);
    const long p = r / 9;
    const int x = (int)(p % W), y = (int)((p / W) % H);
    const long b = p / ((long)W * H);
    const int yy = y + t / 3 - 1, xx = x + t % 3 - 1;
    uint4 v = make_uint4(0, 0, 0, 0);
    if (yy >= 0 && yy < H && xx >= 0 && xx < W)
      v = *reinterpret_cast<const uint4*>(X + (((b * H + yy) * W + xx) * C + ch * 8));
    *reinterpret_cast<uint4*>(col + p * 9 * C + t * C + ch * 8) = v;
  }
}

// colT[t*C + c][p] (pixels contiguous), same values as im2col.
__global__ void im2col_t_kernel(const bf16* __restrict__ X, bf16* __restrict__ colT, int B, int H, int W, int C) {
  const long P = (long)B * H * W;
  const long total = P * 9 * C;
  GRID_STRIDE(i, total) {
    const long p = i % P;
    const long k = i / P;
    const int t = (int)(k / C), c = (int)(k % C);
    const int x = (int)(p % W), y = (int)((p / W) % H);
    const long b = p / ((long)W * H);
    const int yy = y + t / 3 - 1, xx = x + t % 3 - 1;
    bf16 v = __float2bfloat16(0.f);
    if (yy >= 0 && yy < H && xx >= 0 && xx < W) v = X[((b * H + yy) * W + xx) * C + c];
    colT[k * P + p] = v;
  }
}

// dX[b][y][x][c] = sum_t dcol[(b, y-dy+1, x-dx+1)][t*C + c] over outputs inside the image.
__global__ void col2im_kernel(const float* __restrict__ dcol, bf16* __restrict__ dX, int B, int H, int W, int C) {
  const long total = (long)B * H * W * C;
  GRID_STRIDE(i, total) {
    const int c = (int)(i % C);
    const long p = i / C;
    const int x = (int)(p % W), y = (int)((p / W) % H);
    const long b = p / ((long)W * H);
    float s = 0.f;
#pragma unroll
    for (int t = 0; t < 9; ++t) {
      const int yo = y - (t / 3 - 1), xo = x - (t % 3 - 1);
      if (yo >= 0 && yo < H && xo >= 0 && xo < W) s += dcol[((b * H + yo) * W + xo) * 9L * C + t * C + c];
    }
    dX[i] = __float2bfloat16_rn(s);
  }
}

// Weights of the data-gradient convolution: Wf[c][t Cout + co] =
// W[co][(8 - t) C + c] (taps turned by 180 degrees, channels exchanged), so
// that dX = conv3x3(dZ, Wf) equals col2im of dZ W.
__global__ void flip3x3_kernel(const bf16* __restrict__ W, bf16* __restrict__ Wf, int Cout, int C) {
  const long total = 9L * C * Cout;
  GRID_STRIDE(i, total) {
    const int co = (int)(i % Cout);
    const long r = i / Cout;
    const int t = (int)(r % 9), c = (int)(r / 9);
    Wf[i] = W[(long)co * 9 * C + (8 - t) * C + c];
  }
}

__global__ void transpose_kernel(const bf16* __restrict__ in, bf16* __restrict__ out, long R, long Cc) {
  GRID_STRIDE(i, R * Cc) {
    const long r = i % R, c = i / R;
    out[c * R + r] = in[r * Cc + c];
  }
}

__global__ void relu_bwd_kernel(const bf16* __restrict__ y, const bf16* __restrict__ dy, bf16* __restrict__ dz, long n) {
  GRID_STRIDE(i, n) dz[i] = __bfloat162float(y[i]) > 0.f ? dy[i] : __float2bfloat16(0.f);
}

__global__ void avgpool_kernel(const bf16* __restrict__ X, bf16* __restrict__ Y, int B, int H, int W, int C) {
  const int Ho = H / 2, Wo = W / 2;
  GRID_STRIDE(i, (long)B * Ho * Wo * C) {
    const int c = (int)(i % C);
    const long p = i / C;
    const int x = (int)(p % Wo), y = (int)((p / Wo) % Ho);
    const long b = p / ((long)Wo * Ho);
    const bf16* s = X + ((b * H + 2 * y) * W + 2 * x) * C + c;
    const float v = __bfloat162float(s[0]) + __bfloat162float(s[C]) + __bfloat162float(s[(long)W * C]) +
                    __bfloat162float(s[(long)W * C + C]);
    Y[i] = __float2bfloat16_rn(0.25f * v);
  }
}

__global__ void avgpool_bwd_kernel(const bf16* __restrict__ dY, bf16* __restrict__ dX, int B, int H, int W, int C) {
  GRID_STRIDE(i, (long)B * H * W * C) {
    const int c = (int)(i % C);
    const long p = i / C;
    const int x = (int)(p % W), y = (int)((p / W) % H);
    const long b = p / ((long)W * H);
    dX[i] = __float2bfloat16_rn(0.25f * __bfloat162float(dY[((b * (H / 2) + y / 2) * (W / 2) + x / 2) * C + c]));
  }
}

// Y = upsample2(X) + S (nearest neighbour, additive skip).
__global__ void upsample_add_kernel(const bf16* __restrict__ X, const bf16* __restrict__ S, bf16* __restrict__ Y,
                                    int B, int H, int W, int C) {
  GRID_STRIDE(i, (long)B * H * W * C) {
    const int c = (int)(i % C);
    const long p = i / C;
    const int x = (int)(p % W), y = (int)((p / W) % H);
    const long b = p / ((long)W * H);
    const float v = __bfloat162float(X[((b * (H / 2) + y / 2) * (W / 2) + x / 2) * C + c]) + __bfloat162float(S[i]);
    Y[i] = __float2bfloat16_rn(v);
  }
}

// dX = sum over the 2x2 block of dY (gradient of nearest upsampling).
__global__ void upsample_bwd_kernel(const bf16* __restrict__ dY, bf16* __restrict__ dX, int B, int H, int W, int C) {
  GRID_STRIDE(i, (long)B * H * W * C) {
    const int c = (int)(i % C);
    const long p = i / C;
    const int x = (int)(p % W), y = (int)((p / W) % H);
    const long b = p / ((long)W * H);
    const long W2 = 2L * W;
    const bf16* s = dY + ((b * 2 * H + 2 * y) * W2 + 2 * x) * C + c;
    const float v = __bfloat162float(s[0]) + __bfloat162float(s[C]) + __bfloat162float(s[W2 * C]) +
                    __bfloat162float(s[W2 * C + C]);
    dX[i] = __float2bfloat16_rn(v);
  }
}

__global__ void add_kernel(const bf16* __restrict__ a, const bf16* __restrict__ b, bf16* __restrict__ out, long n) {
  GRID_STRIDE(i, n) out[i] = __float2bfloat16_rn(__bfloat162float(a[i]) + __bfloat162float(b[i]));
}

// out[p][c] = a[p] * w[c] (BF16): data gradient of a 1x1 convolution to one channel.
__global__ void outer_kernel(const bf16* __restrict__ a, const float* __restrict__ w, bf16* __restrict__ out, long P,
                             int C) {
  GRID_STRIDE(i, P * C) out[i] = __float2bfloat16_rn(__bfloat162float(a[i / C]) * w[i % C]);
}

__global__ void f32_to_bf16_kernel(const float* __restrict__ in, bf16* __restrict__ out, long n) {
  GRID_STRIDE(i, n) out[i] = __float2bfloat16_rn(in[i]);
}

// out[i] = sum_j part[j * n + i], fixed order.
__global__ void sum_slices_kernel(const float* __restrict__ part, int slices, float* __restrict__ out, long n) {
  GRID_STRIDE(i, n) {
    float s = 0.f;
    for (int j = 0; j < slices; ++j) s += part[(long)j * n + i];
    out[i] = s;
  }
}

// colsum[c] = sum_p in[p][c] for BF16 in [P][C]: one CTA per channel, fixed order.
__global__ void colsum_kernel(const bf16* __restrict__ in, long P, int C, float* __restrict__ out) {
  __shared__ float sh[kT / 32];
  const int c = blockIdx.x;
  float s = 0.f;
  for (long p = threadIdx.x; p < P; p += blockDim.x) s += __bfloat162float(in[p * C + c]);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int w = 0; w < kT / 32; ++w) t += sh[w];
    out[c] = t;
  }
}

// Masked MSE on [B][S][S] predictions (interior m x m region, m <= S):
// per-CTA partial sums of squared errors and the gradient 2 (pred - tgt) / count.
__global__ void mse_kernel(const float* __restrict__ pred, const float* __restrict__ tgt, int B, int S, int m,
                           bf16* __restrict__ grad, float* __restrict__ partial) {
  __shared__ float sh[kT / 32];
  const long total = (long)B * S * S;
  const float inv = 2.f / ((float)B * m * m);
  float acc = 0.f;
  GRID_STRIDE(i, total) {
    const int x = (int)(i % S), y = (int)((i / S) % S);
    float g = 0.f;
    if (x < m && y < m) {
      const float d = pred[i] - tgt[i];
      acc += d * d;
      g = inv * d;
    }
    grad[i] = __float2bfloat16_rn(g);
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int w = 0; w < kT / 32; ++w) t += sh[w];
    partial[blockIdx.x] = t;
  }
}

// AdamW on FP32 master weights; BF16 copy refreshed.
__global__ void adamw_kernel(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m1,
                             float* __restrict__ m2, bf16* __restrict__ w16, long n, float lr, float b1, float b2,
                             float eps, float wd, float bc1, float bc2) {
  GRID_STRIDE(i, n) {
    const float gi = g[i];
    const float a = b1 * m1[i] + (1.f - b1) * gi;
    const float b = b2 * m2[i] + (1.f - b2) * gi * gi;
    m1[i] = a;
    m2[i] = b;
    float wi = w[i] * (1.f - lr * wd);
    wi -= lr * (a / bc1) / (sqrtf(b / bc2) + eps);
    w[i] = wi;
    if (w16) w16[i] = __float2bfloat16_rn(wi);
  }
}

// ---- eight channels (16 bytes) per thread -------------------------------------
// The layer kernels between the convolutions move activations once, so they
// are bound by memory; a thread takes one 16-byte chunk (8 channels of a
// pixel) with 32-bit index arithmetic.  One channel per thread with 64-bit
// divisions took 50 us where the bytes take 10 (upsampling to 256^2 x 32,
// batch 8).
struct alignas(16) B8 {
  __nv_bfloat162 v[4];
};
__device__ __forceinline__ B8 ldb(const bf16* p) { return *reinterpret_cast<const B8*>(p); }
__device__ __forceinline__ void stb(bf16* p, const B8& x) { *reinterpret_cast<B8*>(p) = x; }
__device__ __forceinline__ void widen(const B8& x, float (&f)[8]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float2 t = __bfloat1622float2(x.v[k]);
    f[2 * k] = t.x;
    f[2 * k + 1] = t.y;
  }
}
__device__ __forceinline__ B8 narrow(const float (&f)[8]) {
  B8 x;
#pragma unroll
  for (int k = 0; k < 4; ++k) x.v[k] = __floats2bfloat162_rn(f[2 * k], f[2 * k + 1]);
  return x;
}
// Chunk i of [B][H][W][C8]: its pixel and channel group.
struct Chunk {
  unsigned c8, x, y, b;
  __device__ __forceinline__ Chunk(unsigned i, unsigned H, unsigned W, unsigned C8) {
    c8 = i % C8;
    const unsigned p = i / C8, r = p / W;
    x = p - r * W;
    b = r / H;
    y = r - b * H;
  }
};
__device__ __forceinline__ size_t at(unsigned b, unsigned y, unsigned x, unsigned c8, unsigned H, unsigned W,
                                     unsigned C8) {
  return ((((size_t)b * H + y) * W + x) * C8 + c8) * 8;
}
// Sum of the 2 x 2 block at (2 y, 2 x), in the order of the scalar kernels.
__device__ __forceinline__ void block_sum(const bf16* X, const Chunk& c, unsigned H2, unsigned W2, unsigned C8,
                                          float (&v)[8]) {
  const bf16* s = X + at(c.b, 2 * c.y, 2 * c.x, c.c8, H2, W2, C8);
  float f0[8], f1[8], f2[8], f3[8];
  widen(ldb(s), f0);
  widen(ldb(s + C8 * 8), f1);
  widen(ldb(s + (size_t)W2 * C8 * 8), f2);
  widen(ldb(s + ((size_t)W2 + 1) * C8 * 8), f3);
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] = f0[k] + f1[k] + f2[k] + f3[k];
}

__global__ void __launch_bounds__(kT) avgpool8_kernel(const bf16* __restrict__ X, bf16* __restrict__ Y, unsigned Ho,
                                                      unsigned Wo, unsigned C8, unsigned total) {
  pdl_enter();
  const unsigned i = blockIdx.x * kT + threadIdx.x;
  if (i >= total) return;
  const Chunk c(i, Ho, Wo, C8);
  float v[8];
  block_sum(X, c, 2 * Ho, 2 * Wo, C8, v);
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] *= 0.25f;
  stb(Y + (size_t)i * 8, narrow(v));
}

__global__ void __launch_bounds__(kT) upsample_add8_kernel(const bf16* __restrict__ X, const bf16* __restrict__ S,
                                                           bf16* __restrict__ Y, unsigned H, unsigned W, unsigned C8,
                                                           unsigned total) {
  pdl_enter();
  const unsigned i = blockIdx.x * kT + threadIdx.x;
  if (i >= total) return;
  const Chunk c(i, H, W, C8);
  float a[8], v[8];
  widen(ldb(X + at(c.b, c.y / 2, c.x / 2, c.c8, H / 2, W / 2, C8)), a);
  widen(ldb(S + (size_t)i * 8), v);
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] = a[k] + v[k];
  stb(Y + (size_t)i * 8, narrow(v));
}

// launch_grad_act (cmg_internal.h).  A thread's chunks share their channel
// group (the stride is a multiple of C8), so the column sums are eight
// running FP32 sums per thread, then the CTA's in a fixed order.  One pass
// instead of four or five (the gradient of the resampling, the skip's sum, the ReLU mask,
// the bias gradient, whose column sums took one CTA per channel: 242 us at
// 256^2 x 32).
template <int MODE>
__global__ void __launch_bounds__(kT) grad_act_kernel(const bf16* __restrict__ y, const bf16* __restrict__ dA,
                                                      const bf16* __restrict__ dB, const float* __restrict__ w,
                                                      bf16* __restrict__ dZ, unsigned H, unsigned W, unsigned C8,
                                                      unsigned total, float* __restrict__ rows, int width) {
  pdl_enter();
  __shared__ float sh[kT][9];
  float sum[8] = {}, hsum[8] = {}, dsum = 0.f, wc[8];
  const unsigned c8 = threadIdx.x % C8;
  if (MODE == kGradHead) {
#pragma unroll
    for (int k = 0; k < 8; ++k) wc[k] = w[c8 * 8 + k];
  }
  for (unsigned i = blockIdx.x * kT + threadIdx.x; i < total; i += gridDim.x * kT) {
    float v[8], yv[8];
    widen(ldb(y + (size_t)i * 8), yv);
    if (MODE == kGradDirect) {
      widen(ldb(dA + (size_t)i * 8), v);
    } else if (MODE == kGradHead) {
      const float d = __bfloat162float(dA[i / C8]);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        v[k] = d * wc[k];
        hsum[k] = fmaf(d, yv[k], hsum[k]);
      }
      if (c8 == 0) dsum += d;
    } else {
      const Chunk c(i, H, W, C8);
      if (MODE == kGradUpsample) {
        block_sum(dA, c, 2 * H, 2 * W, C8, v);
      } else {
        float a[8];
        widen(ldb(dA + at(c.b, c.y / 2, c.x / 2, c.c8, H / 2, W / 2, C8)), a);
        widen(ldb(dB + (size_t)i * 8), v);
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = __bfloat162float(__float2bfloat16_rn(0.25f * a[k])) + v[k];
      }
    }
    B8 o = narrow(v);
    widen(o, v);
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = yv[k] > 0.f ? v[k] : 0.f;
    stb(dZ + (size_t)i * 8, narrow(v));
#pragma unroll
    for (int k = 0; k < 8; ++k) sum[k] += v[k];
  }
  // CTA sums: thread t < 8 C8 adds channel t over the threads of its group
  const auto reduce = [&](const float (&a)[8], int col) {
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 8; ++k) sh[threadIdx.x][k] = a[k];
    __syncthreads();
    if (threadIdx.x < 8 * C8) {
      const unsigned g = threadIdx.x / 8, k = threadIdx.x % 8;
      float t = 0.f;
      for (unsigned r = g; r < kT; r += C8) t += sh[r][k];
      rows[(size_t)blockIdx.x * width + col + threadIdx.x] = t;
    }
  };
  reduce(sum, 0);
  if (MODE == kGradHead) {
    reduce(hsum, 8 * C8);
    const float one[8] = {dsum};
    __syncthreads();
    sh[threadIdx.x][8] = one[0];
    __syncthreads();
    if (threadIdx.x == 0) {
      float t = 0.f;
      for (unsigned r = 0; r < kT; r += C8) t += sh[r][8];
      rows[(size_t)blockIdx.x * width + 16 * C8] = t;
    }
  }
}

// launch_finish_layer.  CTAs 0 .. : 32 entries of gw each, eight threads per
// entry over the slices; the last CTA: the columns of rows, a warp per column.
__global__ void __launch_bounds__(kT) finish_layer_kernel(const float* __restrict__ part, int slices,
                                                          float* __restrict__ gw, int n, int gblocks,
                                                          const float* __restrict__ rows, int nrows, int width,
                                                          float* __restrict__ gb, int C, float* __restrict__ hw,
                                                          float* __restrict__ hb) {
  pdl_enter();
  const int lane = threadIdx.x & 31, wy = threadIdx.x >> 5;
  if ((int)blockIdx.x < gblocks) {
    __shared__ float sh[8][33];
    const int e = blockIdx.x * 32 + lane;
    float t = 0.f;
    if (e < n) {
#pragma unroll 4
      for (int z = wy; z < slices; z += 8) t += part[(size_t)z * n + e];
    }
    sh[wy][lane] = t;
    __syncthreads();
    if (wy == 0 && e < n) {
      for (int k = 1; k < 8; ++k) t += sh[k][lane];
      gw[e] = t;
    }
    return;
  }
  const int col = ((int)blockIdx.x - gblocks) * 8 + wy;
  if (col >= width) return;
  float t = 0.f;
  for (int r = lane; r < nrows; r += 32) t += rows[(size_t)r * width + col];
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (lane == 0) {
    if (col < C) gb[col] = t;
    else if (col < 2 * C) hw[col - C] = t;
    else hb[col - 2 * C] = t;
  }
}

// Network input with eight channels: one 16-byte store per pixel.
__global__ void __launch_bounds__(kT) pack_input8_kernel(const double* __restrict__ f0, const double* __restrict__ f1,
                                                         unsigned n, unsigned S, float s0, float s1,
                                                         bf16* __restrict__ X, unsigned total) {
  const unsigned i = blockIdx.x * kT + threadIdx.x;
  if (i >= total) return;
  const Chunk c(i, S, S, 1);
  float v[8] = {};
  if (c.x < n && c.y < n) {
    const size_t node = ((size_t)c.b * n + c.y) * n + c.x;
    v[0] = s0 * (float)f0[node];
    v[1] = s1 * (float)f1[node];
  }
  stb(X + (size_t)i * 8, narrow(v));
}

// Network input [B][S][S][Cp] from two n x n FP64 fields per image (channel 0
// and 1, scaled), zero elsewhere (channels >= 2 and pixels beyond n).
__global__ void pack_input_kernel(const double* __restrict__ f0, const double* __restrict__ f1, int B, int n, int S,
                                  int Cp, float s0, float s1, bf16* __restrict__ X) {
  GRID_STRIDE(i, (long)B * S * S * Cp) {
    const int c = (int)(i % Cp);
    const long p = i / Cp;
    const int x = (int)(p % S), y = (int)((p / S) % S);
    const long b = p / ((long)S * S);
    float v = 0.f;
    if (x < n && y < n && c < 2) {
      const long node = b * (long)n * n + (long)y * n + x;
      v = c == 0 ? s0 * (float)f0[node] : s1 * (float)f1[node];
    }
    X[i] = __float2bfloat16_rn(v);
  }
}

// [B][S][S] FP32 images -> [B][n*n] FP64 (times scale), the inverse of the packing.
__global__ void unpack_output_kernel(const float* __restrict__ img, int B, int n, int S, double scale,
                                     double* __restrict__ out) {
  GRID_STRIDE(i, (long)B * n * n) {
    const int x = (int)(i % n), y = (int)((i / n) % n);
    const long b = i / ((long)n * n);
    out[i] = scale * (double)img[(b * S + y) * S + x];
  }
}

// [B][n*n] FP64 -> [B][S][S] FP32 images (times scale, zero padding).
__global__ void pack_target_kernel(const double* __restrict__ u, int B, int n, int S, double scale,
                                   float* __restrict__ img) {
  GRID_STRIDE(i, (long)B * S * S) {
    const int x = (int)(i % S), y = (int)((i / S) % S);
    const long b = i / ((long)S * S);
    img[i] = (x < n && y < n) ? (float)(scale * u[b * (long)n * n + (long)y * n + x]) : 0.f;
  }
}

}  // namespace
}  // namespace cmg

using namespace cmg;

namespace {
inline cmg_status done(int launches) {
  count_launches(launches);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? CMG_OK : CMG_ERR_CUDA;
}
inline cudaStream_t st(void* s) { return static_cast<cudaStream_t>(s); }
// 16-byte chunks of 8 channels, 32-bit chunk indices (also past the last CTA)
inline bool chunked(long long n, int C, const void* a, const void* b, const void* c) {
  return C % 8 == 0 && n / 8 < (1LL << 31) &&
         ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b) | reinterpret_cast<uintptr_t>(c)) & 15) == 0;
}
inline cmg_status launched(cudaError_t e) {
  count_launches(1);
  if (e == cudaSuccess) e = cudaGetLastError();
  return e == cudaSuccess ? CMG_OK : CMG_ERR_CUDA;
}
inline dim3 ctas(long long n) { return dim3((unsigned)((n + kT - 1) / kT)); }
}  // namespace

namespace cmg {

cudaError_t launch_grad_act(int mode, const void* y, const void* dA, const void* dB, const float* w, void* dZ, int B,
                            int H, int W, int C, float* rows, int* nrows, cudaStream_t s) {
  const long total = (long)B * H * W * (C / 8);
  if ((C != 32 && C != 64) || total >= (1L << 31)) return cudaErrorNotSupported;
  const long want = (total + kT - 1) / kT;
  const unsigned grid = (unsigned)(want < kGradRows ? want : kGradRows);
  *nrows = (int)grid;
  const int width = mode == kGradHead ? 2 * C + 1 : C;
  const auto go = [&](auto* k) {
    return launch_k(k, dim3(grid), dim3(kT), 0, s, (const bf16*)y, (const bf16*)dA, (const bf16*)dB, w, (bf16*)dZ,
                    (unsigned)H, (unsigned)W, (unsigned)(C / 8), (unsigned)total, rows, width);
  };
  count_launches(1);
  switch (mode) {
    case kGradDirect: return go(grad_act_kernel<kGradDirect>);
    case kGradUpsample: return go(grad_act_kernel<kGradUpsample>);
    case kGradPoolSkip: return go(grad_act_kernel<kGradPoolSkip>);
    case kGradHead: return go(grad_act_kernel<kGradHead>);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_finish_layer(const float* part, int slices, float* gw, int n, const float* rows, int nrows, int width,
                                float* gb, int C, float* hw, float* hb, cudaStream_t s) {
  const int gblocks = (n + 31) / 32, cblocks = (width + 7) / 8;
  count_launches(1);
  return launch_k(finish_layer_kernel, dim3((unsigned)(gblocks + cblocks)), dim3(kT), 0, s, part, slices, gw, n, gblocks,
                  rows, nrows, width, gb, C, hw, hb);
}

}  // namespace cmg

extern "C" {

cmg_status cmg_nn_im2col(const void* X, void* col, int B, int H, int W, int C, int transposed, void* stream) {
  if (!X || !col || B < 1 || H < 1 || W < 1 || C < 8 || C % 8) return CMG_ERR_INVALID_ARG;
  if (transposed)
    im2col_t_kernel<<<blocks((long)B * H * W * 9 * C), kT, 0, st(stream)>>>((const bf16*)X, (bf16*)col, B, H, W, C);
  else
    im2col_kernel<<<blocks((long)B * H * W * 9 * C / 8), kT, 0, st(stream)>>>((const bf16*)X, (bf16*)col, B, H, W, C);
  return done(1);
}

cmg_status cmg_nn_col2im(const float* dcol, void* dX, int B, int H, int W, int C, void* stream) {
  if (!dcol || !dX || B < 1 || H < 1 || W < 1 || C < 1) return CMG_ERR_INVALID_ARG;
  col2im_kernel<<<blocks((long)B * H * W * C), kT, 0, st(stream)>>>(dcol, (bf16*)dX, B, H, W, C);
  return done(1);
}

cmg_status cmg_nn_transpose(const void* in, void* out, long long R, long long Cc, void* stream) {
  if (!in || !out || R < 1 || Cc < 1) return CMG_ERR_INVALID_ARG;
  transpose_kernel<<<blocks(R * Cc), kT, 0, st(stream)>>>((const bf16*)in, (bf16*)out, R, Cc);
  return done(1);
}

cmg_status cmg_nn_flip3x3(const void* W, void* Wf, int Cout, int C, void* stream) {
  if (!W || !Wf || Cout < 1 || C < 1) return CMG_ERR_INVALID_ARG;
  flip3x3_kernel<<<blocks(9L * C * Cout), kT, 0, st(stream)>>>((const bf16*)W, (bf16*)Wf, Cout, C);
  return done(1);
}

cmg_status cmg_nn_relu_bwd(const void* y, const void* dy, void* dz, long long n, void* stream) {
  if (!y || !dy || !dz || n < 1) return CMG_ERR_INVALID_ARG;
  relu_bwd_kernel<<<blocks(n), kT, 0, st(stream)>>>((const bf16*)y, (const bf16*)dy, (bf16*)dz, n);
  return done(1);
}

cmg_status cmg_nn_avgpool(const void* X, void* Y, int B, int H, int W, int C, int backward, void* stream) {
  if (!X || !Y || B < 1 || H < 2 || W < 2 || (H | W) & 1 || C < 1) return CMG_ERR_INVALID_ARG;
  if (backward)   // X = dY [B][H/2][W/2][C], Y = dX [B][H][W][C]
    avgpool_bwd_kernel<<<blocks((long)B * H * W * C), kT, 0, st(stream)>>>((const bf16*)X, (bf16*)Y, B, H, W, C);
  else if (chunked((long long)B * H * W * C / 4, C, X, Y, Y))
    return launched(launch_k(avgpool8_kernel, ctas((long long)B * H * W * C / 32), dim3(kT), 0, st(stream),
                             (const bf16*)X, (bf16*)Y, (unsigned)(H / 2), (unsigned)(W / 2), (unsigned)(C / 8),
                             (unsigned)((long long)B * H * W * C / 32)));
  else
    avgpool_kernel<<<blocks((long)B * H * W * C / 4), kT, 0, st(stream)>>>((const bf16*)X, (bf16*)Y, B, H, W, C);
  return done(1);
}

cmg_status cmg_nn_upsample_add(const void* X, const void* S, void* Y, int B, int H, int W, int C, void* stream) {
  if (!X || !S || !Y || B < 1 || H < 2 || W < 2 || (H | W) & 1 || C < 1) return CMG_ERR_INVALID_ARG;
  if (chunked((long long)B * H * W * C, C, X, S, Y))
    return launched(launch_k(upsample_add8_kernel, ctas((long long)B * H * W * C / 8), dim3(kT), 0, st(stream),
                             (const bf16*)X, (const bf16*)S, (bf16*)Y, (unsigned)H, (unsigned)W, (unsigned)(C / 8),
                             (unsigned)((long long)B * H * W * C / 8)));
  upsample_add_kernel<<<blocks((long)B * H * W * C), kT, 0, st(stream)>>>((const bf16*)X, (const bf16*)S, (bf16*)Y, B,
                                                                          H, W, C);
  return done(1);
}

cmg_status cmg_nn_upsample_bwd(const void* dY, void* dX, int B, int H, int W, int C, void* stream) {
  if (!dY || !dX || B < 1 || H < 1 || W < 1 || C < 1) return CMG_ERR_INVALID_ARG;
  upsample_bwd_kernel<<<blocks((long)B * H * W * C), kT, 0, st(stream)>>>((const bf16*)dY, (bf16*)dX, B, H, W, C);
  return done(1);
}

cmg_status cmg_nn_add(const void* a, const void* b, void* out, long long n, void* stream) {
  if (!a || !b || !out || n < 1) return CMG_ERR_INVALID_ARG;
  add_kernel<<<blocks(n), kT, 0, st(stream)>>>((const bf16*)a, (const bf16*)b, (bf16*)out, n);
  return done(1);
}

cmg_status cmg_nn_outer(const void* a, const float* w, void* out, long long P, int C, void* stream) {
  if (!a || !w || !out || P < 1 || C < 1) return CMG_ERR_INVALID_ARG;
  outer_kernel<<<blocks(P * C), kT, 0, st(stream)>>>((const bf16*)a, w, (bf16*)out, P, C);
  return done(1);
}

cmg_status cmg_nn_to_bf16(const float* in, void* out, long long n, void* stream) {
  if (!in || !out || n < 1) return CMG_ERR_INVALID_ARG;
  f32_to_bf16_kernel<<<blocks(n), kT, 0, st(stream)>>>(in, (bf16*)out, n);
  return done(1);
}

cmg_status cmg_nn_sum_slices(const float* part, int slices, float* out, long long n, void* stream) {
  if (!part || !out || slices < 1 || n < 1) return CMG_ERR_INVALID_ARG;
  sum_slices_kernel<<<blocks(n), kT, 0, st(stream)>>>(part, slices, out, n);
  return done(1);
}

cmg_status cmg_nn_colsum(const void* in, long long P, int C, float* out, void* stream) {
  if (!in || !out || P < 1 || C < 1) return CMG_ERR_INVALID_ARG;
  colsum_kernel<<<C, kT, 0, st(stream)>>>((const bf16*)in, P, C, out);
  return done(1);
}

cmg_status cmg_nn_mse(const float* pred, const float* tgt, int B, int S, int m, void* grad, float* partial,
                      int max_partials, int* used_partials, void* stream) {
  if (!pred || !tgt || !grad || !partial || !used_partials || B < 1 || S < 1 || m < 1 || m > S)
    return CMG_ERR_INVALID_ARG;
  const unsigned g = blocks((long)B * S * S);
  if ((int)g > max_partials) return CMG_ERR_INVALID_ARG;
  mse_kernel<<<g, kT, 0, st(stream)>>>(pred, tgt, B, S, m, (bf16*)grad, partial);
  *used_partials = (int)g;
  return done(1);
}

cmg_status cmg_nn_adamw(float* w, const float* g, float* m1, float* m2, void* w16, long long n, float lr, float b1,
                        float b2, float eps, float wd, int step, void* stream) {
  if (!w || !g || !m1 || !m2 || n < 1 || step < 1) return CMG_ERR_INVALID_ARG;
  const float bc1 = 1.f - powf(b1, (float)step), bc2 = 1.f - powf(b2, (float)step);
  adamw_kernel<<<blocks(n), kT, 0, st(stream)>>>(w, g, m1, m2, (bf16*)w16, n, lr, b1, b2, eps, wd, bc1, bc2);
  return done(1);
}

cmg_status cmg_nn_pack_input(const double* f0, const double* f1, int B, int n, int S, int Cp, float s0, float s1,
                             void* X, void* stream) {
  if (!f0 || !f1 || !X || B < 1 || n < 1 || S < n || Cp < 2) return CMG_ERR_INVALID_ARG;
  if (chunked((long long)B * S * S * Cp, Cp, X, X, X) && Cp == 8) {
    const long long total = (long long)B * S * S;
    pack_input8_kernel<<<ctas(total), kT, 0, st(stream)>>>(f0, f1, (unsigned)n, (unsigned)S, s0, s1, (bf16*)X,
                                                           (unsigned)total);
    return done(1);
  }
  pack_input_kernel<<<blocks((long)B * S * S * Cp), kT, 0, st(stream)>>>(f0, f1, B, n, S, Cp, s0, s1, (bf16*)X);
  return done(1);
}

cmg_status cmg_nn_unpack_output(const float* img, int B, int n, int S, double scale, double* out, void* stream) {
  if (!img || !out || B < 1 || n < 1 || S < n) return CMG_ERR_INVALID_ARG;
  unpack_output_kernel<<<blocks((long)B * n * n), kT, 0, st(stream)>>>(img, B, n, S, scale, out);
  return done(1);
}

cmg_status cmg_nn_pack_target(const double* u, int B, int n, int S, double scale, float* img, void* stream) {
  if (!u || !img || B < 1 || n < 1 || S < n) return CMG_ERR_INVALID_ARG;
  pack_target_kernel<<<blocks((long)B * S * S), kT, 0, st(stream)>>>(u, B, n, S, scale, img);
  return done(1);
}

}  // extern "C"
