// 3x3 convolutions of the warm-start network (NHWC BF16, zero padding 1) on
// the 5th-generation tensor cores, reading each input pixel once per tile.
//
// conv3x3_patch_kernel: a CTA walks tiles of 8 x 16 output pixels (the 128 rows of a
// tcgen05.mma) and holds the whole weight matrix in shared memory.  A tile's
// input is the 10 x 18 pixel patch around it, kept as one plane of 16-byte
// chunks (8 channels of a pixel) per 8 input channels.  In the no-swizzle
// core-matrix layout a core matrix is eight 16-byte rows in a line, here
// eight neighbouring pixels of an image row, and the next eight MMA rows are
// the next image row, 10 chunks on; so the operand of filter tap (dy, dx) is
// the same patch read from chunk 10 dy + dx on.  The nine taps are nine start
// addresses, and no patch matrix is built, in memory or in shared memory.
//
// Why: what bounds these layers is how often the activations cross into
// shared memory.  The im2col tensor map (cmg_nn_gemm.cu) brings each pixel
// in nine times, in boxes of 16 to 128 bytes; the patch brings it in 1.4 times
// (180 pixels for 128), by cp.async, each of four producer warps a whole
// patch at a time.  Now the tensor cores' own operand reads are the limit: an
// MMA of 128 x 64 x 16 reads 6 KB, 48 of the 50 cycles it takes, and while a
// tile's queued MMAs drain the other roles' shared-memory accesses wait
// (about 650 cycles per tile), with some 5 us to start (weights, first patch).  Batch 8, ReLU layers,
// im2col map -> patch: 256^2 8->32 81 -> 16 us, 32->32 74 -> 28, 128^2 64->64
// 28 -> 22, 32->64 27 -> 15.
//
// K runs tap by tap, then over the channels, 16 per MMA: the order of the
// im2col GEMM, hence its bits (tests/test_gpu_nn_conv.py).
//
// TB: the data gradient.  dX is the convolution of dZ with the taps turned by
// 180 degrees and the channels exchanged; the weight matrix is read in its
// forward layout and presented as an MN-major operand, so no turned copy is
// made.
#include <cuda_bf16.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>

#include "cmg_common.cuh"
#include "cmg_nn_mma.cuh"

namespace cmg {
namespace nn {
namespace {

constexpr int kPW = 8, kPH = 16;                         // output pixels of a tile
constexpr int kIW = kPW + 2, kIH = kPH + 2;              // its input patch
constexpr int kPatch = kIW * kIH;                        // 180 pixels
constexpr int kProd = 128;                               // producer threads (warps 0-3), then the MMA warp, then
constexpr int kEpi = 256;                                // two epilogue groups of four warps (one per TMEM lane
constexpr int kConvThreads = kProd + 32 + kEpi;          // quadrant), taking alternate tiles
constexpr int kAcc = 4;                                  // patches in shared memory, and accumulators

// Chunks from one plane to the next: odd multiples so that the producers'
// writes (consecutive channels of a pixel in consecutive lanes) spread over
// the banks.
constexpr uint32_t patch_pitch(int c8) { return (c8 == 8 ? 181u : 182u) * 16u; }

__device__ __forceinline__ void cp16(uint32_t dst, const void* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
__device__ __forceinline__ void fence_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// The two words of a no-swizzle descriptor (smem_desc): address and leading
// offset, stride offset and version; and the MMA that takes them.
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr, uint32_t lbo) { return ((addr & 0x3FFFF) >> 4) | (lbo >> 4) << 16; }
__device__ __forceinline__ uint32_t desc_hi(uint32_t sbo) { return (sbo >> 4) | 1u << 14; }
__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint32_t alo, uint32_t ahi, uint32_t blo, uint32_t bhi,
                                         uint32_t idesc, bool accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n .reg .b64 da, db;\n mov.b64 da, {%1, %2};\n mov.b64 db, {%3, %4};\n setp.ne.u32 p, %6, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n}\n" ::"r"(tmem_d),
      "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc), "r"((uint32_t)accumulate)
      : "memory");
}

// Tiles of an image batch; tile t is image t / (tx ty), row band, column.
struct Tiles {
  int B, H, W, tx, ty, count;
};
__device__ __forceinline__ void tile_pos(const Tiles& g, int t, int& b, int& y0, int& x0) {
  const int per = g.tx * g.ty;
  b = t / per;
  const int r = t - b * per;
  const int ty = r / g.tx;
  y0 = ty * kPH;
  x0 = (r - ty * g.tx) * kPW;
}

// One warp brings the 10 x 18 x C patch around tile (y0, x0) of image b into
// planes of pitch `pitch`: a 16-byte asynchronous copy per chunk, zeros
// outside the image (a copy of size 0 from the valid base address).  A lane
// keeps to one channel group and walks the patch 32 / C8 pixels at a time.
template <int C8>
__device__ __forceinline__ void load_patch(uint32_t dst, uint32_t pitch, const __nv_bfloat16* __restrict__ X,
                                           const Tiles& g, int b, int y0, int x0, int lane) {
  constexpr int kStep = 32 / C8, kRows = kStep / kIW, kCols = kStep % kIW;   // a step in rows and columns
  constexpr int kN = (kPatch + kStep - 1) / kStep;
  const int c8 = lane % C8, px0 = lane / C8;
  int py = px0 / kIW, pc = px0 - py * kIW;
  const long row = (long)g.W * (C8 * 8);
  const __nv_bfloat16* src = X + (((long)b * g.H + y0 + py - 1) * g.W + x0 + pc - 1) * (C8 * 8) + c8 * 8;
  dst += c8 * pitch + px0 * 16;
  const bool interior = y0 > 0 && x0 > 0 && y0 + kPH < g.H && x0 + kPW < g.W;
#pragma unroll 4
  for (int i = 0; i < kN; ++i) {
    const bool ok = interior || ((unsigned)(y0 + py - 1) < (unsigned)g.H && (unsigned)(x0 + pc - 1) < (unsigned)g.W);
    if ((i + 1) * kStep <= kPatch || px0 + i * kStep < kPatch) cp16(dst + i * kStep * 16, ok ? src : X, ok);
    src += kRows * row + kCols * (C8 * 8);
    py += kRows;
    pc += kCols;
    if (pc >= kIW) {
      pc -= kIW;
      ++py;
      src += row - kIW * (C8 * 8);
    }
  }
}

// Store of 32 bytes (16 BF16) to a 32-byte aligned address: a whole sector.
__device__ __forceinline__ void st32(void* p, const uint32_t* v) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]),
               "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}

// One warp brings 128 pixels of C8 channel groups into planes of pitch
// `pitch`; where(px, src) gives pixel px's address, or false for zeros.
template <int C8, typename Where>
__device__ __forceinline__ void load_pixels(uint32_t dst, uint32_t pitch, const __nv_bfloat16* __restrict__ X, int lane,
                                            Where where) {
  constexpr int kStep = 32 / C8;
  const int c8 = lane % C8, px0 = lane / C8;
#pragma unroll 4
  for (int i = 0; i < 128 / kStep; ++i) {
    const int px = px0 + i * kStep;
    long p;
    const bool ok = where(px, p);
    cp16(dst + c8 * pitch + px * 16, ok ? X + p * (C8 * 8) + c8 * 8 : X, ok);
  }
}

template <int C, int NP>
struct ConvTile {
  static constexpr int C8 = C / 8;
  static constexpr uint32_t kPitch = patch_pitch(C8);
  static constexpr uint32_t kStage = C8 * kPitch;
  static constexpr int kPlanesB = C == 8 ? 10 : 9 * C8;   // C = 8: tap 9 pairs with a plane of zeros
  static constexpr uint32_t kPitchB = (NP + 1) * 16;      // odd chunk count: the loaders' plane-wise writes spread over the banks
  static constexpr uint32_t kBf = kPlanesB * kPitchB, kBt = 9u * (NP / 8) * (C + 1) * 16;   // forward, turned
  static constexpr uint32_t kB = kBf > kBt ? kBf : kBt;
  static constexpr uint32_t kZero = C == 8 ? kPitch : 0;  // zeros that stand for tap 9's pixels
  static constexpr int S = kAcc;
  static constexpr int kSmem = (int)(kB + S * kStage + kZero);
  static constexpr uint32_t kCols = kAcc * NP;
  // CTAs that fit an SM beside each other (shared memory; TMEM holds 512 columns)
  static constexpr int kFit = 227 * 1024 / (kSmem + 1536);
  static constexpr int kCtas = kFit > 2 ? 2 : kFit;
  static_assert(kCtas >= 1 && kCtas * (int)kCols <= 512, "shared memory and TMEM of an SM");
};

template <int C, int NP, bool TB>
__global__ void __launch_bounds__(kConvThreads)
    conv3x3_patch_kernel(const __nv_bfloat16* __restrict__ X, Tiles g, const __nv_bfloat16* __restrict__ Wt, int Cout,
                         const float* __restrict__ bias, int relu, __nv_bfloat16* __restrict__ Y, int vec,
                         int* __restrict__ status, long long wlimit, int early) {
  using T = ConvTile<C, NP>;
  constexpr int C8 = T::C8, S = T::S;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t full[S], done[S], acc_empty[S], wfull;
  __shared__ uint32_t tmem_base;
  __shared__ volatile int failed;
  __shared__ __align__(16) float sbias[NP];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t sB = smem_u32(smem), sA = sB + T::kB;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                 "r"(T::kCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 32) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&done[s], 1);
      mbar_init(&acc_empty[s], 4);
    }
    mbar_init(&wfull, kEpi / 32);
    failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;

  if (warp < kProd / 32) {
    pdl_enter();
    // producers: each warp brings whole patches (every fourth one), so that four
    // patches' waits, copies and proxy fences run side by side
    for (int it = warp, t = blockIdx.x + warp * gridDim.x; t < g.count; it += 4, t += 4 * gridDim.x) {
      const int s = it % S;
      int b, y0, x0;
      tile_pos(g, t, b, y0, x0);
      if (it >= S && !mbar_wait(&done[s], (uint32_t)((it / S - 1) & 1), &failed, wlimit)) failed = 1;
      if (__any_sync(0xffffffffu, failed)) break;
      load_patch<C8>(sA + s * T::kStage, T::kPitch, X, g, b, y0, x0, lane);
      cp_commit();
      cp_wait<0>();
      fence_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(&full[s]);
    }
  } else if (warp == kProd / 32) {
    // MMA issuer.  A single commit per tile (done) frees the patch and hands the accumulator over.  Descriptors are a
    // low word (address / 16, leading offset) that advances by constants and a fixed high word.
    // The preceding kernel first: nothing can be issued before it ends, and its time is not the waits' (their poll limit
    // is for this launch's copies).
    pdl_wait();
    const uint32_t idesc = instr_desc(128, NP) | (TB ? 1u << 16 : 0u);
    const uint32_t ahi = desc_hi(kIW * 16), bhi = desc_hi(TB ? (C + 1) * 16 : 128);
    const uint32_t blo = desc_lo(sB, TB ? 128 : T::kPitchB);
    if (lane == 0) {
      int it = 0;
      if (!mbar_wait(&wfull, 0, &failed, wlimit)) failed = 1;
      for (int t = blockIdx.x; t < g.count && !failed; t += gridDim.x, ++it) {
        const int s = it % S;
        if ((it >= S && !mbar_wait(&acc_empty[s], (uint32_t)((it / S - 1) & 1), &failed, wlimit)) ||
            !mbar_wait(&full[s], (uint32_t)((it / S) & 1), &failed, wlimit)) {
          failed = 1;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t acc = tmem + (uint32_t)(s * NP), p0 = sA + s * T::kStage;
        if constexpr (C == 8) {
          // K = 16 takes two taps; tap 9 is zeros on both sides
#pragma unroll
          for (int i = 0; i < 5; ++i) {
            const int t0 = 2 * i, t1 = 2 * i + 1;
            const uint32_t a0 = p0 + ((t0 / 3) * kIW + t0 % 3) * 16;
            const uint32_t a1 = t1 < 9 ? p0 + ((t1 / 3) * kIW + t1 % 3) * 16 : sA + S * T::kStage;
            mma_bf16(acc, desc_lo(a0, a1 - a0), ahi, blo + t0 * T::kPitchB / 16, bhi, idesc, i > 0);
          }
        } else {
          // rolled over the taps: a short loop stays in the instruction cache beside the other roles' code
          uint32_t al = desc_lo(p0, T::kPitch), bl = blo;
          const uint32_t bstep = TB ? (NP / 8) * (C + 1) : C8 * T::kPitchB / 16;
#pragma unroll 1
          for (int t9 = 0; t9 < 9; ++t9, bl += bstep) {
#pragma unroll
            for (int j = 0; j < C / 16; ++j)
              // turned weights, MN-major: eight-output groups C + 1 chunks apart (stride), eight K rows 128 bytes (leading)
              mma_bf16(acc, al + 2 * j * T::kPitch / 16, ahi, bl + j * (TB ? 16 : 2 * T::kPitchB / 16), bhi, idesc,
                       t9 > 0 || j > 0);
            al += (t9 == 2 || t9 == 5) ? kIW - 2 : 1;
          }
        }
        mma_commit(&done[s]);
      }
      // every MMA issued has completed before the CTA ends
      for (int j = it > S ? it - S : 0; j < it; ++j)
        if (!mbar_wait(&done[j % S], (uint32_t)((j / S) & 1))) failed = 1;
    }
  } else {
    // First the weights and the bias, once per CTA, while the producers fetch
    // the first patches.  With `early` they do not depend on the preceding
    // kernel of the stream and are read while it still runs.
    if (!early) pdl_wait();
    const int et = threadIdx.x - kProd - 32;
    if (et < NP) sbias[et] = (bias && et < Cout) ? bias[et] : 0.f;
    if constexpr (!TB) {
      // plane k8 of the K dimension: [NP outputs] x 8 of K
      for (int i = et; i < T::kPlanesB * NP; i += kEpi) {
        const int n = i / T::kPlanesB, k8 = i - n * T::kPlanesB;
        const bool ok = n < Cout && k8 < 9 * C8;
        cp16(sB + k8 * T::kPitchB + n * 16, ok ? Wt + (long)n * 9 * C + k8 * 8 : Wt, ok);
      }
    } else {
      // chunk (tap t, eight outputs n8, k): row k of the forward weights [C][9 Cout], tap 8 - t
      for (int i = et; i < 9 * (NP / 8) * C; i += kEpi) {
        const int n8 = i % (NP / 8), r = i / (NP / 8), t = r % 9, k = r / 9;
        const bool ok = n8 * 8 < Cout;
        cp16(sB + (uint32_t)((t * (NP / 8) + n8) * (C + 1) + k) * 16, ok ? Wt + ((long)k * 9 + 8 - t) * Cout + n8 * 8 : Wt,
             ok);
      }
    }
    if constexpr (C == 8) {
      for (uint32_t i = et; i < T::kZero / 16; i += kEpi)
        *reinterpret_cast<uint4*>(smem + T::kB + S * T::kStage + i * 16) = make_uint4(0, 0, 0, 0);
    }
    cp_commit();
    cp_wait<0>();
    fence_async();
    asm volatile("bar.sync 1, 256;" ::: "memory");   // the bias is read by all epilogue warps
    if (lane == 0) mbar_arrive(&wfull);
    pdl_wait();
    // epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31 = pixels of the tile, lane by lane
    const int q = warp & 3, m = q * 32 + lane, my = m / kPW, mx = m % kPW;
    int it = et / 128;   // this group's tiles: every other one
    for (int t = blockIdx.x + it * gridDim.x; t < g.count; t += 2 * gridDim.x, it += 2) {
      const int a = it % kAcc;
      int b, y0, x0;
      tile_pos(g, t, b, y0, x0);
      if (!__all_sync(0xffffffffu, mbar_wait(&done[a], (uint32_t)((it / kAcc) & 1), &failed, wlimit))) {
        failed = 1;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int gy = y0 + my, gx = x0 + mx;
      const bool inside = gy < g.H && gx < g.W;
      __nv_bfloat16* row = Y + (((long)b * g.H + gy) * g.W + gx) * Cout;
#pragma unroll 1
      for (int c0 = 0; c0 < NP; c0 += 32) {
        uint32_t r[32];
        tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(a * NP + c0), r);
        if (c0 + 32 >= NP) {   // the accumulator is free for the tile after next
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(&acc_empty[a]);
        }
        if (!inside) continue;
        uint32_t pk[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const float2 bv = *reinterpret_cast<const float2*>(sbias + c0 + 2 * j);
          float v0 = __uint_as_float(r[2 * j]) + bv.x, v1 = __uint_as_float(r[2 * j + 1]) + bv.y;
          if (relu) {
            v0 = fmaxf(v0, 0.f);
            v1 = fmaxf(v1, 0.f);
          }
          const __nv_bfloat162 b2 = __floats2bfloat162_rn(v0, v1);
          pk[j] = *reinterpret_cast<const uint32_t*>(&b2);
        }
        if (vec == 2) {   // whole sectors: Cout a multiple of 16, 32-byte aligned rows
#pragma unroll
          for (int j = 0; j < 2; ++j)
            if (c0 + 16 * j < Cout) st32(row + c0 + 16 * j, pk + 8 * j);
        } else if (vec) {   // whole 16-byte chunks of a 16-byte aligned row
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (c0 + 8 * j < Cout)
              *reinterpret_cast<uint4*>(row + c0 + 8 * j) =
                  make_uint4(pk[4 * j], pk[4 * j + 1], pk[4 * j + 2], pk[4 * j + 3]);
        } else {
#pragma unroll
          for (int j = 0; j < 32; ++j)
            if (c0 + j < Cout)
              reinterpret_cast<unsigned short*>(row)[c0 + j] = (unsigned short)(pk[j / 2] >> (16 * (j & 1)));
        }
      }
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(T::kCols) : "memory");
  if (failed && threadIdx.x == 0) atomicExch(status, 1);
}

template <int C, int NP, bool TB>
cudaError_t launch_patch(const __nv_bfloat16* X, const Tiles& g, const __nv_bfloat16* Wt, int Cout, const float* bias,
                         int relu, __nv_bfloat16* Y, int* status, cudaStream_t s, int early) {
  using T = ConvTile<C, NP>;
  static std::once_flag once;
  static cudaError_t attr = cudaSuccess;
  std::call_once(once, [] {
    attr = cudaFuncSetAttribute(conv3x3_patch_kernel<C, NP, TB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                T::kSmem);
  });
  if (attr != cudaSuccess) return attr;
  // A second CTA per SM overlaps the hand-offs of long walks (32 -> 32 channels, 4096 tiles: 28 against 31 us) but
  // loads the weights twice (32 -> 64, 1024 tiles: 19 against 15 us): from eight tiles per CTA on.
  const long sms = sm_count() > 0 ? sm_count() : 1;
  const long cap = sms * (T::kCtas > 1 && g.count >= 16 * sms ? 2 : 1);
  const unsigned grid = (unsigned)(g.count < cap ? g.count : cap);
  const uintptr_t ya = reinterpret_cast<uintptr_t>(Y);
  const int vec = Cout % 16 == 0 && ya % 32 == 0 ? 2 : Cout % 8 == 0 && ya % 16 == 0 ? 1 : 0;
  const cudaError_t e = launch_k(conv3x3_patch_kernel<C, NP, TB>, dim3(grid), dim3(kConvThreads), T::kSmem, s, X, g, Wt,
                                 Cout, bias, relu, Y, vec, status, wait_limit(), early);
  count_launches(1);
  return e;
}

// ---- weight gradient -------------------------------------------------------
//
// gw[co][t C + c] = sum over pixels p of dZ[p][co] X[p shifted by tap t][c].
// The contraction runs over pixels, so both operands are MN-major: dZ of a
// tile as planes of 16-byte chunks (8 output channels of a pixel), X as the
// forward kernel's patch, eight pixels of an image row being a core matrix;
// a tap again is a start address.  An MMA of 64 x C x 16 takes two image rows
// of the tile; a CTA sums a slice of at most 32 tiles (4096 pixels, the depth
// of the FP32 accumulation) into one accumulator of C columns per tap, and the
// slices are added in a fixed order by finish_layer (cmg_nn_ops.cu).
//
// Why: the GEMM form needed dZ transposed and the patch matrix transposed
// ([9 C][pixels], 302 MB at 256^2, batch 8), which took ten times the
// multiplications' time: 320 us of transposing per layer on average and 63 us
// of GEMM.  Here X and dZ are read once (twice for C = 64, whose nine
// accumulators exceed the 512 TMEM columns: five taps in one CTA, four in
// another).  256^2 32->32, batch 8: 67 us in all; 128^2 64->64 31 us.  Bound by
// the tensor cores' operand reads (3 to 4 KB per MMA of 64 x C x 16).
template <int C, int CO>
struct WgradTile {
  static constexpr int C8 = C / 8, CO8 = CO / 8;
  static constexpr int kTaps = C == 64 ? 5 : 9;              // taps of a CTA
  static constexpr int kGroups = (9 + kTaps - 1) / kTaps;
  static constexpr uint32_t kPitch = patch_pitch(C8);
  static constexpr uint32_t kPitchZ = (CO8 == 8 ? 129u : 130u) * 16u;   // 128 pixels
  static constexpr uint32_t kZ = CO8 * kPitchZ;
  static constexpr uint32_t kStage = kZ + C8 * kPitch;
  static constexpr int S = 4;
  // the MMA's 64 rows read eight planes of dZ; with CO = 32 the last four are whatever follows (rows not stored)
  static constexpr uint32_t kSlack = CO8 < 8 ? 4 * kPitchZ : 0;
  static constexpr int kUse = (int)(S * kStage + kSlack);
  static constexpr int kSmem = kUse > 116 * 1024 ? kUse : 116 * 1024;   // one CTA per SM (TMEM)
  static constexpr uint32_t kCols = kTaps * C <= 128 ? 128 : 512;
  static_assert(kTaps * C <= (int)kCols && kSmem <= 227 * 1024, "TMEM and shared memory");
};
constexpr int kWgThreads = kProd + 32 + 128;

template <int C, int CO>
__global__ void __launch_bounds__(kWgThreads, 1)
    conv3x3_wgrad_kernel(const __nv_bfloat16* __restrict__ X, const __nv_bfloat16* __restrict__ dZ, Tiles g, int per,
                         float* __restrict__ part, int* __restrict__ status, long long wlimit) {
  using T = WgradTile<C, CO>;
  constexpr int C8 = T::C8, CO8 = T::CO8, S = T::S;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t full[S], done[S], fin;
  __shared__ uint32_t tmem_base;
  __shared__ volatile int failed;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t s0 = smem_u32(smem);
  const int z = blockIdx.x, tap0 = blockIdx.y * T::kTaps, taps = tap0 + T::kTaps < 9 ? T::kTaps : 9 - tap0;
  const int first = z * per, last = first + per < g.count ? first + per : g.count;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                 "r"(T::kCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 32) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&done[s], 1);
    }
    mbar_init(&fin, 1);
    failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;
  pdl_enter();

  if (warp < kProd / 32) {
    for (int it = warp, t = first + warp; t < last; it += 4, t += 4) {
      const int s = it % S;
      int b, y0, x0;
      tile_pos(g, t, b, y0, x0);
      if (it >= S && !mbar_wait(&done[s], (uint32_t)((it / S - 1) & 1), &failed, wlimit)) failed = 1;
      if (__any_sync(0xffffffffu, failed)) break;
      const uint32_t dz = s0 + s * T::kStage;
      load_pixels<CO8>(dz, T::kPitchZ, dZ, lane, [&](int px, long& p) {
        const int gy = y0 + px / kPW, gx = x0 + px % kPW;
        p = ((long)b * g.H + gy) * g.W + gx;
        return gy < g.H && gx < g.W;
      });
      load_patch<C8>(dz + T::kZ, T::kPitch, X, g, b, y0, x0, lane);
      cp_commit();
      cp_wait<0>();
      fence_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(&full[s]);
    }
  } else if (warp == kProd / 32) {
    const uint32_t idesc = instr_desc(64, C) | 1u << 15 | 1u << 16;   // both operands MN-major
    const uint32_t ahi = desc_hi(T::kPitchZ), bhi = desc_hi(T::kPitch);
    if (lane == 0) {
      int it = 0;
      for (int t = first; t < last && !failed; ++t, ++it) {
        const int s = it % S;
        if (!mbar_wait(&full[s], (uint32_t)((it / S) & 1), &failed, wlimit)) {
          failed = 1;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t al = desc_lo(s0 + s * T::kStage, 128), bl = desc_lo(s0 + s * T::kStage + T::kZ, kIW * 16);
#pragma unroll 1
        for (int k = 0; k < taps; ++k) {
          const int t9 = tap0 + k, toff = t9 + (kIW - 3) * (t9 / 3);   // 10 dy + dx
#pragma unroll
          for (int j = 0; j < kPH / 2; ++j)
            mma_bf16(tmem + k * C, al + j * 16, ahi, bl + toff + j * 2 * kIW, bhi, idesc, it > 0 || j > 0);
        }
        mma_commit(&done[s]);
      }
      mma_commit(&fin);   // completes once every MMA issued above has completed
      if (!mbar_wait(&fin, 0)) failed = 1;
    }
  } else {
    const int q = warp & 3;
    const bool ok = __all_sync(0xffffffffu, mbar_wait(&fin, 0, &failed, wlimit > kSpinLimit ? wlimit : kSpinLimit));
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (ok && !failed) {
      // M = 64: row 16 q + l of the product in lane l < 16 of quadrant q
      const int co = q * 16 + lane;
      float* row = part + ((long)z * CO + co) * (9 * C) + tap0 * C;
#pragma unroll 1
      for (int c0 = 0; c0 < taps * C; c0 += 8) {
        uint32_t r[8];
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                     : "r"(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c0)
                     : "memory");
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (lane < 16 && co < CO) st32(row + c0, r);
      }
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(T::kCols) : "memory");
  if (failed && threadIdx.x == 0) atomicExch(status, 1);
}

// ---- 1x1 head ---------------------------------------------------------------
//
// out[p] = sum_c X[p][c] w[c] + bias over C = 32 channels, one output: two MMAs
// of 128 x 16 x 16 per 128 pixels (the sums of the 64-wide GEMM, bit for bit),
// bound by reading X.  The GEMM (cmg_nn_gemm.cu) took 34 us for 256^2, batch 8,
// moving 32 output columns through its transposing epilogue for one.
constexpr int kHeadN = 16, kHeadS = 4;
constexpr uint32_t kHeadPitch = 130 * 16, kHeadStage = 4 * kHeadPitch;
constexpr int kHeadSmem = (int)(kHeadS * kHeadStage + 4 * kHeadN * 16);

__global__ void __launch_bounds__(kWgThreads)
    head1x1_kernel(const __nv_bfloat16* __restrict__ X, const __nv_bfloat16* __restrict__ w,
                   const float* __restrict__ bias, long P, long tiles, float* __restrict__ out, float* __restrict__ out2,
                   int* __restrict__ status, long long wlimit) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t full[kHeadS], done[kHeadS], acc_empty[kHeadS];
  __shared__ uint32_t tmem_base;
  __shared__ volatile int failed;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t sA = smem_u32(smem), sB = sA + kHeadS * kHeadStage;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                 "r"(kHeadS * kHeadN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 32) {
    for (int s = 0; s < kHeadS; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&done[s], 1);
      mbar_init(&acc_empty[s], 4);
    }
    failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  pdl_wait();
  // weight plane k8: row 0 the weights, rows 1 .. 15 zero
  if (threadIdx.x < 4 * kHeadN) {
    const int k8 = threadIdx.x / kHeadN, n = threadIdx.x % kHeadN;
    *reinterpret_cast<uint4*>(smem + kHeadS * kHeadStage + threadIdx.x * 16) =
        n == 0 ? *reinterpret_cast<const uint4*>(w + k8 * 8) : make_uint4(0, 0, 0, 0);
  }
  fence_async();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;
  pdl_enter();

  if (warp < kProd / 32) {
    long t = (long)blockIdx.x + (long)warp * gridDim.x;
    for (int it = warp; t < tiles; it += 4, t += 4L * gridDim.x) {
      const int s = it % kHeadS;
      if (it >= kHeadS && !mbar_wait(&done[s], (uint32_t)((it / kHeadS - 1) & 1), &failed, wlimit)) failed = 1;
      if (__any_sync(0xffffffffu, failed)) break;
      load_pixels<4>(sA + s * kHeadStage, kHeadPitch, X, lane, [&](int px, long& p) {
        p = t * 128 + px;
        return p < P;
      });
      cp_commit();
      cp_wait<0>();
      fence_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(&full[s]);
    }
  } else if (warp == kProd / 32) {
    if (lane == 0) {
      const uint32_t idesc = instr_desc(128, kHeadN), hi = desc_hi(128);
      int it = 0;
      for (long t = blockIdx.x; t < tiles && !failed; t += gridDim.x, ++it) {
        const int s = it % kHeadS;
        if ((it >= kHeadS && !mbar_wait(&acc_empty[s], (uint32_t)((it / kHeadS - 1) & 1), &failed, wlimit)) ||
            !mbar_wait(&full[s], (uint32_t)((it / kHeadS) & 1), &failed, wlimit)) {
          failed = 1;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t al = desc_lo(sA + s * kHeadStage, kHeadPitch), bl = desc_lo(sB, kHeadN * 16);
#pragma unroll
        for (int j = 0; j < 2; ++j)
          mma_bf16(tmem + s * kHeadN, al + 2 * j * kHeadPitch / 16, hi, bl + 2 * j * kHeadN, hi, idesc, j > 0);
        mma_commit(&done[s]);
      }
      for (int j = it > kHeadS ? it - kHeadS : 0; j < it; ++j)
        if (!mbar_wait(&done[j % kHeadS], (uint32_t)((j / kHeadS) & 1))) failed = 1;
    }
  } else {
    const int q = warp & 3;
    const float bv = bias[0];
    int it = 0;
    for (long t = blockIdx.x; t < tiles; t += gridDim.x, ++it) {
      const int s = it % kHeadS;
      if (!__all_sync(0xffffffffu, mbar_wait(&done[s], (uint32_t)((it / kHeadS) & 1), &failed, wlimit))) {
        failed = 1;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      uint32_t r;
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];"
                   : "=r"(r)
                   : "r"(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(s * kHeadN))
                   : "memory");
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[s]);
      const long p = t * 128 + q * 32 + lane;
      if (p < P) {
        out[p] = __uint_as_float(r) + bv;
        if (out2) out2[p] = __uint_as_float(r) + bv;
      }
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kHeadS * kHeadN) : "memory");
  if (failed && threadIdx.x == 0) atomicExch(status, 1);
}

// Tiles per slice: an even share of the SMs, at most 32 tiles.
int wgrad_per(long tiles, int groups) {
  const long sms = sm_count() > 0 ? sm_count() : 1;
  const long per = (tiles * groups + sms - 1) / sms;
  return (int)(per < 1 ? 1 : per > 32 ? 32 : per);
}

template <int C, int CO>
cudaError_t launch_wgrad(const __nv_bfloat16* X, const __nv_bfloat16* dZ, const Tiles& g, float* part, int* slices,
                         int* status, cudaStream_t s) {
  using T = WgradTile<C, CO>;
  static std::once_flag once;
  static cudaError_t attr = cudaSuccess;
  std::call_once(once, [] {
    attr = cudaFuncSetAttribute(conv3x3_wgrad_kernel<C, CO>, cudaFuncAttributeMaxDynamicSharedMemorySize, T::kSmem);
  });
  if (attr != cudaSuccess) return attr;
  const int per = wgrad_per(g.count, T::kGroups);
  *slices = (g.count + per - 1) / per;
  const cudaError_t e = launch_k(conv3x3_wgrad_kernel<C, CO>, dim3((unsigned)*slices, T::kGroups), dim3(kWgThreads),
                                 T::kSmem, s, X, dZ, g, per, part, status, wait_limit());
  count_launches(1);
  return e;
}

}  // namespace
}  // namespace nn

cudaError_t launch_head(const void* X, const void* w16, const float* b, long P, float* out, float* out2, int* status,
                        cudaStream_t s) {
  using namespace nn;
  const long tiles = (P + 127) / 128, sms = sm_count() > 0 ? sm_count() : 1;
  const unsigned grid = (unsigned)(tiles < 4 * sms ? tiles : 4 * sms);
  const cudaError_t e = launch_k(head1x1_kernel, dim3(grid), dim3(kWgThreads), kHeadSmem, s,
                                 static_cast<const __nv_bfloat16*>(X), static_cast<const __nv_bfloat16*>(w16), b, P,
                                 tiles, out, out2, status, wait_limit());
  count_launches(1);
  return e;
}

long wgrad_max_slices(int B, int H, int W) {
  const long tiles = (long)B * ((W + nn::kPW - 1) / nn::kPW) * ((H + nn::kPH - 1) / nn::kPH);
  const long sms = nn::sm_count() > 0 ? nn::sm_count() : 1;
  return std::max(sms, (tiles + 31) / 32) + 1;
}

cudaError_t launch_conv3x3_wgrad(const void* X, const void* dZ, int B, int H, int W, int C, int Cout, float* part,
                                 int* slices, int* status, cudaStream_t s) {
  using namespace nn;
  Tiles g{B, H, W, (W + kPW - 1) / kPW, (H + kPH - 1) / kPH, 0};
  const long tiles = (long)B * g.tx * g.ty;
  if (tiles > 0x7fffffffL) return cudaErrorNotSupported;
  g.count = (int)tiles;
  const __nv_bfloat16 *x = static_cast<const __nv_bfloat16*>(X), *d = static_cast<const __nv_bfloat16*>(dZ);
  if (C == 8 && Cout == 32) return launch_wgrad<8, 32>(x, d, g, part, slices, status, s);
  if (C == 32 && Cout == 32) return launch_wgrad<32, 32>(x, d, g, part, slices, status, s);
  if (C == 32 && Cout == 64) return launch_wgrad<32, 64>(x, d, g, part, slices, status, s);
  if (C == 64 && Cout == 32) return launch_wgrad<64, 32>(x, d, g, part, slices, status, s);
  if (C == 64 && Cout == 64) return launch_wgrad<64, 64>(x, d, g, part, slices, status, s);
  return cudaErrorNotSupported;
}

// Times (us) by the tiles that an SM works off, fitted to 30 image shapes per
// channel pair on a GB300, batches included: a patch tile costs a third (C =
// 64) to an eighth (C = 8) of an im2col tile, but its 8 x 16 pixels end at the
// image's edge while im2col tiles run on over rows and images, and C = 64
// starts by loading 74 KB of weights.  So thin and small images stay with im2col
// (C = Cout = 64: 64 images of 1 x 4096 343 against 59, 4096 of 4 x 4 51 against 21,
// 8 of 40^2 10.8 against 8.4; the network's levels are on the patches' side,
// 8 of 128^2 21 against 32).
bool conv3x3_patch_pays(int B, int H, int W, int C, int Cout) {
  using namespace nn;
  const long sms = sm_count() > 0 ? sm_count() : 1;
  const long tiles = (long)B * ((W + kPW - 1) / kPW) * ((H + kPH - 1) / kPH), dense = ((long)B * H * W + 127) / 128;
  const double rp = (double)((tiles + sms - 1) / sms), ri = (double)((dense + sms - 1) / sms);
  const bool narrow = Cout <= 32;
  if (C == 8) return 3.9 + (narrow ? 0.38 : 0.48) * rp <= 4.8 + 3.0 * ri;
  if (C == 32) return std::min(4.5 + (narrow ? 1.3 : 1.4) * rp, 10.0 + 0.68 * rp) <= 4.6 + 3.6 * ri;
  return (2 * tiles <= sms ? 8.0 : 9.0 + 1.7 * rp) <= 4.2 + 4.1 * ri;
}

cudaError_t launch_conv3x3_patch(const void* X, int B, int H, int W, int C, const void* Wt, int Cout,
                                 const float* bias, int relu, int turned, void* Y16, int* status, cudaStream_t s, int early) {
  using namespace nn;
  if (Cout < 1 || Cout > 64) return cudaErrorNotSupported;
  Tiles g{B, H, W, (W + kPW - 1) / kPW, (H + kPH - 1) / kPH, 0};
  const long tiles = (long)B * g.tx * g.ty;
  if (tiles > 0x7fffffffL) return cudaErrorNotSupported;
  g.count = (int)tiles;
  const __nv_bfloat16 *x = static_cast<const __nv_bfloat16*>(X), *w = static_cast<const __nv_bfloat16*>(Wt);
  __nv_bfloat16* y = static_cast<__nv_bfloat16*>(Y16);
  const bool narrow = Cout <= 32;
  if (turned) {
    if (Cout % 8) return cudaErrorNotSupported;
    if (C == 32) return narrow ? launch_patch<32, 32, true>(x, g, w, Cout, bias, relu, y, status, s, early)
                               : launch_patch<32, 64, true>(x, g, w, Cout, bias, relu, y, status, s, early);
    if (C == 64) return narrow ? launch_patch<64, 32, true>(x, g, w, Cout, bias, relu, y, status, s, early)
                               : launch_patch<64, 64, true>(x, g, w, Cout, bias, relu, y, status, s, early);
    return cudaErrorNotSupported;
  }
  if (C == 8) return narrow ? launch_patch<8, 32, false>(x, g, w, Cout, bias, relu, y, status, s, early)
                            : launch_patch<8, 64, false>(x, g, w, Cout, bias, relu, y, status, s, early);
  if (C == 32) return narrow ? launch_patch<32, 32, false>(x, g, w, Cout, bias, relu, y, status, s, early)
                             : launch_patch<32, 64, false>(x, g, w, Cout, bias, relu, y, status, s, early);
  if (C == 64) return narrow ? launch_patch<64, 32, false>(x, g, w, Cout, bias, relu, y, status, s, early)
                             : launch_patch<64, 64, false>(x, g, w, Cout, bias, relu, y, status, s, early);
  return cudaErrorNotSupported;
}

}  // namespace cmg
