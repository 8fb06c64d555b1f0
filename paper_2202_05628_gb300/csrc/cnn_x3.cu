// The FP32 shading network's 3x3 convolutions on the tensor cores (arXiv
// 2202.05628, Sec. 3.1 "Neural Shading"), at FP32 precision.
//
// An FP32 value is the sum of three BF16 parts (x = x1 + x2 + x3, each part
// the rounding of what the earlier ones leave; exactly from 2^-110 up, below
// that bits under 2^-133, the smallest BF16 value, are lost), so a product is
//   w x = w1 x1 + (w1 x2 + w2 x1) + (w2 x2 + w1 x3 + w3 x1) + O(2^-24 |w x|),
// six BF16 products of which each is exact in FP32.  tcgen05.mma truncates
// its FP32 sums, so two things keep the error below that of a chain of FP32
// FMAs: the products x1 w1 go to an accumulator of their own (the others,
// 2^-8 as large, are summed apart), and that accumulator never runs over more
// than 96 channels x taps: it is read out and added to FP32 registers (rounded
// to nearest) while the tensor cores fill the other row's.  Relative error of
// a sum over K = 320 / 1152 / 3456 ReLU'd inputs (against FP64): 7e-8 / 9e-8 /
// 1.4e-7, an FP32 FMA chain 2.2e-7 / 4.1e-7 / 7.3e-7; one accumulator
// for all six products 2e-6 / 7e-6 / 2e-5.
//
// Activations are stored as their parts, [y][x][part][channel] (6 bytes a
// value), written by the producing layer; the decoders' skip tensors x-phase
// split (even pixels of a row, then odd).  A work unit is 128 pixels x N
// output channels x two "rows": two image rows, or, in the decoders' first
// convolution (sub-pixel form, as in cnn_sub.cu: 9 taps of the skip tensor
// and 4 summed taps of the low-resolution one), the two column phases of
// one output row.  One TMA box brings 130 pixels x 32 channels x 3 parts of
// an input row, which serves the three horizontal taps of both rows; one
// box the N x 32 x 3 weights of a tap, which serves both rows.  Per tap and
// 16 channels the parts are stacked along N: x1 meets [w1 w2 w3], x2
// [w1 w2], x3 [w1] (accumulators a | b | c side by side): N = 32 costs 144
// instead of 240 cycles, N = 64 208 instead of 288 (an MMA takes
// max(N / 2, 32 + N / 4)).  Warp 0 issues TMA, warp 1 MMAs, warps 2-5 and 6-9
// are the two rows' epilogues: they drain their row's a per (tap row, 32
// channels), and at the unit's end add b and c, the bias, ReLU, split and store
// through TMA (with the fused 2x2 pooling, or the fused 1x1 head + sigmoid).
// N = 128 (an eighth fewer MMA cycles) measured slower: its sums fill the
// registers, its drains outlast the other row's MMAs, and small images have
// half as many units.
//
// Bounds: at these N operand reads alone take ~125 B of shared memory a clock of
// MMA time, and the TMA boxes and the staged stores come on top: 49-61 %
// tensor-pipe time for N = 64; for N = 32 (36-42 %) also the epilogue between
// its short units.
// Measured: FP32 frame of 1M voxels at 1024x1024 10.21 ms with the CUDA-core
// kernels (36 TFLOP/s) -> 1.74 ms; the U-Net at 424x248 1720 -> 351 us.
//
// A result that is not finite (an infinite or NaN input, or parts whose
// products overflow) is recomputed as the FP32 FMA chain over taps and
// channels, which such values propagate through as in any FP32 network.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>

#include "internal.cuh"
#include "tc.cuh"

namespace art {
namespace {

constexpr int kThreads = 320;  // warp 0 TMA, warp 1 MMA + TMEM, warps 2..9 epilogue (two groups of four)
constexpr int kKC = 32;        // channels per K chunk
constexpr int kKCB = 64;       // ... in bytes (64-B swizzle)
constexpr int kHalo = 130;     // input pixels of a box (128 + 2)
constexpr int kPlaneA = kHalo * kKCB;
constexpr int kSlotA = (3 * kPlaneA + 1023) / 1024 * 1024;
constexpr int kBoxA = 3 * kPlaneA;
constexpr int kMaxCout = 512;
constexpr int kOutStage = 3 * 128 * kKCB;  // one group's output tile of 32 channels

template <int N>
struct Cfg {
  static constexpr int kPlaneB = N * kKCB;
  static constexpr int kSlotB = 3 * kPlaneB;
  static constexpr int kSet = 3 * N;                  // TMEM columns of one row: accumulators a | b | c
  static constexpr int kScratch = 2 * kSet;           // N = 64: the two rows' finished sums, N columns each
  static constexpr int kTmem = N == 32 ? 256 : 512;
  static constexpr int kSlotsA = 4;
  static constexpr int kSlotsB = N == 32 ? 9 : 6;
  static constexpr int kSmem = 1024 + kSlotsA * kSlotA + kSlotsB * kSlotB + 2 * kOutStage +
                               8 * (2 * (kSlotsA + kSlotsB) + 4) + 16 + 16 + 4 * kMaxCout + 4 * (4 * 32 + 4);
};
static_assert(Cfg<64>::kSmem <= 232448 && Cfg<32>::kSmem <= 232448, "shared memory");

struct Params {
  int H, W;              // output size
  int tiles_x, n_tiles;  // 128-pixel tiles per row, N-channel tiles
  int n_units;
  int c0, c1;            // 32-channel chunks of the input (sub: of the skip tensor, of the low-resolution tensor)
  int act;               // 1 ReLU, 2 sigmoid
  int cout;
  const float* bias;
  int store;             // output planes through TMA
  int psplit;            // ... x-phase split
  __nv_bfloat16* pool;   // fused 2x2 max pooling: [H/2][W/2][3][cout] planes
  // FP32 outputs instead of planes: the fused 1x1 head (cout 32 -> head_n) + sigmoid, or the layer's own channels
  float* out;
  const float* head_w;   // [head_n][32] or null
  const float* head_b;
  int out_n, out_ld, out_off, out_vec;
  // the FP32 chain for results that are not finite
  const __nv_bfloat16 *in, *up;
  int cin, cs, cu;       // weight channels, stored channels of in, of up (0 unless sub)
  const float* w32;
  unsigned long long* err;
};

struct RingPos {
  int i = 0;
  uint32_t ph = 0;
  __device__ __forceinline__ void next(int n) {
    if (++i == n) {
      i = 0;
      ph ^= 1u;
    }
  }
};

__device__ __forceinline__ float part_sum(const __nv_bfloat16* p, int plane) {
  return (__bfloat162float(p[0]) + __bfloat162float(p[plane])) + __bfloat162float(p[2 * plane]);
}

// The parts of x (x = sum, exactly from 2^-110 up): rounded to nearest, the first toward
// zero where rounding would overflow; an infinity or NaN is its own first part.
__device__ __forceinline__ void split3(float x, __nv_bfloat16& a, __nv_bfloat16& b, __nv_bfloat16& c) {
  a = __float2bfloat16_rn(x);
  float fa = __bfloat162float(a);
  if (fabsf(fa) == __int_as_float(0x7f800000) && fabsf(x) < __int_as_float(0x7f800000)) {
    fa = __uint_as_float(__float_as_uint(x) & 0xFFFF0000u);
    a = __float2bfloat16_rn(fa);
  }
  float r = x - fa;
  if (!(fabsf(x) < __int_as_float(0x7f800000))) r = 0.0f;
  b = __float2bfloat16_rn(r);
  c = __float2bfloat16_rn(r - __bfloat162float(b));
}

// The parts of eight non-negative values (o: one 16-byte chunk per part): two
// values per conversion; values a BF16 rounding would overflow go one by one.
__device__ __forceinline__ void split3x8(const float* x, uint4 (&o)[3]) {
  float m = x[0];
#pragma unroll
  for (int j = 1; j < 8; ++j) m = fmaxf(m, x[j]);
  if (m < 3.38e38f) {
    uint32_t w[3][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float a = x[2 * j], b = x[2 * j + 1];
#pragma unroll
      for (int pl = 0; pl < 3; ++pl) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
        w[pl][j] = *reinterpret_cast<const uint32_t*>(&h);
        if (pl < 2) {
          a -= __uint_as_float(w[pl][j] << 16);
          b -= __uint_as_float(w[pl][j] & 0xFFFF0000u);
        }
      }
    }
#pragma unroll
    for (int pl = 0; pl < 3; ++pl) o[pl] = make_uint4(w[pl][0], w[pl][1], w[pl][2], w[pl][3]);
  } else {
    __align__(16) __nv_bfloat16 v[3][8];
#pragma unroll
    for (int j = 0; j < 8; ++j) split3(x[j], v[0][j], v[1][j], v[2][j]);
#pragma unroll
    for (int pl = 0; pl < 3; ++pl) o[pl] = *reinterpret_cast<uint4*>(v[pl]);
  }
}

// The output (Y, X, co) as one FP32 FMA chain over taps, then channels (the
// concatenation [up2(up), in] where there is a low-resolution tensor).
template <bool SUB>
__device__ __noinline__ float chain(const Params& p, int co, int Y, int X) {
  float acc = 0.0f;
  for (int t = 0; t < 9; ++t) {
    const int yy = Y + t / 3 - 1, xx = X + t % 3 - 1;
    const float* w = p.w32 + ((size_t)co * 9 + t) * p.cin;
    if (yy < 0 || yy >= p.H || xx < 0 || xx >= p.W) {
      for (int c = 0; c < p.cin; ++c) acc = fmaf(0.0f, w[c], acc);
      continue;
    }
    for (int c = 0; c < p.cu; ++c)
      acc = fmaf(part_sum(p.up + ((size_t)(yy >> 1) * (p.W >> 1) + (xx >> 1)) * 3 * p.cu + c, p.cu), w[c], acc);
    const int xs = SUB ? (xx & 1) * (p.W >> 1) + (xx >> 1) : xx;
    const __nv_bfloat16* s = p.in + ((size_t)yy * p.W + xs) * 3 * p.cs;
    for (int c = 0; c < p.cin - p.cu; ++c) acc = fmaf(part_sum(s + c, p.cs), w[p.cu + c], acc);
  }
  return acc;
}

// One tap of one row: 32 channels of A (three parts, kPlaneA apart) against
// N x 32 weights (three parts, stacked), into the accumulators a | b | c at d.
// kFreshA: the tap starts a K block (a begins anew, b and c go on);
// kFreshAll: it starts the unit.  Descriptors advance by constants.
enum Start { kGoOn, kFreshA, kFreshAll };
template <int N>
__device__ __forceinline__ void tap_mma(uint32_t d, uint64_t a1, uint64_t w1, Start start) {
  constexpr uint64_t kA = kPlaneA >> 4, kB = Cfg<N>::kPlaneB >> 4;
#pragma unroll
  for (int kk = 0; kk < kKCB / 32; ++kk, a1 += 2, w1 += 2) {
    if (kk == 0 && start == kFreshA) {
      umma<false>(d, a1, w1, idesc_bf16(128, N), 0u);                // a = x1 w1
      umma<false>(d + N, a1, w1 + kB, idesc_bf16(128, 2 * N), 1u);   // b, c += x1 (w2, w3)
    } else {
      umma<false>(d, a1, w1, idesc_bf16(128, 3 * N), kk == 0 && start == kFreshAll ? 0u : 1u);  // a, b, c += x1 (w1, w2, w3)
    }
    umma<false>(d + N, a1 + kA, w1, idesc_bf16(128, 2 * N), 1u);     // b, c += x2 (w1, w2)
    umma<false>(d + 2 * N, a1 + 2 * kA, w1, idesc_bf16(128, N), 1u);  // c += x3 w1
  }
}

// The 32 columns at t and the 32 at u.
__device__ __forceinline__ void tmem_ld32x2(uint32_t t, uint32_t u, uint32_t (&a)[32], uint32_t (&b)[32]) {
#define ART_R32(r)                                                                                             \
  "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),  \
      "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),   \
      "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),  \
      "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%64];\n"
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, "
      "%46, %47, %48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63}, [%65];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : ART_R32(a), ART_R32(b)
      : "r"(t), "r"(u)
      : "memory");
#undef ART_R32
}

// 32 values into this warp's lanes of the 32 columns at t.
__device__ __forceinline__ void tmem_st32(uint32_t t, const float* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(t),
      "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "f"(v[8]), "f"(v[9]),
      "f"(v[10]), "f"(v[11]), "f"(v[12]), "f"(v[13]), "f"(v[14]), "f"(v[15]), "f"(v[16]), "f"(v[17]), "f"(v[18]),
      "f"(v[19]), "f"(v[20]), "f"(v[21]), "f"(v[22]), "f"(v[23]), "f"(v[24]), "f"(v[25]), "f"(v[26]), "f"(v[27]),
      "f"(v[28]), "f"(v[29]), "f"(v[30]), "f"(v[31])
      : "memory");
}

// Barrier over the `count` threads (whole warps) that name it.
__device__ __forceinline__ void bar_sync(int id, int count) {
  asm volatile("barrier.cta.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}

// The sums v of 32 output channels from n0 on of this thread's pixel (Y, X):
// bias, activation, outputs.
template <int N, bool SUB>
__device__ __forceinline__ void finish(const Params& p, float (&v)[32], int n0, int Y, int X, int x0, int yy, int q, int g,
                                       int gt, bool inside, const float* s_bias, const float* s_head, uint8_t* sO,
                                       const CUtensorMap* tmO) {
  uint8_t* st = sO + g * kOutStage;
  // a sum that is not finite (zero times it is NaN) as the FP32 chain
  float odd0 = 0.0f, odd1 = 0.0f;
#pragma unroll
  for (int j = 0; j < 32; j += 2) {
    odd0 = fmaf(v[j], 0.0f, odd0);
    odd1 = fmaf(v[j + 1], 0.0f, odd1);
  }
  if (odd0 + odd1 != 0.0f && inside) {
    float fix[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) fix[j] = v[j];
#pragma unroll 1
    for (int j = 0; j < 32 && n0 + j < p.cout; ++j)
      if (fix[j] - fix[j] != 0.0f) fix[j] = chain<SUB>(p, n0 + j, Y, X);
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = fix[j];
  }
#pragma unroll
  for (int j = 0; j < 32; j += 4) {
    const float4 b = *reinterpret_cast<const float4*>(s_bias + n0 + j);
    v[j] += b.x;
    v[j + 1] += b.y;
    v[j + 2] += b.z;
    v[j + 3] += b.w;
  }
  if (p.act == 1) {
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = fmaxf(v[j], 0.0f);
  }
  if (p.out) {  // FP32 outputs
    float* o = p.out + ((size_t)Y * p.W + X) * p.out_ld + p.out_off;
    if (p.head_w) {
      float h[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
      for (int j = 0; j < 32; j += 4)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float4 w = *reinterpret_cast<const float4*>(s_head + k * 32 + j);
          h[k] = fmaf(v[j + 3], w.w, fmaf(v[j + 2], w.z, fmaf(v[j + 1], w.y, fmaf(v[j], w.x, h[k]))));
        }
#pragma unroll
      for (int k = 0; k < 4; ++k) h[k] = 1.0f / (1.0f + expf(-(h[k] + s_head[128 + k])));
      if (inside) {
        if (p.out_vec) {
          *reinterpret_cast<float4*>(o) = make_float4(h[0], h[1], h[2], h[3]);
        } else {
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if (k < p.out_n) o[k] = h[k];
        }
      }
    } else if (inside) {
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (n0 + j < p.out_n) o[n0 + j] = p.act == 2 ? 1.0f / (1.0f + expf(-v[j])) : v[j];
    }
  }
  if (!p.store) return;
  // the staging tile is free once its last store has read it
  if (gt == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
  bar_sync(1 + g, 128);
  {
    // chunk k of part pl of this pixel's row: the row's start, and the chunk's swizzled offset in it
    const int r = p.psplit ? q >> 1 : q, plane = (p.psplit ? 64 : 128) * kKCB;
    uint8_t* row = st + (p.psplit ? (q & 1) * (kOutStage / 2) : 0) + r * kKCB;
    const int x = (r >> 1) & 3;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      uint4 o[3];
      split3x8(v + 8 * k, o);
      uint8_t* d = row + ((k ^ x) << 4);
#pragma unroll
      for (int pl = 0; pl < 3; ++pl) *reinterpret_cast<uint4*>(d + pl * plane) = o[pl];
    }
  }
  fence_proxy_async_smem();
  if (p.pool)
    bar_sync(3, 256);
  else
    bar_sync(1 + g, 128);
  if (gt == 0) {
    if (p.psplit) {
      tma_store_5d(tmO, st, n0, x0 >> 1, 0, 0, Y);
      tma_store_5d(tmO, st + kOutStage / 2, n0, x0 >> 1, 0, 1, Y);
    } else {
      tma_store_5d(tmO, st, n0, x0, 0, SUB ? g : 0, Y);
    }
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
  }
  if (p.pool) {  // 2x2 maxima of both groups' rows (x-phase split): pooled pixel e / 4, channels 8 (e % 4) .. + 7
    const int e = g * 128 + gt, pq = e >> 2, k = e & 3;
    const uint8_t* src = sO + pq * kKCB + ((k ^ ((pq >> 1) & 3)) << 4);
    float m[8];
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      uint4 w[3];
#pragma unroll
      for (int pl = 0; pl < 3; ++pl)
        w[pl] = *reinterpret_cast<const uint4*>(src + (s >> 1) * kOutStage + (s & 1) * (kOutStage / 2) + pl * 64 * kKCB);
      const __nv_bfloat16* h = reinterpret_cast<const __nv_bfloat16*>(w);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float f = part_sum(h + j, 8);
        m[j] = s == 0 ? f : fmaxf(m[j], f);
      }
    }
    const int hx = (x0 >> 1) + pq, hw = p.W >> 1;
    if (hx < hw && yy < (p.H >> 1)) {
      uint4 o[3];
      split3x8(m, o);
#pragma unroll
      for (int pl = 0; pl < 3; ++pl)
        *reinterpret_cast<uint4*>(p.pool + (((size_t)yy * hw + hx) * 3 + pl) * p.cout + n0 + 8 * k) = o[pl];
    }
    bar_sync(3, 256);  // (both groups' tiles are read: they may be staged again)
  }
}

template <int N, bool SUB>
__global__ void __launch_bounds__(kThreads, 1)
    conv_x3_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmU,
                   const __grid_constant__ CUtensorMap tmB, const __grid_constant__ CUtensorMap tmV,
                   const __grid_constant__ CUtensorMap tmO, const __grid_constant__ Params p) {
  using C = Cfg<N>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  uint8_t* sm = smem_raw + (((raw + 1023u) & ~1023u) - raw);
  uint8_t* sA = sm;
  uint8_t* sB = sA + C::kSlotsA * kSlotA;
  uint8_t* sO = sB + C::kSlotsB * C::kSlotB;
  uint64_t* fullA = reinterpret_cast<uint64_t*>(sO + 2 * kOutStage);
  uint64_t* emptyA = fullA + C::kSlotsA;
  uint64_t* fullB = emptyA + C::kSlotsA;
  uint64_t* emptyB = fullB + C::kSlotsB;
  uint64_t* accf = emptyB + C::kSlotsB;
  uint64_t* acce = accf + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acce + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  // the layer's biases (every unit reads them: from global memory each would wait for them)
  float* s_bias = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(tmem_slot + 4) + 15) & ~(uintptr_t)15);
  float* s_head = s_bias + kMaxCout;  // [4][32] weights, [4] biases

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < C::kSlotsA; ++s) {
      mbar_init(&fullA[s], 1);
      mbar_init(&emptyA[s], 1);
    }
    for (int s = 0; s < C::kSlotsB; ++s) {
      mbar_init(&fullB[s], 1);
      mbar_init(&emptyB[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&acce[b], 128);
    }
    *abort_flag = 0;
    fence_mbar_init();
  }
  for (int i = threadIdx.x; i < p.n_tiles * N; i += kThreads) s_bias[i] = i < p.cout ? p.bias[i] : 0.0f;
  if (p.head_w)
    for (int i = threadIdx.x; i < 4 * 32 + 4; i += kThreads)  // outputs beyond out_n are zero
      s_head[i] = i < 128 ? (i < p.out_n * 32 ? p.head_w[i] : 0.0f) : (i - 128 < p.out_n ? p.head_b[i - 128] : 0.0f);
  if (warp == 1) tmem_alloc(tmem_slot, C::kTmem);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  grid_dep_launch();
  grid_dep_wait();  // the previous layers' outputs (this one's inputs) are complete

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA
    if (lane == 0) {
      RingPos ra, rb;
      bool ok = true;
      auto box = [&](const CUtensorMap* tm, int c, int x, int phase, int y) {
        if (!ok || !(ok = mbar_wait(&emptyA[ra.i], ra.ph ^ 1u, abort_flag))) return;
        mbar_expect_tx(&fullA[ra.i], kBoxA);
        tma_load_5d(sA + ra.i * kSlotA, tm, &fullA[ra.i], c * kKC, x, 0, phase, y);
        ra.next(C::kSlotsA);
      };
      auto weights = [&](const CUtensorMap* tm, int c, int n0, int tap) {
        if (!ok || !(ok = mbar_wait(&emptyB[rb.i], rb.ph ^ 1u, abort_flag))) return;
        mbar_expect_tx(&fullB[rb.i], C::kSlotB);
        tma_load_4d(sB + rb.i * C::kSlotB, tm, &fullB[rb.i], c * kKC, n0, 0, tap);
        rb.next(C::kSlotsB);
      };
      for (int u = blockIdx.x; ok && u < p.n_units && !*abort_flag; u += gridDim.x) {
        const int t = u / p.n_tiles, n0 = (u - t * p.n_tiles) * N;
        const int yy = t / p.tiles_x, x0 = (t - yy * p.tiles_x) * 128;
        if constexpr (!SUB) {
          for (int c = 0; c < p.c0; ++c) {
            box(&tmA, c, x0 - 1, 0, 2 * yy - 1);
            for (int dy = 0; dy < 3; ++dy) {
              for (int dx = 0; dx < 3; ++dx) weights(&tmB, c, n0, dy * 3 + dx);
              box(&tmA, c, x0 - 1, 0, 2 * yy + dy);
            }
          }
        } else {
          const int i = yy >> 1, py = yy & 1;
          for (int c = 0; c < p.c0; ++c)
            for (int dy = 0; dy < 3; ++dy) {
              box(&tmA, c, x0 - 1, 0, yy + dy - 1);
              box(&tmA, c, x0 - 1, 1, yy + dy - 1);
              for (int dx = 0; dx < 3; ++dx) weights(&tmB, c, n0, dy * 3 + dx);
            }
          for (int c = 0; c < p.c1; ++c)
            for (int oy = 0; oy < 2; ++oy) {
              box(&tmU, c, x0 - 1, 0, i + py - 1 + oy);
              for (int px = 0; px < 2; ++px)
                for (int ox = 0; ox < 2; ++ox) weights(&tmV, c, n0, ((py * 2 + px) * 2 + oy) * 2 + ox);
            }
        }
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA
    // The whole warp runs the loop and one elected lane issues, so that operand
    // addresses stay in uniform registers (a lone lane's ~68 cycles per MMA were
    // more than N = 32 executes in).  The tensor pipe queues about one MMA beyond
    // the running one, so everything the next row waits for is waited for before
    // this row's last tap: ~270 cycles between rows were idle.
    const bool el = elect_one();
    RingPos ra, rb;
    uint32_t aph = 0;  // both rows' accumulators are used once per K block
    bool ok = true;
    const uint64_t a_base = umma_desc<kKCB>(smem_u32(sA)), b_base = umma_desc<kKCB>(smem_u32(sB));
    auto wait = [&](uint64_t* bar, uint32_t ph) { ok = ok && __all_sync(0xffffffffu, mbar_wait(bar, ph, abort_flag)); };
    auto wait_a = [&](const RingPos& r) { wait(&fullA[r.i], r.ph); };
    auto wait_b = [&](const RingPos& r) { wait(&fullB[r.i], r.ph); };
    auto A = [&](const RingPos& r, int off) { return a_base + (uint32_t)((r.i * kSlotA + off * kKCB) >> 4); };
    auto B = [&](const RingPos& r) { return b_base + (uint32_t)((r.i * C::kSlotB) >> 4); };
    const uint32_t d[2] = {tmem_base, tmem_base + (uint32_t)C::kSet};
    auto tap = [&](int r, uint64_t a1, uint64_t w1, Start st) {
      tc_fence_after();
      if (ok && el) tap_mma<N>(d[r], a1, w1, st);
    };
    auto commit = [&](uint64_t* bar) {
      if (ok && el) umma_commit(bar);
    };
    auto free_b = [&]() {  // the weights in hand have served both rows
      commit(&emptyB[rb.i]);
      rb.next(C::kSlotsB);
    };
    // (the first row's accumulators of a block are waited for in the block before)
    for (int u = blockIdx.x; ok && u < p.n_units && !*abort_flag; u += gridDim.x) {
      Start start = kFreshAll;  // of a block's first tap
      if constexpr (!SUB) {
        for (int c = 0; ok && c < p.c0; ++c) {
          wait_a(ra);
          for (int dy = 0; ok && dy < 3; ++dy) {  // first row: input row dy of the four; second: dy + 1
            RingPos b = rb, an = ra;
            an.next(C::kSlotsA);
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) {
              wait_b(b);
              if (dx == 2) {
                wait_a(an);
                wait(&acce[1], aph ^ 1u);
              }
              tap(0, A(ra, dx), B(b), dx == 0 ? start : kGoOn);
              b.next(C::kSlotsB);
            }
            commit(&accf[0]);
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) {
              if (dx == 2) wait(&acce[0], aph);
              tap(1, A(an, dx), B(rb), dx == 0 ? start : kGoOn);
              if (dx == 0) commit(&emptyA[ra.i]);
              free_b();
            }
            commit(&accf[1]);
            aph ^= 1u;
            start = kFreshA;
            ra = an;
          }
          commit(&emptyA[ra.i]);
          ra.next(C::kSlotsA);
        }
      } else {
        for (int k = 0; ok && k < 3 * p.c0; ++k) {  // skip taps: even box E, odd box O
          const RingPos e = ra;
          ra.next(C::kSlotsA);
          const RingPos o = ra;
          ra.next(C::kSlotsA);
          RingPos b = rb;
          wait_a(e);
          wait_a(o);
#pragma unroll
          for (int dx = 0; dx < 3; ++dx) {  // even column 2j: input columns 2j - 1, 2j, 2j + 1
            wait_b(b);
            if (dx == 2) wait(&acce[1], aph ^ 1u);
            tap(0, dx == 1 ? A(e, 1) : A(o, dx / 2), B(b), dx == 0 ? start : kGoOn);
            b.next(C::kSlotsB);
          }
          commit(&accf[0]);
#pragma unroll
          for (int dx = 0; dx < 3; ++dx) {  // odd column 2j + 1: input columns 2j, 2j + 1, 2j + 2
            if (dx == 2) wait(&acce[0], aph);
            tap(1, dx == 1 ? A(o, 1) : A(e, 1 + dx / 2), B(rb), dx == 0 ? start : kGoOn);
            free_b();
          }
          commit(&accf[1]);
          commit(&emptyA[e.i]);
          commit(&emptyA[o.i]);
          aph ^= 1u;
          start = kFreshA;
        }
        for (int k = 0; ok && k < 2 * p.c1; ++k) {  // low-resolution taps: columns j - 1, j | j, j + 1
          wait_a(ra);
#pragma unroll
          for (int px = 0; px < 2; ++px) {
#pragma unroll
            for (int ox = 0; ox < 2; ++ox) {
              wait_b(rb);
              if (ox == 1) wait(&acce[px ^ 1], px == 0 ? aph ^ 1u : aph);
              tap(px, A(ra, px + ox), B(rb), ox == 0 ? kFreshA : kGoOn);
              free_b();
            }
            commit(&accf[px]);
          }
          commit(&emptyA[ra.i]);
          ra.next(C::kSlotsA);
          aph ^= 1u;
        }
      }
    }
  } else {
    // ---------------------------------------------------------------- epilogue
    const int g = (warp - 2) >> 2;     // this group's row (sub: column phase)
    const int qd = warp & 3;           // TMEM lane quarter this warp may access
    const int q = qd * 32 + lane;      // pixel of the tile
    const int gt = threadIdx.x - 64 - 128 * g;  // thread of the group
    const uint32_t tl = tmem_base + ((uint32_t)(qd * 32) << 16);
    const uint32_t tq = tl + (uint32_t)(g * C::kSet), ts = tl + (uint32_t)(C::kScratch + g * N);
    const int n_blocks = SUB ? 3 * p.c0 + 2 * p.c1 : 3 * p.c0;
    uint32_t aph = 0;
    // (after an abort the loops run on without waiting, so that every thread passes every barrier)
    for (int u = blockIdx.x; u < p.n_units; u += gridDim.x) {
      const int t = u / p.n_tiles, n0 = (u - t * p.n_tiles) * N;
      const int yy = t / p.tiles_x, x0 = (t - yy * p.tiles_x) * 128;
      const int Y = SUB ? yy : 2 * yy + g, X = SUB ? 2 * (x0 + q) + g : x0 + q;
      float acc[N];
#pragma unroll
      for (int j = 0; j < N; ++j) acc[j] = 0.0f;
      for (int k = 0; k < n_blocks; ++k) {
        if (!*abort_flag) mbar_wait(&accf[g], aph, abort_flag);
        tc_fence_after();
        if constexpr (N == 32) {
          uint32_t a[32];
          tmem_ld32(tq, a);
#pragma unroll
          for (int j = 0; j < 32; ++j) acc[j] += __uint_as_float(a[j]);
        } else {
          uint32_t a[32], b[32];
          tmem_ld32x2(tq, tq + 32, a, b);
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            acc[j] += __uint_as_float(a[j]);
            acc[32 + j] += __uint_as_float(b[j]);
          }
        }
        if (k == n_blocks - 1) {  // the corrections, summed over the whole unit
#pragma unroll
          for (int c = 0; c < N; c += 32) {
            uint32_t a[32], b[32];
            tmem_ld32x2(tq + (uint32_t)(N + c), tq + (uint32_t)(2 * N + c), a, b);
#pragma unroll
            for (int j = 0; j < 32; ++j) acc[c + j] += __uint_as_float(a[j]) + __uint_as_float(b[j]);
          }
        }
        tc_fence_before();
        mbar_arrive(&acce[g]);
        aph ^= 1u;
      }
      // The sums of N = 64 pass through TMEM, so that one copy of the code below
      // takes both groups of 32 channels: unrolled over registers it runs once
      // per unit out of a cold instruction cache.
      if constexpr (N > 32) {
#pragma unroll
        for (int c = 0; c < N; c += 32) tmem_st32(ts + (uint32_t)c, acc + c);
        tmem_wait_st();
      }
      const bool inside = Y < p.H && X < p.W;
#pragma unroll 1
      for (int c = 0; c < N; c += 32) {
        float v[32];
        if constexpr (N > 32) {
          uint32_t a[32];
          tmem_ld32(ts + (uint32_t)c, a);
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(a[j]);
        } else {
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = acc[j];
        }
        finish<N, SUB>(p, v, n0 + c, Y, X, x0, yy, q, g, gt, inside, s_bias, s_head, sO, &tmO);
      }
    }
    if (gt == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem_base, C::kTmem);
  if (threadIdx.x == 0 && *abort_flag) atomicAdd(p.err, 1ull);
}

// Weight parts [taps][3][coutp][cinp] from w32 [cout][3][3][cin], channels
// [off, off + cnt) (zero beyond cnt and cout).  16 taps: the decoder's
// low-resolution part, tap ((py 2 + px) 2 + oy) 2 + ox = the sum of the 3x3
// taps that land on low-resolution row i + py - 1 + oy, column
// j + px - 1 + ox of output pixel (2i + py, 2j + px), summed in FP64 and
// rounded once to FP32.
__global__ void x3_weights_kernel(const float* __restrict__ w32, int cout, int cin, int off, int cnt, int taps,
                                  int coutp, int cinp, __nv_bfloat16* __restrict__ out) {
  const int64_t n = (int64_t)taps * coutp * cinp;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int c = (int)(i % cinp), co = (int)(i / cinp % coutp), t = (int)(i / ((int64_t)cinp * coutp));
    float w = 0.0f;
    if (c < cnt && co < cout) {
      const float* wc = w32 + (size_t)co * 9 * cin + off + c;
      if (taps == 9) {
        w = wc[(size_t)t * cin];
      } else {
        const int py = t >> 3, px = (t >> 2) & 1, oy = (t >> 1) & 1, ox = t & 1;
        double s = 0.0;
        for (int dy = -1; dy <= 1; ++dy)
          for (int dx = -1; dx <= 1; ++dx)
            if ((py + dy + 2) / 2 - 1 == py - 1 + oy && (px + dx + 2) / 2 - 1 == px - 1 + ox)
              s += (double)wc[(size_t)((dy + 1) * 3 + dx + 1) * cin];
        w = (float)s;
      }
    }
    __nv_bfloat16 a, b, d;
    split3(w, a, b, d);
    __nv_bfloat16* o = out + ((int64_t)t * 3 * coutp + co) * cinp + c;
    o[0] = a;
    o[(int64_t)coutp * cinp] = b;
    o[2 * (int64_t)coutp * cinp] = d;
  }
}

// FP32 [pixel][c] -> parts [pixel][3][cp] (channels beyond c zero); eight channels per thread.
__global__ void __launch_bounds__(256) x3_split_kernel(const float* __restrict__ in, int64_t npx, int c, int cp, int vec,
                                                       __nv_bfloat16* __restrict__ out) {
  ART_PDL_ENTRY();
  const int k8 = cp / 8;
  const int64_t n = npx * k8;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t px = i / k8;
    const int c0 = (int)(i - px * k8) * 8;
    const float* s = in + px * c + c0;
    float f[8];
    if (vec && c0 + 8 <= c) {
      const float4 u = __ldg(reinterpret_cast<const float4*>(s)), v = __ldg(reinterpret_cast<const float4*>(s) + 1);
      f[0] = u.x, f[1] = u.y, f[2] = u.z, f[3] = u.w, f[4] = v.x, f[5] = v.y, f[6] = v.z, f[7] = v.w;
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j) f[j] = c0 + j < c ? s[j] : 0.0f;
    }
    __align__(16) __nv_bfloat16 v[3][8];
#pragma unroll
    for (int j = 0; j < 8; ++j) split3(f[j], v[0][j], v[1][j], v[2][j]);
#pragma unroll
    for (int pl = 0; pl < 3; ++pl)
      *reinterpret_cast<uint4*>(out + (px * 3 + pl) * cp + c0) = *reinterpret_cast<uint4*>(v[pl]);
  }
}

// Parts tensor as (channel, x, part, x phase, y): ph = 1, 2 phases stored
// one after the other per row (split), or 2 interleaved ones (pixel 2x + phase).
bool parts_map(PFN_cuTensorMapEncodeTiled_v12000 enc, CUtensorMap* tm, const void* p, int C, int W, int H, int phases,
               bool split, int box_px) {
  const cuuint64_t px = (cuuint64_t)3 * C * 2;
  const int wx = W / phases;
  cuuint64_t dims[5] = {(cuuint64_t)C, (cuuint64_t)wx, 3, (cuuint64_t)phases, (cuuint64_t)H};
  cuuint64_t strides[4] = {phases == 2 && !split ? 2 * px : px, (cuuint64_t)C * 2,
                           phases == 2 && split ? (cuuint64_t)wx * px : px, (cuuint64_t)W * px};
  cuuint32_t box[5] = {(cuuint32_t)kKC, (cuuint32_t)box_px, 3, 1, 1};
  cuuint32_t es[5] = {1, 1, 1, 1, 1};
  return enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(p), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool weights_map(PFN_cuTensorMapEncodeTiled_v12000 enc, CUtensorMap* tm, const void* w, int cinp, int coutp, int taps,
                 int n) {
  cuuint64_t dims[4] = {(cuuint64_t)cinp, (cuuint64_t)coutp, 3, (cuuint64_t)taps};
  cuuint64_t strides[3] = {(cuuint64_t)cinp * 2, (cuuint64_t)cinp * coutp * 2, (cuuint64_t)cinp * coutp * 6};
  cuuint32_t box[4] = {(cuuint32_t)kKC, (cuuint32_t)n, 3, 1};
  cuuint32_t es[4] = {1, 1, 1, 1};
  return enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(w), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int N, bool SUB>
art_status launch_n(art_ctx* ctx, const X3Conv& c) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
  const ConvLayer& L = *c.layer;
  const int coutp = x3_cout_pad(L.cout);
  CUtensorMap tmA, tmU, tmB, tmV, tmO;
  bool ok = parts_map(enc, &tmA, c.in, c.cs, c.W, c.H, SUB ? 2 : 1, true, kHalo) &&
            weights_map(enc, &tmB, L.wx, c.cs, coutp, 9, N);
  tmU = tmA;
  tmV = tmB;
  if (SUB)
    ok = ok && parts_map(enc, &tmU, c.up, c.cu, c.W / 2, c.H / 2, 1, false, kHalo) &&
         weights_map(enc, &tmV, L.wxu, c.cu, coutp, 16, N);
  tmO = tmA;
  if (c.planes)
    ok = ok && parts_map(enc, &tmO, c.planes, L.cout, c.W, c.H, SUB || c.psplit ? 2 : 1, c.psplit != 0,
                         c.psplit ? 64 : 128);
  if (!ok) return fail(ctx, ART_ERR_CUDA, "cuTensorMapEncodeTiled (FP32 parts) failed");
  Params p{};
  p.H = c.H;
  p.W = c.W;
  p.tiles_x = ((SUB ? c.W / 2 : c.W) + 127) / 128;
  p.n_tiles = coutp / N;
  p.n_units = p.tiles_x * (SUB ? c.H : (c.H + 1) / 2) * p.n_tiles;  // (sub: output rows, else row pairs)
  p.c0 = c.cs / kKC;
  p.c1 = SUB ? c.cu / kKC : 0;
  p.act = c.act;
  p.cout = L.cout;
  p.bias = L.b32;
  p.store = c.planes != nullptr;
  p.psplit = c.psplit;
  p.pool = (__nv_bfloat16*)c.pool;
  p.out = c.out;
  p.head_w = c.head ? c.head->w32 : nullptr;
  p.head_b = c.head ? c.head->b32 : nullptr;
  p.out_n = c.head ? c.head->cout : L.cout;
  p.out_ld = c.out_ld;
  p.out_off = c.out_off;
  p.out_vec = p.out_n == 4 && c.out_ld == 4 && c.out_off == 0 && (reinterpret_cast<uintptr_t>(c.out) & 15) == 0;
  p.in = (const __nv_bfloat16*)c.in;
  p.up = (const __nv_bfloat16*)c.up;
  p.cin = L.cin;
  p.cs = c.cs;
  p.cu = SUB ? c.cu : 0;
  p.w32 = L.w32;
  p.err = ctx->d_status + kStTcError;
  auto kfn = conv_x3_kernel<N, SUB>;
  cudaError_t e = cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<N>::kSmem);
  if (e != cudaSuccess) return cuda_fail(ctx, e, "conv_x3 shared memory attribute");
  ART_LAUNCH_PDL(ctx, "conv_x3", kfn, std::min(p.n_units, ctx->num_sms), kThreads, Cfg<N>::kSmem, tmA, tmU, tmB, tmV, tmO,
                 p);
  return ART_OK;
}

}  // namespace

int x3_cin_pad(int c) { return (c + kKC - 1) / kKC * kKC; }
int x3_cout_pad(int c) { return c <= 32 ? 32 : c; }

bool x3_net_ok(const art_net_desc& d) {
  if (tensor_map_encoder() == nullptr) return false;
  auto width_ok = [](int c) { return c <= kMaxCout && (c == 32 || c % 64 == 0); };
  if (d.arch == ART_NET_TINY) return d.ch[0] == 32 && d.cout <= 32;
  bool ok = d.ch[0] == 32 && d.cout <= 4;
  for (int c : d.ch) ok = ok && width_ok(c);
  if (d.arch == ART_NET_TWO_BRANCH) ok = ok && d.ach[0] == 32 && width_ok(d.ach[1]);
  return ok;
}

size_t x3_weight_elems(int cout, int cin, int taps) { return (size_t)taps * 3 * x3_cout_pad(cout) * x3_cin_pad(cin); }

void launch_x3_weights(art_ctx* ctx, const ConvLayer& L, int off, int cnt, int taps, __nv_bfloat16* out) {
  const int64_t n = (int64_t)taps * x3_cout_pad(L.cout) * x3_cin_pad(cnt);
  const int grid = (int)std::min<int64_t>((n + 255) / 256, 4096);
  ART_LAUNCH(ctx, "x3_weights", x3_weights_kernel, grid, 256, 0, L.w32, L.cout, L.cin, off, cnt, taps,
             x3_cout_pad(L.cout), x3_cin_pad(cnt), out);
}

void launch_x3_split(art_ctx* ctx, const float* in, int64_t npx, int c, __nv_bfloat16* out) {
  const int cp = x3_cin_pad(c);
  const int vec = c % 4 == 0 && (reinterpret_cast<uintptr_t>(in) & 15) == 0;
  const int64_t n = npx * (cp / 8);
  const int grid = (int)std::min<int64_t>((n + 255) / 256, (int64_t)ctx->num_sms * 16);
  ART_LAUNCH_PDL(ctx, "x3_split", x3_split_kernel, grid, 256, 0, in, npx, c, cp, vec, out);
}

art_status launch_x3_conv(art_ctx* ctx, const X3Conv& c) {
  if (c.layer->cout <= 32) return c.up ? launch_n<32, true>(ctx, c) : launch_n<32, false>(ctx, c);
  return c.up ? launch_n<64, true>(ctx, c) : launch_n<64, false>(ctx, c);
}

}  // namespace art
