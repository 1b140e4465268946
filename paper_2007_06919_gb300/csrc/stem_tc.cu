// stem_tc.cu -- the network's first convolution (Eq. 4 on the 8-bit image codes, then the
// integer epilogue: Eq. 6 bias and Eq. 2 rescale + clip) on the tcgen05 tensor cores.
//
// The image has 3 channels of 8-bit codes (0..255) and the weights are signed integers
// |w| <= 127, so the implicit GEMM has K = 7 * 7 * 3 = 147 and codes too wide for the E4M3
// embedding of conv_tc.cu. Here both operands are F16 (kind::f16): integers up to 2048 are
// exact in F16, every product is an integer, and the FP32 accumulator is exact while
// K * 255 * max|w| < 2^24 (the host checks it; 147 * 255 * 128 < 2^23).
//
// Activation encoding: the F16 bit pattern 0x6400 | x is exactly 1024 + x for x in
// [0, 1023], so one byte permute (PRMT) turns two code bytes into two F16 values 1024 + x
// and one exact F16x2 subtraction of 1024 leaves x. Padding positions (outside the image)
// hold x = 0; K positions past the receptive field meet zero weights.
//
// K order: kernel row r, then the 21 contiguous bytes (7 columns x 3 channels) of that row
// of the receptive field, padded to 22 so that element pairs stay 4-byte aligned:
// kk = 22 r + j. 7 x 22 = 154 is padded to 160 = 10 MMAs of K = 16. Operands use the
// no-swizzle K-major layout of 8-row x 16-byte core matrices (K-adjacent core matrices 128 B
// apart, 8-row groups 2560 B apart).
//
// Two kernels: stem_rows_kernel for stride 2 (a network's first conv), whose operand is the image
// row itself, and stem_kernel for other strides, small maps and widths that leave strips of 128 columns
// partly empty, which builds each pixel's receptive field.
//
// stem_kernel, per CTA (one per SM, persistent over tiles of 128 consecutive output pixels):
//   warps 0..7   epilogue: tcgen05.ld (warp w reads TMEM lanes 32 (w % 4).., the two warps of a
//                lane quarter every other 32-column group), Eq. 6 + Eq. 2, bit-pack, store
//   warp  8      TMEM allocation + one thread issuing tcgen05.mma (M=128, N=cout, K=16)
//   warps 9..16  im2col producers: two threads per tile row (kernel rows 0..3 / 4..6),
//                word loads of the receptive field, PRMT to F16, 16-byte stores
// The weights (cout x 160 F16) stay in shared memory for the whole launch. Every wait is
// bounded: on expiry the CTA latches kStatusTimeout and unwinds.
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <mutex>

#include "common.cuh"
#include "epilogue.cuh"
#include "kernels.h"
#include "tc_ptx.cuh"

namespace aqd {
namespace stem {

using namespace aqd::tc;

constexpr int kKH = 7, kKW = 7, kC = 3;
constexpr int kSeg = kKW * kC;             // 21 bytes of one receptive-field row
constexpr int kLs = kSeg + (kSeg & 1);     // 22: K elements per kernel row
constexpr int kKUsed = kKH * kLs;          // 154
constexpr int kK = (kKUsed + 15) / 16 * 16;  // 160
constexpr int kKSteps = kK / 16;
constexpr int kLBO = 128;                  // K-adjacent core matrices
constexpr int kSBO = (kK / 8) * 128;       // 8-row groups
constexpr int kStageA = 128 * kK * 2;      // one tile's A operand
constexpr int kSplitR = 4;                 // producer half 0: kernel rows [0, 4); half 1: [4, 7)
static_assert((kSplitR * kLs) % 8 == 0, "the producer halves must meet on a core-matrix boundary");
static_assert(kLs <= 24, "a receptive-field row must fit six realigned words");
// 17 warps: at most 5 per SM sub-partition, so 96 registers per thread. (4 epilogue warps, one per
// sub-partition, ran two 32-column groups each per tile as one chain of dependent instructions:
// 8 x 400 x 672 x 64 outputs 203 -> 173 us.)
constexpr int kEpiWarps = 8, kWarpMma = kEpiWarps, kWarpProd0 = kEpiWarps + 1, kProdWarps = 8;
constexpr int kThreads = (kWarpProd0 + kProdWarps) * 32;
constexpr uint32_t kF16Pair1024 = 0x64006400u;

struct StemParams {
  const uint8_t* x;       // [n][h][w][3] 8-bit codes
  uint8_t* y;             // [n][ho][wo] rows of y_row_bytes
  int64_t x_bytes;        // bytes of x (bounds of the word loads)
  int32_t n, h, w, ho, wo, stride, pad;
  int32_t m_total, hw_out; // n * ho * wo (< 2^31, checked on the host), ho * wo
  int32_t cout, n_pad, out_bits, level, total_tiles, stages, tmem_cols;
  int32_t strips, nbuf_log2;  // (rows kernel) strips of 128 output columns, accumulators
  int64_t y_row_bytes;
  const int32_t* m0;
  const int8_t* shift;
  const int32_t* bias;
  const uint16_t* w_f16;  // [cout][147] F16 values, K order (r, s, c)
  uint32_t off_b, off_cst, off_bar;
  uint32_t* status;
};


__device__ __forceinline__ uint64_t sdesc_noswz(uint32_t saddr) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)(kLBO >> 4) << 16;
  d |= (uint64_t)(kSBO >> 4) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version; swizzle field 0 = none
  return d;
}

// Two code bytes (bytes 0-1 or 2-3 of u) -> two F16 values: 1024 + x by a byte permute,
// then 1024 subtracted (exact).
__device__ __forceinline__ uint32_t f16_pair(uint32_t u, bool high) {
  const uint32_t b = __byte_perm(u, 0x64646464u, high ? 0x4342u : 0x4140u);
  uint32_t r;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(b), "r"(kF16Pair1024));
  return r;
}

// One producer thread: tile row m's K elements of kernel rows [R0, R1) (plus the zero tail
// past 154 when kTail), written as core-matrix rows of 16 bytes. Kernel row r of the
// receptive field is 21 contiguous code bytes; inside the image they are read as seven
// aligned words and realigned with funnel shifts (the 22nd byte meets a zero weight), at the
// image border byte by byte with out-of-image columns and rows read as code 0.
template <int R0, int R1, bool kTail>
__device__ __forceinline__ void build_half(const StemParams& p, int mg, uint8_t* row_dst) {
  constexpr int kWordsRows = (R1 - R0) * kLs / 2;
  constexpr int kWords = kWordsRows + (kTail ? (kK - kKUsed) / 2 : 0);
  static_assert(kWords % 4 == 0, "whole core-matrix rows");
  uint32_t o[kWords];
  const bool valid = mg < p.m_total;
  int img = 0, ho = 0, wo = 0;
  if (valid) {
    img = mg / p.hw_out;
    const int rem = mg - img * p.hw_out;
    ho = rem / p.wo;
    wo = rem - ho * p.wo;
  }
  const int wi0 = wo * p.stride - p.pad;
  const int hi0 = ho * p.stride - p.pad;
  // byte offset of (img, hi0 + R0, wi0): one kernel row further is one image row further
  const int64_t a0 = (((int64_t)img * p.h + hi0 + R0) * p.w + wi0) * kC;
  const int64_t row_step = (int64_t)p.w * kC;
  const int64_t a4_last = (a0 + (R1 - 1 - R0) * row_step) & ~(int64_t)3;
  const bool interior = valid && hi0 + R0 >= 0 && hi0 + R1 <= p.h && wi0 >= 0 && wi0 + kKW <= p.w &&
                        a4_last + 28 <= p.x_bytes;
  if (interior) {
#pragma unroll
    for (int r = R0; r < R1; ++r) {
      const int64_t a = a0 + (r - R0) * row_step;
      const uint32_t* src = reinterpret_cast<const uint32_t*>(p.x + (a & ~(int64_t)3));
      const uint32_t shr = 8u * (uint32_t)(a & 3);
      uint32_t w[7];
#pragma unroll
      for (int i = 0; i < 7; ++i) w[i] = __ldg(src + i);
#pragma unroll
      for (int q = 0; q < kLs / 2; ++q)
        o[(r - R0) * (kLs / 2) + q] = f16_pair(__funnelshift_r(w[q / 2], w[q / 2 + 1], shr), q & 1);
    }
  } else {
#pragma unroll
    for (int r = R0; r < R1; ++r) {
      const int hi = hi0 + r;
      uint32_t u[6] = {0u, 0u, 0u, 0u, 0u, 0u};
      if (valid && hi >= 0 && hi < p.h) {
        const int64_t a = a0 + (r - R0) * row_step;
#pragma unroll
        for (int j = 0; j < kSeg; ++j) {
          const int wi = wi0 + j / kC;
          if (wi >= 0 && wi < p.w) u[j / 4] |= (uint32_t)__ldg(p.x + a + j) << (8 * (j % 4));
        }
      }
#pragma unroll
      for (int q = 0; q < kLs / 2; ++q) o[(r - R0) * (kLs / 2) + q] = f16_pair(u[q / 2], q & 1);
    }
  }
#pragma unroll
  for (int q = kWordsRows; q < kWords; ++q) o[q] = 0u;
#pragma unroll
  for (int c = 0; c < kWords / 4; ++c)
    *reinterpret_cast<uint4*>(row_dst + (R0 * kLs / 8 + c) * kLBO) = make_uint4(o[4 * c], o[4 * c + 1], o[4 * c + 2], o[4 * c + 3]);
}

// Eq. 6 -> Eq. 2 of 16 columns as the definition states them (some R < 33): byte-words of the codes. Not inlined: its registers and code stay out of the common form.
__device__ __noinline__ uint4 general_cols(uint32_t taddr, const EpiChan* c, int out_bits) {
  uint32_t v[16];
  tmem_ld16(taddr, v);
  tmem_wait_ld();
  reg_fence16(v);
  uint32_t bw[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int i = 0; i < 16; ++i)
    bw[i / 4] |= (uint32_t)requant64(add_sat(__float2int_rn(__uint_as_float(v[i])), c[i].bias), c[i].m0, c[i].r,
                                     (1 << out_bits) - 1) << (8 * (i % 4));
  return make_uint4(bw[0], bw[1], bw[2], bw[3]);
}

// int32 outputs of 16 columns: sum + bias, saturating.
__device__ __noinline__ void sums_int32(uint32_t taddr, const EpiChan* c, uint4* y, bool valid) {
  uint32_t v[16];
  tmem_ld16(taddr, v);
  tmem_wait_ld();
  reg_fence16(v);
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = (uint32_t)add_sat(__float2int_rn(__uint_as_float(v[i])), c[i].bias);
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (valid) y[q] = make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
  __syncwarp();
}

// One float add turns an exact sum v, |v| < 2^22, into the int32 v + kMagicBits: the mantissa of
// 1.5 x 2^23 + v. (The conversion instruction runs at a sixteenth of the add's rate.)
constexpr float kMagic = 12582912.0f;
constexpr uint32_t kMagicBits = 0x4B400000u;

// Per-channel constants of the launch's level: {bias - kMagicBits, M0, 2^(R-33), R-32} and the int64
// form. The 32-bit form holds (and 1 stays in *s_fast) where every R >= 33 (code outputs), |bias| <= 2^30, and
// every |sum| < 2^22 (weights_small); int32 outputs then need no saturation either.
__device__ __forceinline__ void load_channels(const StemParams& p, int4* cst4, EpiChan* cste, int* s_fast) {
  int fast = 1;
  for (int n = threadIdx.x; n < p.n_pad; n += blockDim.x) {
    EpiChan ec{};
    int4 c4 = make_int4(0, 0, 0, 0);
    if (n < p.cout) {
      const int64_t idx = (int64_t)p.level * p.cout + n;
      ec.bias = p.bias ? p.bias[idx] : 0;
      if (ec.bias < -(1 << 30) || ec.bias > (1 << 30)) fast = 0;
      c4.x = (int)((uint32_t)ec.bias - kMagicBits);
      if (p.out_bits != 32) {
        ec.m0 = p.m0[idx];
        const int r = 31 + p.shift[idx];
        ec.r = (int8_t)r;
        if (r >= 33) c4 = make_int4(c4.x, ec.m0, 1 << (r - 33), r - 32);
        else fast = 0;
      }
    }
    cst4[n] = c4;
    cste[n] = ec;
  }
  if (!fast) atomicAnd(s_fast, 0);
}

__device__ __forceinline__ uint32_t abs_f16(uint16_t w) {
  return (uint32_t)__half2int_rn(__ushort_as_half(w & 0x7FFFu));
}
// a channel's sum of |w| (the warp's lanes each hold a part): every |sum of products| < 2^22
__device__ __forceinline__ bool weights_small(uint32_t part) { return __reduce_add_sync(0xffffffffu, part) * 255u < (1u << 22); }

// kTiles accumulators' columns of one output pixel each: the 32-column groups 0, 2, .. (odd = 0)
// or 1, 3, .. (odd = 1), 16 columns at a time (cout is a multiple of 16). Constants are read from
// shared memory once for all tiles; release() hands the accumulators back after the last read.
// kInt: int32 outputs (an instantiation of its own: beside the codes' form in one loop, codes took 2 to 9% longer).
template <int kTiles, bool kInt, class Release>
__device__ __forceinline__ void drain_pixels(const StemParams& p, const uint32_t (&tbase)[kTiles], uint8_t* const (&yrow)[kTiles],
                                             const bool (&valid)[kTiles], int odd, bool fast, const int4* cst4,
                                             const EpiChan* cste, Release&& release) {
  const int qmax = (1 << (p.out_bits & 15)) - 1;
  uint32_t top[kTiles] = {};  // (3-bit codes: see store_codes16)
  [[maybe_unused]] const bool sectors = (reinterpret_cast<uintptr_t>(p.y) & 31) == 0;  // (int32 rows are multiples of 64 bytes)
  if (fast) {
    if (32 * odd >= p.cout) release();
#pragma unroll 1
    for (int c0 = 32 * odd, next; c0 < p.cout; c0 = next) {
      next = c0 + ((c0 & 16) ? 48 : 16);
      uint32_t v[kTiles][16], bw[kTiles][4] = {};
#pragma unroll
      for (int k = 0; k < kTiles; ++k) tmem_ld16(tbase[k] + (uint32_t)c0, v[k]);
      tmem_wait_ld();
#pragma unroll
      for (int k = 0; k < kTiles; ++k) reg_fence16(v[k]);
      if (next >= p.cout) release();
      if constexpr (kInt) {
        // (a tile's row at a time, whole sectors where the rows allow it: the two tiles' 16-byte pieces in turn
        // left half-written sectors behind, 256 channels of 4 x 240 x 320 outputs 230 us against 112)
#pragma unroll
        for (int k = 0; k < kTiles; ++k) {
#pragma unroll
          for (int i = 0; i < 16; ++i) v[k][i] = (uint32_t)(__float_as_int(__uint_as_float(v[k][i]) + kMagic) + cst4[c0 + i].x);
          if (!valid[k]) continue;
          uint8_t* row = yrow[k] + 4 * c0;
          if (sectors) {
            store_words8(row, &v[k][0]);
            store_words8(row + 32, &v[k][8]);
          } else {
#pragma unroll
            for (int q = 0; q < 4; ++q)
              reinterpret_cast<uint4*>(row)[q] = make_uint4(v[k][4 * q], v[k][4 * q + 1], v[k][4 * q + 2], v[k][4 * q + 3]);
          }
        }
      } else {
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int4 c = cst4[c0 + i];
#pragma unroll
          for (int k = 0; k < kTiles; ++k)
            bw[k][i / 4] += requant32(__float_as_int(__uint_as_float(v[k][i]) + kMagic) + c.x, c, qmax) << (8 * (i % 4));
        }
#pragma unroll
        for (int k = 0; k < kTiles; ++k)
          if (valid[k]) store_codes16(yrow[k], c0, bw[k], p.out_bits, top[k]);
      }
    }
    return;
  }
#pragma unroll
  for (int k = 0; k < kTiles; ++k) {
#pragma unroll 1
    for (int c0 = 32 * odd; c0 < p.cout; c0 += (c0 & 16) ? 48 : 16) {
      if constexpr (kInt) {
        sums_int32(tbase[k] + (uint32_t)c0, cste + c0, reinterpret_cast<uint4*>(yrow[k]) + (c0 >> 2), valid[k]);
      } else {
        const uint4 r = general_cols(tbase[k] + (uint32_t)c0, cste + c0, p.out_bits);
        __syncwarp();
        const uint32_t bw[4] = {r.x, r.y, r.z, r.w};
        if (valid[k]) store_codes16(yrow[k], c0, bw, p.out_bits, top[k]);
      }
    }
  }
  release();
}

template <bool kInt>
__global__ void __launch_bounds__(kThreads, 1) stem_kernel(const __grid_constant__ StemParams p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t s_a = smem_u32(smem);
  const uint32_t s_b = s_a + p.off_b;
  // per output channel of the launch's level: {bias, M0, 2^(R-33), R-32} and the int64 form
  int4* cst4 = reinterpret_cast<int4*>(smem + p.off_cst);
  EpiChan* cste = reinterpret_cast<EpiChan*>(smem + p.off_cst + 256 * sizeof(int4));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + p.off_bar);
  const int S = p.stages;
  const uint32_t b_full = smem_u32(bars);
  const uint32_t b_empty = b_full + 8 * S;
  const uint32_t b_tfull = b_empty + 8 * S;
  const uint32_t b_tempty = b_tfull + 16;
  const uint32_t b_final = b_tempty + 16;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * S + 5);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* s_fast = reinterpret_cast<int*>(tmem_slot + 2);  // AND over channels of "R >= 33"
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(b_full + 8 * s, kProdWarps);
      mbar_init(b_empty + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(b_tfull + 8 * b, 1);
      mbar_init(b_tempty + 8 * b, kEpiWarps);
    }
    mbar_init(b_final, 1);
    *abort_flag = 0;
    *s_fast = 1;
    fence_barrier_init();
  }
  if (warp == kWarpMma) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(tmem_slot)), "r"(p.tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  grid_dep_wait();
  if (threadIdx.x == 0) grid_dep_launch();

  // weights -> F16 B operand (n_pad rows x 160, core-matrix layout), a warp per channel with all its loads
  // issued together (element by element over the block, and the sums of |w| in a pass of their own, a call of 256
  // channels and 32 x 32 outputs took 30 us, now 16)
#pragma unroll 2
  for (int n = warp; n < p.n_pad; n += kThreads / 32) {
    uint32_t part = 0;
#pragma unroll
    for (int q = 0; q < (kK / 2 + 31) / 32; ++q) {
      const int kk = 2 * (lane + 32 * q);  // (kLs is even: a pair lies in one kernel row)
      const int r = kk / kLs, j = kk - r * kLs;
      uint16_t w0 = 0, w1 = 0;  // (F16 zero)
      if (n < p.cout && r < kKH) {
        const uint16_t* w = p.w_f16 + (int64_t)n * (kKH * kSeg) + r * kSeg + j;
        w0 = w[0];
        if (j + 1 < kSeg) w1 = w[1];
      }
      part += abs_f16(w0) + abs_f16(w1);
      if (kk < kK)
        *reinterpret_cast<uint32_t*>(smem + p.off_b + (n / 8) * kSBO + (kk / 8) * kLBO + (n % 8) * 16 + (kk % 8) * 2) =
            (uint32_t)w0 | ((uint32_t)w1 << 16);
    }
    if (!weights_small(part) && lane == 0) atomicAnd(s_fast, 0);
  }
  load_channels(p, cst4, cste, s_fast);
  fence_proxy_async();  // generic-proxy stores of B -> visible to the MMA
  __syncthreads();
  const bool fast = *s_fast != 0;

  const int first = blockIdx.x, stride_t = gridDim.x;
  if (warp == kWarpMma) {
    // ------------------------------------------------------------ MMA issuer
    if (elect_one()) {
      const uint32_t idesc = idesc_e4m3(p.n_pad);  // F16 has the same type code 0
      const uint64_t db0 = sdesc_noswz(s_b);
      uint32_t s = 0, ph = 0, lt = 0;
      bool ok = true;
      for (int t = first; t < p.total_tiles && ok; t += stride_t, ++lt) {
        const uint32_t buf = lt & 1;
        if (!mbar_poll(b_tempty + 8 * buf, ((lt >> 1) & 1) ^ 1, abort_flag)) { ok = false; break; }
        tc_fence_after();
        if (!mbar_poll(b_full + 8 * s, ph, abort_flag)) { ok = false; break; }
        const uint64_t da0 = sdesc_noswz(s_a + s * kStageA);
        const uint32_t d = tmem_base + buf * (uint32_t)p.n_pad;
#pragma unroll
        for (int i = 0; i < kKSteps; ++i)  // K = 16 = two core matrices per step
          mma_f16(d, da0 + (uint64_t)((2 * i * kLBO) >> 4), db0 + (uint64_t)((2 * i * kLBO) >> 4), idesc,
                  i > 0 ? 1u : 0u);
        mma_commit(b_empty + 8 * s);
        mma_commit(b_tfull + 8 * buf);
        if (++s == (uint32_t)S) { s = 0; ph ^= 1; }
      }
      if (!ok) fail(abort_flag, p.status);
      mma_commit(b_final);
      if (!mbar_wait(b_final, 0, abort_flag)) fail(abort_flag, p.status);
    }
  } else if (warp >= kWarpProd0) {
    // ------------------------------------------------------------ im2col producers
    const int pt = threadIdx.x - kWarpProd0 * 32;  // 0..255
    const int row = pt & 127, half = pt >> 7;
    uint32_t s = 0, ph = 0;
    bool ok = true;
    for (int t = first; t < p.total_tiles; t += stride_t) {
      if (!mbar_wait(b_empty + 8 * s, ph ^ 1, abort_flag)) { ok = false; break; }
      uint8_t* dst = smem + s * kStageA + (row / 8) * kSBO + (row % 8) * 16;
      const int mg = t * 128 + row;
      if (half == 0) build_half<0, kSplitR, false>(p, mg, dst);
      else build_half<kSplitR, kKH, true>(p, mg, dst);
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(b_full + 8 * s);
      if (++s == (uint32_t)S) { s = 0; ph ^= 1; }
    }
    if (!ok) fail(abort_flag, p.status);
  } else {
    // ------------------------------------------------------------ epilogue (warps 0..7)
    const int quarter = warp & 3;
    const uint32_t lane_base = tmem_base + ((uint32_t)(quarter * 32) << 16);
    uint32_t lt = 0;
    bool ok = true;
    for (int t = first; t < p.total_tiles; t += stride_t, ++lt) {
      const uint32_t buf = lt & 1;
      const int mg = t * 128 + quarter * 32 + lane;
      const bool valid = mg < p.m_total;
      uint8_t* yrow = p.y + (int64_t)(valid ? mg : 0) * p.y_row_bytes;
      if (!mbar_wait(b_tfull + 8 * buf, (lt >> 1) & 1, abort_flag)) { ok = false; break; }
      tc_fence_after();
      const uint32_t tbase[1] = {lane_base + buf * (uint32_t)p.n_pad};
      uint8_t* const yrows[1] = {yrow};
      const bool valids[1] = {valid};
      drain_pixels<1, kInt>(p, tbase, yrows, valids, warp >> 2, fast, cst4, cste, [&] {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_relaxed(b_tempty + 8 * buf);
      });
    }
    if (!ok) fail(abort_flag, p.status);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kWarpMma) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(p.tmem_cols) : "memory");
  }
}

// ------------------------------------------------------------------ stride 2: no im2col
// With 4 channels per pixel (the fourth 0) in F16 a pixel is 8 bytes, so at stride 2 the receptive
// fields of neighbouring output pixels start 16 bytes apart in an image row: one core-matrix row.
// The image row itself is then the A operand of one kernel row: 8 output pixels are 128 contiguous
// bytes, the next 16 bytes of K lie 16 bytes further (leading offset 16: core matrices overlap), the
// next 8 pixels 128. Seven pixels and an eighth with zero weights are K = 32 per kernel row, 224 in
// all. An image pixel is converted once per tile row pair instead of 12 times, and a CTA's tiles
// go down the rows of a strip of 128 output columns, so that each tile brings two new image rows.
// What bounds it is the epilogue: a sum was converted by F2I (a sixteenth of the add's rate) and added
// with saturation, and 16 bytes of constants were read per output. Two tiles now share each read, and
// one float add converts. 8 x 400 x 672 x 64 4-bit outputs 171 -> 130 us (HBM alone 14); 16 epilogue
// warps in two sets take 141. With the requant left out 93 remain: no one pipe, the issue of its 19 warps.
//   warps 0..7    epilogue, two tiles at a time
//   warp  8       TMEM allocation + one thread issuing tcgen05.mma (M=128, N=cout, 14 of K=16)
//   warps 9..18   producers: two sets of 5 take row pairs in turn, 4 pixels per thread, the words
//                 of the next pair loaded before this one is written
constexpr int kRK = 32 * kKH;                // K
constexpr int kRSBO = (kRK / 8) * 128;       // 8-row groups of the weights
constexpr int kRowUnits = 132;               // 2-pixel units of a strip's row: 127 + 4, and one to make groups whole
constexpr int kRowBytes = kRowUnits * 16;
constexpr int kPairBytes = 2 * kRowBytes;
constexpr int kPairs = 16;                   // ring of row pairs (a tile reads 4)
constexpr int kRowGroups = kRowUnits / 2;    // 4-pixel groups
constexpr int kRSets = 2, kRSetWarps = (2 * kRowGroups + 31) / 32;
constexpr int kREpiWarps = 8, kRWarpMma = kREpiWarps, kRWarpProd0 = kREpiWarps + 1;
constexpr int kRThreads = (kRWarpProd0 + kRSets * kRSetWarps) * 32;
constexpr int kMaxBufs = 4;
static_assert((kPairs & (kPairs - 1)) == 0 && kPairs > 4, "ring");

// A CTA's contiguous tiles [t, end), numbered (image, strip, output row), as runs down one strip.
struct Run {
  int t, end, img, strip, h0, len;
  __device__ __forceinline__ Run(const StemParams& p, int t0, int t1) : t(t0), end(t1) {
    const int col = t / p.ho;
    h0 = t - col * p.ho;
    img = col / p.strips;
    strip = col - img * p.strips;
    len = min(p.ho - h0, end - t);
  }
  __device__ __forceinline__ bool done() const { return t >= end; }
  __device__ __forceinline__ void next(const StemParams& p) {
    t += len;
    h0 = 0;
    if (++strip == p.strips) { strip = 0; ++img; }
    len = min(p.ho, end - t);
  }
};

// 12 code bytes of 4 pixels as loaded: aligned words and the shift that realigns them, and the bytes to keep.
struct Group {
  uint32_t w[4];
  uint32_t shr, keep;  // keep: bit i = pixel i lies inside the image
};

__device__ __forceinline__ Group load_group(const StemParams& p, int img, int hi, int wi) {
  Group g{};
  if (hi < 0 || hi >= p.h || wi <= -4 || wi >= p.w) return g;
  const int64_t a = (((int64_t)img * p.h + hi) * p.w + wi) * kC;
  const int64_t a4 = a & ~(int64_t)3;
  g.shr = 8u * (uint32_t)(a & 3);
  g.keep = 15u;
  if (wi < 0) g.keep &= 15u << -wi;
  if (wi + 4 > p.w) g.keep &= 15u >> (wi + 4 - p.w);
  if (a4 >= 0 && a4 + 16 <= p.x_bytes) {
    const uint32_t* src = reinterpret_cast<const uint32_t*>(p.x + a4);
#pragma unroll
    for (int i = 0; i < 4; ++i) g.w[i] = __ldg(src + i);
  } else {  // the first and last bytes of the tensor
#pragma unroll
    for (int i = 0; i < 16; ++i)
      if (a4 + i >= 0 && a4 + i < p.x_bytes) g.w[i / 4] |= (uint32_t)__ldg(p.x + a4 + i) << (8 * (i % 4));
  }
  return g;
}

__device__ __forceinline__ uint32_t f16_bytes(uint32_t a, uint32_t sel) {  // 1024 + x, minus 1024
  uint32_t r;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(__byte_perm(a, kF16Pair1024, sel)), "r"(kF16Pair1024));
  return r;
}

__device__ __forceinline__ void store_group(const Group& g, uint8_t* dst) {
  uint32_t b[4];
#pragma unroll
  for (int i = 0; i < 3; ++i) b[i] = __funnelshift_r(g.w[i], g.w[i + 1], g.shr);
  b[3] = b[2] >> 8;                              // pixel 3
  b[2] = __funnelshift_r(b[1], b[2], 16);        // pixel 2
  b[1] = __funnelshift_r(b[0], b[1], 24);        // pixel 1
#pragma unroll
  for (int i = 0; i < 4; ++i) b[i] = (g.keep >> i) & 1u ? b[i] : 0u;
  // {x0, x1}, {x2, 0}: bytes of the permute are x, 0x64 and, for the fourth channel, 0x00, 0x64
  *reinterpret_cast<uint4*>(dst) = make_uint4(f16_bytes(b[0], 0x5150u), f16_bytes(b[0], 0x5452u),
                                              f16_bytes(b[1], 0x5150u), f16_bytes(b[1], 0x5452u));
  *reinterpret_cast<uint4*>(dst + 16) = make_uint4(f16_bytes(b[2], 0x5150u), f16_bytes(b[2], 0x5452u),
                                                   f16_bytes(b[3], 0x5150u), f16_bytes(b[3], 0x5452u));
}

__device__ __forceinline__ uint64_t sdesc_offsets(uint32_t saddr, int lbo, int sbo) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)(lbo >> 4) << 16;
  d |= (uint64_t)(sbo >> 4) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version; swizzle field 0 = none
  return d;
}

template <bool kInt>
__global__ void __launch_bounds__(kRThreads, 1) stem_rows_kernel(const __grid_constant__ StemParams p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t s_a = smem_u32(smem);
  const uint32_t s_b = s_a + p.off_b;
  int4* cst4 = reinterpret_cast<int4*>(smem + p.off_cst);
  EpiChan* cste = reinterpret_cast<EpiChan*>(smem + p.off_cst + 256 * sizeof(int4));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + p.off_bar);
  const uint32_t b_full = smem_u32(bars);
  const uint32_t b_empty = b_full + 8 * kPairs;
  const uint32_t b_tfull = b_empty + 8 * kPairs;
  const uint32_t b_tempty = b_tfull + 8 * kMaxBufs;
  const uint32_t b_final = b_tempty + 8 * kMaxBufs;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kPairs + 2 * kMaxBufs + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* s_fast = reinterpret_cast<int*>(tmem_slot + 2);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kPairs; ++s) {
      mbar_init(b_full + 8 * s, kRSetWarps);
      mbar_init(b_empty + 8 * s, 1);
    }
    for (int b = 0; b < kMaxBufs; ++b) {
      mbar_init(b_tfull + 8 * b, 1);
      mbar_init(b_tempty + 8 * b, kREpiWarps);
    }
    mbar_init(b_final, 1);
    *abort_flag = 0;
    *s_fast = 1;
    fence_barrier_init();
  }
  if (warp == kRWarpMma) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(tmem_slot)), "r"(p.tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  grid_dep_wait();
  if (threadIdx.x == 0) grid_dep_launch();

  // weights -> F16 B operand (n_pad rows x 224): kk = 32 r + 4 s + c, zero at s = 7 and c = 3; a
  // warp per channel
  for (int n = warp; n < p.n_pad; n += kRThreads / 32) {
    uint32_t part = 0;
#pragma unroll
    for (int j = 0; j < (kRK / 2 + 31) / 32; ++j) {
      const int kk = 2 * (lane + 32 * j);
      const int r = kk / 32, s = (kk % 32) / 4, c = kk % 4;  // (c is 0 or 2)
      uint16_t w0 = 0, w1 = 0;
      if (n < p.cout && kk < kRK && s < kKW) {
        const uint16_t* w = p.w_f16 + (int64_t)n * (kKH * kSeg) + r * kSeg + s * kC + c;
        w0 = w[0];
        if (c == 0) w1 = w[1];
      }
      part += abs_f16(w0) + abs_f16(w1);
      if (kk < kRK)
        *reinterpret_cast<uint32_t*>(smem + p.off_b + (n / 8) * kRSBO + (kk / 8) * kLBO + (n % 8) * 16 + (kk % 8) * 2) =
            (uint32_t)w0 | ((uint32_t)w1 << 16);
    }
    if (!weights_small(part) && lane == 0) atomicAnd(s_fast, 0);
  }
  load_channels(p, cst4, cste, s_fast);
  fence_proxy_async();  // generic-proxy stores of B -> visible to the MMA
  __syncthreads();
  const bool fast = *s_fast != 0;

  const int share = p.total_tiles / gridDim.x, extra = p.total_tiles - share * gridDim.x;
  const int first = blockIdx.x * share + min((int)blockIdx.x, extra);
  Run run(p, first, first + share + ((int)blockIdx.x < extra));
  bool ok = true;
  if (warp == kRWarpMma) {
    // ------------------------------------------------------------ MMA issuer
    if (elect_one()) {
      const uint32_t idesc = idesc_e4m3(p.n_pad);  // F16 has the same type code 0
      const uint64_t da0 = sdesc_offsets(s_a, 16, 128);
      const uint64_t db0 = sdesc_offsets(s_b, kLBO, kRSBO);
      const uint32_t buf_mask = (1u << p.nbuf_log2) - 1u;
      uint32_t pair = 0, lt = 0;  // first row pair of the tile, tiles done
      for (; !run.done() && ok; run.next(p)) {
        for (uint32_t i = 0; i < 3 && ok; ++i)  // the run's first tile reads four new pairs
          ok = mbar_poll(b_full + 8 * ((pair + i) % kPairs), ((pair + i) / kPairs) & 1, abort_flag);
        for (int i = 0; i < run.len && ok; ++i, ++pair, ++lt) {
          const uint32_t buf = lt & buf_mask;
          ok = mbar_poll(b_tempty + 8 * buf, ((lt >> p.nbuf_log2) & 1) ^ 1, abort_flag) &&
               mbar_poll(b_full + 8 * ((pair + 3) % kPairs), ((pair + 3) / kPairs) & 1, abort_flag);
          if (!ok) break;
          tc_fence_after();
          const uint32_t d = tmem_base + buf * (uint32_t)p.n_pad;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint64_t da = da0 + ((pair + q) % kPairs) * (kPairBytes >> 4);
#pragma unroll
            for (int h = 0; h < 4; ++h) {  // (row, K half) of the pair
              const int r = 2 * q + h / 2;
              if (r < kKH)
                mma_f16(d, da + (uint64_t)(((h / 2) * kRowBytes + (h & 1) * 32) >> 4),
                        db0 + (uint64_t)((4 * r + 2 * (h & 1)) * kLBO >> 4), idesc, q + h > 0 ? 1u : 0u);
            }
          }
          mma_commit(b_tfull + 8 * buf);
          mma_commit(b_empty + 8 * (pair % kPairs));
        }
        for (int i = 0; i < 3 && ok; ++i, ++pair) mma_commit(b_empty + 8 * (pair % kPairs));
      }
      if (!ok) fail(abort_flag, p.status);
      mma_commit(b_final);
      if (!mbar_wait(b_final, 0, abort_flag)) fail(abort_flag, p.status);
    }
  } else if (warp >= kRWarpProd0) {
    // ------------------------------------------------------------ producers
    const int set = (warp - kRWarpProd0) / kRSetWarps;
    const int item = (warp - kRWarpProd0 - set * kRSetWarps) * 32 + lane;
    const bool busy = item < 2 * kRowGroups;
    const int row = item >= kRowGroups, grp = item - row * kRowGroups;
    uint8_t* dst = smem + row * kRowBytes + grp * 32;
    int i = set;  // pair of the run
    auto settle = [&] {  // to the run that holds pair i
      while (!run.done() && i >= run.len + 3) { i -= run.len + 3; run.next(p); }
    };
    auto load = [&] {
      return busy && !run.done()
                 ? load_group(p, run.img, 2 * (run.h0 + i) + row - p.pad, 256 * run.strip - p.pad + 4 * grp)
                 : Group{};
    };
    settle();
    Group cur = load();
    for (uint32_t pair = set; !run.done(); pair += kRSets) {
      i += kRSets;
      settle();
      const Group nxt = load();
      const uint32_t s = pair % kPairs;
      if (!mbar_wait(b_empty + 8 * s, ((pair / kPairs) & 1) ^ 1, abort_flag)) { ok = false; break; }
      if (busy) store_group(cur, dst + s * kPairBytes);
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(b_full + 8 * s);
      cur = nxt;
    }
    if (!ok) fail(abort_flag, p.status);
  } else {
    // ------------------------------------------------------------ epilogue
    const int quarter = warp & 3;
    const uint32_t lane_base = tmem_base + ((uint32_t)(quarter * 32) << 16);
    const uint32_t buf_mask = (1u << p.nbuf_log2) - 1u;
    const int col = quarter * 32 + lane, total = run.end - run.t;
    int i = 0;  // tile of the run
    uint8_t* yrow[2];
    bool valid[2];
    auto take = [&](int k) {  // the next tile's output row of this lane
      valid[k] = false;
      yrow[k] = p.y;
      if (run.done()) return;
      const int wo = run.strip * 128 + col;
      valid[k] = wo < p.wo;
      if (valid[k]) yrow[k] += (((int64_t)run.img * p.ho + run.h0 + i) * p.wo + wo) * p.y_row_bytes;
      if (++i == run.len) { i = 0; run.next(p); }
    };
    for (int lt = 0; lt < total; lt += 2) {
      const uint32_t b0 = lt & buf_mask, b1 = (lt + 1) & buf_mask;
      const bool two = lt + 1 < total;
      take(0);
      take(1);
      if (!mbar_wait(b_tfull + 8 * b0, (lt >> p.nbuf_log2) & 1, abort_flag) ||
          (two && !mbar_wait(b_tfull + 8 * b1, ((lt + 1) >> p.nbuf_log2) & 1, abort_flag))) { ok = false; break; }
      tc_fence_after();
      const uint32_t tbase[2] = {lane_base + b0 * (uint32_t)p.n_pad, lane_base + b1 * (uint32_t)p.n_pad};
      drain_pixels<2, kInt>(p, tbase, yrow, valid, warp >> 2, fast, cst4, cste, [&] {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive_relaxed(b_tempty + 8 * b0);
          if (two) mbar_arrive_relaxed(b_tempty + 8 * b1);
        }
      });
    }
    if (!ok) fail(abort_flag, p.status);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kRWarpMma) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(p.tmem_cols) : "memory");
  }
}

}  // namespace stem

bool stem_applicable(const ConvArgs& a) {
  return a.njobs == 1 && a.x_bits == 8 && a.cin == stem::kC && a.kh == stem::kKH && a.kw == stem::kKW &&
         !a.has_skip && a.cout % 16 == 0 && a.cout <= 256 && a.k_total == stem::kKH * stem::kSeg &&
         a.acc_bound < (1LL << 24);  // K * 255 * max|w|: the FP32 sum is exact
}

int launch_stem(const ConvArgs& a, cudaStream_t stream, std::string* err) {
  using namespace stem;
  const ConvJobDev& jb = a.jobs[0];
  StemParams p{};
  p.x = jb.x;
  p.y = jb.y;
  p.x_bytes = (int64_t)jb.n * jb.h * jb.w * kC;
  p.n = jb.n; p.h = jb.h; p.w = jb.w; p.ho = jb.ho; p.wo = jb.wo;
  p.stride = a.stride; p.pad = a.pad;
  p.cout = a.cout;
  p.n_pad = (a.cout + 15) / 16 * 16;
  p.out_bits = a.out_bits;
  p.level = jb.level;
  p.y_row_bytes = a.y_row_bytes;
  p.m0 = a.m0; p.shift = a.shift; p.bias = a.bias;
  p.w_f16 = a.w_f16;
  p.status = a.status;
  const int64_t m_total = (int64_t)jb.n * jb.ho * jb.wo;
  if (m_total + 128 >= (1LL << 31)) { *err = "stem conv: more than 2^31 output pixels"; return 2; }
  p.m_total = (int32_t)m_total;
  p.hw_out = jb.ho * jb.wo;
  if (m_total == 0) return 0;
  int dev = 0, sms = 0, max_smem = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const uint32_t cst_bytes = (uint32_t)(256 * (sizeof(int4) + sizeof(EpiChan)));
  const uint32_t bar_rest = 16 + 1024;  // TMEM slot + 2 flags, alignment
  p.strips = (jb.wo + 127) / 128;
  // Stride 2: image rows as the operand where there is more than one tile per SM and the strips of 128
  // columns are full enough: a tile of a strip costs the same whatever its columns, 0.4 of a built tile of 128
  // pixels with 16 channels, 0.55 with 32, 0.6, 0.75 and 0.95 with 64, 128 and 256 (the epilogue has the larger
  // share). Rows / built in us, 4-bit or, with 16 channels, int32 outputs: 16 channels, 64 images of 32 x 48 outputs
  // 11.3 / 13.4; 32 channels, 64 of 64 x 64 26.2 / 29.1; 64 channels, 32 of 64 x 72 20.1 / 19.2, of 64 x 80 20.3 /
  // 20.9; 128 channels, 32 of 64 x 80 30.5 / 28.5, of 64 x 96 30.5 / 32.4; 256 channels, 32 of 64 x 96 58 / 54, of 64
  // x 128 59 / 67. Within one tile per SM built tiles start sooner: 64 channels, one image of 100 x 128 8.4 / 7.6.
  const int full = a.cout <= 16 ? 38 : (a.cout <= 32 ? 58 : (a.cout <= 64 ? 77 : (a.cout <= 128 ? 96 : 115)));
  const bool rows = a.stride == 2 && jb.wo >= full * p.strips && (int64_t)jb.n * p.strips * jb.ho > sms;
  uint32_t total = 0;
  if (rows) {
    p.total_tiles = (int32_t)((int64_t)jb.n * p.strips * jb.ho);
    p.nbuf_log2 = 4 * p.n_pad <= 512 ? 2 : 1;
    p.off_b = kPairs * kPairBytes;
    p.off_cst = p.off_b + (uint32_t)p.n_pad * kRK * 2;
    p.off_bar = (p.off_cst + cst_bytes + 15) / 16 * 16;
    total = p.off_bar + 8 * (2 * kPairs + 2 * kMaxBufs + 1) + bar_rest;
  } else {
    p.total_tiles = (int32_t)((m_total + 127) / 128);
    p.nbuf_log2 = 1;
    for (p.stages = 4; p.stages >= 2; --p.stages) {
      p.off_b = (uint32_t)p.stages * kStageA;
      p.off_cst = p.off_b + (uint32_t)p.n_pad * kK * 2;
      p.off_bar = (p.off_cst + cst_bytes + 15) / 16 * 16;
      total = p.off_bar + 8 * (2 * p.stages + 5) + bar_rest;
      if ((int)total <= max_smem) break;
    }
  }
  if ((int)total > max_smem) { *err = "stem conv: shared memory too small"; return 2; }
  p.tmem_cols = 32;
  while (p.tmem_cols < (p.n_pad << p.nbuf_log2)) p.tmem_cols *= 2;
  const auto kern = rows ? (a.out_bits == 32 ? stem_rows_kernel<true> : stem_rows_kernel<false>)
                         : (a.out_bits == 32 ? stem_kernel<true> : stem_kernel<false>);
  static std::once_flag attr_once;
  static cudaError_t attr_err = cudaSuccess;
  std::call_once(attr_once, [&] {
    for (auto k : {stem_rows_kernel<true>, stem_rows_kernel<false>, stem_kernel<true>, stem_kernel<false>})
      if (attr_err == cudaSuccess) attr_err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
  });
  if (attr_err != cudaSuccess) {
    *err = std::string("stem conv: shared-memory attribute: ") + cudaGetErrorString(attr_err);
    return 3;
  }
  const int grid = (int)(p.total_tiles < sms ? p.total_tiles : sms);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(rows ? kRThreads : kThreads);
  cfg.dynamicSmemBytes = total;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, p);
  if (e != cudaSuccess) {
    *err = std::string("stem conv launch: ") + cudaGetErrorString(e);
    return 3;
  }
  return 0;
}

}  // namespace aqd
