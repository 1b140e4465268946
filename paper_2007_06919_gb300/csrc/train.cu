// train.cu -- the training-side steps of AQD (Sec. 3.1.2, Sec. 3.2.2) on the GPU:
//   * the quantizers with learnable intervals, Eq. 2 (activations, [0, nu]) and Eq. 3
//     (weights, [-nu, nu]): fake-quantized values and their integer codes;
//   * their backward under the Straight-Through Estimator: the input gradient and the
//     interval's gradient (a sum over the tensor);
//   * the per-level batch statistics of the multi-level batch normalization.
// All three stream their tensors once (HBM-bound). Every rounding decision is taken in float32
// with explicit round-to-nearest operations in the order the equations state (no fused
// multiply-adds), so a code is decided exactly as a float32 restatement decides it; sums run
// in float32 over short runs and in float64 beyond.
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "kernels.h"

namespace aqd {
namespace trn {

constexpr int kThreads = 256;

// x / b correctly rounded, for a divisor known in advance with its correctly rounded reciprocal r
// (Markstein, "Computation of elementary functions on the IBM RISC System/6000 processor", 1990):
// q0 = x r is within 2 ulp of the quotient; one correction by the remainder makes it faithful;
// the remainder is then exact, and the second correction rounds as the exact quotient does.
// Needs the remainders not to underflow: |x| >= 2^-100 or x = 0, 2^-20 <= b <= 2^20.
// 5 instructions and no branch; the compiler's division is a call-like sequence with a slow path,
// and two of them per element bounded the backward pass.
__device__ __forceinline__ float div_known(float x, float b, float r) {
  const float q0 = __fmul_rn(x, r);
  const float q1 = __fmaf_rn(__fmaf_rn(-q0, b, x), r, q0);
  return __fmaf_rn(__fmaf_rn(-q1, b, x), r, q1);
}

// The constants of one call.
struct Quant {
  float nu, rnu;  // the interval and its reciprocal
  float q, rq;    // Q = 2^b - 1 and its reciprocal
  float s;        // nu / Q
};

// x / nu. Beyond twice the interval only its side matters (every use is a clip or a comparison with
// +-1; a NaN counts as the lower side, as the clips below take it), so x is clamped there first.
// kKnown: 2^-20 <= nu <= 2^20 (the host's choice); tiny x take the division itself.
template <bool kKnown>
__device__ __forceinline__ float ratio(float x, const Quant& k) {
  if constexpr (!kKnown) return __fdiv_rn(x, k.nu);
  const float c = fminf(fmaxf(x, -2.0f * k.nu), 2.0f * k.nu);
  const float v = div_known(c, k.nu, k.rnu);
  if (__builtin_expect(fabsf(c) < 0x1p-100f && c != 0.0f, 0)) return __fdiv_rn(c, k.nu);
  return v;
}
// floor(t) for 0 <= t < 2^22: the sum with 2^23 rounded down holds it in its low bits
__device__ __forceinline__ float floor_code(float t, uint32_t& code) {
  const float m = __fadd_rd(t, 8388608.0f);
  code = __float_as_uint(m) & 0xFFu;
  return __fsub_rn(m, 8388608.0f);
}

// One element of Eq. 2 / Eq. 3: the code eta and the fake-quantized value.
template <bool kWeight, bool kKnown>
__device__ __forceinline__ float quant_one(float x, const Quant& k, uint32_t& eta_out) {
  const float v = ratio<kKnown>(x, k);
  if constexpr (kWeight) {
    // eta = round((clip(w / nu, -1, 1) + 1) / 2 * Q), w_bar = (2 eta / Q - 1) nu
    const float c = fminf(fmaxf(v, -1.0f), 1.0f);
    const float eta = floor_code(__fadd_rn(__fmul_rn(__fmul_rn(__fadd_rn(c, 1.0f), 0.5f), k.q), 0.5f), eta_out);
    return __fmul_rn(__fsub_rn(div_known(__fmul_rn(eta, 2.0f), k.q, k.rq), 1.0f), k.nu);
  } else {
    // eta = round(clip(x / nu, 0, 1) * Q), x_bar = eta * nu / Q (s = nu / Q)
    const float c = fminf(fmaxf(v, 0.0f), 1.0f);
    return __fmul_rn(floor_code(__fadd_rn(__fmul_rn(c, k.q), 0.5f), eta_out), k.s);
  }
}

// Streaming passes, bound by HBM. Each thread takes kUnroll units a grid apart per step with all their
// loads issued first: one at a time left too few bytes in flight. A unit is four values, or one where
// an address is not a multiple of 16. Measured on 16x100x168x256 values: forward 113 -> 91 us (9 bytes a
// value), backward 240 -> 120 us (12), backward at odd addresses 387 -> 170.
// kStream: evict-first accesses, for tensors larger than L2 together (33M values 50.5 -> 49.4 us); smaller
// ones are left for what reads them next (8M values read and written again from L2 11.7 -> 9.8).
template <int kVec>
struct Unit;
template <>
struct Unit<4> {
  using F = float4;
  using C = uint32_t;
  static constexpr int kUnroll = 4;
};
template <>
struct Unit<1> {
  using F = float;
  using C = uint8_t;
  static constexpr int kUnroll = 8;
};
template <bool kStream, class T>
__device__ __forceinline__ T load(const T* p) {
  if constexpr (kStream) return __ldcs(p);
  else return __ldg(p);
}
template <bool kStream, class T>
__device__ __forceinline__ void store(T* p, T v) {
  if constexpr (kStream) __stcs(p, v);
  else *p = v;
}

template <bool kWeight, bool kKnown>
__device__ __forceinline__ float quant_unit(float v, const Quant& k, uint8_t& code) {
  uint32_t e;
  const float o = quant_one<kWeight, kKnown>(v, k, e);
  code = (uint8_t)e;
  return o;
}
template <bool kWeight, bool kKnown>
__device__ __forceinline__ float4 quant_unit(const float4& v, const Quant& k, uint32_t& codes) {
  uint32_t e0, e1, e2, e3;
  const float4 o = make_float4(quant_one<kWeight, kKnown>(v.x, k, e0), quant_one<kWeight, kKnown>(v.y, k, e1),
                               quant_one<kWeight, kKnown>(v.z, k, e2), quant_one<kWeight, kKnown>(v.w, k, e3));
  codes = e0 | (e1 << 8) | (e2 << 16) | (e3 << 24);
  return o;
}

template <bool kWeight, bool kKnown, int kVec, bool kStream>
__global__ void __launch_bounds__(kThreads) fake_quant_kernel(const float* __restrict__ x, int64_t n, const Quant k,
                                                              float* __restrict__ y, uint8_t* __restrict__ codes) {
  using F = typename Unit<kVec>::F;
  using C = typename Unit<kVec>::C;
  constexpr int kUnroll = Unit<kVec>::kUnroll;
  const int64_t units = n / kVec, step = (int64_t)gridDim.x * kThreads;
  for (int64_t u0 = (int64_t)blockIdx.x * kThreads + threadIdx.x; u0 < units; u0 += step * kUnroll) {
    F v[kUnroll];
#pragma unroll
    for (int j = 0; j < kUnroll; ++j)
      if (u0 + j * step < units) v[j] = load<kStream>(reinterpret_cast<const F*>(x) + u0 + j * step);
#pragma unroll
    for (int j = 0; j < kUnroll; ++j) {
      const int64_t u = u0 + j * step;
      if (u >= units) break;
      C c;
      const F o = quant_unit<kWeight, kKnown>(v[j], k, c);
      if (y) store<kStream>(reinterpret_cast<F*>(y) + u, o);
      if (codes) store<kStream>(reinterpret_cast<C*>(codes) + u, c);
    }
  }
  // the tail past the last whole vector (kVec = 4: at most 3 elements), by block 0
  if (kVec > 1 && blockIdx.x == 0 && threadIdx.x < n - units * kVec) {
    const int64_t i = units * kVec + threadIdx.x;
    uint32_t e;
    const float o = quant_one<kWeight, kKnown>(x[i], k, e);
    if (y) y[i] = o;
    if (codes) codes[i] = (uint8_t)e;
  }
}

// One element of the STE backward: the input gradient and d y / d nu.
template <bool kWeight, bool kKnown>
__device__ __forceinline__ float dquant_one(float x, float gy, const Quant& k, float& dnu) {
  const float v = ratio<kKnown>(x, k);
  uint32_t code;
  bool inside;
  if constexpr (kWeight) {
    inside = v > -1.0f && v < 1.0f;
    const float c = fminf(fmaxf(v, -1.0f), 1.0f);
    const float eta = floor_code(__fadd_rn(__fmul_rn(__fmul_rn(__fadd_rn(c, 1.0f), 0.5f), k.q), 0.5f), code);
    const float slope = __fsub_rn(__fsub_rn(div_known(__fmul_rn(eta, 2.0f), k.q, k.rq), 1.0f), v);  // 2 eta / Q - 1 - w / nu
    dnu = inside ? slope : (v >= 1.0f ? 1.0f : -1.0f);
  } else {
    inside = v > 0.0f && v < 1.0f;
    const float c = fminf(fmaxf(v, 0.0f), 1.0f);
    const float eta = floor_code(__fadd_rn(__fmul_rn(c, k.q), 0.5f), code);
    const float slope = __fsub_rn(div_known(eta, k.q, k.rq), v);  // eta / Q - x / nu
    dnu = inside ? slope : (v >= 1.0f ? 1.0f : 0.0f);
  }
  return inside ? gy : 0.0f;
}

template <bool kWeight, bool kKnown>
__device__ __forceinline__ float dquant_unit(float x, float g, const Quant& k, float& acc) {
  float d;
  const float o = dquant_one<kWeight, kKnown>(x, g, k, d);
  acc = __fadd_rn(acc, __fmul_rn(g, d));
  return o;
}
template <bool kWeight, bool kKnown>
__device__ __forceinline__ float4 dquant_unit(const float4& x, const float4& g, const Quant& k, float& acc) {
  float d0, d1, d2, d3;
  const float4 o = make_float4(dquant_one<kWeight, kKnown>(x.x, g.x, k, d0), dquant_one<kWeight, kKnown>(x.y, g.y, k, d1),
                               dquant_one<kWeight, kKnown>(x.z, g.z, k, d2), dquant_one<kWeight, kKnown>(x.w, g.w, k, d3));
  acc = __fadd_rn(acc, __fadd_rn(__fadd_rn(__fmul_rn(g.x, d0), __fmul_rn(g.y, d1)),
                                 __fadd_rn(__fmul_rn(g.z, d2), __fmul_rn(g.w, d3))));
  return o;
}

// gx (STE) and one float64 partial of sum(gy * dy/dnu) per block: float32 over runs of 16 units
// of a thread, float64 across runs and threads.
template <bool kWeight, bool kKnown, int kVec, bool kStream>
__global__ void __launch_bounds__(kThreads) fake_quant_backward_kernel(const float* __restrict__ x,
                                                                       const float* __restrict__ gy, int64_t n,
                                                                       const Quant k, float* __restrict__ gx,
                                                                       double* __restrict__ partial) {
  using F = typename Unit<kVec>::F;
  constexpr int kUnroll = Unit<kVec>::kUnroll;
  static_assert(16 % kUnroll == 0, "a run is whole steps");
  __shared__ double red[kThreads / 32];
  float acc = 0.0f;
  double accd = 0.0;
  int run = 0;
  const int64_t units = n / kVec, step = (int64_t)gridDim.x * kThreads;
  for (int64_t u0 = (int64_t)blockIdx.x * kThreads + threadIdx.x; u0 < units; u0 += step * kUnroll) {
    F xv[kUnroll], gv[kUnroll];
#pragma unroll
    for (int j = 0; j < kUnroll; ++j) {
      if (u0 + j * step >= units) break;
      xv[j] = load<kStream>(reinterpret_cast<const F*>(x) + u0 + j * step);
      gv[j] = load<kStream>(reinterpret_cast<const F*>(gy) + u0 + j * step);
    }
#pragma unroll
    for (int j = 0; j < kUnroll; ++j) {
      const int64_t u = u0 + j * step;
      if (u >= units) break;
      const F o = dquant_unit<kWeight, kKnown>(xv[j], gv[j], k, acc);
      if (gx) store<kStream>(reinterpret_cast<F*>(gx) + u, o);
    }
    run += kUnroll;
    if (run == 16) { accd += (double)acc; acc = 0.0f; run = 0; }
  }
  if (kVec > 1 && blockIdx.x == 0 && threadIdx.x < n - units * kVec) {
    const int64_t i = units * kVec + threadIdx.x;
    float d;
    const float o = dquant_one<kWeight, kKnown>(x[i], gy[i], k, d);
    if (gx) gx[i] = o;
    accd += (double)__fmul_rn(gy[i], d);
  }
  accd += (double)acc;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) accd += __shfl_xor_sync(0xffffffffu, accd, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = accd;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kThreads / 32; ++w) t += red[w];
    partial[blockIdx.x] = t;
  }
}

// the blocks' partials summed in a fixed order (deterministic)
__global__ void sum_partials_kernel(const double* __restrict__ partial, int nparts, double* __restrict__ out) {
  __shared__ double red[kThreads];
  double t = 0.0;
  for (int i = threadIdx.x; i < nparts; i += kThreads) t += partial[i];
  red[threadIdx.x] = t;
  __syncthreads();
  for (int w = kThreads / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = red[0];
}

// Per-level batch statistics: a 1D grid whose blocks are dealt to the levels in proportion to
// their pixels (at least one each); block b of level l (of B_l) takes pixels b, b + B_l, ...;
// thread t channels t, t + 256, ... (consecutive threads read consecutive channels of one
// pixel). Each channel's values are shifted by the level's first pixel
// (k = z[0][ch]) and summed as (z - k) and (z - k)^2: float32 over runs of 32 pixels, float64
// beyond, written as one float64 partial pair per (level, block, channel). A thread's loads for 8
// pixels are issued before they are summed.
struct StatsArgs {
  const float* z[kMaxJobs];
  int64_t pixels[kMaxJobs];
  int32_t nblk[kMaxJobs], blk0[kMaxJobs];  // blocks of level l: [blk0[l], blk0[l] + nblk[l])
  int32_t levels, c;
};

__global__ void __launch_bounds__(kThreads) bn_stats_partial_kernel(const StatsArgs a, double* __restrict__ s1,
                                                                    double* __restrict__ s2) {
  int l = 0;
  while (l + 1 < a.levels && (int)blockIdx.x >= a.blk0[l + 1]) ++l;
  const int b = (int)blockIdx.x - a.blk0[l], B = a.nblk[l];
  const float* z = a.z[l];
  const int64_t P = a.pixels[l];
  for (int ch = threadIdx.x; ch < a.c; ch += kThreads) {
    const float k = P > 0 ? __ldg(z + ch) : 0.0f;
    double d1 = 0.0, d2 = 0.0;
    float f1 = 0.0f, f2 = 0.0f;
    int run = 0;
    // 8 of this block's pixels per step, their loads issued together (pixels past the level
    // contribute d = 0)
    constexpr int kU = 8;
    for (int64_t p0 = b; p0 < P; p0 += (int64_t)B * kU) {
      float d[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int64_t p = p0 + (int64_t)u * B;
        d[u] = p < P ? __fsub_rn(__ldg(z + p * a.c + ch), k) : 0.0f;
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        f1 = __fadd_rn(f1, d[u]);
        f2 = __fadd_rn(f2, __fmul_rn(d[u], d[u]));
      }
      run += kU;
      if (run >= 32) { d1 += (double)f1; d2 += (double)f2; f1 = f2 = 0.0f; run = 0; }
    }
    d1 += (double)f1;
    d2 += (double)f2;
    const int64_t o = (int64_t)blockIdx.x * a.c + ch;
    s1[o] = d1;
    s2[o] = d2;
  }
}

// The same for c % 4 == 0 and 16-byte aligned levels: a thread sums four channels over the pixels of
// its block's rows (16-byte loads, 8 pixels' loads issued together), and the block's rows of one
// channel are added in a fixed order in shared memory. One channel per thread kept a quarter of
// the bytes in flight. 367 MB in five levels of 256 channels: 111 -> 58 us.
__global__ void __launch_bounds__(kThreads) bn_stats_partial4_kernel(const StatsArgs a, double* __restrict__ s1,
                                                                     double* __restrict__ s2) {
  __shared__ double red1[kThreads * 4], red2[kThreads * 4];
  int l = 0;
  while (l + 1 < a.levels && (int)blockIdx.x >= a.blk0[l + 1]) ++l;
  const int b = (int)blockIdx.x - a.blk0[l], B = a.nblk[l];
  const float* z = a.z[l];
  const int64_t P = a.pixels[l];
  const int quads = a.c >> 2;
  // quads <= kThreads: kThreads / quads rows of threads, else one row over kThreads quads at a time
  const int qt = quads < kThreads ? quads : kThreads;
  const int rows = kThreads / qt;
  const int row = threadIdx.x / qt, q0 = threadIdx.x - row * qt;
  for (int qb = 0; qb < quads; qb += qt) {
    const int quad = qb + q0;
    double d1[4] = {0.0, 0.0, 0.0, 0.0}, d2[4] = {0.0, 0.0, 0.0, 0.0};
    if (row < rows && quad < quads && P > 0) {
      const float4 k = __ldg(reinterpret_cast<const float4*>(z) + quad);
      float f1[4] = {0.0f, 0.0f, 0.0f, 0.0f}, f2[4] = {0.0f, 0.0f, 0.0f, 0.0f};
      int run = 0;
      constexpr int kU = 8;
      const int64_t stride = (int64_t)B * rows;
      for (int64_t p0 = (int64_t)b * rows + row; p0 < P; p0 += stride * kU) {
        float4 v[kU];
        if (p0 + (kU - 1) * stride < P) {  // (no branch between the loads)
#pragma unroll
          for (int u = 0; u < kU; ++u)
            v[u] = __ldcs(reinterpret_cast<const float4*>(z + (p0 + u * stride) * a.c) + quad);
        } else {
#pragma unroll
          for (int u = 0; u < kU; ++u) {
            const int64_t p = p0 + u * stride;
            v[u] = p < P ? __ldcs(reinterpret_cast<const float4*>(z + p * a.c) + quad) : k;  // (past the level: d = 0)
          }
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
          const float e[4] = {__fsub_rn(v[u].x, k.x), __fsub_rn(v[u].y, k.y), __fsub_rn(v[u].z, k.z), __fsub_rn(v[u].w, k.w)};
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            f1[i] = __fadd_rn(f1[i], e[i]);
            f2[i] = __fadd_rn(f2[i], __fmul_rn(e[i], e[i]));
          }
        }
        run += kU;
        if (run >= 32) {
#pragma unroll
          for (int i = 0; i < 4; ++i) { d1[i] += (double)f1[i]; d2[i] += (double)f2[i]; f1[i] = f2[i] = 0.0f; }
          run = 0;
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) { d1[i] += (double)f1[i]; d2[i] += (double)f2[i]; }
    }
    __syncthreads();  // the previous quads' sums have been read
#pragma unroll
    for (int i = 0; i < 4; ++i) { red1[i * kThreads + threadIdx.x] = d1[i]; red2[i * kThreads + threadIdx.x] = d2[i]; }
    __syncthreads();
    if (row == 0 && quad < quads) {
      const int64_t o = (int64_t)blockIdx.x * a.c + 4 * quad;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        double t1 = 0.0, t2 = 0.0;
        for (int r = 0; r < rows; ++r) { t1 += red1[i * kThreads + r * qt + q0]; t2 += red2[i * kThreads + r * qt + q0]; }
        s1[o + i] = t1;
        s2[o + i] = t2;
      }
    }
  }
}

// mean = k + S1 / N, var = S2 / N - (S1 / N)^2 (biased, as batch normalization's training
// statistics), in float64 from the blocks' partials. Block (g, l) finishes channels 8 g .. of level
// l (channels along x: y takes 65,535 blocks, 524,280 channels): thread (r, ch), r < 32, adds the
// partials of blocks r, r + 32, ..., then one thread per channel the 32 sums, both in a fixed order.
// One thread per channel over all partials was a serial chain of about 600 loads and double additions
// on five SMs: 120 -> 17 us.
constexpr int kFinCh = 8;
__global__ void __launch_bounds__(kThreads) bn_stats_final_kernel(const StatsArgs a, const double* __restrict__ s1,
                                                                  const double* __restrict__ s2,
                                                                  double* __restrict__ mean, double* __restrict__ var) {
  constexpr int kR = kThreads / kFinCh;
  __shared__ double r1[kR][kFinCh], r2[kR][kFinCh];
  const int l = blockIdx.y, c8 = threadIdx.x % kFinCh, r = threadIdx.x / kFinCh;
  const int64_t ch = (int64_t)kFinCh * blockIdx.x + c8;
  const int64_t P = a.pixels[l];
  double t1 = 0.0, t2 = 0.0;
  if (ch < a.c) {
    const double* p1 = s1 + (int64_t)a.blk0[l] * a.c + ch;
    const double* p2 = s2 + (int64_t)a.blk0[l] * a.c + ch;
#pragma unroll 4
    for (int b = r; b < a.nblk[l]; b += kR) {
      t1 += __ldg(p1 + (int64_t)b * a.c);
      t2 += __ldg(p2 + (int64_t)b * a.c);
    }
  }
  r1[r][c8] = t1;
  r2[r][c8] = t2;
  __syncthreads();
  if (r != 0 || ch >= a.c) return;
#pragma unroll 8
  for (int i = 1; i < kR; ++i) { t1 += r1[i][c8]; t2 += r2[i][c8]; }
  const double k = P > 0 ? (double)a.z[l][ch] : 0.0;
  const double m1 = P > 0 ? t1 / (double)P : 0.0;
  const double v = P > 0 ? t2 / (double)P - m1 * m1 : 0.0;
  mean[(int64_t)l * a.c + ch] = k + m1;
  var[(int64_t)l * a.c + ch] = v > 0.0 ? v : 0.0;
}

inline Quant quant_of(float nu, int32_t bits) {
  const float q = (float)((1 << bits) - 1);
  return Quant{nu, 1.0f / nu, q, 1.0f / q, nu / q};
}
// the intervals div_known takes (anything a trained network has); others use the division itself
inline bool known_divisor(float nu) { return nu >= 0x1p-20f && nu <= 0x1p20f; }

// Blocks for a pass over n values: a step of kUnroll units per thread, but two blocks per SM before a thread
// takes more than one (65,536 values forward in 16 blocks took 2.7 us, in 64 2.0); at most cap.
template <int kVec>
inline unsigned grid_for(int64_t n, int sms, int cap) {
  const int64_t units = n / kVec, per = kThreads * Unit<kVec>::kUnroll;
  const int64_t one = (units + kThreads - 1) / kThreads, full = (units + per - 1) / per;
  int64_t b = one < 2 * sms ? one : 2 * sms;
  if (full > b) b = full;
  return (unsigned)(b < 1 ? 1 : (b > cap ? cap : b));
}
// Tensors that leave L2 (129 MB) anyway
inline bool stream_size(int64_t bytes) { return bytes > (int64_t)128 << 20; }

// go(weight, known divisor, values per unit) with the choice as types
template <class Go>
void dispatch(bool weight, bool known, bool v4, Go&& go) {
  using std::integral_constant;
  auto vec = [&](auto w, auto kn) { v4 ? go(w, kn, integral_constant<int, 4>{}) : go(w, kn, integral_constant<int, 1>{}); };
  auto kn = [&](auto w) { known ? vec(w, std::true_type{}) : vec(w, std::false_type{}); };
  weight ? kn(std::true_type{}) : kn(std::false_type{});
}

}  // namespace trn

static int check_launch_t(const char* what, std::string* err) {
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { *err = std::string(what) + ": " + cudaGetErrorString(e); return 3; }
  return 0;
}

int launch_fake_quant(const float* x, int64_t n, float nu, int32_t bits, bool weight, float* y, uint8_t* codes,
                      cudaStream_t stream, std::string* err) {
  if (n == 0) return 0;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const trn::Quant k = trn::quant_of(nu, bits);
  const bool known = trn::known_divisor(nu);
  const bool v4 = ((uintptr_t)x % 16 == 0) && ((uintptr_t)y % 16 == 0) && ((uintptr_t)codes % 4 == 0);
  if (sms <= 0) sms = 152;
  const unsigned g = v4 ? trn::grid_for<4>(n, sms, sms * 8) : trn::grid_for<1>(n, sms, sms * 8);
  const bool big = trn::stream_size(n * (4 + (y ? 4 : 0) + (codes ? 1 : 0)));
  auto go = [&](auto w, auto kn, auto vec) {
    if (big) trn::fake_quant_kernel<w.value, kn.value, vec.value, true><<<g, trn::kThreads, 0, stream>>>(x, n, k, y, codes);
    else trn::fake_quant_kernel<w.value, kn.value, vec.value, false><<<g, trn::kThreads, 0, stream>>>(x, n, k, y, codes);
  };
  trn::dispatch(weight, known, v4, go);
  return check_launch_t("fake_quant launch", err);
}

int launch_fake_quant_backward(const float* x, const float* gy, int64_t n, float nu, int32_t bits, bool weight,
                               float* gx, double* gnu, double* partial, int32_t max_parts, cudaStream_t stream,
                               std::string* err) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const trn::Quant k = trn::quant_of(nu, bits);
  const bool known = trn::known_divisor(nu);
  const bool v4 = ((uintptr_t)x % 16 == 0) && ((uintptr_t)gy % 16 == 0) && ((uintptr_t)gx % 16 == 0);
  if (sms <= 0) sms = 152;
  int cap = sms * 3;  // one wave
  if (cap > max_parts) cap = max_parts;
  const unsigned g = v4 ? trn::grid_for<4>(n, sms, cap) : trn::grid_for<1>(n, sms, cap);
  const bool big = trn::stream_size(n * (gx ? 12 : 8));
  auto go = [&](auto w, auto kn, auto vec) {
    if (big) trn::fake_quant_backward_kernel<w.value, kn.value, vec.value, true><<<g, trn::kThreads, 0, stream>>>(x, gy, n, k, gx, partial);
    else trn::fake_quant_backward_kernel<w.value, kn.value, vec.value, false><<<g, trn::kThreads, 0, stream>>>(x, gy, n, k, gx, partial);
  };
  trn::dispatch(weight, known, v4, go);
  trn::sum_partials_kernel<<<1, trn::kThreads, 0, stream>>>(partial, (int)g, gnu);
  return check_launch_t("fake_quant_backward launch", err);
}

// blocks of the statistics pass over all levels together: about 4 per SM
int bn_stats_blocks(int32_t levels) { return 152 * 4 > levels ? 152 * 4 : levels; }

int launch_bn_level_stats(const float* const* z, const int64_t* pixels, int32_t levels, int32_t c, double* mean,
                          double* var, double* work, cudaStream_t stream, std::string* err) {
  trn::StatsArgs a{};
  int64_t ptot = 0;
  for (int l = 0; l < levels; ++l) { a.z[l] = z[l]; a.pixels[l] = pixels[l]; ptot += pixels[l]; }
  a.levels = levels; a.c = c;
  // four channels per thread where every level's pixels are whole 16-byte pieces
  bool v4 = c % 4 == 0;
  for (int l = 0; l < levels; ++l) v4 = v4 && (pixels[l] == 0 || (uintptr_t)z[l] % 16 == 0);
  // one block per level, the rest in proportion to the pixels: the sum stays within the cap (one
  // wave: 3 blocks per SM of the four-channel form, whose threads hold 8 loads of 16 bytes)
  const int cap = v4 ? bn_stats_blocks(levels) / 4 * 3 : bn_stats_blocks(levels);
  int total = 0;
  for (int l = 0; l < levels; ++l) {
    const int extra = ptot > 0 ? (int)((double)(cap - levels) * (double)pixels[l] / (double)ptot) : 0;
    a.nblk[l] = 1 + extra;
    a.blk0[l] = total;
    total += a.nblk[l];
  }
  double* s1 = work;
  double* s2 = work + (size_t)cap * c;
  if (v4) trn::bn_stats_partial4_kernel<<<(unsigned)total, trn::kThreads, 0, stream>>>(a, s1, s2);
  else trn::bn_stats_partial_kernel<<<(unsigned)total, trn::kThreads, 0, stream>>>(a, s1, s2);
  const dim3 fin(((unsigned)c + trn::kFinCh - 1) / trn::kFinCh, (unsigned)levels);
  trn::bn_stats_final_kernel<<<fin, trn::kThreads, 0, stream>>>(a, s1, s2, mean, var);
  return check_launch_t("bn_level_stats launch", err);
}

}  // namespace aqd
