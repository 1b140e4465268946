// epilogue.cuh -- the common 32-bit forms of the integer epilogue (Eq. 2 on Eq. 6's sum) and the
// packed stores that the tensor-core kernels share.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "common.cuh"

namespace aqd {
namespace tc {

// The 32-bit requant (every R = 31 + shift >= 33): rhu(u M0, R) = (mulhi(u, M0) + 2^(R-33)) >>
// (R-32), as the low product word cannot carry into the rounded result; the clip of Eq. 2 is
// one min.relu (max(min(x, qmax), 0)).
__device__ __forceinline__ uint32_t requant32(int32_t u, const int4& f, int qmax) {
  return (uint32_t)__vimin_s32_relu((__mulhi(u, f.y) + f.z) >> f.w, qmax);
}

// The same for any R: rhu in one variable shift, floor((v + 2^(r-1)) / 2^r) = floor((floor(v / 2^(r-1)) + 1) / 2)
__device__ __forceinline__ int64_t rhu1(int64_t v, int r) { return r > 0 ? ((v >> (r - 1)) + 1) >> 1 : v; }
__device__ __forceinline__ int32_t requant64(int32_t u, int32_t m0, int r, int32_t qmax) {
  const int64_t v = rhu1((int64_t)u * m0, r);
  return v < 0 ? 0 : (v > qmax ? qmax : (int32_t)v);
}

// 16 codes < 2^bits as byte-words (word j: channels 4j..4j+3, one per byte) -> their place in the
// packed row (the layout of common.cuh: word w of the 2/4/8-bit layout holds its channels 4k..4k+3
// in bit field k of every byte; a 3-bit group of 32 channels is two 2-bit words of the low bits
// and one word of bit 2, channel i at bit 8 (i%4) + i/4). ch: the first channel, a multiple of
// 16; top: bit 2 of the group's first half (3-bit codes), kept for the second.
__device__ __forceinline__ void store_codes16(uint8_t* yrow, int ch, const uint32_t (&bw)[4], int bits, uint32_t& top) {
  if (bits == 4) {
    *reinterpret_cast<uint2*>(yrow + (ch >> 1)) = make_uint2(bw[0] | (bw[1] << 4), bw[2] | (bw[3] << 4));
  } else if (bits == 2) {
    *reinterpret_cast<uint32_t*>(yrow + (ch >> 2)) = bw[0] | (bw[1] << 2) | (bw[2] << 4) | (bw[3] << 6);
  } else if (bits == 8) {
    *reinterpret_cast<uint4*>(yrow + ch) = make_uint4(bw[0], bw[1], bw[2], bw[3]);
  } else {
    const int half = (ch >> 4) & 1;
    uint32_t* g = reinterpret_cast<uint32_t*>(yrow + (ch >> 5) * 12);
    g[half] = (bw[0] & 0x03030303u) | ((bw[1] & 0x03030303u) << 2) | ((bw[2] & 0x03030303u) << 4) |
              ((bw[3] & 0x03030303u) << 6);
    uint32_t h = 0u;
#pragma unroll
    for (int j = 0; j < 4; ++j) h |= ((bw[j] >> 2) & 0x01010101u) << j;
    if (half) g[2] = top | (h << 4);
    else top = h;
  }
}

// 32 bytes of a row, 32-byte aligned: one store of a whole sector
__device__ __forceinline__ void store_sector(uint8_t* p, const uint32_t (&a)[4], const uint32_t (&b)[4]) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(a[0]), "r"(a[1]), "r"(a[2]),
               "r"(a[3]), "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3])
               : "memory");
}
__device__ __forceinline__ void store_words8(uint8_t* p, const uint32_t* w) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(w[0]), "r"(w[1]), "r"(w[2]),
               "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
               : "memory");
}
// A whole 32-channel group: the byte-words of its halves to their place in the packed row (see
// store_codes16)
__device__ __forceinline__ void store_codes32(uint8_t* yrow, int ch, const uint32_t (&a)[4], const uint32_t (&b)[4], int bits) {
  if (bits == 4) {
    *reinterpret_cast<uint4*>(yrow + (ch >> 1)) =
        make_uint4(a[0] | (a[1] << 4), a[2] | (a[3] << 4), b[0] | (b[1] << 4), b[2] | (b[3] << 4));
  } else if (bits == 2) {
    *reinterpret_cast<uint2*>(yrow + (ch >> 2)) =
        make_uint2(a[0] | (a[1] << 2) | (a[2] << 4) | (a[3] << 6), b[0] | (b[1] << 2) | (b[2] << 4) | (b[3] << 6));
  } else if (bits == 8) {
    *reinterpret_cast<uint4*>(yrow + ch) = make_uint4(a[0], a[1], a[2], a[3]);
    *reinterpret_cast<uint4*>(yrow + ch + 16) = make_uint4(b[0], b[1], b[2], b[3]);
  } else {
    uint32_t top = 0u;
    store_codes16(yrow, ch, a, bits, top);
    store_codes16(yrow, ch + 16, b, bits, top);
  }
}
}  // namespace tc
}  // namespace aqd
