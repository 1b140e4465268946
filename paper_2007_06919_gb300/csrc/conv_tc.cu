// conv_tc.cu -- AQD's integer convolution (Eq. 4) as a persistent tcgen05 implicit GEMM
// on sm_103a, with the integer epilogue (Eq. 6 bias, Eq. 7/8 skip, Eq. 2 rescale + clip)
// fused after the TMEM accumulator.
//
// Exact integer arithmetic on the FP8 tensor pipe. sm_103a has no integer tcgen05 MMA
// (kind::i8), so codes are embedded in E4M3 bit patterns: the raw byte n (0..15) of an
// E4M3 value is exactly n * 2^-9 (0..7 subnormal, 8..15 exponent field 1), and a signed
// weight |w| <= 15 is the same byte with the sign bit set. Every product is an integer
// times 2^-18, and the FP32 accumulator holds the exact integer sum times 2^-18 as long as
// K * max|x| * max|w| < 2^24, which the host checks before choosing this kernel.
//
// 2-bit codes on the FP4 pipe (kFp4): E2M1 holds n / 2 exactly for n <= 4, so a code n and a
// weight |w| <= 4 become the E2M1 values n / 2 and w / 2 (raw nibbles n and sign | |w|), every
// product is an integer / 4, and kind::mxf4nvf4 (K = 64 per instruction, one UE8M0 scale
// per 32 K elements, all set to 2^0 in TMEM) accumulates the exact integer sum / 4 in FP32.
// Operands are nibble images (two codes per byte), so a 128-byte K chunk holds 256 codes. A
// nibble image keeps the byte image's row stride (cin bytes) and fills the first cin / 2
// bytes of each row, so its zero border lies where a byte image's does in the same workspace.
//
// 8-bit codes on the F16 pipe (kF16): F16 holds them and weights of any width exactly, every product is an
// integer, and with 8-bit weights the FP32 accumulator is exact over 512 K elements (512 * 255 * 128 <
// 2^24). K runs in segments of that length, each in its own TMEM accumulator; the epilogue warps
// add the segments as int32 in registers. (With narrower weights one segment holds all of K.) The image
// holds F16 values (2 cin bytes a row).
//
// Per CTA (one per SM, persistent over tiles of 128 output pixels x BN channels):
//   warps 0..E-1  epilogue (E = 16, or 8 beside activation producers): tcgen05.ld of the
//              accumulator, integer epilogue, bit-pack, store (warp w reads TMEM lanes
//              32*(w%4)..; the E / 4 warps of a lane quarter split the columns)
//   warp  E    TMEM allocation + one thread issuing tcgen05.mma (kind::f8f6f4, M=128)
//   warp  E+1.. one thread each loading operands with TMA (cp.async.bulk.tensor, SW128)
//   then 8 warps of activation producers (in-kernel variant): im2col gather of packed k-bit codes
//              (zero-fill = the padding code 0), unpack to E4M3 bytes, store into the
//              128B-swizzled K-major operand layout, signal an mbarrier
// Stages of 128 K-bytes (one 128B swizzle atom) circulate between producers and the MMA
// thread; two or four TMEM accumulators let the epilogue of tile i overlap the next MMAs.
// Every wait is bounded: on expiry the CTA latches kStatusTimeout and unwinds.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdio>
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "epilogue.cuh"
#include "kernels.h"
#include "tc_ptx.cuh"

namespace aqd {
namespace tc {

constexpr int BM = 128;            // output pixels per tile and CTA
constexpr int kStageA = BM * 128;  // bytes of A per stage (128-byte K chunks)
constexpr int BK = 128;            // K bytes per stage
// Epilogue warps. The epilogue is a chain of dependent integer instructions per output, and a
// scheduler that holds two such warps issued in a third of its cycles; with four it covers the
// latencies. The in-kernel-unpack variant keeps 8: its producer warps need the registers.
__host__ __device__ constexpr int epi_warps(bool flat) { return flat ? 16 : 8; }
// Producers of the in-kernel-unpack variant: two threads per tile row, each 64 channels of a K chunk, with
// four chunks in flight. (One thread per row and a 128-channel chunk was a chain of 150 instructions on one
// warp per scheduler: ragged 3-bit conv 10.4 -> 9.4 us, small 2-bit conv 11.1 -> 9.6, the 3x3 stride-2 64 -> 128
// conv at batch 8 34 -> 30.)
constexpr int kProdWarps = 8;
// The expanded-activation ("flat") variant has no producer warps: TMA loads both operands, one
// thread the activations and two the weights.
//
// Activations come in slabs: the 128 + kw - 1 image rows that the kw taps of one kernel row read,
// once, and the tap s multiplies the 128 rows from row s of the slab on. The swizzle of an operand
// row depends on its address alone, so a later first row is only a later start address in the
// MMA's descriptor. Weights stay in shared memory for the whole launch where all of them fit, and
// come per tap otherwise. L2 delivers about 70 bytes per clock to each SM, and a 128 x 128-byte
// piece of each operand per 4 MMAs needed all of that: a 3x3 layer's 32 KB per tap are 21.7 KB this
// way, and with 64 channels and resident weights 2.9 KB instead of 10. Together with the MMA
// thread's loop below, at batch 8: 64-channel layer 58 -> 49 us, 256-channel tower layer 72 -> 68, the
// whole detector 1397 -> 1343 (slabs alone, with the loop as it was: 64 and 68 us, 1399).
constexpr int kTmaWarpsFlat = 3;
__host__ __device__ constexpr int tma_warps(bool flat) { return flat ? kTmaWarpsFlat : 1; }
__host__ __device__ constexpr int threads_for(bool flat) {
  return (epi_warps(flat) + 1 + tma_warps(flat) + (flat ? 0 : kProdWarps)) * 32;
}
constexpr int kMaxBufs = 4;    // TMEM accumulators
constexpr int kMaxStages = 16;
constexpr int kStageRow = 20;  // words per row of an int32 staging block: 16 and a pad (conflict-free)

// One layer of a launch: its per-channel tables, the packed output of each job and the
// zero-padded byte image its epilogue writes for the next layer (NULL: none).
struct LayerDev {
  const int32_t* m0;
  const int8_t* shift;
  const int32_t* bias;
  uint8_t* y[kMaxJobs];
  uint8_t* ws_out;
  int32_t ws_nib;  // ws_out holds two 2-bit codes per byte (the next layer runs on the FP4 pipe)
};

// The tensor maps of a launch: the weights of each layer, the weights with half-height
// boxes (half-width tiles), and the two byte images that chained layers read in turn.
struct Maps {
  CUtensorMap w[kMaxLayers];
  CUtensorMap wh;
  CUtensorMap a[2];
};

struct Params {
  ConvJobDev jobs[kMaxJobs];
  int32_t njobs, total_tiles, n_tiles, num_kchunks;
  int32_t cin, cout, kh, kw, stride, pad, k_total;
  int32_t out_bits, skip_bits;
  int64_t x_row_bytes, y_row_bytes, skip_row_bytes;
  const int32_t* skip_c;
  const int8_t* skip_d;
  int32_t upsample, scale_main, has_skip;
  int32_t bn, stages, tmem_cols;
  int32_t nbuf_log2;   // log2 of the TMEM accumulators (2, or 4 where four fit)
  // The epilogue warps of a lane quarter split a tile's 32-column groups epi_groups ways; where a
  // tile has fewer groups than there are warps, epi_sets sets of warps take tiles in turn.
  int32_t epi_groups, epi_sets;
  uint64_t div_layer, div_nt;  // fast_div of layer_tiles and n_tiles
  int32_t acc_small;  // |acc| < 2^22 guaranteed by K * max|x| * max|w|
  int32_t cin_chunks; // cin / 128 (flat path)
  int32_t dp_tiles;   // tiles [0, dp_tiles) are bn wide; later ones are the two bn/2 halves of the remaining
                      // full tiles (the last, partial wave)
  int32_t tile_stride; // from one tile of a CTA (pair) to its next
  int32_t contig;     // each CTA takes one contiguous range of tiles (single CTAs, one layer, no half tiles)
                      // instead of every gridDim-th tile:
  int32_t share, extra; // tiles per CTA, CTAs with one more
  // flat path: a ring of `stages` activation slabs and one of stages_b weight tiles (resident: all
  // weight tiles, loaded once)
  int32_t stages_b, resident;
  uint32_t slab_bytes;
  int32_t taps;        // taps that share a slab: kw, or 1 for kernels too wide for that
  uint32_t off_b, off_epi, off_bar;
  uint32_t off_sktab;   // table of 2- to 4-bit skip codes
  uint32_t off_ostage;  // int32 outputs: per-warp staging blocks for row-contiguous stores (0: none)
  int32_t out_pad;
  int32_t seg_chunks; // kF16: K chunks per exact FP32 segment
  int32_t a_planes;   // K runs over this many planes of the byte image (2: 8-bit codes in halves)
  int32_t plane_rows; // workspace rows per plane
  int32_t split_w;    // weights in the split layout: a tile's bn B rows give bn/2 channels
  uint32_t* status;
  // Several chained stride-1 layers of one shape in one launch (workspace path, CTA pairs,
  // one N tile, no half-width tiles): layer l covers the tiles [l * layer_tiles, (l + 1) *
  // layer_tiles), in that order over the persistent CTAs. Tile t of layer l reads the
  // previous layer's output rows written by its tiles t - K .. t + K of the same image
  // (K = 1 + wp / 256), which are also the only tiles of that layer that read the rows tile
  // t writes. Each epilogue warp of a tile of layer l < nlayers - 1 adds 1 to
  // dep[l * layer_tiles + t] (release) after its stores; the TMA issuers of a tile of layer
  // l > 0 wait (acquire, bounded) for dep[(l - 1) * layer_tiles + t'] >= dep_target on those
  // tiles before loading A.
  int32_t nlayers, layer_tiles;
  LayerDev layers[kMaxLayers];
  int32_t sf_col;     // FP4: first of the 32 TMEM columns that hold the unit block scales
  uint32_t* dep;
  uint32_t dep_target;
};

static_assert(BM == kMmaM, "a CTA's tile rows are one M=128 MMA operand");

// ---------------------------------------------------------------- tile bookkeeping

struct TileInfo {
  int layer;
  int job, mt;
  int bn;    // MMA N of this tile (weight rows): p.bn, or p.bn / 2 for a half tile
  int col0;  // first output channel
  int brow;  // first weight row
  int cn;    // output channels of this tile: bn, or bn / 2 with split weights
};
// Flat path: M tile mt of a job covers virtual rows [v0, v0 + 128) of image img, where the
// virtual grid holds the output rows at the padded input width wp (stride 1).
struct FlatTile {
  int img, v0;
};
__device__ __forceinline__ FlatTile flat_tile(const ConvJobDev& jb, int mt, int rows = 128) {
  FlatTile f;
  f.img = fast_div(mt, jb.div_img);
  f.v0 = (mt - f.img * jb.tpi) * rows;
  return f;
}
// Waits until every tile of layer l - 1 that writes the rows M tile mt of job j (of layer l)
// reads has been stored (see Params::dep), then orders those stores before this thread's TMA
// loads. kTileRows: rows of a tile (every layer of a launch has the same tiles).
template <int kTileRows>
__device__ __forceinline__ bool wait_dep_tiles(const Params& p, int l, int j, int mt, volatile int* abort_flag) {
  const ConvJobDev& jb = p.jobs[j];
  const int img = fast_div(mt, jb.div_img), m_in = mt - img * jb.tpi;
  const int K = 1 + jb.wp / kTileRows;
  const int lo = m_in - K < 0 ? 0 : m_in - K;
  const int hi = m_in + K > jb.tpi - 1 ? jb.tpi - 1 : m_in + K;
  const uint32_t* c = p.dep + (size_t)(l - 1) * p.layer_tiles + jb.tile_begin + img * jb.tpi;
  if (!counters_wait(c + lo, hi - lo + 1, p.dep_target, abort_flag)) return false;
  fence_proxy_async_global();
  return true;
}

// Global tile t -> (job, M tile, channel range). Tiles past dp_tiles split the remaining
// full tiles into two halves of N, so the last, partial wave covers more SMs.
__device__ __forceinline__ TileInfo tile_info(const Params& p, int t) {
  const int layer = p.nlayers > 1 ? fast_div(t, p.div_layer) : 0;
  t -= layer * p.layer_tiles;
  int half = -1;
  if (t >= p.dp_tiles) {
    const int h = t - p.dp_tiles;
    t = p.dp_tiles + (h >> 1);
    half = h & 1;
  }
  int j = 0;
#pragma unroll 1
  while (j + 1 < p.njobs && t >= p.jobs[j + 1].tile_begin) ++j;
  int local = t - p.jobs[j].tile_begin;
  TileInfo ti;
  ti.layer = layer;
  ti.job = j;
  ti.mt = fast_div(local, p.div_nt);
  const int nt = local - ti.mt * p.n_tiles;
  ti.bn = half < 0 ? p.bn : p.bn / 2;
  ti.brow = nt * p.bn + (half > 0 ? p.bn / 2 : 0);
  // split weights (no half tiles): rows [brow, brow + bn/2) hold w_lo of bn/2 channels and
  // the next bn/2 rows their w_hi
  ti.cn = p.split_w ? ti.bn / 2 : ti.bn;
  ti.col0 = p.split_w ? nt * (p.bn / 2) : ti.brow;
  return ti;
}

// ---------------------------------------------------------------- epilogue

// Per-column constants of a tile's level and channel range, in shared memory: the int64 form's
// (EpiChan), the 32-bit requant's {bias - kMagicBits, M0, 2^(R-33), R-32} and the 32-bit skip
// rescale's {c, rounding term, shift, 0}.
struct EpiTab {
  uint8_t* base;
  static constexpr size_t kBytes = 256 * (sizeof(EpiChan) + 2 * sizeof(int4));
  __device__ __forceinline__ EpiChan* gen() const { return reinterpret_cast<EpiChan*>(base); }
  __device__ __forceinline__ int4* fast() const { return reinterpret_cast<int4*>(base + 256 * sizeof(EpiChan)); }
  __device__ __forceinline__ int4* skip() const { return fast() + 256; }
};
// What the tables of the current tile allow
enum : int {
  kFlagReq = 1,   // every R >= 33 and |bias| <= 2^30: the 32-bit requant
  kFlagBias = 2,  // |bias| <= 2^30
  kFlagSkip = 4   // the 32-bit skip rescale (skip_const below), with kFlagReq
};

// 1.5 * 2^23: adding it to an integer-valued float |x| < 2^22 puts x in the low mantissa bits
constexpr float kMagic = 12582912.0f;
constexpr uint32_t kMagicBits = 0x4B400000u;

// Eq. 7's rescaled skip rhu(s c, d) in 32-bit arithmetic: with s pre-scaled by 2^k so that
// |s 2^k| < 2^31, rhu(s c, d) = (mulhi(s 2^k, c) + 2^(d+k-33)) >> (d+k-32) for d + k >= 33 (the
// same identity as the requant's). k = 23 for 8-bit codes, 3 for int32 skips below 2^28 in
// magnitude (checked per value). A d so large that |s c| < 2^(d-1) for every s gives 0. The sum
// acc + bias + rescaled skip then stays within int32 (|bias| <= 2^30, |acc| < 2^24, the skip term
// below 2^29), so Eq. 7 needs no saturation. (Narrower codes take a table, below.)
__device__ __forceinline__ int skip_prescale(int skip_bits) { return skip_bits == 32 ? 3 : 23; }
__device__ __forceinline__ bool skip_const(int skip_bits, int32_t c, int d, int4& o) {
  const int r = d + skip_prescale(skip_bits);
  if (r < 33) return false;
  // |s c| < 2^(bits + 31) for codes (bits <= 8), 2^59 for int32 skips below 2^28
  if (d > (skip_bits == 32 ? 59 : skip_bits + 31)) o = make_int4(0, 0, 1, 0);
  else o = make_int4(c, 1 << (r - 33), r - 32, 0);
  return true;
}
__device__ __forceinline__ uint32_t magnitude(int32_t s) { return s < 0 ? 0u - (uint32_t)s : (uint32_t)s; }
__device__ __forceinline__ int32_t skip32(int32_t s_scaled, const int4& e) {
  return (__mulhi(s_scaled, e.x) + e.y) >> e.z;
}

// Chained output: the 16 codes at their place in the row of the zero-padded image that the next
// stride-1 conv reads: one byte per code, or, when that conv runs on the FP4 pipe (nib), two
// codes per byte (channel 2k in the low nibble of byte k) in the first half of the row.
__device__ __forceinline__ void store_image16(uint8_t* irow, int ch, const uint32_t (&bw)[4], int nib) {
  if (nib) {
    // bytes 0 and 2 of t hold the nibble pairs (c0, c1) and (c2, c3) of a byte-word
    uint32_t t[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) t[j] = bw[j] | (bw[j] >> 4);
    *reinterpret_cast<uint2*>(irow + (ch >> 1)) =
        make_uint2(__byte_perm(t[0], t[1], 0x6420), __byte_perm(t[2], t[3], 0x6420));
  } else {
    *reinterpret_cast<uint4*>(irow + ch) = make_uint4(bw[0], bw[1], bw[2], bw[3]);
  }
}

// A whole 32-channel group.
__device__ __forceinline__ void store_image32(uint8_t* irow, int ch, const uint32_t (&a)[4], const uint32_t (&b)[4], int nib) {
  if (nib) {
    // bytes 0 and 2 of t hold the nibble pairs (c0, c1) and (c2, c3) of a byte-word
    uint32_t t[8];
#pragma unroll
    for (int j = 0; j < 4; ++j) { t[j] = a[j] | (a[j] >> 4); t[4 + j] = b[j] | (b[j] >> 4); }
    *reinterpret_cast<uint4*>(irow + (ch >> 1)) = make_uint4(__byte_perm(t[0], t[1], 0x6420), __byte_perm(t[2], t[3], 0x6420),
                                                             __byte_perm(t[4], t[5], 0x6420), __byte_perm(t[6], t[7], 0x6420));
  } else {
    store_sector(irow + ch, a, b);  // (rows are cout bytes, cout % 32 == 0, in a 256-byte aligned workspace)
  }
}

// Skip codes of 2 to 4 bits: Eq. 6's bias and Eq. 7's rescaled skip together are one of 2^bits values per
// column, bias + rhu(s c, d) - kMagicBits, kept in a shared-memory table (built in int64, any c and
// d). Entry (s, col) at s kSkipStride + col words: the lanes of a warp, which look up one column
// with their own codes, read different banks. The form holds where every entry's sum part is
// within 2^30 (|acc| < 2^22 then cannot leave int32, so Eq. 7 needs no saturation).
constexpr int kSkipStride = 257;
__host__ __device__ constexpr size_t skip_tab_bytes(int skip_bits) {
  return skip_bits >= 2 && skip_bits <= 4 ? (((size_t)1 << skip_bits) * kSkipStride * 4 + 15) / 16 * 16 : 0;
}

// int32 skips: each warp stages the next 16 columns of its 32 rows (64 bytes a row) in shared memory
// by cp.async, two steps in flight. A lane that reads its own row takes 16 bytes of 32 different rows
// per load; four lanes per row take whole 64-byte pieces. The 16-byte pieces of a row are
// rotated by its index, so that both the copies and the row reads are conflict-free.
constexpr int kSkipStage = 32 * 64;  // bytes of one step of one warp
__device__ __forceinline__ uint32_t skip_stage_off(int row, int piece) {
  return (uint32_t)(row * 64 + ((piece ^ (row >> 1)) & 3) * 16);
}

// The packed words of a row's 32 skip codes from channel ch on (2- to 4-bit codes: the layout needs
// cout % 32 == 0, so they all exist), a half's in x and y, the other's in z and w; a half's byte-words.
// (One 16-byte load per group instead of two of 8: 1x1 convs with a skip, 30 -> 28 us.)
__device__ __forceinline__ uint4 load_skip_group(const uint8_t* srow, int ch, int sb, bool ok) {
  uint4 g = make_uint4(0u, 0u, 0u, 0u);
  if (!ok) return g;
  if (sb == 4) {
    g = __ldg(reinterpret_cast<const uint4*>(srow + (ch >> 1)));
  } else if (sb == 2) {
    const uint2 t = __ldg(reinterpret_cast<const uint2*>(srow + (ch >> 2)));
    g.x = t.x; g.z = t.y;
  } else {
    const uint32_t* g3 = reinterpret_cast<const uint32_t*>(srow + (ch >> 5) * 12);
    const uint32_t top = __ldg(g3 + 2);
    g = make_uint4(__ldg(g3), top, __ldg(g3 + 1), top >> 4);
  }
  return g;
}
__device__ __forceinline__ void skip_bytewords(const uint2& g, int sb, uint32_t (&b)[4]) {
  if (sb == 4) {
    b[0] = g.x & 0x0F0F0F0Fu; b[1] = (g.x >> 4) & 0x0F0F0F0Fu;
    b[2] = g.y & 0x0F0F0F0Fu; b[3] = (g.y >> 4) & 0x0F0F0F0Fu;
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      b[j] = (g.x >> (2 * j)) & 0x03030303u;
      if (sb == 3) b[j] |= ((g.y >> j) & 0x01010101u) << 2;
    }
  }
}

// ---- the general form: any shift, any skip direction and width, any row size, int32 outputs with a skip, biases
// beyond 2^30. Eq. 6 -> Eq. 7 -> Eq. 2 as the definition states them, in int64 where a value needs it. Functions
// of their own, not inlined: their registers and code stay out of the common forms. Skips are loaded and int32
// outputs stored in whole pieces where rows allow it. Against element by element, on two 100 x 168 maps: 3x3 256 ->
// 256 with a 4-bit skip and R = 32 151 -> 52 us, 1x1 64 -> 256 with a 4-bit skip and int32 outputs 156 -> 44.

// A column's constants (EpiChan) from their shared-memory address
struct ColConst {
  int32_t bias, m0, c;
  int r, d;
};
__device__ __forceinline__ ColConst col_const(uint32_t addr) {
  int32_t w;
  ColConst k;
  asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(k.bias), "=r"(k.m0), "=r"(k.c), "=r"(w) : "r"(addr));
  k.r = w & 0xFF;
  k.d = (w >> 8) & 0xFF;
  return k;
}
static_assert(sizeof(EpiChan) == 16 && offsetof(EpiChan, r) == 12 && offsetof(EpiChan, d) == 13, "col_const");

__device__ __forceinline__ int32_t sat_s32(int64_t v) { return (int32_t)sat32(v); }

// The row's skip values of nc columns from channel ch on.
__device__ __forceinline__ void general_skip(const Params& p, const uint8_t* srow, int ch, int nc, int32_t (&sk)[16]) {
  const int sb = p.skip_bits;
  const bool whole = (p.skip_row_bytes & 15) == 0;  // (then nc is a multiple of 4, and 16 with 8-bit codes)
#pragma unroll
  for (int i = 0; i < 16; ++i) sk[i] = 0;
  if (sb == 32 && whole) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      int4 v = make_int4(0, 0, 0, 0);
      if (4 * q < nc) v = __ldg(reinterpret_cast<const int4*>(srow) + (ch >> 2) + q);
      sk[4 * q] = v.x; sk[4 * q + 1] = v.y; sk[4 * q + 2] = v.z; sk[4 * q + 3] = v.w;
    }
  } else if (sb == 32) {
#pragma unroll
    for (int i = 0; i < 16; ++i)
      if (i < nc) sk[i] = __ldg(reinterpret_cast<const int32_t*>(srow) + ch + i);
  } else if (sb == 8 && !whole) {
#pragma unroll
    for (int i = 0; i < 16; ++i)
      if (i < nc) sk[i] = __ldg(srow + ch + i);
  } else {
    uint32_t b[4];
    if (sb == 8) {
      const uint4 v = __ldg(reinterpret_cast<const uint4*>(srow + ch));
      b[0] = v.x; b[1] = v.y; b[2] = v.z; b[3] = v.w;
    } else {
      // (2- to 4-bit codes: whole groups, of which these are a half)
      uint2 g = make_uint2(0u, 0u);
      if (sb == 4) g = __ldg(reinterpret_cast<const uint2*>(srow + (ch >> 1)));
      else if (sb == 2) g.x = __ldg(reinterpret_cast<const uint32_t*>(srow + (ch >> 2)));
      else {
        const uint32_t* g3 = reinterpret_cast<const uint32_t*>(srow + (ch >> 5) * 12);
        const int half = (ch >> 4) & 1;
        g = make_uint2(__ldg(g3 + half), __ldg(g3 + 2) >> (4 * half));
      }
      skip_bytewords(g, sb, b);
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) sk[i] = (int32_t)((b[i / 4] >> (8 * (i % 4))) & 0xFFu);
  }
}

// nc columns (at most 16) of one row from channel ch on (srow and yrow stand at the tile's first channel; ep: the
// columns' constants): the codes as byte-words, or the outputs of int32 rows and of 8-bit rows of no whole groups
// stored here.
template <bool kSkip>
__device__ __forceinline__ uint4 general_finish(const Params& p, uint32_t ep, const uint8_t* srow, uint8_t* yrow, int ch,
                                                int nc, int flags, int32_t (&acc)[16]) {
  const int out_bits = p.out_bits;
  const int32_t qmax = (1 << (out_bits & 15)) - 1;
  const auto at = [ep](int i) { return ep + (uint32_t)(i * sizeof(EpiChan)); };
  auto requant = [qmax](int32_t u, const ColConst& k) { return requant64(u, k.m0, k.r, qmax); };
  if constexpr (kSkip) {
    int32_t sk[16];
    general_skip(p, srow, ch, nc, sk);
    if (p.scale_main == 0) {
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const ColConst k = col_const(at(i));
        acc[i] = sat_s32((int64_t)acc[i] + k.bias + rhu1((int64_t)sk[i] * k.c, k.d));
        if (out_bits != 32) acc[i] = requant(acc[i], k);
      }
    } else {
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const ColConst k = col_const(at(i));
        acc[i] = sat_s32(rhu1((int64_t)add_sat(acc[i], k.bias) * k.c, k.d) + sk[i]);
        if (out_bits != 32) acc[i] = requant(acc[i], k);
      }
    }
  } else if (out_bits == 32) {
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[i] = add_sat(acc[i], col_const(at(i)).bias);
  } else if (flags & kFlagReq) {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const ColConst k = col_const(at(i));
      acc[i] = __vimin_s32_relu((__mulhi(add_sat(acc[i], k.bias), k.m0) + (1 << (k.r - 33))) >> (k.r - 32), qmax);
    }
  } else {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const ColConst k = col_const(at(i));
      acc[i] = requant(add_sat(acc[i], k.bias), k);
    }
  }
  if (out_bits == 32) {
    int32_t* yr = reinterpret_cast<int32_t*>(yrow) + ch;
    if ((p.cout & 3) == 0) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (4 * q < nc) reinterpret_cast<int4*>(yr)[q] = make_int4(acc[4 * q], acc[4 * q + 1], acc[4 * q + 2], acc[4 * q + 3]);
    } else {
#pragma unroll
      for (int i = 0; i < 16; ++i)
        if (i < nc) yr[i] = acc[i];
    }
  } else if (out_bits == 8 && (p.cout & 31) != 0) {
#pragma unroll
    for (int i = 0; i < 16; ++i)
      if (i < nc) yrow[ch + i] = (uint8_t)acc[i];
  }
  uint32_t bw[4];
#pragma unroll
  for (int j = 0; j < 4; ++j)
    bw[j] = (uint32_t)acc[4 * j] | ((uint32_t)acc[4 * j + 1] << 8) | ((uint32_t)acc[4 * j + 2] << 16) |
            ((uint32_t)acc[4 * j + 3] << 24);
  return make_uint4(bw[0], bw[1], bw[2], bw[3]);
}

// A warp's columns of a tile in the general form. (In memory: as arguments they would be registers of the caller.)
struct GenTile {
  uint32_t taddr;       // TMEM address of the tile's first column
  int cn;               // split weights: columns from there to the w_hi accumulator
  uint32_t ep;          // shared address of the first column's constants
  int c_lo, c_hi, flags, nib;
  const uint8_t* srow;  // the lane's row of the skip (kSkip), of the output (NULL: none) and of the chained image, at the
  uint8_t *yrow, *irow; // tile's first channel
};
template <bool kSkip>
__device__ __forceinline__ void general_step(const Params& p, const GenTile& g, int c0, int32_t (&acc)[16], uint32_t& top) {
  const uint4 r = general_finish<kSkip>(p, g.ep + (uint32_t)(c0 * sizeof(EpiChan)), g.srow, g.yrow, c0,
                                        g.c_hi - c0 < 16 ? g.c_hi - c0 : 16, g.flags, acc);
  if (p.out_bits == 32 || (p.out_bits == 8 && (p.cout & 31) != 0)) return;  // (stored by general_finish)
  const uint32_t bw[4] = {r.x, r.y, r.z, r.w};
  store_codes16(g.yrow, c0, bw, p.out_bits, top);
  if (g.irow) store_image16(g.irow, c0, bw, g.nib);
}
// From the accumulators in TMEM, which hold the integer sum / sc.
template <bool kSkip, bool kSplit>
__device__ __noinline__ void general_tile(const Params& p, const GenTile& g, float sc) {
  uint32_t top = 0u;  // (3-bit codes: see store_codes16)
#pragma unroll 1
  for (int c0 = g.c_lo; c0 < g.c_hi; c0 += 16) {
    uint32_t v[16];
    tmem_ld16(g.taddr + (uint32_t)c0, v);
    tmem_wait_ld();
    reg_fence16(v);
    int32_t acc[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[i] = __float2int_rn(__uint_as_float(v[i]) * sc);
    if constexpr (kSplit) {
      tmem_ld16(g.taddr + (uint32_t)(g.cn + c0), v);
      tmem_wait_ld();
      reg_fence16(v);
#pragma unroll
      for (int i = 0; i < 16; ++i) acc[i] += 16 * __float2int_rn(__uint_as_float(v[i]) * sc);
    }
    if (g.yrow) general_step<kSkip>(p, g, c0, acc, top);
    __syncwarp();
  }
}
// From a lane's sums of the columns from c_lo on (kF16).
__device__ __noinline__ void general_sums(const Params& p, const GenTile& g, const int32_t* sums) {
  uint32_t top = 0u;
#pragma unroll 1
  for (int c0 = g.c_lo; c0 < g.c_hi; c0 += 16, sums += 16) {
    int32_t acc[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[i] = sums[i];
    general_step<false>(p, g, c0, acc, top);
  }
}

// ---------------------------------------------------------------- the kernel

// Loads the packed codes of half (64 channels) of a 128-channel K chunk of one output row into
// registers (2 * kXBits words; group g = 32 channels at words [g * kXBits, ...)). Taps outside the
// image (and rows past the end of the job) read zeros = code 0.
template <int kXBits>
struct RowCursor {
  const uint8_t* xbase;  // image base of this row's pixel
  int hb, wb, H, W;      // top-left input coordinate of the window, image size
  bool valid;
  int tr, ts, tc0;       // tap (r, s) and channel offset of the next 32-channel group
};

template <int kXBits>
__device__ __forceinline__ void skip_groups(const Params& p, RowCursor<kXBits>& rc, int n) {
  for (int g = 0; g < n; ++g) {
    rc.tc0 += 32;
    if (rc.tc0 == p.cin) { rc.tc0 = 0; if (++rc.ts == p.kw) { rc.ts = 0; ++rc.tr; } }
  }
}

// The cursor stands at this half's first group of chunk q, and is left at that of chunk q + 1.
template <int kXBits, bool kChunkInTap>
__device__ __forceinline__ void load_half(const Params& p, RowCursor<kXBits>& rc, int q, int half, uint32_t (&w)[2 * kXBits]) {
  constexpr int kGB = 4 * kXBits;
  if constexpr (kChunkInTap) {
    // cin % 128 == 0: the chunk is 128 consecutive channels of one tap
    const int hi = rc.hb + rc.tr, wi = rc.wb + rc.ts;
    const bool ok = rc.valid && hi >= 0 && hi < rc.H && wi >= 0 && wi < rc.W;
    // (3-bit halves are 24 bytes: 8-byte pieces)
    using Piece = std::conditional_t<kXBits == 3, uint2, uint4>;
    constexpr int kPieces = 2 * kGB / (int)sizeof(Piece), kPw = (int)sizeof(Piece) / 4;
    const Piece* src = reinterpret_cast<const Piece*>(rc.xbase + ((int64_t)hi * rc.W + wi) * p.x_row_bytes + (rc.tc0 >> 5) * kGB);
#pragma unroll
    for (int i = 0; i < kPieces; ++i) {
      Piece v{};
      if (ok) v = __ldg(src + i);
      w[kPw * i] = v.x; w[kPw * i + 1] = v.y;
      if constexpr (kPw == 4) { w[kPw * i + 2] = v.z; w[kPw * i + 3] = v.w; }
    }
    rc.tc0 += 128;
    if (rc.tc0 >= p.cin) { rc.tc0 -= p.cin; if (++rc.ts == p.kw) { rc.ts = 0; ++rc.tr; } }
  } else {
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      const int k0 = q * BK + 64 * half + 32 * g;
      bool ok = false;
      const uint8_t* src = rc.xbase;
      if (k0 < p.k_total) {
        const int hi = rc.hb + rc.tr, wi = rc.wb + rc.ts;
        ok = rc.valid && hi >= 0 && hi < rc.H && wi >= 0 && wi < rc.W;
        src = rc.xbase + ((int64_t)hi * rc.W + wi) * p.x_row_bytes + (rc.tc0 >> 5) * kGB;
        skip_groups(p, rc, 1);
      }
      if constexpr (kXBits == 2) {
        uint2 v = make_uint2(0, 0);
        if (ok) v = __ldg(reinterpret_cast<const uint2*>(src));
        w[2 * g] = v.x; w[2 * g + 1] = v.y;
      } else if constexpr (kXBits == 4) {
        uint4 v = make_uint4(0, 0, 0, 0);
        if (ok) v = __ldg(reinterpret_cast<const uint4*>(src));
        w[4 * g] = v.x; w[4 * g + 1] = v.y; w[4 * g + 2] = v.z; w[4 * g + 3] = v.w;
      } else {
#pragma unroll
        for (int i = 0; i < 3; ++i) w[3 * g + i] = ok ? __ldg(reinterpret_cast<const uint32_t*>(src) + i) : 0u;
      }
    }
    skip_groups(p, rc, 2);  // (the other half's)
  }
}

// kSkip: the instantiation that handles a skip tensor (Eq. 7); the others carry no skip code,
// which keeps the common path's registers free.
// kSplit: the 8-bit split form (split weights combined as D1 + 16 D2 in the epilogue).
// kOStage: int32 outputs, through per-warp shared-memory staging blocks, or on the F16 pipe stored as they are
// (an instantiation of its own, so that the other forms keep their registers)
template <int kXBits, bool kChunkInTap, bool kFlat, bool kPair, bool kSkip, bool kSplit, int kBK, bool kFp4,
          bool kOStage>
__global__ void __launch_bounds__(threads_for(kFlat), 1)
conv_tc_kernel(const __grid_constant__ Maps maps, const __grid_constant__ Params p) {
  static_assert(!kPair || kFlat, "the CTA-pair form exists for the workspace path only");
  static_assert(kBK == BK || kFlat, "64-byte K chunks exist for the workspace path only");
  static_assert(!kFp4 || (kFlat && kBK == BK && !kSplit), "the FP4 pipe reads nibble images in 128-byte chunks");
  constexpr bool kF16 = kXBits == 8;  // (flat kernels read images: kXBits names the pipe only here)
  static_assert(!kF16 || (kFlat && kBK == BK && !kSplit && !kFp4 && !kSkip), "the F16 pipe's form");
  // the FP32 accumulator holds the integer sum / kAccSc
  constexpr float kAccSc = kFp4 ? 4.0f : 262144.0f;
  constexpr int kStA = BM * kBK;  // bytes of one stage's A operand
  constexpr int kTma = tma_warps(kFlat);
  constexpr int kEpiWarps = epi_warps(kFlat);
  constexpr int kEpiThreads = kEpiWarps * 32;
  constexpr int kWarpMma = kEpiWarps, kWarpTma = kEpiWarps + 1, kWarpProd0 = kWarpTma + kTma;
  // CTA pair: this CTA's rank; the even CTA issues the MMAs; a tile has 256 rows
  const uint32_t rank = kPair ? cluster_ctarank() : 0u;
  const bool leader = rank == 0;
  constexpr int kTileRows = kPair ? 256 : 128;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  // align by pointer arithmetic on the shared array itself (no integer round trip), so the
  // compiler keeps every access through `smem` in the shared state space (lds/sts)
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t sbase = smem_u32(smem);
  const uint32_t s_a = sbase;
  const uint32_t s_b = sbase + p.off_b;
  const EpiTab epi{smem + p.off_epi};
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + p.off_bar);
  // barrier slots: tfull[nbuf], tempty[nbuf] (kMaxBufs each), final, then full[0..S), empty[0..S), on
  // the flat path of the slabs, and of the weight tiles wfull[0..SB), wempty[0..SB)
  const uint32_t b_tfull = smem_u32(bars), b_tempty = b_tfull + 8 * kMaxBufs;
  const uint32_t b_final = b_tempty + 8 * kMaxBufs, b_full = b_final + 8;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kMaxBufs + 1 + 4 * kMaxStages);
  const uint32_t buf_mask = (1u << p.nbuf_log2) - 1u;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x / 32;
  const int lane = threadIdx.x % 32;
  const int BN = p.bn;
  const uint32_t stage_b_bytes = (uint32_t)(kPair ? BN / 2 : BN) * kBK;  // this CTA's rows of B

  // (the roles that use them work these out for themselves: the epilogue has no register to spare)
  auto slots = [&](uint32_t& empty, uint32_t& wfull, uint32_t& wempty) {
    empty = b_full + 8 * p.stages;
    wfull = empty + 8 * p.stages;
    wempty = wfull + 8 * (kFlat ? p.stages_b : 0);
  };
  if (threadIdx.x == 0) {
    const int S = p.stages, SB = kFlat ? p.stages_b : 0;
    uint32_t b_empty, b_wfull, b_wempty;
    slots(b_empty, b_wfull, b_wempty);
    for (int s = 0; s < S; ++s) {
      mbar_init(b_full + 8 * s, kFlat ? 1 : kProdWarps + 1);  // per producer warp + TMA
      mbar_init(b_empty + 8 * s, 1);
    }
    for (int s = 0; s < SB; ++s) {
      mbar_init(b_wfull + 8 * s, 1);
      mbar_init(b_wempty + 8 * s, 1);
    }
    for (int b = 0; b < kMaxBufs; ++b) {
      mbar_init(b_tfull + 8 * b, 1);
      mbar_init(b_tempty + 8 * b, (kPair ? 8 : 4) * p.epi_groups);  // one arrive per epilogue warp of a tile
    }
    mbar_init(b_final, 1);
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == kWarpMma) {
    if constexpr (kPair) {
      // one warp of each CTA of the pair allocates, collectively, the same columns in both
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                   ::"r"(smem_u32(tmem_slot)), "r"(p.tmem_cols) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                   ::"r"(smem_u32(tmem_slot)), "r"(p.tmem_cols) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  if (warp >= kWarpTma && warp < kWarpTma + kTma && lane == 0) {
    for (int l = 0; l < p.nlayers; ++l) asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&maps.w[l]) : "memory");
    if (p.dp_tiles < p.layer_tiles) asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&maps.wh) : "memory");
    if (kFlat) {
      asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&maps.a[0]) : "memory");
      if (p.nlayers > 1) asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&maps.a[1]) : "memory");
    }
  }
  tc_fence_before();
  __syncthreads();
  // the peer signals this CTA's barriers (and the leader's MMAs read the peer's shared
  // memory) only after both CTAs have initialised them
  if constexpr (kPair) cluster_sync();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  if constexpr (kFp4) {
    // unit block scales (UE8M0 127 = 2^0) in the 32 TMEM columns from sf_col, every lane of
    // both CTAs of a pair: the MMAs read the A scales from the first 16, the B scales from
    // the next 16, whatever the scale vectors' layout inside them
    if (warp < 4) {
      const uint32_t ta = tmem_base + ((uint32_t)(32 * warp) << 16) + (uint32_t)p.sf_col;
      tmem_st16_fill(ta, 0x7F7F7F7Fu);
      tmem_st16_fill(ta + 16, 0x7F7F7F7Fu);
      tmem_wait_st();
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (kPair) cluster_sync();
    tc_fence_after();
  }
  // everything above overlaps the previous kernel; global memory is touched only after this
  grid_dep_wait();
  if (threadIdx.x == 0) grid_dep_launch();

  const int nk = p.num_kchunks * p.a_planes;  // K chunks, over every plane of the image
  // This CTA's tiles: every tile_stride-th from first_tile, or (contig) the range
  // [first_tile, tile_end) of a balanced split of the tiles over the grid, so that a CTA's
  // consecutive tiles are neighbours (one level's table, adjacent rows in L2)
  // (contig: share tiles each, one more for the first `extra` CTAs)
  const int bid = (int)blockIdx.x;
  const bool contig = !kPair && p.contig;
  const int first_tile = kPair ? bid >> 1 : (contig ? bid * p.share + (bid < p.extra ? bid : p.extra) : bid);
  const int tile_end = contig ? first_tile + p.share + (bid < p.extra ? 1 : 0) : p.total_tiles;

  if (warp == kWarpMma) {
    // ------------------------------------------------------------ MMA issuer
    if (leader && elect_one()) {
      const int S = p.stages, SB = kFlat ? p.stages_b : 0;
      uint32_t b_empty, b_wfull, b_wempty;
      slots(b_empty, b_wfull, b_wempty);
      const uint32_t idesc_full = kFp4 ? idesc_fp4(BN, kPair ? 2 * kMmaM : kMmaM) : idesc_e4m3(BN, kPair ? 2 * kMmaM : kMmaM);
      const uint32_t idesc_half =
          kFp4 ? idesc_fp4(BN / 2, kPair ? 2 * kMmaM : kMmaM) : idesc_e4m3(BN / 2, kPair ? 2 * kMmaM : kMmaM);
      const uint32_t sfa = tmem_base + (uint32_t)p.sf_col, sfb = sfa + 16;  // (FP4 only)
      // descriptors of stage 0, k-step 0; later stages / k-steps add
      // (byte offset >> 4) to the 14-bit start-address field (shared addresses < 2^18)
      // the descriptors' high words are constant; stages / k-steps only move the
      // 14-bit start-address field in the low word (shared addresses < 2^18, no carry)
      const uint64_t da0 = sdesc_k<kBK>(s_a), db0 = sdesc_k<kBK>(s_b);
      const uint32_t a_lo0 = (uint32_t)da0, b_lo0 = (uint32_t)db0;
      const uint32_t a_hi = (uint32_t)(da0 >> 32), b_hi = (uint32_t)(db0 >> 32);
      // one instruction of K = 32 bytes: operand rows at da, db
      auto mma = [&](uint32_t d0, uint32_t a_lo, uint32_t b_lo, uint32_t idesc, uint32_t acc) {
        const uint64_t da = ((uint64_t)a_hi << 32) | a_lo, db = ((uint64_t)b_hi << 32) | b_lo;
        if constexpr (kPair && kFp4) mma_fp4_pair(d0, da, db, idesc, sfa, sfb, acc);
        else if constexpr (kPair && kF16) mma_f16_pair(d0, da, db, idesc, acc);
        else if constexpr (kPair) mma_e4m3_pair(d0, da, db, idesc, acc);
        else if constexpr (kF16) mma_f16(d0, da, db, idesc, acc);
        else if constexpr (kFp4) mma_fp4(d0, da, db, idesc, sfa, sfb, acc);
        else mma_e4m3(d0, da, db, idesc, acc);
      };
      auto commit = [&](uint32_t bar) {
        if constexpr (kPair) mma_commit_pair_both(bar);
        else mma_commit(bar);
      };
      uint32_t lt = 0;
      bool ok = true;
      // (operands written by TMA, or by producer threads followed by fence.proxy.async, are ordered
      // for the MMA by the mbarrier phase alone; tcgen05.fence is needed only where TMEM changes
      // hands, after the accumulator-empty wait)
      if constexpr (kFlat) {
        // The issuing thread runs one instruction at a time between the epilogue's warps, about 10
        // cycles each, while the MMAs queue behind it: with narrow tiles its bookkeeping, not the
        // tensor pipe, set the pace (330 of 450 cycles per chunk). So addresses advance by additions,
        // the taps of a slab are unrolled (1 and 3 of them), and a barrier is tested once, where
        // it is needed: the queued MMAs cover that.
        const bool resident = p.resident != 0;
        if (resident && !mbar_poll(b_wfull, 0, abort_flag)) ok = false;
        uint32_t sa = 0, pa = 0, a_cur = a_lo0;              // slab stage, its phase, its descriptor
        uint32_t fw = b_wfull, pw = 0, w_cur = b_lo0;        // weight barrier, its phase, descriptor
        const uint32_t a_step = p.slab_bytes >> 4, w_step = stage_b_bytes >> 4;
        const uint32_t w_end = b_lo0 + (uint32_t)SB * w_step, w_empty = b_wempty - b_wfull;
        uint32_t buf = 0, d0 = 0, acc = 0;
        int sq = 0;  // kF16: chunks of this accumulator
        auto open = [&]() {  // the next accumulator
          buf = lt & buf_mask;
          if (!mbar_poll(b_tempty + 8 * buf, ((lt >> p.nbuf_log2) & 1) ^ 1, abort_flag)) return false;
          tc_fence_after();
          d0 = tmem_base + buf * (uint32_t)BN;
          acc = 0;
          sq = 0;
          return true;
        };
        // the MMAs of one slab: false if a wait ran out
        auto slab = [&](auto taps_c, uint32_t idesc) {
          constexpr int kTaps = decltype(taps_c)::value;  // 0: p.taps
          if (!mbar_poll(b_full + 8 * sa, pa, abort_flag)) return false;
          const int taps = kTaps > 0 ? kTaps : p.taps;
#pragma unroll(kTaps > 0 ? kTaps : 1)
          for (int tap = 0; tap < taps; ++tap) {
            if (kF16 && sq == p.seg_chunks) {  // (a tile's segments take accumulators in turn)
              commit(b_tfull + 8 * buf);
              ++lt;
              if (!open()) return false;
            }
            if (!resident && !mbar_poll(fw, pw, abort_flag)) return false;
#pragma unroll
            for (int kk = 0; kk < kBK / 32; ++kk) {
              mma(d0, a_cur + (uint32_t)(tap * (kBK >> 4) + 2 * kk), w_cur + 2 * kk, idesc, acc);
              acc = 1;
            }
            w_cur += w_step;
            if (!resident) {
              commit(fw + w_empty);
              fw += 8;
              if (w_cur == w_end) { w_cur = b_lo0; fw = b_wfull; pw ^= 1; }
            }
            if constexpr (kF16) ++sq;
          }
          commit(b_empty + 8 * sa);
          a_cur += a_step;
          if (++sa == (uint32_t)S) { sa = 0; a_cur = a_lo0; pa ^= 1; }
          return true;
        };
        for (int t = first_tile; t < tile_end && ok; t += p.tile_stride, ++lt) {
          // (a launch of several layers has no half-width tiles)
          const uint32_t idesc = p.nlayers > 1 || t < p.dp_tiles ? idesc_full : idesc_half;
          if (!open()) { ok = false; break; }
          for (int plane = 0; plane < p.a_planes && ok; ++plane) {
            // resident weights: the tiles of this N range (a second plane meets the same ones)
            if (resident)
              w_cur = b_lo0 + (p.n_tiles > 1 ? (uint32_t)(tile_info(p, t).brow / BN * p.num_kchunks) * w_step : 0u);
            for (int q = 0; q < p.num_kchunks && ok; q += p.taps)
              ok = p.taps == 3 ? slab(std::integral_constant<int, 3>{}, idesc)
                               : p.taps == 1 ? slab(std::integral_constant<int, 1>{}, idesc)
                                             : slab(std::integral_constant<int, 0>{}, idesc);
          }
          if (ok) commit(b_tfull + 8 * buf);
        }
      } else {
        uint32_t s = 0, ph = 0;
        bool next_ready = false;  // the stage after the current one is known to be full
        for (int t = first_tile; t < tile_end && ok; t += p.tile_stride, ++lt) {
          const uint32_t buf = lt & buf_mask;
          const uint32_t idesc = t < p.dp_tiles ? idesc_full : idesc_half;
          if (!mbar_poll(b_tempty + 8 * buf, ((lt >> p.nbuf_log2) & 1) ^ 1, abort_flag)) { ok = false; break; }
          tc_fence_after();
          const uint32_t d0 = tmem_base + buf * (uint32_t)BN;
          for (int q = 0; q < nk; ++q) {
            if (!next_ready && !mbar_poll(b_full + 8 * s, ph, abort_flag)) { ok = false; break; }
            const uint32_t a_lo = a_lo0 + ((s * kStA) >> 4);
            const uint32_t b_lo = b_lo0 + ((s * stage_b_bytes) >> 4);
            const uint32_t s_next = s + 1 == (uint32_t)S ? 0u : s + 1;
            const uint32_t ph_next = s_next == 0 ? ph ^ 1u : ph;
#pragma unroll
            for (int kk = 0; kk < kBK / 32; ++kk) {
              if (kk == kBK / 32 - 1) next_ready = mbar_test(b_full + 8 * s_next, ph_next);
              mma(d0, a_lo + 2 * kk, b_lo + 2 * kk, idesc, (q > 0 || kk > 0) ? 1u : 0u);
            }
            commit(b_empty + 8 * s);
            s = s_next;
            ph = ph_next;
          }
          if (ok) commit(b_tfull + 8 * buf);
        }
      }
      if (!ok) fail(abort_flag, p.status);
      // drain: every MMA issued above has completed once this barrier flips
      if constexpr (kPair) mma_commit_pair(b_final);
      else mma_commit(b_final);
      if (!mbar_wait(b_final, 0, abort_flag)) fail(abort_flag, p.status);
    }
  } else if (warp >= kWarpTma && warp < kWarpTma + kTma) {
    // ------------------------------------------------------------ operand loaders (TMA)
    const int tw = warp - kWarpTma;
    if (elect_one()) {
      const int S = p.stages, SB = kFlat ? p.stages_b : 0;
      uint32_t b_empty, b_wfull, b_wempty;
      slots(b_empty, b_wfull, b_wempty);
      bool ok = true;
      // arms a barrier of this CTA, or of a pair's leader, which counts both CTAs' copies, and loads
      // one box into this CTA's shared memory
      auto load = [&](uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar, uint32_t bytes) {
        if (leader) {
          if (bytes > 0) mbar_arrive_expect_tx(bar, (kPair ? 2u : 1u) * bytes);
          tma_load_2d(dst, map, x, y, bar);
        } else {
          tma_load_2d_pair(dst, map, x, y, mapa_shared(bar, 0));
        }
      };
      if constexpr (!kFlat) {
        uint32_t s = 0, ph = 0;
        for (int t = first_tile; t < tile_end && ok; t += p.tile_stride) {
          const TileInfo ti = tile_info(p, t);
          const CUtensorMap* wm = ti.bn == BN ? &maps.w[0] : &maps.wh;
          for (int q = 0; q < nk; ++q, s = (s + 1 == (uint32_t)S) ? 0 : s + 1, ph ^= (s == 0)) {
            if (!mbar_wait(b_empty + 8 * s, ph ^ 1, abort_flag)) { ok = false; break; }
            load(s_b + s * stage_b_bytes, wm, q * kBK, ti.brow, b_full + 8 * s, (uint32_t)ti.bn * kBK);
          }
        }
      } else if (tw == 0) {
        // slabs: the rows that the taps of kernel row r (p.taps at a time) read of channel block cb, for
        // each plane of the image (8-bit activations in two planes: x_lo, then 16 x_hi)
        const uint32_t bytes = (uint32_t)(BM + p.taps - 1) * kBK;
        uint32_t s = 0, ph = 0;
        for (int t = first_tile; t < tile_end && ok; t += p.tile_stride) {
          const TileInfo ti = tile_info(p, t);
          const ConvJobDev& jb = p.jobs[ti.job];
          const FlatTile ft = flat_tile(jb, ti.mt, kTileRows);
          const int row0 = jb.row_off + ft.img * jb.hp * jb.wp + ft.v0 + (int)rank * 128;
          const CUtensorMap* am = &maps.a[ti.layer & 1];  // layers read the two images in turn
          // the previous layer's tiles that this tile reads (and that read what it writes)
          if (ti.layer > 0 && !wait_dep_tiles<kTileRows>(p, ti.layer, ti.job, ti.mt, abort_flag)) { ok = false; break; }
          for (int pr = 0; pr < p.a_planes * p.kh && ok; ++pr) {
            const int plane = pr >= p.kh ? 1 : 0;
            const int row = row0 + plane * p.plane_rows + (pr - plane * p.kh) * jb.wp;
            for (int cb = 0; cb < p.cin_chunks && ok; ++cb)
              for (int sx = 0; sx < p.kw; sx += p.taps, s = (s + 1 == (uint32_t)S) ? 0 : s + 1, ph ^= (s == 0)) {
                if (!mbar_wait(b_empty + 8 * s, ph ^ 1, abort_flag)) { ok = false; break; }
                load(s_a + s * p.slab_bytes, am, cb * kBK, row + sx, b_full + 8 * s, bytes);
              }
          }
        }
      } else if (p.resident) {
        // all weight tiles, once, by one thread; their barrier counts them all
        if (tw == 1) {
          for (int nt = 0, i = 0; nt < p.n_tiles; ++nt)
            for (int r = 0; r < p.kh; ++r)
              for (int cb = 0; cb < p.cin_chunks; ++cb)
                for (int sx = 0; sx < p.kw; ++sx, ++i)
                  load(s_b + i * stage_b_bytes, &maps.w[0], ((r * p.kw + sx) * p.cin_chunks + cb) * kBK,
                       nt * BN + (int)rank * (BN / 2), b_wfull,
                       i == 0 ? (uint32_t)(p.n_tiles * p.num_kchunks) * stage_b_bytes : 0u);
        }
      } else {
        // weight tiles in the MMA's order (r, cb, s), the two threads taking every other one
        uint32_t it = 0, s = 0, ph = 0;
        for (int t = first_tile; t < tile_end && ok; t += p.tile_stride) {
          const TileInfo ti = tile_info(p, t);
          const CUtensorMap* wm = ti.bn == BN ? &maps.w[ti.layer] : &maps.wh;
          const int rows = kPair ? ti.bn / 2 : ti.bn, brow = ti.brow + (int)rank * rows;
          for (int pr = 0; pr < p.a_planes * p.kh && ok; ++pr) {
            const int r = pr >= p.kh ? pr - p.kh : pr;
            for (int cb = 0; cb < p.cin_chunks && ok; ++cb)
              for (int sx = 0; sx < p.kw; ++sx, ++it, s = (s + 1 == (uint32_t)SB) ? 0 : s + 1, ph ^= (s == 0)) {
                if ((int)(it & 1) != tw - 1) continue;
                if (!mbar_wait(b_wempty + 8 * s, ph ^ 1, abort_flag)) { ok = false; break; }
                load(s_b + s * stage_b_bytes, wm, ((r * p.kw + sx) * p.cin_chunks + cb) * kBK, brow, b_wfull + 8 * s,
                     (uint32_t)rows * kBK);
              }
          }
        }
      }
      if (!ok) fail(abort_flag, p.status);
    }
  } else if (!kFlat && warp >= kWarpProd0) {
    // ------------------------------------------------------------ activation producers
    const int row = (threadIdx.x - kWarpProd0 * 32) & (BM - 1);  // tile row of this thread,
    const int half = (warp - kWarpProd0) / (BM / 32);             // and its half of every K chunk
    const int r7 = row & 7;
    uint8_t* arow = smem + row * BK;
    int my_tiles = 0;
    for (int t = first_tile; t < tile_end; t += p.tile_stride) ++my_tiles;
    const int total = my_tiles * nk;

    RowCursor<kXBits> rc{};
    int l_tile = first_tile, l_q = 0;  // load cursor (runs four chunks ahead)
    auto start_tile = [&](int t) {
      const TileInfo ti = tile_info(p, t);
      const ConvJobDev& jb = p.jobs[ti.job];
      const int m = ti.mt * BM + row;
      rc.valid = m < jb.m_total;
      const int mm = rc.valid ? m : 0;
      const int img = fast_div(mm, jb.div_img);
      const int rem = mm - img * (jb.ho * jb.wo);
      const int ho = fast_div(rem, jb.div_row), wo = rem - ho * jb.wo;
      rc.hb = ho * p.stride - p.pad;
      rc.wb = wo * p.stride - p.pad;
      rc.H = jb.h;
      rc.W = jb.w;
      rc.xbase = jb.x + (int64_t)img * jb.h * jb.w * p.x_row_bytes;
      rc.tr = 0; rc.ts = 0; rc.tc0 = 0;
      if constexpr (kChunkInTap) rc.tc0 = 64 * half;
      else skip_groups(p, rc, 2 * half);
    };
    auto load_next = [&](uint32_t (&w)[2 * kXBits]) {
      if (l_q == 0) start_tile(l_tile);
      load_half<kXBits, kChunkInTap>(p, rc, l_q, half, w);
      if (++l_q == nk) { l_q = 0; l_tile += p.tile_stride; }
    };
    bool ok = true;
    const int S = p.stages;
    uint32_t b_empty, b_wfull, b_wempty;
    slots(b_empty, b_wfull, b_wempty);
    uint32_t s = 0, ph = 0;
    auto consume = [&](const uint32_t (&w)[2 * kXBits]) -> bool {
      if (!mbar_wait(b_empty + 8 * s, ph ^ 1, abort_flag)) return false;
      uint8_t* dst = arow + (size_t)s * kStageA;
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        uint32_t o[8];
        unpack_group_bytes<kXBits>(w + g * kXBits, o);  // raw E4M3 byte = code
        const int c16 = 4 * half + 2 * g;               // 16-byte column of the operand row
        *reinterpret_cast<uint4*>(dst + 16 * (c16 ^ r7)) = make_uint4(o[0], o[1], o[2], o[3]);
        *reinterpret_cast<uint4*>(dst + 16 * ((c16 + 1) ^ r7)) = make_uint4(o[4], o[5], o[6], o[7]);
      }
      fence_proxy_async();  // this thread's generic-proxy stores -> visible to the MMA
      __syncwarp();
      if (lane == 0) mbar_arrive(b_full + 8 * s);
      if (++s == (uint32_t)S) { s = 0; ph ^= 1; }
      return true;
    };
    uint32_t w[4][2 * kXBits];  // chunks in flight
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (i < total) load_next(w[i]);
    for (int c = 0; c < total && ok; c += 4) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (c + i >= total) break;
        if (!consume(w[i])) { ok = false; break; }
        if (c + i + 4 < total) load_next(w[i]);
      }
    }
    if (!ok) fail(abort_flag, p.status);
  } else {
    // ------------------------------------------------------------ epilogue (warps 0..E-1)
    // Warp w reads TMEM lanes 32*(w%4).. (the hardware lane quarter of its warp index), one lane
    // per output row, in steps of 16 columns. The warps of a quarter split a tile's 32-column groups
    // into epi_groups ranges; sets of epi_groups warps take tiles in turn (epi_sets > 1: narrow
    // tiles).
    //
    // What bounds it: for 256-channel tiles, stores to rows that lie apart (see store16 below); then the
    // issue of dependent integer instructions, about 9 per output and lane without a skip and 14 with
    // one, in about half of the cycles. So everything that does not depend on the column is done once per tile and lane (the
    // output pixel, by multiply-high divisions, and the row pointers), the rare forms live in a
    // function of their own, and four warps per scheduler cover the chains' latencies. Against two
    // warps per scheduler, 25 and 40 instructions per output (divisions per 32 columns, 64-bit
    // skip arithmetic): the whole detector at batch 8 1987 -> 1687 us, its third stage's entry
    // block 104 -> 78 us, a 1x1 128->512 conv with a skip on 30,400 pixels 49 -> 36 us.
    const int quarter = warp & 3;
    const int gset = (warp >> 2) / p.epi_groups, grp = (warp >> 2) - gset * p.epi_groups;
    const int et = threadIdx.x;  // 0 .. kEpiThreads-1
    // (read again for every tile: no register to spare)
    auto lane_base = [&]() {
      const uint32_t base = kF16 ? tmem_base : *const_cast<volatile uint32_t*>(tmem_slot);
      return base + ((uint32_t)(quarter * 32) << 16);
    };
    uint32_t lt = 0;
    bool ok = true;
    const int out_bits = p.out_bits;
    const int qmax = (1 << (out_bits & 15)) - 1;
    // the per-column constant tables of the last tile's level and channel range: rebuilt only
    // when a tile needs others (tiles of one job and N range keep them), so most tiles start
    // without table loads or barriers
    uint32_t cur_key = 0xFFFFFFFFu;  // (first channel, half width, job, layer) of the tables
    int flags = 0;
    for (;; ++lt) {
      // (worked out anew for every tile: no register to spare for the range)
      int t = (kPair ? (int)(blockIdx.x >> 1) : (int)blockIdx.x) + (int)lt * p.tile_stride;
      if (!kPair && p.contig) {
        const int b = (int)blockIdx.x;
        t = b * p.share + (b < p.extra ? b : p.extra) + (int)lt;
        if ((int)lt >= p.share + (b < p.extra ? 1 : 0)) break;
      } else if (t >= p.total_tiles) {
        break;
      }
      const TileInfo ti = tile_info(p, t);
      const ConvJobDev& jb = p.jobs[ti.job];
      // this tile's output channels that exist (a last N tile may reach past cout; packed
      // groups past it must not be written)
      const int TBN = ti.cn < p.cout - ti.col0 ? ti.cn : p.cout - ti.col0;
      const LayerDev& ly = p.layers[ti.layer];
      const uint32_t key = ((uint32_t)ti.col0 << 6) | (ti.bn != BN ? 32u : 0u) | ((uint32_t)ti.job << 2) | (uint32_t)ti.layer;
      if (key != cur_key) {
        // (the same decision in every epilogue thread: all of them see the same tiles)
        named_bar(1, kEpiThreads);  // every epilogue warp is done with the previous tables
        int fq = 1, sbias = 1, fsk = 1;
        for (int col = et; col < 256; col += kEpiThreads) {
          const int ch = ti.col0 + col;
          EpiChan ec{};
          int4 ef = make_int4((int32_t)(0u - kMagicBits), 0, 0, 1), es = make_int4(0, 0, 1, 0);
          if (col < TBN && ch < p.cout) {
            const int64_t idx = (int64_t)jb.level * p.cout + ch;
            ec.bias = ly.bias ? ly.bias[idx] : 0;
            const bool sb = ec.bias >= -(1 << 30) && ec.bias <= (1 << 30);
            sbias &= sb;
            ef.x = (int32_t)((uint32_t)ec.bias - kMagicBits);
            if (out_bits != 32) {
              ec.m0 = ly.m0[idx];
              const int r = 31 + ly.shift[idx];
              ec.r = (int8_t)r;
              if (r >= 33 && sb) { ef.y = ec.m0; ef.z = 1 << (r - 33); ef.w = r - 32; }
              else fq = 0;
            }
            if constexpr (kSkip) {
              ec.c = p.skip_c[idx]; ec.d = p.skip_d[idx];
              if (p.skip_bits > 4) fsk &= skip_const(p.skip_bits, ec.c, ec.d, es) ? 1 : 0;
            }
          }
          epi.gen()[col] = ec;
          epi.fast()[col] = ef;
          if constexpr (kSkip) epi.skip()[col] = es;
        }
        if constexpr (kSkip) {
          if (p.skip_bits <= 4) {
            int32_t* tab = reinterpret_cast<int32_t*>(smem + p.off_sktab);
            const int col = et & 255, ch = ti.col0 + col;
            if (col < TBN && ch < p.cout) {
              const int64_t idx = (int64_t)jb.level * p.cout + ch;
              const int64_t bias = ly.bias ? ly.bias[idx] : 0, c = p.skip_c[idx];
              const int dd = p.skip_d[idx];
              for (int s = et >> 8; s < (1 << p.skip_bits); s += kEpiThreads / 256) {
                const int64_t v = bias + rhu(s * c, dd);
                fsk &= v >= -(1LL << 30) && v <= (1LL << 30);
                tab[s * kSkipStride + col] = (int32_t)((uint32_t)v - kMagicBits);
              }
            }
          }
        }
        fq = named_bar_and(1, kEpiThreads, fq);
        sbias = named_bar_and(1, kEpiThreads, sbias);
        flags = (fq ? kFlagReq : 0) | (sbias ? kFlagBias : 0);
        if constexpr (kSkip) {
          fsk = named_bar_and(1, kEpiThreads, fsk);
          if (fsk && p.scale_main == 0) flags |= kFlagSkip;
        }
        cur_key = key;
      }
      if (!takes_tile(ok, lt, p.epi_sets, gset)) continue;  // another set's tile (or an idle warp, or a wait ran out)
      // (below, a warp's lanes give up on a wait together: they go on to warp-wide instructions and barriers)
      if constexpr (kF16) {
        // this warp's columns: whole 32-column groups, at most 64 (one int32 sum each per lane)
        const int per = ((TBN + 31) / 32 + p.epi_groups - 1) / p.epi_groups * 32;
        const int c_lo = grp * per, c_hi = c_lo + per < TBN ? c_lo + per : TBN;
        int32_t sum[64];
#pragma unroll
        for (int i = 0; i < 64; ++i) sum[i] = 0;
        const int nseg = (nk + p.seg_chunks - 1) / p.seg_chunks;
#pragma unroll 1
        for (int sg = 0; sg < nseg; ++sg) {
          const uint32_t un = lt * (uint32_t)nseg + (uint32_t)sg, b = un & buf_mask;
          // (no call here, where 64 sums are live: 3x3 128 -> 128 on four 100 x 168 maps and below 40.4 -> 39.6 us)
          if (!__all_sync(0xffffffffu, mbar_wait_inline(b_tfull + 8 * b, (un >> p.nbuf_log2) & 1, abort_flag))) { ok = false; break; }
          tc_fence_after();
          // (8 columns a load: beside 64 sums, 16 spill)
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            if (c_lo + 8 * j >= c_hi) break;
            uint32_t v[8];
            tmem_ld8(lane_base() + b * (uint32_t)BN + (uint32_t)(c_lo + 8 * j), v);
            tmem_wait_ld();
            reg_fence8(v);
#pragma unroll
            for (int i = 0; i < 8; ++i) sum[8 * j + i] += __float2int_rn(__uint_as_float(v[i]));
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) {
            if (kPair && !leader) mbar_arrive_cluster_relaxed(mapa_shared(b_tempty + 8 * b, 0));
            else mbar_arrive_relaxed(b_tempty + 8 * b);
          }
        }
        if (!ok) {
          fail(abort_flag, p.status);
          continue;
        }
        const FlatTile ft = flat_tile(jb, ti.mt, kTileRows);
        const int vr = ft.v0 + (int)rank * 128 + quarter * 32 + lane;
        const int oh = fast_div(vr, jb.div_row), ow = vr - oh * jb.wp;
        if (vr < jb.vimg && ow < jb.wo) {  // else a junk column or past the image
          // (the row pointers stand at the tile's first channel, a multiple of 32)
          const int grp0 = ti.col0 >> 5, nib = ly.ws_nib;
          uint8_t* yrow = ly.y[ti.job] + (int64_t)((ft.img * jb.ho + oh) * jb.wo + ow) * p.y_row_bytes + grp0 * group_bytes(out_bits);
          uint8_t* irow = ly.ws_out ? ly.ws_out + (size_t)(jb.orow_off + (ft.img * jb.ohp + oh + p.out_pad) * jb.owp + ow +
                                                           p.out_pad) * p.cout + grp0 * (nib ? 16 : 32)
                                    : nullptr;
          const bool lean = kOStage ? (flags & kFlagBias) && (p.cout & 3) == 0
                                    : (flags & kFlagReq) && (out_bits != 8 || (p.cout & 31) == 0);
          if (__builtin_expect(lean, 1)) {
            // (|sum| < 2^28 and |bias| <= 2^30)
            uint32_t top = 0u;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const int c0 = c_lo + 16 * j;
              if (c0 >= c_hi) break;
              const int4* ef = epi.fast() + c0;
              auto biased = [&](int i) { return sum[16 * j + i] + (int32_t)((uint32_t)ef[i].x + kMagicBits); };
              if constexpr (kOStage) {  // sum + bias in whole 16-byte pieces
                int4* yr = reinterpret_cast<int4*>(yrow) + (c0 >> 2);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                  if (c0 + 4 * q < c_hi) yr[q] = make_int4(biased(4 * q), biased(4 * q + 1), biased(4 * q + 2), biased(4 * q + 3));
              } else {
                uint32_t bw[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                for (int i = 0; i < 16; ++i) bw[i / 4] += requant32(biased(i), ef[i], qmax) << (8 * (i % 4));
                store_codes16(yrow, c0, bw, out_bits, top);
                if (irow) store_image16(irow, c0, bw, nib);
              }
            }
          } else {
            int32_t all[64];
#pragma unroll
            for (int i = 0; i < 64; ++i) all[i] = sum[i];
            general_sums(p, GenTile{0u, 0, smem_u32(epi.gen()), c_lo, c_hi, flags, nib, nullptr, yrow, irow}, all);
          }
        }
        __syncwarp();
        continue;
      }
      const uint32_t buf = lt & buf_mask;

      // this lane's output row
      int m;  // output pixel index within the job
      bool row_ok;
      int img = 0, oh = 0, ow = 0;
      if constexpr (kFlat) {
        const FlatTile ft = flat_tile(jb, ti.mt, kTileRows);
        const int vr = ft.v0 + (int)rank * 128 + quarter * 32 + lane;  // virtual row at the padded width
        img = ft.img;
        oh = fast_div(vr, jb.div_row);
        ow = vr - oh * jb.wp;
        row_ok = vr < jb.vimg && ow < jb.wo;  // else a junk column or past the image
        m = (img * jb.ho + oh) * jb.wo + ow;
      } else {
        m = ti.mt * BM + quarter * 32 + lane;
        row_ok = m < jb.m_total;
        if constexpr (kSkip) {
          img = fast_div(m, jb.div_img);
          const int rem = m - img * (jb.ho * jb.wo);
          oh = fast_div(rem, jb.div_row);
          ow = rem - oh * jb.wo;
        }
      }
      // the row pointers stand at the tile's first channel (a multiple of 32)
      const int grp0 = ti.col0 >> 5;
      uint8_t* yrow = ly.y[ti.job] + (int64_t)m * p.y_row_bytes + grp0 * group_bytes(out_bits);
      uint8_t* irow = nullptr;  // this row of the chained image
      const int nib = ly.ws_nib;
      if (kFlat && ly.ws_out)
        irow = ly.ws_out +
               (size_t)(jb.orow_off + (img * jb.ohp + oh + p.out_pad) * jb.owp + ow + p.out_pad) * p.cout +
               grp0 * (nib ? 16 : 32);
      const uint8_t* srow = nullptr;
      if constexpr (kSkip) {
        const int up = p.upsample == 2 ? 1 : 0;
        srow = jb.skip + (((int64_t)img * jb.skip_h + (oh >> up)) * jb.skip_w + (ow >> up)) * p.skip_row_bytes +
               grp0 * group_bytes(p.skip_bits);
      }

      // this warp's columns [c_lo, c_hi), whole 32-column groups but for the tile's last one
      const int per = ((TBN + 31) / 32 + p.epi_groups - 1) / p.epi_groups * 32;
      const int c_lo = grp * per, c_hi = c_lo + per < TBN ? c_lo + per : TBN;
      const uint32_t tbuf = lane_base() + buf * (uint32_t)BN;
      // The common forms; everything else goes through general_tile.
      //  codes:  the 32-bit requant of FP32 accumulators below 2^22 (or split sums), and, with a
      //          skip, the 32-bit rescale;  int32 outputs: the sum alone
      bool common;
      [[maybe_unused]] const bool lean32 = p.acc_small && (flags & kFlagBias);  // int32 outputs without saturation
      if constexpr (kOStage) common = true;
      else if constexpr (kSkip)
        common = p.acc_small && out_bits != 32 && (flags & (kFlagReq | kFlagSkip)) == (kFlagReq | kFlagSkip);
      else if constexpr (kSplit) common = out_bits != 32 && (flags & kFlagReq);
      else common = p.acc_small && (flags & (out_bits == 32 ? kFlagBias : kFlagReq));
      // rows whose pieces would not be aligned, or not whole
      if ((out_bits == 8 && (p.cout & 31) != 0) || (out_bits == 32 && (p.cout & 3) != 0)) common = false;
      if (kSkip && p.skip_bits >= 8 && (p.skip_row_bytes & 15) != 0) common = false;
      // int32 skips: the skip pixels of the four rows whose pieces this lane copies (-1: none)
      [[maybe_unused]] int sp4[4] = {-1, -1, -1, -1};
      [[maybe_unused]] const uint32_t sk_stage = sbase + p.off_sktab + (uint32_t)warp * (2 * kSkipStage);
      // Columns c0 .. c0 + 15, or an empty group past the end: the wait of the last step then completes
      // every copy, before the next tile's copies (which nothing would order against them) go to the same places.
      auto copy_skip32 = [&](int c0, int step) {
        if (c0 < c_hi) {
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const bool on = sp4[k] >= 0;
            const uint8_t* src = jb.skip;
            if (on) src += (int64_t)sp4[k] * p.skip_row_bytes + (int64_t)(ti.col0 + c0) * 4 + (lane & 3) * 16;
            cp_async<16>(sk_stage + (uint32_t)(step & 1) * kSkipStage + skip_stage_off(8 * k + (lane >> 2), lane & 3), src, on);
          }
        }
        cp_async_commit();
      };
      const bool sk_int = kSkip && p.skip_bits == 32 && common;
      if constexpr (kSkip) {
        if (sk_int) {
          const int up = p.upsample == 2 ? 1 : 0;
          const int sp = row_ok ? (img * jb.skip_h + (oh >> up)) * jb.skip_w + (ow >> up) : -1;
#pragma unroll
          for (int k = 0; k < 4; ++k) sp4[k] = __shfl_sync(0xffffffffu, sp, 8 * k + (lane >> 2));
          copy_skip32(c_lo, 0);
          copy_skip32(c_lo + 16, 1);
        }
      }
      uint4 sw = make_uint4(0u, 0u, 0u, 0u);  // a group's skip codes (a half's in x and y), loaded a step ahead
      const bool sk_codes = kSkip && p.skip_bits <= 4;
      if (sk_codes && c_lo < c_hi) sw = load_skip_group(srow, c_lo, p.skip_bits, row_ok);
      __syncwarp();
      if (!__all_sync(0xffffffffu, mbar_wait_inline(b_tfull + 8 * buf, (lt >> p.nbuf_log2) & 1, abort_flag))) {
        if constexpr (kSkip) cp_async_wait<0>();  // (no copy outlives the block)
        ok = false;
        fail(abort_flag, p.status);
        continue;
      }
      tc_fence_after();
      auto release = [&]() {  // every TMEM read of this warp is complete
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (kPair && !leader) mbar_arrive_cluster_relaxed(mapa_shared(b_tempty + 8 * buf, 0));
          else mbar_arrive_relaxed(b_tempty + 8 * buf);
        }
      };
      // A warp's columns are whole 32-channel groups (where pieces are stored at all), whose halves are
      // stored together: a lane's 16 or 32 bytes are whole sectors' parts. (Its rows lie a row of the
      // output apart, so a warp's store goes to 32 sectors whatever its width.) 256-channel layer of
      // a detector tower with a chained image 67.5 -> 60.8 us (58 with no stores at all), batch-8 detector 1286 -> 1234.
      uint32_t first[4] = {0u, 0u, 0u, 0u};  // the group's first half
      auto store16 = [&](int c0, const uint32_t (&bw)[4]) {
        if (!(c0 & 16)) {
#pragma unroll
          for (int q = 0; q < 4; ++q) first[q] = bw[q];
          return;
        }
        if (!row_ok) return;
        store_codes32(yrow, c0 - 16, first, bw, out_bits);
        if (kFlat && irow) store_image32(irow, c0 - 16, first, bw, nib);
      };
      // int32 skips may turn out to need the general form, which reads the accumulator again
      const bool late = !common || (kSkip && p.skip_bits == 32);
      uint32_t big = 0u;  // bits above 27 set: an int32 skip beyond the 32-bit form
      if (common) {
        if (c_lo >= c_hi && !late) release();
#pragma unroll 1
        for (int c0 = c_lo; c0 < c_hi; c0 += 16) {
          const bool last = c0 + 16 >= c_hi;
          const int4* ef = epi.fast() + c0;
          const int4* es = epi.skip() + c0;
          uint32_t bw[4] = {0u, 0u, 0u, 0u};
          uint32_t v[16];
          tmem_ld16(tbuf + c0, v);
          // One FMA turns the accumulator float acc / sc into the int32 acc + kMagicBits; ef.x
          // holds bias - kMagicBits (no int32 overflow under the stated bounds).
          if constexpr (kSkip) {
            auto sum = [&](int i, const int4& c, int32_t scaled) {
              return __float_as_int(__fmaf_rn(__uint_as_float(v[i]), kAccSc, kMagic)) + c.x + skip32(scaled, es[i]);
            };
            if (sk_codes) {
              uint32_t sb[4];
              skip_bytewords(make_uint2(sw.x, sw.y), p.skip_bits, sb);
              if (!(c0 & 16)) { sw.x = sw.z; sw.y = sw.w; }
              else if (!last) sw = load_skip_group(srow, c0 + 16, p.skip_bits, row_ok);
              const int32_t* tab = reinterpret_cast<const int32_t*>(smem + p.off_sktab) + c0;
              tmem_wait_ld();
              reg_fence16(v);
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                const int s = (int)((sb[i / 4] >> (8 * (i % 4))) & 0xFFu);
                const int32_t u = __float_as_int(__fmaf_rn(__uint_as_float(v[i]), kAccSc, kMagic)) + tab[s * kSkipStride + i];
                bw[i / 4] += requant32(u, ef[i], qmax) << (8 * (i % 4));  // codes < 256: the add is an or
              }
            } else {
              // 8-bit or int32 skips, four columns at a time
              tmem_wait_ld();
              reg_fence16(v);
              const int step = (c0 - c_lo) >> 4;
              if (p.skip_bits == 32) {
                cp_async_wait<1>();  // this step's copies (the next step's may be in flight)
                __syncwarp();
              }
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                int4 x = make_int4(0, 0, 0, 0);
                if (p.skip_bits == 8) {
                  const uint32_t w = row_ok ? __ldg(reinterpret_cast<const uint32_t*>(srow + c0) + q) : 0u;
                  x = make_int4((int)(__byte_perm(w, 0u, 0x0444) >> 1), (int)(__byte_perm(w, 0u, 0x1444) >> 1),
                                (int)(__byte_perm(w, 0u, 0x2444) >> 1), (int)(__byte_perm(w, 0u, 0x3444) >> 1));
                } else {
                  x = *reinterpret_cast<const int4*>(smem + (sk_stage - sbase) + (step & 1) * kSkipStage + skip_stage_off(lane, q));
                  big |= magnitude(x.x) | magnitude(x.y) | magnitude(x.z) | magnitude(x.w);
                  x = make_int4((int)((uint32_t)x.x << 3), (int)((uint32_t)x.y << 3), (int)((uint32_t)x.z << 3),
                                (int)((uint32_t)x.w << 3));
                }
                const int4 k0 = ef[4 * q], c1 = ef[4 * q + 1], c2 = ef[4 * q + 2], c3 = ef[4 * q + 3];
                bw[q] = requant32(sum(4 * q, k0, x.x), k0, qmax) | (requant32(sum(4 * q + 1, c1, x.y), c1, qmax) << 8) |
                        (requant32(sum(4 * q + 2, c2, x.z), c2, qmax) << 16) |
                        (requant32(sum(4 * q + 3, c3, x.w), c3, qmax) << 24);
              }
              if (p.skip_bits == 32) {
                __syncwarp();  // every lane has read its row
                copy_skip32(c0 + 32, step);
              }
            }
            if (last && !late) release();
          } else if constexpr (kSplit) {
            // split weights: v holds D1 (w_lo rows); D2 (w_hi rows) sits cn columns on; the exact
            // sum is D1 + 16 D2, each an integer x 2^-18 below 2^24 (|sum| < 2^29, |bias| <= 2^30)
            uint32_t vb[16];
            tmem_ld16(tbuf + (uint32_t)(ti.cn + c0), vb);
            tmem_wait_ld();
            reg_fence16(v);
            reg_fence16(vb);
            if (last) release();
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const int4 c = ef[i];
              const int32_t d1 = __float2int_rn(__uint_as_float(v[i]) * kAccSc);
              const int32_t d2 = __float2int_rn(__uint_as_float(vb[i]) * kAccSc);
              bw[i / 4] += requant32(d1 + 16 * d2 + (int32_t)((uint32_t)c.x + kMagicBits), c, qmax) << (8 * (i % 4));
            }
          } else {
            tmem_wait_ld();
            reg_fence16(v);
            if (last) release();
            if (kOStage || out_bits == 32) {
              // int32 outputs: acc + bias
              if (!kOStage || lean32) {
#pragma unroll
                for (int i = 0; i < 16; ++i)
                  v[i] = (uint32_t)(__float_as_int(__fmaf_rn(__uint_as_float(v[i]), kAccSc, kMagic)) + ef[i].x);
              } else {
#pragma unroll
                for (int i = 0; i < 16; ++i)
                  v[i] = (uint32_t)add_sat(__float2int_rn(__uint_as_float(v[i]) * kAccSc), (int32_t)((uint32_t)ef[i].x + kMagicBits));
              }
              const int nq = (c_hi - c0 < 16 ? c_hi - c0 : 16) >> 2;  // whole 16-byte pieces (cout % 4 == 0)
              if constexpr (kOStage) {
                // through this warp's staging block: each lane holds its row's 16 values; stored
                // back eight rows at a time, so a warp store covers whole sectors of eight row
                // segments instead of 32 scattered 16-byte pieces
                uint32_t* stg = reinterpret_cast<uint32_t*>(smem + p.off_ostage) + warp * (32 * kStageRow);
                const uint32_t rows_ok = __ballot_sync(0xffffffffu, row_ok);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                  *reinterpret_cast<uint4*>(stg + lane * kStageRow + 4 * q) =
                      make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
                __syncwarp();
#pragma unroll
                for (int r8 = 0; r8 < 4; ++r8) {
                  const int r = 8 * r8 + (lane >> 2), c4 = lane & 3;
                  const int mr = __shfl_sync(0xffffffffu, m, r);
                  if (((rows_ok >> r) & 1u) && c4 < nq)
                    *reinterpret_cast<uint4*>(ly.y[ti.job] + (int64_t)mr * p.y_row_bytes + (int64_t)(ti.col0 + c0 + 4 * c4) * 4) =
                        *reinterpret_cast<const uint4*>(stg + r * kStageRow + 4 * c4);
                }
                __syncwarp();
              } else if (row_ok) {
                uint4* yr = reinterpret_cast<uint4*>(yrow) + (c0 >> 2);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                  if (q < nq) yr[q] = make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
              }
              continue;
            }
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const int4 c = ef[i];
              const int32_t u = __float_as_int(__fmaf_rn(__uint_as_float(v[i]), kAccSc, kMagic)) + c.x;
              bw[i / 4] += requant32(u, c, qmax) << (8 * (i % 4));  // codes < 256: the add is an or
            }
          }
          store16(c0, bw);
        }
        if constexpr (kSkip) common = !__any_sync(0xffffffffu, (big >> 28) != 0u);
      }
      if (!common) {
        const GenTile g{tbuf, ti.cn, smem_u32(epi.gen()), c_lo, c_hi, flags, nib, srow, row_ok ? yrow : nullptr, irow};
        general_tile<kSkip, kSplit>(p, g, kAccSc);
      }
      if (late) release();
      const int tile = (int)(blockIdx.x >> 1) + (int)lt * p.tile_stride;  // (t, worked out again)
      if (kPair && p.dep && tile < (p.nlayers - 1) * p.layer_tiles) {
        // this warp's stores of tile t are done: order them for the next layer's TMA (async
        // proxy) loads, gather the warp (__syncwarp orders its lanes' stores before lane 0's
        // next operations), and count the warp in with one release (cumulative over them)
        fence_proxy_async_global();
        __syncwarp();
        // (a tower launch has no half-width tiles: t is layer * layer_tiles + the tile)
        if (lane == 0) red_release_gpu_add(p.dep + tile, 1u);
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  // neither CTA of a pair leaves while the leader's MMAs may still read the peer's shared
  // memory or write its TMEM (the leader's MMA thread drained them before the barrier)
  if constexpr (kPair) cluster_sync();
  if (warp == kWarpMma) {
    tc_fence_after();
    if constexpr (kPair)
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;"
                   ::"r"(tmem_base), "r"(p.tmem_cols) : "memory");
    else
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                   ::"r"(tmem_base), "r"(p.tmem_cols) : "memory");
  }
}

// ---------------------------------------------------------------- activation expansion

// Writes every job's input as a zero-padded byte image: workspace row
// row_off + (img * hp + hp_i) * wp + wp_i holds the cin E4M3 bytes (raw byte = code) of
// input pixel (img, hp_i - pad, wp_i - pad), or zeros in the padding border.
struct ExpandArgs {
  ConvJobDev jobs[kMaxJobs];
  int32_t njobs, cin, pad;
  int64_t x_row_bytes;
  int64_t total_rows;     // rows of one plane
  uint8_t* ws;
  // per-tile counters of a chained tower, cleared here (before the first layer, which waits
  // for this grid, can raise them)
  uint32_t* zero;
  int32_t zero_words;
};

// E4M3 byte of the value 16 n * 2^-9 = n * 2^-5, n in [0, 15] (the raw byte n is n * 2^-9):
// n = 2^e (1 + m/8) with 8-bit exponent field e + 2, packed as two 64-bit tables of 8 bytes.
__device__ __forceinline__ uint32_t e4m3_times16(uint32_t n) {
  constexpr uint64_t lo = 0x26242220'1C181000ull;  // n = 7 .. 0
  constexpr uint64_t hi = 0x2F2E2D2C'2B2A2928ull;  // n = 15 .. 8
  return (uint32_t)(((n < 8 ? lo : hi) >> (8 * (n & 7))) & 0xFFu);
}

// Position of one workspace row: its job, image, padded row / column and input pointer.
struct ExpandPos {
  int row, job, img, hr, wc;  // workspace row; job; image; padded row and column
  int next_off;               // first row of the next job (INT_MAX for the last)
};

__device__ __forceinline__ void expand_locate(const ExpandArgs& a, int row, ExpandPos& ps) {
  int j = 0;
#pragma unroll 1
  while (j + 1 < a.njobs && row >= a.jobs[j + 1].row_off) ++j;
  const ConvJobDev& jb = a.jobs[j];
  const int local = row - jb.row_off;
  const int plane = jb.hp * jb.wp;
  ps.row = row;
  ps.job = j;
  ps.img = local / plane;
  const int rem = local - ps.img * plane;
  ps.hr = rem / jb.wp;
  ps.wc = rem - ps.hr * jb.wp;
  ps.next_off = j + 1 < a.njobs ? a.jobs[j + 1].row_off : 0x7fffffff;
}

// Moves the position forward by d rows (d small: at most 4 here).
__device__ __forceinline__ void expand_advance(const ExpandArgs& a, int d, ExpandPos& ps) {
  ps.row += d;
  if (ps.row >= ps.next_off) { expand_locate(a, ps.row, ps); return; }
  const ConvJobDev& jb = a.jobs[ps.job];
  ps.wc += d;
#pragma unroll 1
  while (ps.wc >= jb.wp) {
    ps.wc -= jb.wp;
    if (++ps.hr == jb.hp) { ps.hr = 0; ++ps.img; }
  }
}

// kXBits = 16: 8-bit codes as F16 values (the F16 pipe's image), 8 codes per 16 bytes of the image.
template <int kXBits>
__global__ void __launch_bounds__(256) expand_kernel(const __grid_constant__ ExpandArgs a) {
  // The (row, 16-byte chunk) pairs of the workspace, row-major, are split into runs of
  // 32 * kPerLane; a warp takes one run, lane l the pairs l, l + 32, ... of it, so every
  // warp-wide step reads consecutive packed words and writes 512 consecutive bytes. The
  // position is divided out once per lane and then advanced incrementally; the loads of
  // all steps are issued before the stores. All index arithmetic is 32-bit (the host
  // checks rows * cin / 16 < 2^31).
  constexpr int kPerLane = 4;  // (measured: 4 beats 8 and 2 on the head step, 120.6 / 121.7 / 121.5 us)
  // the previous kernel in the stream may still be reading the workspace or writing x
  grid_dep_wait();
  if (threadIdx.x == 0) grid_dep_launch();
  if (blockIdx.x == 0)
    for (int i = threadIdx.x; i < a.zero_words; i += blockDim.x) a.zero[i] = 0u;
  constexpr bool kF16 = kXBits == 16;
  const int chunks = kF16 ? a.cin >> 3 : a.cin >> 4;
  const int row_bytes = kF16 ? 2 * a.cin : a.cin;
  const int total = (int)a.total_rows * chunks;
  const int lane = threadIdx.x & 31;
  const int e0 = (blockIdx.x * 8 + (threadIdx.x >> 5)) * (32 * kPerLane) + lane;
  if (e0 >= total) return;
  const int drow = 32 / chunks, dq = 32 - drow * chunks;
  ExpandPos ps;
  int q = e0 % chunks;
  expand_locate(a, e0 / chunks, ps);
  uint32_t w[kPerLane][kXBits == 2 ? 1 : (kXBits == 8 ? 4 : 2)];  // (16: 8 codes)
  uint8_t* dst[kPerLane];
  bool inside[kPerLane];
  int hsel[kPerLane];
#pragma unroll
  for (int i = 0; i < kPerLane; ++i) {
    const int e = e0 + 32 * i;
    const bool live = e < total;
    const ConvJobDev& jb = a.jobs[ps.job];
    const int hi = ps.hr - a.pad, wi = ps.wc - a.pad;
    inside[i] = live && hi >= 0 && hi < jb.h && wi >= 0 && wi < jb.w;
    dst[i] = live ? a.ws + (size_t)ps.row * row_bytes + q * 16 : nullptr;
    hsel[i] = q & 1;
    if (inside[i]) {
      const uint32_t* grp = reinterpret_cast<const uint32_t*>(
          jb.x + ((size_t)(ps.img * jb.h + hi) * jb.w + wi) * a.x_row_bytes + (q >> 1) * 4 * kXBits);
      if constexpr (kF16) {
        const uint2 v = __ldg(reinterpret_cast<const uint2*>(jb.x + ((size_t)(ps.img * jb.h + hi) * jb.w + wi) *
                                                             a.x_row_bytes) + q);
        w[i][0] = v.x; w[i][1] = v.y;
      } else if constexpr (kXBits == 8) {
        // 16 one-byte codes: channels 16 q .. 16 q + 15
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(jb.x + ((size_t)(ps.img * jb.h + hi) * jb.w + wi) *
                                                             a.x_row_bytes) + q);
        w[i][0] = v.x; w[i][1] = v.y; w[i][2] = v.z; w[i][3] = v.w;
      } else if constexpr (kXBits == 2) {
        w[i][0] = __ldg(grp + (q & 1));
      } else if constexpr (kXBits == 4) {
        const uint2 v = __ldg(reinterpret_cast<const uint2*>(grp) + (q & 1));
        w[i][0] = v.x; w[i][1] = v.y;
      } else {
        w[i][0] = __ldg(grp + (q & 1)); w[i][1] = __ldg(grp + 2);
      }
    }
    if (i + 1 < kPerLane) {
      q += dq;
      int step = drow;
      if (q >= chunks) { q -= chunks; ++step; }
      if (step) expand_advance(a, step, ps);
    }
  }
#pragma unroll
  for (int i = 0; i < kPerLane; ++i) {
    if (!dst[i]) continue;
    uint32_t o[4] = {0u, 0u, 0u, 0u};
    if constexpr (kF16) {
      // the F16 bit pattern 0x6400 | x is 1024 + x; the subtraction of 1024 is exact
      if (inside[i]) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint32_t u = __byte_perm(w[i][k >> 1], 0x64646464u, (k & 1) ? 0x4342u : 0x4140u);
          asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(o[k]) : "r"(u), "r"(0x64006400u));
        }
      }
      *reinterpret_cast<uint4*>(dst[i]) = make_uint4(o[0], o[1], o[2], o[3]);
      continue;
    }
    if constexpr (kXBits == 8) {
      // plane 0: x_lo = x & 15 (raw byte); plane 1, total_rows rows on: 16 x_hi as E4M3
      uint32_t o1[4] = {0u, 0u, 0u, 0u};
      if (inside[i]) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          o[j] = w[i][j] & 0x0F0F0F0Fu;
          const uint32_t hn = (w[i][j] >> 4) & 0x0F0F0F0Fu;
          o1[j] = e4m3_times16(hn & 0xFFu) | (e4m3_times16((hn >> 8) & 0xFFu) << 8) |
                  (e4m3_times16((hn >> 16) & 0xFFu) << 16) | (e4m3_times16(hn >> 24) << 24);
        }
      }
      *reinterpret_cast<uint4*>(dst[i]) = make_uint4(o[0], o[1], o[2], o[3]);
      *reinterpret_cast<uint4*>(dst[i] + (size_t)a.total_rows * a.cin) = make_uint4(o1[0], o1[1], o1[2], o1[3]);
      continue;
    }
    if (inside[i]) {
      const int h = hsel[i];
      if constexpr (kXBits == 2) {
#pragma unroll
        for (int j = 0; j < 4; ++j) o[j] = (w[i][0] >> (2 * j)) & 0x03030303u;
      } else if constexpr (kXBits == 4) {
        o[0] = w[i][0] & 0x0F0F0F0Fu; o[1] = (w[i][0] >> 4) & 0x0F0F0F0Fu;
        o[2] = w[i][1] & 0x0F0F0F0Fu; o[3] = (w[i][1] >> 4) & 0x0F0F0F0Fu;
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          o[j] = ((w[i][0] >> (2 * j)) & 0x03030303u) | (((w[i][1] >> (4 * h + j)) & 0x01010101u) << 2);
      }
    }
    *reinterpret_cast<uint4*>(dst[i]) = make_uint4(o[0], o[1], o[2], o[3]);
  }
}

// The zero-padded nibble image of 2-bit codes for the FP4 pipe: the first cin / 2 bytes of
// workspace row r (rows cin bytes apart, as in the byte image) hold two codes per byte,
// channel 2k in the low nibble of byte k, of input pixel (img, hp - pad, wp - pad), or zeros
// in the border (code 0 is the E2M1 value 0). One thread
// per 16 output bytes, i.e. one 32-channel packed group of 8 input bytes; consecutive threads
// take consecutive groups of a row.
__global__ void __launch_bounds__(256) expand_nib_kernel(const __grid_constant__ ExpandArgs a) {
  grid_dep_wait();
  if (threadIdx.x == 0) grid_dep_launch();
  const int groups = a.cin >> 5;
  const int64_t total = a.total_rows * groups;
  for (int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < total; e += (int64_t)gridDim.x * 256) {
    const int row = (int)(e / groups), g = (int)(e - (int64_t)row * groups);
    ExpandPos ps;
    expand_locate(a, row, ps);
    const ConvJobDev& jb = a.jobs[ps.job];
    const int hi = ps.hr - a.pad, wi = ps.wc - a.pad;
    uint32_t o[4] = {0u, 0u, 0u, 0u};
    if (hi >= 0 && hi < jb.h && wi >= 0 && wi < jb.w) {
      const uint2 v = __ldg(reinterpret_cast<const uint2*>(jb.x + ((size_t)(ps.img * jb.h + hi) * jb.w + wi) *
                                                                   a.x_row_bytes) + g);
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        // output word m: channels 8m .. 8m + 7, the byte-words 2(m % 2) and 2(m % 2) + 1 of
        // packed word m / 2 (byte-word j of a 2-bit word: channels 4j .. 4j + 3, one per byte)
        const uint32_t wd = (m >> 1) ? v.y : v.x;
        const int j0 = 2 * (m & 1);
        const uint32_t b0 = (wd >> (2 * j0)) & 0x03030303u, b1 = (wd >> (2 * j0 + 2)) & 0x03030303u;
        o[m] = __byte_perm(b0 | (b0 >> 4), b1 | (b1 >> 4), 0x6420);
      }
    }
    *reinterpret_cast<uint4*>(a.ws + (size_t)row * a.cin + (size_t)g * 16) = make_uint4(o[0], o[1], o[2], o[3]);
  }
}

// ---------------------------------------------------------------- host side

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn get_encode_fn(std::string* err) {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  static cudaError_t st = cudaSuccess;
  std::call_once(once, [] {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    st = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &q);
    if (st == cudaSuccess && q == cudaDriverEntryPointSuccess) fn = reinterpret_cast<EncodeTiledFn>(ptr);
  });
  if (!fn && err) *err = "cuTensorMapEncodeTiled entry point unavailable";
  return fn;
}

template <int kXBits, bool kChunkInTap, bool kFlat, bool kPair = false, bool kSkip = true, bool kSplit = false,
          int kBK = BK, bool kFp4 = false, bool kOStage = false>
static int launch_bits(const Params& prm, const Maps& maps, int grid, size_t smem, cudaStream_t stream,
                       std::string* err) {
  auto kern = conv_tc_kernel<kXBits, kChunkInTap, kFlat, kPair, kSkip, kSplit, kBK, kFp4, kOStage>;
  // The opt-in limit is raised to the device maximum, never lowered to this call's size:
  // a CUDA graph node captured earlier with a larger plan must stay launchable (a graph
  // node, or a tool relaunching it, is checked against the function's current limit).
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if ((size_t)optin < smem) { *err = "conv_tc: shared memory plan exceeds the device limit"; return 2; }
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  if (e != cudaSuccess) { *err = std::string("cudaFuncSetAttribute: ") + cudaGetErrorString(e); return 3; }
  // programmatic dependent launch: the prologue (barriers, TMEM allocation, tensor-map
  // prefetch) overlaps the previous kernel; the kernel waits for it before touching global
  // memory. CTA pairs run as clusters of two.
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads_for(kFlat));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 2;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = kPair ? 2 : 1;
  e = cudaLaunchKernelEx(&cfg, kern, maps, prm);
  if (e != cudaSuccess) { *err = std::string("conv_tc launch: ") + cudaGetErrorString(e); return 3; }
  e = cudaGetLastError();
  if (e != cudaSuccess) { *err = std::string("conv_tc launch: ") + cudaGetErrorString(e); return 3; }
  return 0;
}

}  // namespace tc

bool conv_tc_uses_pair(const ConvArgs& a) {
  // every N tile width of the workspace path (BN is a multiple of 16, so each CTA's half of
  // the weight tile is whole 8-row swizzle atoms and M = 256 MMAs take N = BN), except narrow
  // tiles on the FP4 pipe. Single CTAs / pairs in us, five levels of a head, expansion included: 3x3 256 -> 84
  // int32 at batch 1 11.3 / 11.9, 2 14.5 / 15.8, 4 21.5 / 23.3, 16 67 / 68; 3x3 256 -> 128 2-bit at batch 2 14.7 /
  // 16.2; 1x1 256 -> 64 at batch 4 14.3 / 17.2. (Of 100 such layers pairs are ahead in three, by 5%: 3x3 to 16, 36 and
  // 128 int32 outputs at batch 16.)
  if (a.fp4 && a.bn <= 128) return false;
  return a.ws != nullptr && a.bn >= 16 && a.bn % 16 == 0 && !a.no_pair;
}

// Last-wave balancing: with `workers` persistent CTAs (or CTA pairs), the full tiles past the
// last complete wave run as two half-width (N/2) tiles each, when those halves still fit in
// one wave; half as long per tile, they end the kernel sooner. A half tile must start on a
// 32-channel packing group (bn / 2 a multiple of 32). Returns the first split tile.
static int split_start(int tiles, int workers, int bn, bool split_w) {
  const int rem = tiles % workers;
  return (bn % 64 == 0 && !split_w && rem > 0 && 2 * rem <= workers) ? tiles - rem : tiles;
}

int64_t conv_tc_pair_tiles(const ConvArgs& a) {
  int64_t tiles = 0;
  for (int j = 0; j < a.njobs; ++j) {
    const ConvJobDev& jb = a.jobs[j];
    const int64_t wp = jb.w + 2 * a.pad;
    tiles += (int64_t)jb.n * ((jb.ho * wp + 255) / 256);
  }
  return tiles;
}

int launch_conv_tc(const ConvArgs& a, cudaStream_t stream, std::string* err) {
  using namespace tc;
  Params prm{};
  // split (8-bit) weights: tiles of 256 weight rows = 128 output channels
  const int BN = a.split_w ? 256 : a.bn;
  const bool f16 = a.f16 != 0;
  const int w_rows = a.split_w ? a.split_rows : a.cout_pad;  // rows of the weight block
  prm.njobs = a.njobs;
  prm.n_tiles = w_rows / BN;
  // flat path: the activations are expanded into the workspace first (stride 1,
  // cin % 128 == 0; the API checks both before passing a workspace)
  const bool flat = a.ws != nullptr;
  // CTA pairs (cta_group::2, M = 256 per tile) on the workspace path: each SM streams half
  // of the weight tile per K chunk, and one MMA instruction covers both SMs' rows
  const bool pair = conv_tc_uses_pair(a);
  const int tile_rows = pair ? 256 : 128;
  int tiles = 0;
  int64_t rows = 0;
  for (int j = 0; j < a.njobs; ++j) {
    prm.jobs[j] = a.jobs[j];
    prm.jobs[j].tile_begin = tiles;
    if (flat) {
      ConvJobDev& jb = prm.jobs[j];
      jb.hp = jb.h + 2 * a.pad;
      jb.wp = jb.w + 2 * a.pad;
      jb.vimg = jb.ho * jb.wp;
      jb.tpi = (jb.vimg + tile_rows - 1) / tile_rows;
      jb.div_img = div_magic(jb.tpi);
      jb.div_row = div_magic(jb.wp);
      jb.row_off = (int32_t)rows;
      rows += (int64_t)jb.n * jb.hp * jb.wp;
      tiles += jb.n * jb.tpi * prm.n_tiles;
    } else {
      tiles += ((a.jobs[j].m_total + BM - 1) / BM) * prm.n_tiles;
      prm.jobs[j].div_img = div_magic(a.jobs[j].ho * a.jobs[j].wo);
      prm.jobs[j].div_row = div_magic(a.jobs[j].wo);
    }
  }
  // K chunk width: 128 bytes of one tap, or on the workspace path with cin % 128 != 0 the 64
  // channels of one tap (cin % 64 == 0; 64-byte swizzled operand rows, two MMAs per chunk)
  const bool fp4 = a.fp4 != 0;
  // bytes per row of the image: one code per byte, or two (nibbles) on the FP4 pipe
  const int img_row = fp4 ? a.cin / 2 : (f16 ? 2 * a.cin : a.cin);
  const int bk = (flat && img_row % BK != 0) ? 64 : BK;
  if (flat && (a.stride != 1 || img_row % bk != 0 || rows > a.ws_rows || (a.split_w && bk != BK))) {
    *err = "conv_tc: workspace path needs stride 1, cin % 64 == 0 (128 for split weights) and a large enough workspace";
    return 1;
  }
  if (fp4 && !(flat && bk == BK && a.x_bits == 2 && !a.split_w && a.a_planes <= 1 && a.zero_words == 0 && !a.ws_out &&
               a.nlayers <= 1 && a.w_fp4)) {
    *err = "conv_tc: the FP4 pipe takes 2-bit codes from a nibble image (cin % 256 == 0), one layer, no chained output";
    return 1;
  }
  if (tiles == 0) return 0;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (sms < 2) sms = 2;
  // Last-wave balancing: with `workers` persistent CTAs (or CTA pairs), the full tiles past
  // the last complete wave run as two half-width (N/2) tiles each, when those halves still
  // fit in one wave; half as long per tile, they end the kernel sooner.
  const int nlayers = a.nlayers > 1 ? a.nlayers : 1;
  if (nlayers > 1 && !(flat && pair && prm.n_tiles == 1 && !a.split_w && a.a_planes <= 1 && a.ws2 && a.dep &&
                       nlayers <= kMaxLayers)) {
    *err = "conv_tc: chained layers in one launch need the workspace path on CTA pairs with one N tile";
    return 1;
  }
  // (a launch of several layers has no half-width tiles: every layer keeps the same tiles)
  prm.dp_tiles = nlayers > 1 ? tiles : split_start(tiles, pair ? sms / 2 : sms, BN, a.split_w != 0);
  prm.total_tiles = nlayers * (prm.dp_tiles + 2 * (tiles - prm.dp_tiles));
  // contiguous tile ranges for single-CTA launches of one layer on the workspace path with no
  // half tiles (the FP4 output conv): neighbouring tiles share a level's tables and halo rows
  prm.contig = (!pair && flat && nlayers <= 1 && prm.dp_tiles == tiles) ? 1 : 0;
  prm.nlayers = nlayers;
  prm.layer_tiles = prm.total_tiles / nlayers;
  prm.div_layer = div_magic(prm.layer_tiles);
  prm.div_nt = div_magic(prm.n_tiles);
  prm.num_kchunks = flat ? (fp4 ? a.k_total / 2 : (f16 ? 2 * a.k_total : a.k_total)) / bk : a.k_pad / BK;
  // (64 K elements per chunk; acc_bound / k_total bounds one product)
  prm.seg_chunks = f16 ? (int)(((1LL << 24) - 1) / (a.acc_bound / a.k_total) / 64) : 0;
  prm.cin = a.cin; prm.cout = a.cout; prm.kh = a.kh; prm.kw = a.kw;
  prm.stride = a.stride; prm.pad = a.pad; prm.k_total = a.k_total;
  prm.out_bits = a.out_bits; prm.skip_bits = a.skip_bits;
  prm.x_row_bytes = a.x_row_bytes; prm.y_row_bytes = a.y_row_bytes; prm.skip_row_bytes = a.skip_row_bytes;
  if (nlayers > 1) {
    for (int l = 0; l < nlayers; ++l) {
      LayerDev& ly = prm.layers[l];
      ly.m0 = a.layer[l].m0; ly.shift = a.layer[l].shift; ly.bias = a.layer[l].bias;
      for (int j = 0; j < a.njobs; ++j) ly.y[j] = a.layer[l].y[j];
      ly.ws_out = a.layer[l].ws_out;
      ly.ws_nib = a.layer[l].ws_nib;
    }
  } else {
    LayerDev& ly = prm.layers[0];
    ly.m0 = a.m0; ly.shift = a.shift; ly.bias = a.bias;
    for (int j = 0; j < a.njobs; ++j) ly.y[j] = a.jobs[j].y;
    ly.ws_out = a.ws_out;
    ly.ws_nib = a.ws_out_nib;
  }
  prm.skip_c = a.skip_c; prm.skip_d = a.skip_d;
  prm.upsample = a.upsample; prm.scale_main = a.scale_main; prm.has_skip = a.has_skip;
  prm.bn = BN;
  prm.acc_small = a.acc_bound < (1LL << 22) ? 1 : 0;
  prm.cin_chunks = img_row / bk;
  prm.out_pad = a.out_pad;
  prm.a_planes = flat ? (a.a_planes > 1 ? a.a_planes : 1) : 1;
  prm.plane_rows = (int32_t)rows;
  prm.split_w = a.split_w;
  bool chained = a.ws_out != nullptr;
  for (int l = 0; l < nlayers && nlayers > 1; ++l) chained |= a.layer[l].ws_out != nullptr;
  if (chained) {
    int64_t orows = 0;
    for (int j = 0; j < a.njobs; ++j) {
      ConvJobDev& jb = prm.jobs[j];
      jb.ohp = jb.ho + 2 * a.out_pad;
      jb.owp = jb.wo + 2 * a.out_pad;
      jb.orow_off = (int32_t)orows;
      orows += (int64_t)jb.n * jb.ohp * jb.owp;
    }
  }
  prm.status = a.status;
  prm.dep = nlayers > 1 ? a.dep : nullptr;
  // 32-column groups of a full tile over the epilogue warps of a lane quarter
  const int warp_groups = epi_warps(flat) / 4;
  const int col_groups = ((a.split_w ? BN / 2 : BN) + 31) / 32;
  prm.epi_groups = col_groups < warp_groups ? col_groups : warp_groups;
  prm.epi_sets = warp_groups / prm.epi_groups;  // 1, 2 or 4: tiles are dealt by their low bits
  prm.dep_target = (uint32_t)(8 * prm.epi_groups);  // a tile's epilogue warps, both CTAs of a pair
  // shared memory plan. Flat path: a ring of activation slabs and one of weight tiles (this CTA's B
  // rows x bk bytes), or all weight tiles resident. Otherwise stages of both operands.
  const int b_rows = pair ? BN / 2 : BN;
  const size_t b_tile = (size_t)b_rows * bk;
  prm.taps = a.kw <= 16 ? a.kw : 1;
  const size_t slab = flat ? ((size_t)(BM + prm.taps - 1) * bk + 1023) / 1024 * 1024 : (size_t)BM * bk;
  const size_t epi_bytes = EpiTab::kBytes;
  const size_t bar_bytes = 8 * (4 * kMaxStages + 2 * kMaxBufs + 1) + 16;
  const size_t sk_bytes = !a.has_skip ? 0 : (a.skip_bits == 32 ? (size_t)epi_warps(flat) * 2 * kSkipStage : skip_tab_bytes(a.skip_bits));
  const size_t budget = 232448 - 1024;  // max dynamic smem per block minus alignment slack
  const size_t fixed = epi_bytes + bar_bytes + sk_bytes + 32;
  // int32 outputs with cout % 4 == 0: per-warp staging blocks when at least two slabs and their weight
  // tiles remain (a 1x1 stride-2 64 -> 128 conv to 134,400 pixels 30 -> 27 us in the in-kernel variant)
  const size_t ostage_bytes = (size_t)epi_warps(flat) * 32 * kStageRow * sizeof(uint32_t);
  const bool ostage = bk == BK && a.out_bits == 32 && a.cout % 4 == 0 && !a.has_skip && !a.split_w && !f16 &&
                      budget >= fixed + ostage_bytes + 2 * (slab + (size_t)(flat ? prm.taps : 1) * b_tile);
  const size_t avail = budget - fixed - (ostage ? ostage_bytes : 0);
  int stages = 0, stages_b = 0;
  if (flat) {
    // Resident weights: every N tile's, where they leave at least 3 slabs and a third of the room. (A
    // half-width tile takes other rows per CTA of a pair: a launch with such tiles streams.) Resident / streamed
    // in us, 4 bits, expansion included: 3x3 on eight 100 x 168 maps 64 -> 96 22.3 / 24.4, 256 -> 32 30.7 / 36.1, 512 -> 32
    // 53 / 63; on one 25 x 42 map, where a CTA has a tile or none, 256 -> 96 9.2 / 8.8. With less room than a third
    // for slabs, 3x3 64 -> 512 on two 50 x 84 maps, resident took 11.5 against 10.2 streamed.
    const size_t all_w = (size_t)prm.n_tiles * prm.num_kchunks * b_tile;
    prm.resident = nlayers <= 1 && prm.dp_tiles == tiles && all_w * 3 <= avail * 2 && all_w + 3 * slab <= avail;
    if (prm.resident) {
      stages = (int)((avail - all_w) / slab);
      stages_b = 1;
    } else {
      stages = (int)(avail / (slab + (size_t)prm.taps * b_tile));
      if (stages < 2) stages = 2;
      if (stages > kMaxStages) stages = kMaxStages;
      if (avail < stages * slab + 2 * b_tile) { *err = "conv_tc: shared memory plan does not fit"; return 2; }
      stages_b = (int)((avail - stages * slab) / b_tile);
      if (stages_b > kMaxStages) stages_b = kMaxStages;
    }
    if (stages > kMaxStages) stages = kMaxStages;
  } else {
    stages = (int)(avail / (slab + b_tile));
    if (stages > kMaxStages) stages = kMaxStages;
    if (stages < 2) { *err = "conv_tc: shared memory plan does not fit"; return 2; }
  }
  // (The weight issuers take tiles round-robin and wait on their stage's "empty" barrier by phase
  // parity, which is unambiguous while there are at least as many stages as issuers: two.)
  prm.stages = stages;
  prm.stages_b = stages_b;
  prm.slab_bytes = (uint32_t)slab;
  prm.off_b = (uint32_t)(stages * slab);
  const size_t b_all = flat ? (prm.resident ? (size_t)prm.n_tiles * prm.num_kchunks : (size_t)stages_b) * b_tile : stages * b_tile;
  prm.off_epi = (uint32_t)((prm.off_b + b_all + 15) / 16 * 16);
  prm.off_bar = prm.off_epi + (uint32_t)epi_bytes;
  // (a launch has a skip table or staging blocks, not both: staged outputs have no skip)
  const uint32_t off_end = (uint32_t)((prm.off_bar + bar_bytes + 15) / 16 * 16);
  prm.off_ostage = prm.off_sktab = off_end;
  const size_t smem = 1024 + off_end + (ostage ? ostage_bytes : sk_bytes);
  // two accumulators of BN fp32 columns, or four where they fit beside the 32 columns of scales
  // of the FP4 pipe
  const int sf_cols = fp4 ? 32 : 0;
  prm.nbuf_log2 = 4 * BN + sf_cols <= 512 ? 2 : 1;
  // A set that takes every epi_sets-th tile waits for an accumulator by phase parity, having last seen
  // the end of its previous tile complete: the use that its wait could mistake for its own, one ring
  // of accumulators earlier, must be among those. A tile uses nseg accumulators in turn, so that is
  // (epi_sets - 1) nseg < accumulators; it bounds the sets only on the F16 pipe (elsewhere nseg is 1 and
  // more than one set means four accumulators).
  const int nseg = f16 ? (prm.num_kchunks + prm.seg_chunks - 1) / prm.seg_chunks : 1;
  while ((prm.epi_sets - 1) * nseg >= 1 << prm.nbuf_log2) prm.epi_sets /= 2;
  const int acc_cols = BN << prm.nbuf_log2;
  if (acc_cols + sf_cols > 512) { *err = "conv_tc: FP4 tiles wider than 240 channels do not fit in TMEM"; return 2; }
  int cols = 32;
  while (cols < acc_cols + sf_cols) cols *= 2;
  prm.tmem_cols = cols;
  prm.sf_col = acc_cols;

  EncodeTiledFn enc = get_encode_fn(err);
  if (!enc) return 3;
  Maps maps{};
  // weight rows: k_pad E4M3 bytes, or k_pad / 2 bytes of E2M1 nibbles on the FP4 pipe
  // (F16: k_total values of 2 bytes, cout rows; a tile's rows past them read as zeros)
  const int w_row = fp4 ? a.k_pad / 2 : (f16 ? 2 * a.k_total : a.k_pad);
  cuuint64_t gdim[2] = {(cuuint64_t)w_row, (cuuint64_t)(f16 ? a.cout : w_rows)};
  cuuint64_t gstride[1] = {(cuuint64_t)w_row};
  cuuint32_t box[2] = {(cuuint32_t)bk, (cuuint32_t)b_rows};
  cuuint32_t estr[2] = {1, 1};
  const CUtensorMapSwizzle swz = bk == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B;
  const uint8_t* w_src = fp4 ? a.w_fp4 : (f16 ? reinterpret_cast<const uint8_t*>(a.w_f16) : a.w_e4m3);
  for (int l = 0; l < nlayers; ++l) {
    const uint8_t* wl = nlayers > 1 ? a.layer[l].w_e4m3 : w_src;
    const CUresult r = enc(&maps.w[l], CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, (void*)wl, gdim, gstride, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) { *err = "cuTensorMapEncodeTiled failed: " + std::to_string((int)r); return 3; }
  }
  // the same weights with boxes of half the rows, for the half-width tiles
  maps.wh = maps.w[0];
  if (prm.dp_tiles < prm.layer_tiles) {
    cuuint32_t box_h[2] = {(cuuint32_t)bk, (cuuint32_t)(b_rows / 2)};
    const CUresult r = enc(&maps.wh, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, (void*)w_src, gdim,
                           gstride, box_h, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) { *err = "cuTensorMapEncodeTiled (half) failed: " + std::to_string((int)r); return 3; }
  }

  const int units = prm.total_tiles;
  int grid = units < sms ? units : sms;
  if (pair) grid = 2 * (units < sms / 2 ? units : sms / 2);
  prm.share = prm.total_tiles / grid;
  prm.extra = prm.total_tiles % grid;
  prm.tile_stride = pair ? grid / 2 : (prm.contig ? 1 : grid);
  const bool in_tap = (a.cin % BK) == 0;
  if (flat) {
    // 1) expand the packed codes of every job into the zero-padded byte workspace (unless
    //    the caller expanded them already)
    if (!a.skip_expand || a.zero_words > 0) {
      // (with skip_expand, only the counters are cleared: an expansion of no rows)
      ExpandArgs ea{};
      for (int j = 0; j < a.njobs; ++j) ea.jobs[j] = prm.jobs[j];
      ea.njobs = a.njobs; ea.cin = a.cin; ea.pad = a.pad; ea.x_row_bytes = a.x_row_bytes;
      ea.total_rows = a.skip_expand ? 0 : rows; ea.ws = a.ws;
      ea.zero = a.zero_words > 0 ? a.zero : nullptr;
      ea.zero_words = a.zero_words;
      // one warp per run of 32 * 4 (row, 16-byte chunk) pairs, 8 warps per block
      const int64_t pairs = ea.total_rows * (a.cin / (f16 ? 8 : 16));
      const unsigned blocks = pairs > 0 ? (unsigned)((pairs + 1023) / 1024) : 1u;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(blocks);
      cfg.blockDim = dim3(256);
      cfg.stream = stream;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[0].val.programmaticStreamSerializationAllowed = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      cudaError_t e;
      if (fp4) {
        // nibble image: one thread per 16 output bytes, grid-strided
        const int64_t chunks = ea.total_rows * (a.cin / 32);
        const int64_t want = (chunks + 255) / 256;
        cfg.gridDim = dim3((unsigned)(want < 4096 ? (want > 0 ? want : 1) : 4096));
        e = cudaLaunchKernelEx(&cfg, expand_nib_kernel, ea);
      } else switch (a.x_bits) {
        case 2: e = cudaLaunchKernelEx(&cfg, expand_kernel<2>, ea); break;
        case 3: e = cudaLaunchKernelEx(&cfg, expand_kernel<3>, ea); break;
        case 4: e = cudaLaunchKernelEx(&cfg, expand_kernel<4>, ea); break;
        case 8: e = f16 ? cudaLaunchKernelEx(&cfg, expand_kernel<16>, ea) : cudaLaunchKernelEx(&cfg, expand_kernel<8>, ea); break;
        default: *err = "conv_tc: activation bits must be 2, 3 or 4"; return 2;
      }
      if (e == cudaSuccess) e = cudaGetLastError();
      if (e != cudaSuccess) { *err = std::string("expand launch: ") + cudaGetErrorString(e); return 3; }
    }
    if (a.expand_only) return 0;
    // 2) tensor maps over the workspace (and, for chained layers in one launch, the second
    //    image) as [rows][cin] byte matrices with boxes of a slab
    // (a nibble image keeps the byte image's row stride: cin bytes, the first cin / 2 used)
    cuuint64_t gd[2] = {(cuuint64_t)img_row, (cuuint64_t)rows * (cuuint64_t)prm.a_planes};
    cuuint64_t gs[1] = {(cuuint64_t)(f16 ? 2 * a.cin : a.cin)};
    cuuint32_t bx[2] = {(cuuint32_t)bk, (cuuint32_t)(BM + prm.taps - 1)};
    for (int i = 0; i < (nlayers > 1 ? 2 : 1); ++i) {
      // (a nibble image row uses 128 of every 256 bytes: fetch 128-byte lines from DRAM)
      const CUresult r2 = enc(&maps.a[i], CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, (void*)(i == 0 ? a.ws : a.ws2), gd, gs, bx,
                              estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
                              fp4 ? CU_TENSOR_MAP_L2_PROMOTION_L2_128B : CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
      if (r2 != CUDA_SUCCESS) {
        *err = "cuTensorMapEncodeTiled (activations) failed: " + std::to_string((int)r2);
        return 3;
      }
    }
    if (ostage) {  // int32 outputs, no skip, 128-byte chunks (see the smem plan)
      if (fp4)
        return pair ? launch_bits<2, true, true, true, false, false, 128, true, true>(prm, maps, grid, smem, stream, err)
                    : launch_bits<2, true, true, false, false, false, 128, true, true>(prm, maps, grid, smem, stream, err);
      return pair ? launch_bits<2, true, true, true, false, false, 128, false, true>(prm, maps, grid, smem, stream, err)
                  : launch_bits<2, true, true, false, false, false, 128, false, true>(prm, maps, grid, smem, stream, err);
    }
    if (fp4) {
      if (pair)
        return a.has_skip ? launch_bits<2, true, true, true, true, false, 128, true>(prm, maps, grid, smem, stream, err)
                          : launch_bits<2, true, true, true, false, false, 128, true>(prm, maps, grid, smem, stream, err);
      return a.has_skip ? launch_bits<2, true, true, false, true, false, 128, true>(prm, maps, grid, smem, stream, err)
                        : launch_bits<2, true, true, false, false, false, 128, true>(prm, maps, grid, smem, stream, err);
    }
    if (f16) {  // (no skip: the API keeps skips off the 8-bit forms)
      if (a.out_bits == 32)
        return pair ? launch_bits<8, true, true, true, false, false, 128, false, true>(prm, maps, grid, smem, stream, err)
                    : launch_bits<8, true, true, false, false, false, 128, false, true>(prm, maps, grid, smem, stream, err);
      return pair ? launch_bits<8, true, true, true, false>(prm, maps, grid, smem, stream, err)
                  : launch_bits<8, true, true, false, false>(prm, maps, grid, smem, stream, err);
    }
    if (a.split_w) {  // (no skip: the API keeps skips off the split form)
      if (pair) return launch_bits<2, true, true, true, false, true>(prm, maps, grid, smem, stream, err);
      return launch_bits<2, true, true, false, false, true>(prm, maps, grid, smem, stream, err);
    }
    if (bk == 64) {
      if (pair)
        return a.has_skip ? launch_bits<2, true, true, true, true, false, 64>(prm, maps, grid, smem, stream, err)
                          : launch_bits<2, true, true, true, false, false, 64>(prm, maps, grid, smem, stream, err);
      return a.has_skip ? launch_bits<2, true, true, false, true, false, 64>(prm, maps, grid, smem, stream, err)
                        : launch_bits<2, true, true, false, false, false, 64>(prm, maps, grid, smem, stream, err);
    }
    if (pair)
      return a.has_skip ? launch_bits<2, true, true, true, true>(prm, maps, grid, smem, stream, err)
                        : launch_bits<2, true, true, true, false>(prm, maps, grid, smem, stream, err);
    return a.has_skip ? launch_bits<2, true, true, false, true>(prm, maps, grid, smem, stream, err)
                      : launch_bits<2, true, true, false, false>(prm, maps, grid, smem, stream, err);
  }
  // in-kernel unpacking; the instantiation without skip code keeps its registers for the
  // common case
#define AQD_INKERNEL(B)                                                                                  \
  if (a.has_skip)                                                                                          \
    return in_tap ? launch_bits<B, true, false, false, true>(prm, maps, grid, smem, stream, err) \
                  : launch_bits<B, false, false, false, true>(prm, maps, grid, smem, stream, err); \
  if (ostage)                                                                                            \
    return in_tap ? launch_bits<B, true, false, false, false, false, BK, false, true>(prm, maps, grid, smem, stream, err) \
                  : launch_bits<B, false, false, false, false, false, BK, false, true>(prm, maps, grid, smem, stream, err); \
  return in_tap ? launch_bits<B, true, false, false, false>(prm, maps, grid, smem, stream, err)   \
                : launch_bits<B, false, false, false, false>(prm, maps, grid, smem, stream, err);
  switch (a.x_bits) {
    case 2: { AQD_INKERNEL(2) }
    case 3: { AQD_INKERNEL(3) }
    case 4: { AQD_INKERNEL(4) }
    default: *err = "conv_tc: activation bits must be 2, 3 or 4"; return 2;
  }
#undef AQD_INKERNEL
}

}  // namespace aqd
