// NVFP4 quantizer for sm_100a: tensor-amax reduction (pass 1) and the fused
// transform + scale + round + pack kernel producing the row-wise and/or the transposed copy (pass 2).
//
// Paper: Appendix B (Eq. 1-4), Appendix C (16x16 random Hadamard transform), Section 4.3 (16x16
// weight blocks, two copies for the two passes), Section 4.4 (stochastic rounding).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>
#include <utility>

#include "async_ptx.cuh"
#include "common.cuh"
#include "quantize.h"
#include "quantize_common.cuh"

namespace nvfp4 {

// Pass 1 without words to clear: the {plain, transformed} maximum of a tile goes to a place of its own and pass 2 takes the
// maximum over the places.  For small tensors, see pass1_in_parts().
__device__ __forceinline__ void store_part(float2* part, const float (&plain)[8], const float (&rot)[8]) {
  if (threadIdx.x != 0) return;
  float2 m = make_float2(plain[0], rot[0]);
#pragma unroll
  for (int w = 1; w < 8; ++w) m = make_float2(fmaxf(m.x, plain[w]), fmaxf(m.y, rot[w]));
  *part = m;
}

// ---------------------------------------------------------------------------------------------
// Pass 1: tensor amax (Appendix B.1), plain and / or in the rotated space of a transformed copy.
// CTA tile 128 rows x 256 columns; a warp owns 16 rows, a lane 8 columns of each of them.
// ---------------------------------------------------------------------------------------------
template <bool PLAIN, bool ROT_ROW, bool ROT_COL, bool PARTS>
__device__ __forceinline__ void amax_tile(const uint16_t* __restrict__ x, int64_t rows, int64_t cols, int64_t ld,
                                          uint32_t sign_mask, int tile, int tiles_c, float* __restrict__ out_plain0,
                                          float* __restrict__ out_plain1, float* __restrict__ out_rot_row,
                                          float* __restrict__ out_rot_col, float2* __restrict__ parts) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t tr = tile / tiles_c, tc = tile % tiles_c;
  const int64_t r0 = tr * 128 + warp * 16;
  const int64_t c0 = tc * 256 + lane * 8;
  const bool in_range = (r0 < rows) && (c0 < cols);  // rows % 16 == 0, cols % 8 == 0
  if (PARTS) griddep_wait();    // the first kernel of its call; otherwise zero_words_kernel has waited for the source
  griddep_launch_dependents();  // pass 2 may set itself up while the last CTAs of this pass run

  uint4 raw[16];
  if (in_range) {
    const uint16_t* p = x + r0 * ld + c0;
#pragma unroll
    for (int j = 0; j < 16; ++j) raw[j] = ldg128_stream(p + j * ld);
  } else {
#pragma unroll
    for (int j = 0; j < 16; ++j) raw[j] = make_uint4(0, 0, 0, 0);
  }

  float m_plain = 0.f, m_row = 0.f, m_col = 0.f;
  if (PLAIN) {
    uint32_t acc = 0;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      acc = absmax_bf16x2(acc, raw[j].x);
      acc = absmax_bf16x2(acc, raw[j].y);
      acc = absmax_bf16x2(acc, raw[j].z);
      acc = absmax_bf16x2(acc, raw[j].w);
    }
    m_plain = amax_of_pair(acc);
  }
  if (ROT_COL) {
    // chunks run down the 16 rows of the warp's slab: one transform per column
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      float a[16], b[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        uint32_t word = (w == 0) ? raw[j].x : (w == 1) ? raw[j].y : (w == 2) ? raw[j].z : raw[j].w;
        word ^= sign_pair(sign_mask, j, j);
        a[j] = bf16_lo(word);
        b[j] = bf16_hi(word);
      }
      fwht16(a);
      fwht16(b);
#pragma unroll
      for (int j = 0; j < 16; ++j) m_col = fmaxf(m_col, fmaxf(fabsf(a[j]), fabsf(b[j])));
    }
    m_col *= 0.25f;
  }
  if (ROT_ROW) {
    // a chunk is 16 consecutive columns = the 8 columns of an even lane and of the next odd lane
    const int half = lane & 1;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      float v[8];
      const uint32_t w4[4] = {raw[j].x, raw[j].y, raw[j].z, raw[j].w};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        uint32_t word = w4[k] ^ sign_pair(sign_mask, half * 8 + 2 * k, half * 8 + 2 * k + 1);
        v[2 * k] = bf16_lo(word);
        v[2 * k + 1] = bf16_hi(word);
      }
#pragma unroll
      for (int h = 1; h < 8; h <<= 1)
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if ((i & h) == 0) {
            float a = v[i], b = v[i | h];
            v[i] = a + b;
            v[i | h] = a - b;
          }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        float other = __shfl_xor_sync(0xffffffffu, v[i], 1);
        float y = half ? (other - v[i]) : (v[i] + other);
        m_row = fmaxf(m_row, fabsf(y));
      }
    }
    m_row *= 0.25f;
  }

  __shared__ float red[3][8];
  m_plain = warp_max(m_plain);
  m_row = warp_max(m_row);
  m_col = warp_max(m_col);
  if (lane == 0) {
    red[0][warp] = m_plain;
    red[1][warp] = m_row;
    red[2][warp] = m_col;
  }
  __syncthreads();
  if (PARTS) {
    store_part(parts + tile, red[0], red[2]);
  } else if (threadIdx.x < 3) {
    griddep_wait();  // the words are zero
    float m = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) m = fmaxf(m, red[threadIdx.x][w]);
    // non-negative floats order like their bit patterns
    uint32_t bits = __float_as_uint(m);
    if (threadIdx.x == 0 && PLAIN) {
      if (out_plain0) atomicMax(reinterpret_cast<unsigned int*>(out_plain0), bits);
      if (out_plain1) atomicMax(reinterpret_cast<unsigned int*>(out_plain1), bits);
    }
    if (threadIdx.x == 1 && ROT_ROW) atomicMax(reinterpret_cast<unsigned int*>(out_rot_row), bits);
    if (threadIdx.x == 2 && ROT_COL) atomicMax(reinterpret_cast<unsigned int*>(out_rot_col), bits);
  }
}

template <bool PLAIN, bool ROT_ROW, bool ROT_COL, bool PARTS>
__global__ void __launch_bounds__(256) amax_kernel(const uint16_t* __restrict__ x, int64_t rows, int64_t cols, int64_t ld,
                                                   uint32_t sign_mask, int tiles_c, float* __restrict__ out_plain0,
                                                   float* __restrict__ out_plain1, float* __restrict__ out_rot_row,
                                                   float* __restrict__ out_rot_col, float2* __restrict__ parts) {
  amax_tile<PLAIN, ROT_ROW, ROT_COL, PARTS>(x, rows, cols, ld, sign_mask, (int)blockIdx.x, tiles_c, out_plain0, out_plain1,
                                            out_rot_row, out_rot_col, parts);
}

// ---------------------------------------------------------------------------------------------
// Pass 1 for a copy transformed down the rows (the transposed copy of a Wgrad operand, Appendix C): the
// 16-point transform of 8 columns at a time is one bf16 tensor-core product  Y(16x8) = A(16x16) * X(16x8)  with
// A[k][j] = s_j * h(k, j) (entries +-1, exact in bf16; FP32 accumulation) and the 1/4 applied to the maximum.
// A lane loads 16 columns of one row; its eight words are fragments of eight 8x8 matrices whose "columns" are an
// interleaved subset of the 64 columns a quad covers - columns are independent under this transform, so any
// assignment works - and movmatrix turns each into the k-pair layout the product wants.
// CTA tile 128 rows x 256 columns; a warp owns 16 rows.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t v) {
  uint32_t r;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(v));
  return r;
}

// d, norm: size of the transform (2, 4, 8 or 16: H_16 is replaced by the block-diagonal matrix of 16 / d copies of
// H_d) and its normalisation 1 / sqrt(d), applied to the maximum.
// FIRST: the source leaves L2 before anything else, see kEvictFirstBytes.
template <bool PLAIN, bool PARTS, bool FIRST>
__device__ __forceinline__ void amax_rot_col_tile(const uint16_t* __restrict__ x, int64_t rows, int64_t cols, int64_t ld,
                                                  uint32_t sign_mask, int tile, int tiles_c, float* __restrict__ out_plain0,
                                                  float* __restrict__ out_plain1, float* __restrict__ out_rot_col, int d,
                                                  float norm, float2* __restrict__ parts) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;
  const int64_t tr = tile / tiles_c, tc = tile % tiles_c;
  const int64_t r0 = tr * 128 + warp * 16;
  if (PARTS) griddep_wait();  // as in amax_tile
  griddep_launch_dependents();

  uint64_t policy = 0;
  if constexpr (FIRST) asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
  uint32_t lo[4][8], hi[4][8];  // rows g and g + 8 of the slab, 16 columns each, four 64-column steps
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int64_t c = tc * 256 + q * 64 + t * 16;
    if (r0 < rows && c < cols) {  // rows % 16 == 0, cols % 16 == 0
      if constexpr (FIRST) {
        ldg256_hint(x + (r0 + g) * ld + c, lo[q], policy);
        ldg256_hint(x + (r0 + 8 + g) * ld + c, hi[q], policy);
      } else {
        ldg256_stream(x + (r0 + g) * ld + c, lo[q]);
        ldg256_stream(x + (r0 + 8 + g) * ld + c, hi[q]);
      }
    } else {
#pragma unroll
      for (int w = 0; w < 8; ++w) lo[q][w] = hi[q][w] = 0u;
    }
  }

  // A fragments: entry (k, j) = +-1 as bf16 inside the d x d diagonal blocks (0 outside), negative iff
  // popc(k & j) is odd XOR sign bit j
  auto entry = [&](int k, int j) -> uint32_t {
    if ((k ^ j) >= d) return 0u;
    return ((__popc(k & j & (d - 1)) ^ (sign_mask >> j)) & 1u) ? 0xBF80u : 0x3F80u;
  };
  const uint32_t a0 = entry(g, 2 * t) | (entry(g, 2 * t + 1) << 16);
  const uint32_t a1 = entry(g + 8, 2 * t) | (entry(g + 8, 2 * t + 1) << 16);
  const uint32_t a2 = entry(g, 2 * t + 8) | (entry(g, 2 * t + 9) << 16);
  const uint32_t a3 = entry(g + 8, 2 * t + 8) | (entry(g + 8, 2 * t + 9) << 16);

  float m_col = 0.f;
  uint32_t acc = 0u;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
#pragma unroll
    for (int w = 0; w < 8; ++w) {
      if (PLAIN) {
        acc = absmax_bf16x2(acc, lo[q][w]);
        acc = absmax_bf16x2(acc, hi[q][w]);
      }
      const uint32_t b0 = movmatrix_trans(lo[q][w]);
      const uint32_t b1 = movmatrix_trans(hi[q][w]);
      float d0, d1, d2, d3;
      asm volatile(
          "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
          "{%10,%10,%10,%10};"
          : "=f"(d0), "=f"(d1), "=f"(d2), "=f"(d3)
          : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
      m_col = fmaxf(fmaxf(m_col, fmaxf(fabsf(d0), fabsf(d1))), fmaxf(fabsf(d2), fabsf(d3)));
    }
  }
  m_col *= norm;
  float m_plain = PLAIN ? amax_of_pair(acc) : 0.f;

  __shared__ float red[2][8];
  m_plain = warp_max(m_plain);
  m_col = warp_max(m_col);
  if (lane == 0) {
    red[0][warp] = m_plain;
    red[1][warp] = m_col;
  }
  __syncthreads();
  if (PARTS) {
    store_part(parts + tile, red[0], red[1]);
  } else if (threadIdx.x < 2) {
    griddep_wait();  // the words are zero
    float m = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) m = fmaxf(m, red[threadIdx.x][w]);
    const uint32_t bits = __float_as_uint(m);  // non-negative floats order like their bit patterns
    if (threadIdx.x == 0 && PLAIN) {
      if (out_plain0) atomicMax(reinterpret_cast<unsigned int*>(out_plain0), bits);
      if (out_plain1) atomicMax(reinterpret_cast<unsigned int*>(out_plain1), bits);
    }
    if (threadIdx.x == 1) atomicMax(reinterpret_cast<unsigned int*>(out_rot_col), bits);
  }
}

// A source of 64 MiB or more, read with the policy "evict first": calls on four tensors in turn, gradient of 8192 x 5120 60.1 -> 57.5
// us, of 8192 x 20480 217 -> 209, activation 45.3 -> 42.9 and 166 -> 158.  Smaller ones gain 1 to 4 % by themselves, but a backward
// call of 2816 x 3328 x 2304, which finds its gradient in L2 again, loses 2 %.  (Weights, whose pass 1 is amax_kernel, lose 1 to
// 3 %; the priority as a qualifier of the load, without a policy, gained nothing and cost 5 % between 27 and 52 MB; keeping the
// end of the source with "evict last" lost 2 to 5 % against this.)
// Nor an activation whose scale bytes leave one by one in both copies (sizes that are no multiples of 64, see store_linear_scales):
// with the policy / without 9360 x 7920 96.4 / 93.1 us, 8736 x 12720 146.7 / 139.4, 4880 x 11216 72.5 / 68.8; one side a multiple, 9344 x
// 7920 80.0 / 84.0, 9360 x 7936 80.1 / 83.8; gradients gain either way (9360 x 7920 107.8 / 112.0).
constexpr int64_t kEvictFirstBytes = 64ll << 20;
static bool evict_first(const QuantArgs& a, bool sr) {
  return 2 * a.rows * a.cols >= kEvictFirstBytes && (sr || a.rows % 64 == 0 || a.cols % 64 == 0);
}
template <bool PLAIN, bool PARTS, bool FIRST = false>
__global__ void __launch_bounds__(256) amax_rot_col_kernel(const uint16_t* __restrict__ x, int64_t rows, int64_t cols,
                                                           int64_t ld, uint32_t sign_mask, int tiles_c,
                                                           float* __restrict__ out_plain0, float* __restrict__ out_plain1,
                                                           float* __restrict__ out_rot_col, int d, float norm,
                                                           float2* __restrict__ parts) {
  amax_rot_col_tile<PLAIN, PARTS, FIRST>(x, rows, cols, ld, sign_mask, (int)blockIdx.x, tiles_c, out_plain0, out_plain1,
                                  out_rot_col, d, norm, parts);
}

// Pass 1 of two tensors in one launch (see quantize_x_and_w_kernel): the first n_x CTAs take tiles of an activation (row-wise
// copy plain, transposed copy rotated), the others of a weight (plain).
template <bool X_COL, bool W_COL, bool PARTS>
__global__ void __launch_bounds__(256) amax_x_and_w_kernel(const __grid_constant__ QuantArgs x, const __grid_constant__ QuantArgs w,
                                                           int n_x, int x_tiles_c, int w_tiles_c) {
  const int b = (int)blockIdx.x;
  if (b >= n_x)
    amax_tile<true, false, false, PARTS>(w.x, w.rows, w.cols, w.ld, 0u, b - n_x, w_tiles_c, w.r_global, W_COL ? w.c_global : nullptr,
                                  nullptr, nullptr, w.parts);
  else if (X_COL)
    amax_rot_col_tile<true, PARTS, false>(x.x, x.rows, x.cols, x.ld, x.sign_mask, b, x_tiles_c, x.r_global, nullptr, x.c_global, 16, 0.25f,
                                   x.parts);
  else
    amax_tile<true, false, false, PARTS>(x.x, x.rows, x.cols, x.ld, 0u, b, x_tiles_c, x.r_global, nullptr, nullptr, nullptr,
                                         x.parts);
}

// Pass 1 of a binary32 source: plain tensor amax.  CTA tile 128 rows x 128 columns; a warp owns 16 rows, a lane 4 columns of each.
__global__ void __launch_bounds__(256) amax_f32_kernel(const float* __restrict__ x, int64_t rows, int64_t cols,
                                                       int64_t ld, int tiles_c, float* __restrict__ out0,
                                                       float* __restrict__ out1) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t tr = blockIdx.x / tiles_c, tc = blockIdx.x % tiles_c;
  const int64_t r0 = tr * 128 + warp * 16, c0 = tc * 128 + lane * 4;
  griddep_launch_dependents();  // pass 2 may load its tiles while the last CTAs of this pass run
  float m = 0.f;  // (the source is complete: zero_words_kernel has waited for it)
  if (r0 < rows && c0 < cols) {  // rows % 16 == 0, cols % 16 == 0
    uint4 v[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = ldg128_stream(x + (r0 + j) * ld + c0);
#pragma unroll
    for (int j = 0; j < 16; ++j)
      m = fmaxf(fmaxf(m, fmaxf(fabsf(__uint_as_float(v[j].x)), fabsf(__uint_as_float(v[j].y)))),
                fmaxf(fabsf(__uint_as_float(v[j].z)), fabsf(__uint_as_float(v[j].w))));
  }
  __shared__ float red[8];
  m = warp_max(m);
  if (lane == 0) red[warp] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    griddep_wait();  // the words are zero
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) t = fmaxf(t, red[w]);
    const uint32_t bits = __float_as_uint(t);  // non-negative floats order like their bit patterns
    if (out0) atomicMax(reinterpret_cast<unsigned int*>(out0), bits);
    if (out1) atomicMax(reinterpret_cast<unsigned int*>(out1), bits);
  }
}

// ---------------------------------------------------------------------------------------------
// Pass 2: persistent CTAs (two per SM), each working through tiles of 128 rows x 128 (few tiles: 64) columns of the source.
// The tiles arrive by TMA (cp.async.bulk.tensor, this GPU's memory, no multicast) in a ring of two buffers: the load of tile
// k + 2 is issued as soon as tile k has been consumed, so a tile is in flight during the whole of the previous one;
// out-of-range parts of a ragged tile are zero-filled by the copy.
//   set-up   once per CTA: Eq. 1, and the table  E4M3 byte -> encode scale  of each copy (the text after Eq. 3:
//            s_enc,b = 1 / (fp32(S_b) * s_dec) has only 127 possible values per tensor), so a block costs one
//            conversion and one shared-memory read instead of an IEEE reciprocal;
//   phase 1  each thread owns four 1x16 chunks of the tile and produces the row-wise copy (and, for stochastic
//            rounding, stages the random bytes of its chunks in shared memory);
//   phase 2  each thread owns 16 rows x 2 columns of the tile and produces the transposed copy into a swizzled
//            staging buffer;
//   phase 3  staged codes and scale bytes leave with 16-byte stores.
// A warp's phase 2 reads only what the same warp staged in phase 1, and the buffers phase 3 reads are double
// buffered, so a tile needs one CTA barrier.  Tiles are visited in reverse order so that the end of the tensor,
// which pass 1 touched last, is read first while it may still sit in L2.
// ---------------------------------------------------------------------------------------------
// TC: columns of a tile; F32: the source is binary32 (tiles of 64 columns).
template <int TC, bool F32 = false>
struct QuantSmem {
  static constexpr int kChunks = TC / 16;                // 1x16 chunks per tile row
  static constexpr int kRow = (F32 ? 4 : 2) * TC;        // bytes per tile row
  static constexpr int kTileBytes = 128 * kRow;
  static constexpr int kTile = 0;                        // 2 tiles, filled by TMA
  static constexpr int kColBytes = TC * 64;
  static constexpr int kColCodes = 2 * kTileBytes;       // 2 x (TC columns x 64 B)
  static constexpr int kSfBytes = 8 * TC;                // 128 rows x kChunks bytes, or TC columns x 8
  static constexpr int kSfRow = kColCodes + 2 * kColBytes;
  static constexpr int kSfCol = kSfRow + 2 * kSfBytes;
  static constexpr int kBlkEnc = kSfCol + 2 * kSfBytes;  // 64 floats (16x16 mode)
  static constexpr int kBlkByte = kBlkEnc + 256;         // 64 bytes
  static constexpr int kGlobalScales = kBlkByte + 64;    // s_enc, s_dec of the row-wise and the column-wise copy
  static constexpr int kEncRow = kGlobalScales + 64;     // 128 floats: encode scale by E4M3 byte, row-wise copy
  static constexpr int kEncCol = kEncRow + 512;          // the same for the transposed copy
  static constexpr int kBars = kEncCol + 512;            // two "tile landed" barriers, then the abort word
  static constexpr int kRand = kBars + 32;               // 128 rows x TC B of complemented draws (stochastic rounding),
                                                         // or 128 rows x TC / 2 B of row-wise codes (16x16, both copies)
  static constexpr int bytes(bool rand, bool row_codes) { return kRand + (rand ? 128 * TC : row_codes ? 64 * TC : 0); }
};

// OWN_DRAWS: 16x16 blocks whose transposed copy is rounded with draws of its own.
// WHOLE: no tile is cut off (rows a multiple of 128, columns of TC).
template <bool HAS_ROW, bool HAS_COL, bool BLOCK2D, bool RHT_ROW, bool RHT_COL, bool SR, int TC, bool F32 = false,
          bool PARTS = false, bool OWN_DRAWS = false, bool WHOLE = false>
__device__ __forceinline__ void quantize_tiles(const CUtensorMap* src_map, const QuantArgs& a, const int block,
                                               const int blocks) {  // this CTA among those of the tensor
  using S = QuantSmem<TC, F32>;
  constexpr int CH = S::kChunks;          // chunks per tile row
  constexpr int RPP = 32 / CH;            // rows a warp covers with one chunk per lane; chunk i of a lane: RPP * i rows down
  constexpr int NP = 16 / RPP;            // chunks per lane
  constexpr int NIT = TC / 64;            // column pairs per lane in phase 2
  extern __shared__ __align__(128) uint8_t smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_cb = (int)(a.cols >> 4);  // 16-blocks per source row
  const int n_rb = (int)(a.rows >> 4);  // 16-blocks per source column
  // 16x16 blocks with both copies requested: the transposed copy holds the very codes of the row-wise one
  // (Section 4.3), so it is made by transposing nibbles; the raw tile is not needed a second time
  constexpr bool kNibbleTranspose = BLOCK2D && HAS_ROW && HAS_COL && !OWN_DRAWS;
  volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem + S::kBars + 16);
  const uint32_t bar0 = smem_u32(smem + S::kBars), tile0 = smem_u32(smem + S::kTile);

  const int total = a.tiles_r * a.tiles_c, stride = blocks;
  const int first = total - 1 - block;  // this CTA's tiles: first, first - stride, ...
  const int n_mine = first >= 0 ? first / stride + 1 : 0;
  auto issue = [&](int j) {  // the CTA's tile j into buffer j & 1 (one thread)
    const int t = first - j * stride, tr = t / a.tiles_c, tc = t - tr * a.tiles_c;
    mbar_expect_tx(bar0 + 8 * (j & 1), S::kTileBytes);
    tma_load_2d(tile0 + (j & 1) * S::kTileBytes, src_map, tc * TC, tr * 128, bar0 + 8 * (j & 1));
  };

  // ------------------------------------------------------------------ set-up ----
  float* g_sc = reinterpret_cast<float*>(smem + S::kGlobalScales);
  if (threadIdx.x == 0) {
    mbar_init(bar0, 1);
    mbar_init(bar0 + 8, 1);
    *abort_flag = 0u;
    fence_mbarrier_init();
    fence_proxy_async_smem();
    if (!a.chained) griddep_wait();  // the source may be the previous kernel's output
    if (n_mine > 0) issue(0);
    if (n_mine > 1) issue(1);
    // the source tiles above are nobody's output in this call; the tensor amax below is the previous kernel's.
    // Every other thread passes the barrier below only after this wait, so no output is written before it either.
    if (!PARTS) griddep_wait();
  }
  float2 m = make_float2(0.f, 0.f);
  if (PARTS) {
    griddep_wait();
    for (int i = threadIdx.x; i < a.n_parts; i += 256) {
      const float2 p = __ldcg(a.parts + i);
      m = make_float2(fmaxf(m.x, p.x), fmaxf(m.y, RHT_COL ? p.y : p.x));
    }
    m = make_float2(warp_max(m.x), warp_max(m.y));
    float2* const red = reinterpret_cast<float2*>(smem + S::kEncRow);  // the table is made behind the next barriers
    if (lane == 0) red[warp] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
      for (int w = 1; w < 8; ++w) m = make_float2(fmaxf(m.x, red[w].x), fmaxf(m.y, red[w].y));
      if (block == 0) {
        if (HAS_ROW) a.r_global[0] = m.x;
        if (HAS_COL) a.c_global[0] = m.y;
      }
    }
  }
  if (threadIdx.x == 0) {
    // Eq. 1 (two IEEE divisions per copy)
    float re = 1.f, rd = 1.f, ce = 1.f, cd = 1.f;
    if (!PARTS) {
      if (HAS_ROW) m.x = a.r_global[0];
      if (HAS_COL) m.y = a.c_global[0];
    }
    if (HAS_ROW || BLOCK2D) global_scales(HAS_ROW ? m.x : m.y, re, rd);
    if (HAS_COL) {
      if (BLOCK2D && HAS_ROW) {
        ce = re;
        cd = rd;
      } else {
        global_scales(m.y, ce, cd);
      }
    }
    g_sc[0] = re; g_sc[1] = rd; g_sc[2] = ce; g_sc[3] = cd;
    if (block == 0) {
      if (HAS_ROW) a.r_global[1] = rd;
      if (HAS_COL) a.c_global[1] = cd;
    }
  }
  __syncthreads();
  griddep_launch_dependents();
  const float r_senc = g_sc[0], r_sdec = g_sc[1], c_senc = g_sc[2], c_sdec = g_sc[3];
  const bool tiny = !BLOCK2D && fmaxf(HAS_ROW ? r_senc : 0.f, HAS_COL ? c_senc : 0.f) > kPlainDivisionLimit;
  const float* enc_row = reinterpret_cast<const float*>(smem + S::kEncRow);
  const float* enc_col = reinterpret_cast<const float*>(smem + S::kEncCol);
  if (!BLOCK2D) {
    // with the transform the kernel works on 4 * y: the 1/4 is folded into the block amax and the encode scale (exact)
    if (threadIdx.x < 128) {
      if (HAS_ROW)
        reinterpret_cast<float*>(smem + S::kEncRow)[threadIdx.x] =
            encode_scale_of_byte(threadIdx.x, r_sdec) * (RHT_ROW ? 0.25f : 1.0f);
    } else {
      if (HAS_COL)
        reinterpret_cast<float*>(smem + S::kEncCol)[threadIdx.x - 128] =
            encode_scale_of_byte(threadIdx.x - 128, c_sdec) * (RHT_COL ? 0.25f : 1.0f);
    }
    __syncthreads();
  }

  // per-thread constants of phase 1: chunk column cb, row rl + RPP * i for chunk i
  const int cb = lane % CH, rl = warp * 16 + lane / CH;
  const uint32_t tile_ld = rl * S::kRow + cb * (F32 ? 64 : 32);  // chunk i of the thread inside a tile buffer: + RPP * kRow * i
  const uint32_t rand_st = S::kRand + rl * TC + cb * 16;  // + RPP * TC * i
  const int sf_row_pos = a.r_swz ? ((cb >> 2) * 512 + (rl & 31) * 16 + (rl >> 5) * 4 + (cb & 3)) : (rl * CH + cb);
  const int sf_row_step = a.r_swz ? RPP * 16 : RPP * CH;
  const int64_t r_pitch = a.cols >> 1;  // bytes per row of the row-wise codes
  // bf16: lanes 4 .. 7 of every eight read the second half of their chunk first, so that a quarter warp covers all banks (32-byte
  // chunks: two lanes of the eight met in every bank), and the codes are swapped back: activation of 8192 x 20480 161.3 -> 158.3
  // us, 8192 x 5120 48.0 -> 47.1.  Not with stochastic rounding (the draws would have to follow: 4096 x 4096 30.1 -> 30.5) and
  // not for weights, which win 1 to 3 % up to 84 M elements and lose as much beyond (20480 x 5120 85.4 -> 89.3).
  constexpr bool kSwapHalves = !F32 && !RHT_ROW && !SR && !BLOCK2D;
  const int swap_halves = kSwapHalves ? (lane >> 2) & 1 : 0;
  // F32: a lane reads the four 16-byte quarters of a chunk beginning with its own rot-th, so that the eight lanes of a quarter
  // warp (chunks 64 bytes, rows 256 bytes apart) cover all banks; the codes are rotated back into place
  const int rot = ((cb >> 1) + 2 * (rl & 1)) & 3;

  // hoisted constants of phase 2: where a thread stages its two columns' codes and scale bytes (iteration it, column
  // parity odd); the 16-byte unit of column pair cp and 16-row group q sits at cp * 128 + ((q ^ spread(cp)) & 7) * 16: eight
  // consecutive column pairs, and every fourth of 32, fall into different units of a 128-byte line
  auto spread = [](int cp) { return cp ^ (cp >> 2); };
  const int col_codes_st = lane * 128 + (((warp ^ spread(lane)) & 7) << 4);  // + 4096 it
  // scale bytes of the transposed copy: two whole atoms (TC = 128) or half of the rows of two atoms (TC = 64: 8 bytes of
  // each 16)
  constexpr int kAtomRow = TC == 128 ? 16 : 8;
  const int sf_col_pos = a.c_swz ? ((warp >> 2) * (32 * kAtomRow) + (lane & 15) * (2 * kAtomRow) + (lane >> 4) * 4 + (warp & 3))
                                 : (lane * 16 + warp);
  const int sf_col_odd = a.c_swz ? kAtomRow : 8, sf_col_it = a.c_swz ? 8 : 512;

  const int step_r = stride / a.tiles_c, step_c = stride - step_r * a.tiles_c;  // tile coordinates move by these
  int tr = first >= 0 ? first / a.tiles_c : 0, tc = first >= 0 ? first - tr * a.tiles_c : 0;
  int j = 0;  // tiles done
  for (; j < n_mine; ++j) {
    const int buf = j & 1;
    const uint8_t* const tile_buf = smem + S::kTile + buf * S::kTileBytes;
    quant_wait(bar0 + 8 * buf, (uint32_t)(j >> 1) & 1u, abort_flag, a.status);  // the tile has landed
    const int64_t row0 = (int64_t)tr * 128, col0 = (int64_t)tc * TC;
    const bool full_tile = WHOLE || ((row0 + 128 <= a.rows) && (col0 + TC <= a.cols));
    uint8_t* const col_codes = smem + S::kColCodes + buf * S::kColBytes;
    uint8_t* const sf_row = smem + S::kSfRow + buf * S::kSfBytes;
    uint8_t* const sf_col = smem + S::kSfCol + buf * S::kSfBytes;

    auto phases_1_2 = [&](auto full_c, auto tiny_c) {
      constexpr bool FULL = decltype(full_c)::value, TINY = decltype(tiny_c)::value;
      // ---------------------------------------------------------------- phase 1 ----
      const int rows_left = FULL ? 128 : (int)(a.rows - row0) - rl;         // chunk i exists iff RPP * i < rows_left
      const bool col_ok = FULL || (col0 + cb * 16 < a.cols);
      uint32_t raw[NP][F32 ? 16 : 8];  // F32: quarter rot first
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        const uint8_t* const src = tile_buf + tile_ld + i * (RPP * S::kRow);
#pragma unroll
        for (int h = 0; h < (F32 ? 4 : 2); ++h) {
          const uint4 v = *reinterpret_cast<const uint4*>(src + (F32 ? ((h + rot) & 3) : h ^ swap_halves) * 16);
          raw[i][4 * h] = v.x; raw[i][4 * h + 1] = v.y; raw[i][4 * h + 2] = v.z; raw[i][4 * h + 3] = v.w;
        }
      }

      uint32_t blk_byte = 0;
      float blk_enc = 0.f;
      if (BLOCK2D) {  // amax of the lane's chunk column over the warp's 16 rows: one scale per 16 x 16 block
        float blk_amax = 0.f;
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          if constexpr (F32) {
#pragma unroll
            for (int k = 0; k < 16; k += 2)
              blk_amax = amax3(blk_amax, __uint_as_float(raw[i][k]), __uint_as_float(raw[i][k + 1]));
          } else {
            uint32_t acc = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) acc = absmax_bf16x2(acc, raw[i][k]);
            blk_amax = fmaxf(blk_amax, amax_of_pair(acc));
          }
        }
#pragma unroll
        for (int o = CH; o < 32; o <<= 1) blk_amax = fmaxf(blk_amax, __shfl_xor_sync(0xffffffffu, blk_amax, o));
        block_scales(blk_amax, r_senc, r_sdec, blk_byte, blk_enc);
        if (lane < CH) {
          reinterpret_cast<float*>(smem + S::kBlkEnc)[warp * CH + cb] = blk_enc;
          smem[S::kBlkByte + warp * CH + cb] = (uint8_t)blk_byte;
        }
      }

      uint64_t g = 0;  // Philox counter of chunk 0: the chunk's index in the source, 16-blocks numbered row by row
      if (SR) g = (uint64_t)(row0 + rl) * (uint64_t)n_cb + (uint64_t)((col0 >> 4) + cb);
      uint8_t* r_out = HAS_ROW ? a.r_codes + (row0 + rl) * r_pitch + ((col0 + cb * 16) >> 1) : nullptr;
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        uint32_t rnd[4] = {0u, 0u, 0u, 0u};
        if (SR) {
          const uint64_t gi = g + (uint64_t)(RPP * i) * (uint64_t)n_cb;
          const uint4 q = philox4x32_10((uint32_t)gi, (uint32_t)(gi >> 32), a.off_lo, HAS_ROW ? a.off_hi : a.off_hi_col, a.rk);
          rnd[0] = q.x; rnd[1] = q.y; rnd[2] = q.z; rnd[3] = q.w;
          if (HAS_COL && !kNibbleTranspose)  // staged complemented: the conversion wants 255 - draw
            *reinterpret_cast<uint4*>(smem + rand_st + i * (RPP * TC)) = make_uint4(~q.x, ~q.y, ~q.z, ~q.w);
        }
        if (HAS_ROW) {
          float f[16];
          if constexpr (F32) {
#pragma unroll
            for (int k = 0; k < 16; ++k) f[k] = __uint_as_float(raw[i][k]);
            if (SR) {  // the draws of the quarters in the order they were read
              const uint32_t a0 = (rot & 1) ? rnd[1] : rnd[0], a1 = (rot & 1) ? rnd[2] : rnd[1];
              const uint32_t a2 = (rot & 1) ? rnd[3] : rnd[2], a3 = (rot & 1) ? rnd[0] : rnd[3];
              rnd[0] = (rot & 2) ? a2 : a0; rnd[1] = (rot & 2) ? a3 : a1;
              rnd[2] = (rot & 2) ? a0 : a2; rnd[3] = (rot & 2) ? a1 : a3;
            }
          } else {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              uint32_t word = raw[i][k];
              if (RHT_ROW) word ^= sign_pair(a.sign_mask, 2 * k, 2 * k + 1);
              f[2 * k] = bf16_lo(word);
              f[2 * k + 1] = bf16_hi(word);
            }
            if (RHT_ROW) fwht16(f);  // values are 4 * y from here on
          }
          uint32_t byte;
          float enc;
          if (BLOCK2D) {
            byte = blk_byte;
            enc = blk_enc;
          } else {
            const float m = amax16_3(f);
            byte = block_scale_byte<TINY>(RHT_ROW ? 0.25f * m : m, r_senc);
            enc = enc_row[byte];
          }
          uint2 codes = convert16<SR>(f, enc, Nu14FromWords{rnd});
          if (kSwapHalves) codes = swap_halves ? make_uint2(codes.y, codes.x) : codes;
          if (F32) {  // 64-bit rotation to the left by rot quarters of 16 bits
            const uint32_t x = (rot & 2) ? codes.y : codes.x, y = (rot & 2) ? codes.x : codes.y;
            codes = make_uint2(__funnelshift_l(y, x, (rot & 1) * 16), __funnelshift_l(x, y, (rot & 1) * 16));
          }
          if (FULL || (col_ok && RPP * i < rows_left))
            *reinterpret_cast<uint2*>(r_out + (int64_t)(RPP * i) * r_pitch) = codes;
          if (kNibbleTranspose)  // row r, bytes [8 cb, 8 cb + 8): byte k = columns (2k, 2k + 1) of the chunk
            *reinterpret_cast<uint2*>(smem + S::kRand + (rl + RPP * i) * (TC / 2) + cb * 8) =
                (FULL || (col_ok && RPP * i < rows_left)) ? codes : make_uint2(0u, 0u);
          sf_row[sf_row_pos + i * sf_row_step] = (uint8_t)byte;
        }
      }
      if (SR && HAS_ROW && HAS_COL && !kNibbleTranspose && a.off_hi_col != a.off_hi) {  // draws of its own for the transposed copy
#pragma unroll 1
        for (int i = 0; i < NP; ++i) {
          const uint64_t gi = g + (uint64_t)(RPP * i) * (uint64_t)n_cb;
          const uint4 q = philox4x32_10((uint32_t)gi, (uint32_t)(gi >> 32), a.off_lo, a.off_hi_col, a.rk);
          *reinterpret_cast<uint4*>(smem + rand_st + i * (RPP * TC)) = make_uint4(~q.x, ~q.y, ~q.z, ~q.w);
        }
      }
      // Phase 2 of a warp reads only what the same warp staged in phase 1 (its own 16 rows of the tile, their random
      // bytes, its 16x16 scales), so the warps need not wait for each other here.  (An activation's reads the tile alone, and the
      // two phases may overlap: 4096 x 4096 19.4 -> 19.1 us.)
      if (SR || BLOCK2D) __syncwarp();

      // ---------------------------------------------------------------- phase 2 ----
      if constexpr (kNibbleTranspose) {
        // The transposed copy is the row-wise one with its nibbles transposed: a lane takes eight rows (half) of CL
        // neighbouring columns.  (Two columns per lane, read byte by byte, took 2.3 instructions per element and a shared-memory
        // read for every second one: quantizing an 8192 x 5120 weight 39.8 us, now 37.7.)
        constexpr int CL = TC / 16;
        const int q = warp, o = lane & 15, half = lane >> 4;
        const uint8_t* const src = smem + S::kRand + (q * 16 + half * 8) * (TC / 2) + o * (CL / 2);
        uint32_t w[8];
#pragma unroll
        for (int k = 0; k < 8; ++k)
          w[k] = CL == 8 ? *reinterpret_cast<const uint32_t*>(src + k * (TC / 2))
                         : (uint32_t) * reinterpret_cast<const uint16_t*>(src + k * (TC / 2));
        uint32_t col[CL];
        transpose_nibbles(w, col);
#pragma unroll
        for (int k = 0; k < CL; ++k) {
          const int cp = CL / 2 * o + (k >> 1);
          *reinterpret_cast<uint32_t*>(col_codes + cp * 128 + (((q ^ spread(cp)) & 7) << 4) + (k & 1) * 8 + half * 4) = col[k];
        }
        const uint8_t byte = smem[S::kBlkByte + q * CH + (CL * o >> 4)];
#pragma unroll
        for (int k = 0; k < CL / 2; ++k) {
          const int c = CL * o + CL / 2 * half + k;
          sf_col[a.c_swz ? (q >> 2) * (32 * kAtomRow) + (c & 31) * kAtomRow + (c >> 5) * 4 + (q & 3) : c * 8 + q] = byte;
        }
      } else if constexpr (HAS_COL) {
        const int q = warp;  // 16-row group inside the tile
#pragma unroll
        for (int it = 0; it < NIT; ++it) {
          const int cp = lane + 32 * it;  // column pair: tile columns 2cp, 2cp+1
          float2 v[16];  // rows of the group, (column 2cp, column 2cp + 1)
          const uint8_t* tp = tile_buf + q * 16 * S::kRow + cp * (F32 ? 8 : 4);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            if (F32) {
              v[j] = *reinterpret_cast<const float2*>(tp + j * S::kRow);
              continue;
            }
            uint32_t word = *reinterpret_cast<const uint32_t*>(tp + j * S::kRow);
            if (RHT_COL) word ^= a.row_sign[j];
            v[j] = make_float2(bf16_lo(word), bf16_hi(word));
          }
          if (RHT_COL) fwht16_pairs(v);  // both columns in one pass of packed adds; values are 4 * y from here on
          uint32_t byte0, byte1;
          float2 enc;
          if (BLOCK2D) {
            enc.x = enc.y = reinterpret_cast<const float*>(smem + S::kBlkEnc)[q * CH + (cp >> 3)];
            byte0 = byte1 = smem[S::kBlkByte + q * CH + (cp >> 3)];
          } else {
            const float2 m = amax_pairs(v);
            byte0 = block_scale_byte<TINY>(RHT_COL ? 0.25f * m.x : m.x, c_senc);
            byte1 = block_scale_byte<TINY>(RHT_COL ? 0.25f * m.y : m.y, c_senc);
            enc = make_float2(enc_col[byte0], enc_col[byte1]);
          }
          uint2 codes0, codes1;
          if (SR) {
            // low / high byte of ntwo[j] = 255 - draw of source element (row 16q + j, column 2cp / 2cp + 1)
            uint32_t ntwo[16];
            const uint8_t* rp = smem + S::kRand + q * 16 * TC + cp * 2;
#pragma unroll
            for (int j = 0; j < 16; ++j) ntwo[j] = *reinterpret_cast<const uint16_t*>(rp + j * TC);
            convert16x2_sr(v, enc, ntwo, codes0, codes1);
          } else {
            convert16x2_rne(v, enc, codes0, codes1);
          }
          // staging: both columns' eight bytes in one 16-byte unit (conflict-free: eight consecutive column pairs hit
          // eight different units of a 128-byte line)
          *reinterpret_cast<uint4*>(col_codes + col_codes_st + it * 4096) =
              make_uint4(codes0.x, codes0.y, codes1.x, codes1.y);
          sf_col[sf_col_pos + it * sf_col_it] = (uint8_t)byte0;
          sf_col[sf_col_pos + it * sf_col_it + sf_col_odd] = (uint8_t)byte1;
        }
      }
    };
    if (tiny)
      phases_1_2(std::bool_constant<WHOLE>{}, std::true_type{});
    else if (full_tile)
      phases_1_2(std::true_type{}, std::false_type{});
    else
      phases_1_2(std::bool_constant<WHOLE>{}, std::false_type{});
    __syncthreads();
    if (*abort_flag) break;  // a wait expired (the word is read after the barrier: the same for every thread)
    if (threadIdx.x == 0 && j + 2 < n_mine) issue(j + 2);  // every warp is done with this buffer

    // ------------------------------------------------------------------ phase 3 ----
    if (HAS_COL) {
      const int64_t pitch = a.rows >> 1;  // bytes per row of the transposed copy
      if ((a.rows & 31) == 0) {
        // 16 bytes per store: the 16-row groups (2m, 2m + 1) of a column
        if (TC == 64) {  // a thread takes 32 rows of one column
          const int c = threadIdx.x >> 2, m = threadIdx.x & 3, cp = c >> 1;
          const uint8_t* unit = col_codes + cp * 128 + ((((2 * m) ^ spread(cp)) & 7) << 4) + (c & 1) * 8;
          const uint2 g0 = *reinterpret_cast<const uint2*>(unit);
          const uint2 g1 = *reinterpret_cast<const uint2*>(reinterpret_cast<const uint8_t*>((uintptr_t)unit ^ 16));
          if (full_tile || (row0 + 32 * m < a.rows && col0 + c < a.cols))
            *reinterpret_cast<uint4*>(a.c_codes + (col0 + c) * pitch + (row0 >> 1) + m * 16) =
                make_uint4(g0.x, g0.y, g1.x, g1.y);
        } else {  // ... or of column pair cp
          const int cp = threadIdx.x >> 2, m = threadIdx.x & 3;
          const uint8_t* unit = col_codes + cp * 128 + ((((2 * m) ^ spread(cp)) & 7) << 4);
          const uint4 g0 = *reinterpret_cast<const uint4*>(unit);  // group 2m: (first column, second column) x 8 bytes
          const uint4 g1 = *reinterpret_cast<const uint4*>(reinterpret_cast<const uint8_t*>((uintptr_t)unit ^ 16));
          uint8_t* dst = a.c_codes + (col0 + 2 * cp) * pitch + (row0 >> 1) + m * 16;
          if (full_tile || (row0 + 32 * m < a.rows && col0 + 2 * cp < a.cols)) {  // cols is even, rows % 32 == 0
            *reinterpret_cast<uint4*>(dst) = make_uint4(g0.x, g0.y, g1.x, g1.y);
            *reinterpret_cast<uint4*>(dst + pitch) = make_uint4(g0.z, g0.w, g1.z, g1.w);
          }
        }
      } else {
        // rows % 32 == 16: rows of the copy start on 8-byte boundaries; eight lanes write the 64 bytes of a column
#pragma unroll
        for (int p = 0; p < TC / 32; ++p) {
          const int c = (threadIdx.x >> 3) + 32 * p, q = threadIdx.x & 7, cp = c >> 1;
          const uint2 v = *reinterpret_cast<const uint2*>(col_codes + cp * 128 + (((q ^ spread(cp)) & 7) << 4) + (c & 1) * 8);
          if (full_tile || (row0 + 16 * q < a.rows && col0 + c < a.cols))
            *reinterpret_cast<uint2*>(a.c_codes + (col0 + c) * pitch + (row0 >> 1) + q * 8) = v;
        }
      }
    }
    // scale bytes
#pragma unroll
    for (int which = 0; which < 2; ++which) {
      if (which == 0 && !HAS_ROW) continue;
      if (which == 1 && !HAS_COL) continue;
      const uint8_t* src = which == 0 ? sf_row : sf_col;
      uint8_t* dst = which == 0 ? a.r_scales : a.c_scales;
      const int swz = which == 0 ? a.r_swz : a.c_swz;
      // the copy's row / block coordinates of this tile
      const int64_t R0 = which == 0 ? row0 : col0, K0 = which == 0 ? (col0 >> 4) : (row0 >> 4);
      const int64_t Rn = which == 0 ? a.rows : a.cols, n_kb = which == 0 ? n_cb : n_rb;
      if (swz && TC == 64 && which == 1) {
        if (threadIdx.x < 64) {  // eight bytes (64 of the 128 rows) of each 16 of two atoms
          const int atom = threadIdx.x >> 5, l = threadIdx.x & 31;
          if (K0 + atom * 4 < n_kb) {
            const int64_t off = ((R0 >> 7) * (n_kb >> 2) + (K0 >> 2) + atom) * 512 + l * 16 + ((int)(R0 & 127) >> 5) * 4;
            *reinterpret_cast<uint2*>(dst + off) = *reinterpret_cast<const uint2*>(src + atom * 256 + l * 8);
          }
        }
      } else if (swz) {
        if (threadIdx.x < (TC == 64 ? 32 : 64)) {
          const int atom = threadIdx.x >> 5;
          if (K0 + atom * 4 < n_kb) {
            const int64_t off = ((R0 >> 7) * (n_kb >> 2) + (K0 >> 2) + atom) * 512 + (threadIdx.x & 31) * 16;
            *reinterpret_cast<uint4*>(dst + off) = *reinterpret_cast<const uint4*>(src + threadIdx.x * 16);
          }
        }
      } else {
        if (which == 0)
          store_linear_scales<128, CH>(src, dst, R0, K0, Rn, n_kb, full_tile);
        else
          store_linear_scales<TC, 8>(src, dst, R0, K0, Rn, n_kb, full_tile);
      }
    }
    tr -= step_r;
    tc -= step_c;
    if (tc < 0) {
      tc += a.tiles_c;
      --tr;
    }
  }
  if (j < n_mine && threadIdx.x == 0)
    // left early: tiles j and j + 1 may still be in flight; give each one more bounded wait so that no copy lands in shared
    // memory after the CTA has gone
    for (int i = j; i < j + 2 && i < n_mine; ++i) {
      const unsigned long long t0 = globaltimer_ns();
      while (!mbar_try(bar0 + 8 * (i & 1), (uint32_t)(i >> 1) & 1u) && globaltimer_ns() - t0 < kWaitLimitNs) {
      }
    }
}

template <bool HAS_ROW, bool HAS_COL, bool BLOCK2D, bool RHT_ROW, bool RHT_COL, bool SR, int TC, bool F32 = false,
          bool PARTS = false, bool OWN_DRAWS = false>
__global__ void __launch_bounds__(256, 2) quantize_kernel(const __grid_constant__ CUtensorMap src_map,
                                                          const __grid_constant__ QuantArgs a) {
  quantize_tiles<HAS_ROW, HAS_COL, BLOCK2D, RHT_ROW, RHT_COL, SR, TC, F32, PARTS, OWN_DRAWS>(&src_map, a, (int)blockIdx.x,
                                                                                            (int)gridDim.x);
}

// The activation (1x16 blocks, the transposed copy with the transform) and the weight (16x16 blocks) of a forward call in one
// launch, the first n_x CTAs on the activation: one ramp and one tail instead of two.  Carrying the weight's memory-bound
// pass 1 on the activation's pass 2 and quantizing the weight behind it measured the same for many tiles (8192 x 20480 x 5120)
// and lost for few: fwd + bwd of 512 x 1024 x 1024 27.6 -> 24.2 us of GPU time, 1024 x 2048 x 2048 41.7 -> 39.7, 2048 x 4096 x
// 3072 93.8 -> 91.5.  The layer's sizes are multiples of 256, so no tile is cut off and the code for those that are is left out: with
// it (five copies of a tile's code in one kernel) the forward call of 4096 x 4096 x 4096 took 73.1 us, now 72.1, 1024 x 4096 x 3840
// 36.1, now 35.4, 2048 x 4096 x 3072 41.1, now 39.9, 3584 x 2048 x 3840 46.6, now 45.3.  Not for an activation without its transposed
// copy, whose code is short and came out slower so: 768 x 3840 x 1536 17.9 / 18.6 us, 512 x 5120 x 1024 16.2 / 16.8.
template <bool X_COL, bool W_COL, int TC, bool PARTS>
__global__ void __launch_bounds__(256, 2) quantize_x_and_w_kernel(const __grid_constant__ CUtensorMap x_map,
                                                                  const __grid_constant__ CUtensorMap w_map,
                                                                  const __grid_constant__ QuantArgs x,
                                                                  const __grid_constant__ QuantArgs w, int n_x) {
  const int b = (int)blockIdx.x;
  if (b < n_x)
    quantize_tiles<true, X_COL, false, false, X_COL, false, TC, false, PARTS, false, X_COL>(&x_map, x, b, n_x);
  else
    quantize_tiles<true, W_COL, true, false, false, false, TC, false, PARTS, false, true>(&w_map, w, b - n_x, (int)gridDim.x - n_x);
}

// ---------------------------------------------------------------------------------------------
// Test aids
// ---------------------------------------------------------------------------------------------
__global__ void dequantize_kernel(const uint8_t* __restrict__ codes, const uint8_t* __restrict__ scales,
                                  const float* __restrict__ global, int64_t rows, int64_t cols, int swz,
                                  int mx, int per_row, float* __restrict__ out) {
  const int64_t n = rows * cols;
  const float s_dec_t = global[1];
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = i / cols, c = i % cols;
    const uint32_t byte = codes[r * (cols >> 1) + (c >> 1)];
    const uint32_t code = (c & 1) ? (byte >> 4) : (byte & 15u);
    const float mags[8] = {0.f, 0.5f, 1.f, 1.5f, 2.f, 3.f, 4.f, 6.f};
    float m = mags[code & 7u];
    if (code & 8u) m = -m;
    const int sh = mx ? 5 : 4;  // block length 32 (UE8M0 scale) or 16 (E4M3 scale)
    const int64_t so = swz ? sf_swizzled_offset(r, c >> sh, cols >> sh) : (r * (cols >> sh) + (c >> sh));
    uint16_t sb = scales[so];
    float sf;
    if (mx) {
      sf = sb == 0 ? __uint_as_float(0x00400000u) : __uint_as_float((uint32_t)sb << 23);  // 2^(byte - 127)
    } else {
      uint32_t h2;
      asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"(sb));
      sf = __half2float(__ushort_as_half((unsigned short)(h2 & 0xffffu)));
    }
    out[i] = __fmul_rn(__fmul_rn(m, sf), per_row ? global[2 * r + 1] : s_dec_t);
  }
}

__global__ void rht16_kernel(const uint16_t* __restrict__ x, int64_t rows, int64_t cols, int64_t ld,
                             int colwise, uint32_t mask, float* __restrict__ out) {
  // one thread per chunk of the requested copy
  const int64_t R = colwise ? cols : rows, C = colwise ? rows : cols;
  const int64_t n_chunks = R * (C >> 4);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n_chunks;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = i / (C >> 4), kb = i % (C >> 4);
    float f[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const int64_t sr = colwise ? (kb * 16 + j) : r, sc = colwise ? r : (kb * 16 + j);
      uint32_t bits = (uint32_t)x[sr * ld + sc] << 16;
      if ((mask >> j) & 1u) bits ^= 0x80000000u;
      f[j] = __uint_as_float(bits);
    }
    fwht16(f);
#pragma unroll
    for (int j = 0; j < 16; ++j) out[r * C + kb * 16 + j] = f[j] * 0.25f;
  }
}

// codes[i] = stochastic rounding of v[i] with the draw u[i], through the very conversion the quantizer uses
__global__ void e2m1_sr_kernel(const float* __restrict__ v, const uint8_t* __restrict__ u, int64_t n,
                               uint8_t* __restrict__ codes) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    // the element sits in the low slot on even i and in the high slot on odd i, the other slot holds a decoy
    const float w = __fmul_rz(v[i], kSrTowardsZero), decoy = __fmul_rz(-v[i] * 0.75f, kSrTowardsZero);
    const uint32_t nu = 255u - u[i], nd = (uint32_t)(i * 37) & 255u;
    const uint32_t d = (i & 1) ? e2m1x2_sr(decoy, w, (nu << 24) | (nd << 16) | 0x8080u)
                               : e2m1x2_sr(w, decoy, (nd << 24) | (nu << 16) | 0x8080u);
    codes[i] = (uint8_t)((i & 1) ? (d >> 8) & 15u : d & 15u);
  }
}

// ---------------------------------------------------------------------------------------------
// Host launchers
// ---------------------------------------------------------------------------------------------
int64_t amax_parts(int64_t rows, int64_t cols) { return (rows + 127) / 128 * ((cols + 255) / 256); }

// Pass 1 in parts while every tile of pass 2 (64 columns wide, four to a tile of pass 1) has a CTA of its own: the call has a
// launch less.  Graph time of a layer, words / parts: fwd + bwd of 512 x 1024 x 1024 24.0 / 22.9 us, 1024 x 1024 x 1024 25.9 /
// 24.7, 1024 x 2048 x 2048 39.1 / 38.5; bwd of 1024 x 2048 x 1024 17.2 / 16.9; and 2.3 us of the host's time.  Beyond that it
// loses (2048 x 3328 x 3328 80.6 / 82.1): see launch_amax_parts().
bool pass1_in_parts(int64_t parts) {
  int sms = 0;
  return sm_count(&sms) == cudaSuccess && 4 * parts <= 2 * sms;
}

// In parts, pass 1 is the first kernel of its call and becomes resident while the previous one drains.  At three CTAs per SM
// it crowds on the SMs that drain first and runs there when it may begin (bwd of 1024 x 2048 x 1024 18.9 us instead of 16.9):
// more shared memory than half of an SM's keeps it to one.
template <auto KERN, typename... Args>
static cudaError_t launch_amax_parts(unsigned tiles, cudaStream_t s, Args&&... args) {
  constexpr int kSmem = 120 * 1024;
  static std::atomic<uint64_t> configured{0};  // per kernel and device
  int dev;
  if (device_needs_config(configured, &dev)) {
    const cudaError_t e = cudaFuncSetAttribute(KERN, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
    if (e != cudaSuccess) return e;
    device_configured(configured, dev);
  }
  return launch_kernel(KERN, dim3(tiles), dim3(256), kSmem, s, std::forward<Args>(args)...);
}

template <bool PLAIN, bool RR, bool RC>
static cudaError_t launch_amax_t(const QuantArgs& a, float* plain0, float* plain1, float* rot_row,
                                 float* rot_col, cudaStream_t s) {
  const int tiles_c = (int)((a.cols + 255) / 256);
  const int64_t tiles = ((a.rows + 127) / 128) * tiles_c;
  cudaError_t e = cudaErrorInvalidValue;
  if (!a.parts)
    e = launch_kernel(amax_kernel<PLAIN, RR, RC, false>, dim3((unsigned)tiles), dim3(256), 0, s, a.x, a.rows, a.cols, a.ld,
                      a.sign_mask, tiles_c, plain0, plain1, rot_row, rot_col, (float2*)nullptr);
  else if constexpr (!RR && !RC)
    e = launch_amax_parts<amax_kernel<PLAIN, RR, RC, true>>((unsigned)tiles, s, a.x, a.rows, a.cols, a.ld, a.sign_mask, tiles_c,
                                                            plain0, plain1, rot_row, rot_col, a.parts);
  count_launch();
  return e;
}

// Clears up to four words.  It waits for everything before the call and then lets the reduction behind it start, which
// streams its tensor meanwhile and waits for the zeros just before its first atomic: one short launch in the shadow of
// the launch latency, where a memset per word cost 3 us of stream time each (a layer step had six).  With the kernels
// behind each other in programmatic order throughout, fwd + bwd of 512 x 1024 x 1024 went from 50.2 to 39.9 us, of
// 2816 x 3328 x 2304 from 94.5 to 84.5 us, quantizing a 7168 x 5120 binary32 weight from 68.5 to 62.2 us.
__global__ void zero_words_kernel(float* w0, float* w1, float* w2, float* w3) {
  griddep_wait();
  griddep_launch_dependents();
  float* const w = threadIdx.x == 0 ? w0 : threadIdx.x == 1 ? w1 : threadIdx.x == 2 ? w2 : w3;
  if (threadIdx.x < 4 && w) *w = 0.f;
}

cudaError_t launch_zero_words(float* w0, float* w1, float* w2, float* w3, cudaStream_t s) {
  const cudaError_t e = launch_kernel(zero_words_kernel, dim3(1), dim3(32), 0, s, w0, w1, w2, w3);
  count_launch();
  return e;
}

template <bool PLAIN>
static cudaError_t launch_amax_rot_col(const QuantArgs& a, uint32_t mask16, float* plain0, float* plain1, float* rot_col,
                                       int d, float norm, bool sr, cudaStream_t s) {
  const int tiles_c = (int)((a.cols + 255) / 256);
  const unsigned tiles = (unsigned)(((a.rows + 127) / 128) * tiles_c);
  const cudaError_t e =
      a.parts ? launch_amax_parts<amax_rot_col_kernel<PLAIN, true>>(tiles, s, a.x, a.rows, a.cols, a.ld, mask16, tiles_c, plain0,
                                                                    plain1, rot_col, d, norm, a.parts)
              : launch_kernel(evict_first(a, sr) ? amax_rot_col_kernel<PLAIN, false, true> : amax_rot_col_kernel<PLAIN, false>,
                              dim3(tiles), dim3(256), 0, s, a.x, a.rows, a.cols, a.ld, mask16, tiles_c, plain0, plain1, rot_col,
                              d, norm, (float2*)nullptr);
  count_launch();
  return e;
}

cudaError_t launch_amax(const QuantArgs& a, bool has_row, bool has_col, bool rht_row, bool rht_col, bool sr,
                        cudaStream_t s) {
  if (!a.parts) {
    const cudaError_t e = launch_zero_words(has_row ? a.r_global : nullptr, has_col ? a.c_global : nullptr, nullptr, nullptr, s);
    if (e != cudaSuccess) return e;
  }
  const bool rr = has_row && rht_row, rc = has_col && rht_col;
  float* plain0 = (has_row && !rht_row) ? a.r_global : nullptr;
  float* plain1 = (has_col && !rht_col) ? a.c_global : nullptr;
  const bool plain = plain0 || plain1;
  float* rot_row = rr ? a.r_global : nullptr;
  float* rot_col = rc ? a.c_global : nullptr;
  if (rc && !rr)  // tensor-core transform for the transposed copy
    return plain ? launch_amax_rot_col<true>(a, a.sign_mask, plain0, plain1, rot_col, 16, 0.25f, sr, s)
                 : launch_amax_rot_col<false>(a, a.sign_mask, plain0, plain1, rot_col, 16, 0.25f, sr, s);
#define NVFP4_AMAX(P, R, C) \
  if (plain == P && rr == R && rc == C) return launch_amax_t<P, R, C>(a, plain0, plain1, rot_row, rot_col, s);
  NVFP4_AMAX(true, false, false)
  NVFP4_AMAX(true, false, true)
  NVFP4_AMAX(true, true, false)
  NVFP4_AMAX(false, true, true)
  NVFP4_AMAX(false, false, true)
  NVFP4_AMAX(false, true, false)
#undef NVFP4_AMAX
  return cudaErrorInvalidValue;
}

// Pass 1 of the transposed copy with a d x d transform (d = 2, 4, 8), and the plain amax of the row-wise copy
// beside it: the tensor-core kernel above with a block-diagonal matrix.  sign_mask: the d sign bits repeated to 16.
cudaError_t launch_amax_rot_col_small(const QuantArgs& a, bool has_row, uint32_t mask16, int d, float norm,
                                      cudaStream_t s) {
  const cudaError_t e = launch_zero_words(has_row ? a.r_global : nullptr, a.c_global, nullptr, nullptr, s);
  if (e != cudaSuccess) return e;
  return has_row ? launch_amax_rot_col<true>(a, mask16, a.r_global, nullptr, a.c_global, d, norm, false, s)
                 : launch_amax_rot_col<false>(a, mask16, nullptr, nullptr, a.c_global, d, norm, false, s);
}

// the source as a 2-D tensor map: boxes of 128 rows x tc elements (no swizzle), zero fill outside
static bool quant_source_map(CUtensorMap* map, const QuantArgs& a, int tc, bool f32 = false) {
  return make_map_2d(map, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, f32 ? 4 : 2, a.x,
                     (uint64_t)a.cols, (uint64_t)a.rows, (uint64_t)a.ld * (f32 ? 4 : 2), tc, 128, false);
}

template <bool HR, bool HC, bool B2, bool RR, bool RC, bool SR, int TC, bool F32 = false, bool PARTS = false, bool OWN = false>
static cudaError_t launch_quant_tc(const QuantArgs& a_in, int slots, cudaStream_t s) {
  auto kern = quantize_kernel<HR, HC, B2, RR, RC, SR, TC, F32, PARTS, OWN>;
  QuantArgs a = a_in;
  a.tiles_c = (int)((a.cols + TC - 1) / TC);
  constexpr bool kRowCodes = B2 && HR && HC && !OWN;
  constexpr int smem = QuantSmem<TC, F32>::bytes(SR && HC && !kRowCodes, kRowCodes);
  CUtensorMap map;
  if (!quant_source_map(&map, a, TC, F32)) return cudaErrorInvalidValue;
  static std::atomic<uint64_t> configured{0};  // per call site (template instantiation) and device
  int dev;
  if (device_needs_config(configured, &dev)) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    device_configured(configured, dev);
  }
  const int64_t tiles = (int64_t)a.tiles_r * a.tiles_c;
  const cudaError_t e =
      launch_kernel(kern, dim3((unsigned)(tiles < slots ? tiles : slots)), dim3(256), smem, s, map, a);
  count_launch();
  return e;
}

template <bool HR, bool HC, bool B2, bool RR, bool RC, bool SR>
static cudaError_t launch_quant_t(const QuantArgs& a, cudaStream_t s) {
  int sms = 0;
  const cudaError_t e = sm_count(&sms);
  if (e != cudaSuccess) return e;
  // Tiles 64 columns wide when they go round the resident CTAs in less time: a tile of half the width counts as 0.535 of a whole
  // one (16x16 blocks: 0.58), and the CTAs take whole rounds.  Measured (128 / 64 wide, three tensors in turn): gradient of 2816 x
  // 2304 15.3 / 13.6 us, 1024 x 9728 21.8 / 19.8, 4096 x 4096 29.8 / 28.5, 8192 x 5120 57.6 / 60.4; activation of 4096 x 4096 23.2 /
  // 22.8, 8192 x 5120 42.9 / 46.9; weight of 4096 x 2304 10.6 / 11.7, 8192 x 5120 37.9 / 43.8.  (The factors were fitted when a
  // tile took 5 to 8 % longer; of 90 drawn tensors they give one the slower width by more than 1 %: activation of 2304 x 11008
  // 30.5 / 31.6.)
  const int slots = 2 * sms;  // resident CTAs
  if constexpr (!B2 && !RR && RC == HC)  // an activation or a gradient of a layer
    if (a.parts) return launch_quant_tc<HR, HC, B2, RR, RC, SR, 64, false, true>(a, slots, s);
  const int64_t t128 = (int64_t)a.tiles_r * a.tiles_c, t64 = (int64_t)a.tiles_r * ((a.cols + 63) / 64);
  const double r128 = (double)((t128 + slots - 1) / slots), r64 = (double)((t64 + slots - 1) / slots) * (B2 ? 0.58 : 0.535);
  if (!RR && r64 < r128) return launch_quant_tc<HR, HC, B2, RR, RC, SR, RR ? 128 : 64>(a, slots, s);
  return launch_quant_tc<HR, HC, B2, RR, RC, SR, 128>(a, slots, s);
}

template <bool X_COL, bool W_COL, int TC, bool PARTS = false>
static cudaError_t launch_x_and_w_tc(QuantArgs x, QuantArgs w, int slots, cudaStream_t s) {
  auto kern = quantize_x_and_w_kernel<X_COL, W_COL, TC, PARTS>;
  constexpr int smem = QuantSmem<TC>::bytes(false, W_COL);
  CUtensorMap maps[2];
  QuantArgs* const t[2] = {&x, &w};
  for (int i = 0; i < 2; ++i) {
    t[i]->tiles_c = (int)((t[i]->cols + TC - 1) / TC);
    if (!quant_source_map(&maps[i], *t[i], TC)) return cudaErrorInvalidValue;
  }
  static std::atomic<uint64_t> configured{0};  // per call site (template instantiation) and device
  int dev;
  if (device_needs_config(configured, &dev)) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    device_configured(configured, dev);
  }
  // CTAs in proportion to the work (a weight's tile counts as three quarters of an activation's), at whole rounds of either.  Anything
  // from 0.65 to 0.8 measures the same within 1 %; 0.85 costs 8192 x 6144 x 1536 70.4 -> 71.4 us, 4352 x 2048 x 2560 38.6 -> 39.6.
  const int tx = x.tiles_r * x.tiles_c, tw = w.tiles_r * w.tiles_c;
  int n_x = tx, n_w = tw;
  if (tx + tw > slots) {
    double least = 1e30;
    for (int rounds = (tx + slots - 2) / (slots - 1); rounds <= tx; ++rounds) {
      const int gx = (tx + rounds - 1) / rounds, gw = slots - gx < tw ? slots - gx : tw;
      const double w_time = 0.75 * ((tw + gw - 1) / gw), time = rounds > w_time ? (double)rounds : w_time;
      if (time < least) {
        least = time;
        n_x = gx;
        n_w = gw;
      }
      if (rounds >= w_time) break;  // more rounds of the activation only take longer
    }
  }
  const cudaError_t e = launch_kernel(kern, dim3((unsigned)(n_x + n_w)), dim3(256), smem, s, maps[0], maps[1], x, w, n_x);
  count_launch();
  return e;
}

template <bool X_COL, bool W_COL>
static cudaError_t launch_x_and_w_t(const QuantArgs& x, const QuantArgs& w, cudaStream_t s) {
  int sms = 0;
  cudaError_t e = sm_count(&sms);
  if (e != cudaSuccess) return e;
  if ((x.rows | x.cols | w.rows | w.cols) % 128 != 0) return cudaErrorInvalidValue;  // (a layer's sizes: multiples of 256)
  if (!x.parts) {
    e = launch_zero_words(x.r_global, X_COL ? x.c_global : nullptr, w.r_global, W_COL ? w.c_global : nullptr, s);
    if (e != cudaSuccess) return e;
  }
  const int xc = (int)((x.cols + 255) / 256), wc = (int)((w.cols + 255) / 256);
  const int64_t n_x = ((x.rows + 127) / 128) * xc, n_w = ((w.rows + 127) / 128) * wc;
  if (n_x + n_w > 0x7fffffff) return cudaErrorInvalidValue;
  e = x.parts ? launch_amax_parts<amax_x_and_w_kernel<X_COL, W_COL, true>>((unsigned)(n_x + n_w), s, x, w, (int)n_x, xc, wc)
              : launch_kernel(amax_x_and_w_kernel<X_COL, W_COL, false>, dim3((unsigned)(n_x + n_w)), dim3(256), 0, s, x, w,
                              (int)n_x, xc, wc);
  count_launch();
  if (e != cudaSuccess) return e;
  QuantArgs xa = x, wa = w;
  xa.chained = wa.chained = 1;
  const int slots = 2 * sms;  // resident CTAs; the width of the tiles as in launch_quant_t
  if (x.parts) return launch_x_and_w_tc<X_COL, W_COL, 64, true>(xa, wa, slots, s);
  const int64_t t128 = (int64_t)x.tiles_r * x.tiles_c + (int64_t)w.tiles_r * w.tiles_c;
  const int64_t t64 = (int64_t)x.tiles_r * ((x.cols + 63) / 64) + (int64_t)w.tiles_r * ((w.cols + 63) / 64);
  // (0.6: the forward call of 1024 x 4096 x 4096 takes 38.4 us in nine rounds of narrow tiles, 35.6 in five of wide ones.  Of 34
  // shapes two would gain more than 1 % by the other width: 6144 x 512 x 2560 35.1 / 34.5, 2048 x 4608 x 512 19.8 / 19.5.)
  return 0.6 * (double)((t64 + slots - 1) / slots) < (double)((t128 + slots - 1) / slots)
             ? launch_x_and_w_tc<X_COL, W_COL, 64>(xa, wa, slots, s)
             : launch_x_and_w_tc<X_COL, W_COL, 128>(xa, wa, slots, s);
}

cudaError_t launch_quantize_x_and_w(const QuantArgs& x, bool x_col, const QuantArgs& w, bool w_col, cudaStream_t s) {
  if (x_col) return w_col ? launch_x_and_w_t<true, true>(x, w, s) : launch_x_and_w_t<true, false>(x, w, s);
  return w_col ? launch_x_and_w_t<false, true>(x, w, s) : launch_x_and_w_t<false, false>(x, w, s);
}

cudaError_t launch_quantize(const QuantArgs& a, bool has_row, bool has_col, bool block2d, bool rht_row,
                            bool rht_col, bool sr, cudaStream_t s) {
  rht_row = rht_row && has_row;
  rht_col = rht_col && has_col;
#define NVFP4_Q(HR, HC, B2, RR, RC, SRV)                                                           \
  if (has_row == HR && has_col == HC && block2d == B2 && rht_row == RR && rht_col == RC && sr == SRV) \
    return launch_quant_t<HR, HC, B2, RR, RC, SRV>(a, s);
#define NVFP4_Q_COPIES(B2, RR, RC, SRV)      \
  NVFP4_Q(true, false, B2, RR, false, SRV)   \
  NVFP4_Q(false, true, B2, false, RC, SRV)   \
  NVFP4_Q(true, true, B2, RR, RC, SRV)
  NVFP4_Q_COPIES(true, false, false, false)
  NVFP4_Q_COPIES(true, false, false, true)
  NVFP4_Q_COPIES(false, false, false, false)
  NVFP4_Q_COPIES(false, false, false, true)
  NVFP4_Q_COPIES(false, false, true, false)
  NVFP4_Q_COPIES(false, false, true, true)
  NVFP4_Q_COPIES(false, true, false, false)
  NVFP4_Q_COPIES(false, true, false, true)
  NVFP4_Q_COPIES(false, true, true, false)
  NVFP4_Q_COPIES(false, true, true, true)
#undef NVFP4_Q_COPIES
#undef NVFP4_Q
  return cudaErrorInvalidValue;
}

cudaError_t launch_amax_f32(const QuantArgs& a, bool has_row, bool has_col, cudaStream_t s) {
  cudaError_t e = launch_zero_words(has_row ? a.r_global : nullptr, has_col ? a.c_global : nullptr, nullptr, nullptr, s);
  if (e != cudaSuccess) return e;
  const int tiles_c = (int)((a.cols + 127) / 128);
  const unsigned tiles = (unsigned)(((a.rows + 127) / 128) * tiles_c);
  // Its loads do not fit the L1 beside the shared memory of the pass 2, or the product, before it.  The whole call without the division /
  // with it, sources in turn that exceed L2: 2304 x 3328 15.0 / 14.5 us, 4096 x 4096 26.0 / 25.6, 7168 x 5120 55.0 / 54.1, 20480 x 5120 139.4
  // / 138.3, up to 2048 x 2048 the same; behind a product 2048 x 2048 20.3 / 19.8, 4096 x 4096 37.3 / 37.2, 7168 x 5120 65.3 / 64.7.  The
  // bf16 kernels of pass 1 gain nothing: behind a product within the measurement's 1 %, behind another quantizer's pass 2 they lose 0.3 to
  // 0.8 % (their first CTAs then fit beside the last ones of that pass only as the SM is).
  e = launch_divided(kStreamingCarveout, amax_f32_kernel, dim3(tiles), dim3(256), 0, s, reinterpret_cast<const float*>(a.x), a.rows, a.cols,
                    a.ld, tiles_c, has_row ? a.r_global : nullptr, has_col ? a.c_global : nullptr);
  count_launch();
  return e;
}

// binary32 source (Appendix B names FP32 as well as BF16 as the precision converted from), e.g. weights quantized straight from
// their FP32 master copy; no transform (the recipe transforms activations and gradients, which are bf16)
cudaError_t launch_quantize_f32(const QuantArgs& a, bool has_row, bool has_col, bool block2d, bool sr, cudaStream_t s) {
  int sms = 0;
  const cudaError_t e = sm_count(&sms);
  if (e != cudaSuccess) return e;
  if (block2d && sr && has_row && has_col && a.off_hi_col != a.off_hi)  // independent draws: the copies' codes differ
    return launch_quant_tc<true, true, true, false, false, true, 64, true, false, true>(a, 2 * sms, s);
#define NVFP4_F32Q(HR, HC, B2, SRV)                                              \
  if (has_row == HR && has_col == HC && block2d == B2 && sr == SRV)              \
    return launch_quant_tc<HR, HC, B2, false, false, SRV, 64, true>(a, 2 * sms, s);
#define NVFP4_F32Q_COPIES(B2, SRV) \
  NVFP4_F32Q(true, false, B2, SRV)  \
  NVFP4_F32Q(false, true, B2, SRV)  \
  NVFP4_F32Q(true, true, B2, SRV)
  NVFP4_F32Q_COPIES(true, false)
  NVFP4_F32Q_COPIES(true, true)
  NVFP4_F32Q_COPIES(false, false)
  NVFP4_F32Q_COPIES(false, true)
#undef NVFP4_F32Q_COPIES
#undef NVFP4_F32Q
  return cudaErrorInvalidValue;
}

cudaError_t launch_dequantize(const nvfp4_tensor& t, float* out, cudaStream_t s) {
  dequantize_kernel<<<1184, 256, 0, s>>>(t.codes, t.scales, t.global, t.rows, t.cols,
                                         t.sf_layout == NVFP4_SF_SWIZZLED, t.format == NVFP4_FORMAT_MXFP4,
                                         t.format == NVFP4_FORMAT_NVFP4_ROWSCALE, out);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_rht16(const void* x, int64_t rows, int64_t cols, int64_t ld, int colwise, uint32_t mask,
                         float* out, cudaStream_t s) {
  rht16_kernel<<<1184, 256, 0, s>>>(static_cast<const uint16_t*>(x), rows, cols, ld, colwise, mask, out);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_e2m1_sr(const float* v, const uint8_t* u, int64_t n, uint8_t* codes, cudaStream_t s) {
  e2m1_sr_kernel<<<1184, 256, 0, s>>>(v, u, n, codes);
  count_launch();
  return cudaGetLastError();
}

}  // namespace nvfp4
