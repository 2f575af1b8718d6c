// Device helpers shared by the NVFP4 and the MXFP4 quantizer kernels (included by quantize.cu and quantize_mx.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "async_ptx.cuh"
#include "common.cuh"

namespace nvfp4 {

// just more dynamic shared memory than two | three CTAs of an SM (228 KB, 1 KB of it taken per CTA) can have
constexpr int kSmemOfHalf = 116 * 1024, kSmemOfThird = 76 * 1024;

// ---------------------------------------------------------------------------------------------
// small PTX helpers
// ---------------------------------------------------------------------------------------------
// Loads of a tensor that is read once.  Coherent ones (no .nc): a kernel that is resident before its source has been written may read it
// only that way, and the non-coherent path was no faster (quantizers of every role: within the 1 % that two runs differ).
__device__ __forceinline__ void ldg256_stream(const void* p, uint32_t (&r)[8]) {
  asm volatile("ld.global.L1::no_allocate.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                 "=r"(r[7])
               : "l"(p));
}
__device__ __forceinline__ void ldg256_hint(const void* p, uint32_t (&r)[8], uint64_t policy) {
  asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8], %9;"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                 "=r"(r[7])
               : "l"(p), "l"(policy));
}
__device__ __forceinline__ uint4 ldg128_stream(const void* p) {
  uint4 r;
  asm volatile("ld.global.L1::no_allocate.v4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
               : "l"(p));
  return r;
}

// magnitudes of `acc` become the larger ones of both operands; its signs mean nothing (amax_of_pair drops them)
__device__ __forceinline__ uint32_t absmax_bf16x2(uint32_t acc, uint32_t v) {
  asm("max.xorsign.abs.bf16x2 %0, %0, %1;" : "+r"(acc) : "r"(v));
  return acc;
}
__device__ __forceinline__ float amax_of_pair(uint32_t acc) { return fmaxf(fabsf(bf16_lo(acc)), fabsf(bf16_hi(acc))); }

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// sign word for a bf16 pair whose two elements are inputs j0 and j1 of a Hadamard chunk
__device__ __forceinline__ uint32_t sign_pair(uint32_t mask, int j0, int j1) {
  return (((mask >> j0) & 1u) << 15) | (((mask >> j1) & 1u) << 31);
}

// Bounded wait for a tile (2 s): on expiry the abort word of the CTA and the device status word are set.
constexpr uint32_t kQuantWaitCode = 0x51000001u;
__device__ __forceinline__ bool quant_wait(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag,
                                           unsigned int* status) {
  if (mbar_try(bar, parity)) return true;
  const unsigned long long t0 = globaltimer_ns();
  uint32_t spins = 0;
  while (true) {
    if (mbar_try(bar, parity)) return true;
    if ((++spins & 63u) == 0u) {
      if (*abort_flag) return false;
      if (globaltimer_ns() - t0 > kWaitLimitNs) {
        *abort_flag = kQuantWaitCode;
        if (status) atomicCAS(status, 0u, kQuantWaitCode);
        return false;
      }
    }
  }
}

// Eq. 2-3: the stored E4M3 byte of a block, S_b = e4m3(fl(fl(amax_b / 6) * s_enc)).  TINY: s_enc > kPlainDivisionLimit; the other
// form has no branch.  A branch per block (this one, and one around the transposed copy's own draws) cut the code of a tile into
// pieces that could not overlap, at four warps per scheduler: activation of 8192 x 5120 43.5 -> 41.0 us without, gradient 59.2 ->
// 55.6, 4096 x 4096 20.2 -> 19.4 and 26.4 -> 24.5.
template <bool TINY>
__device__ __forceinline__ uint32_t block_scale_byte(float amax_b, float s_enc) {
  const float t = __fmul_rn(TINY ? div6_rn(amax_b) : div6_fast(amax_b), s_enc);
  uint16_t packed;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(packed) : "f"(0.f), "f"(t));
  return packed;
}
// the text after Eq. 3: encode scale of a block from its stored byte, fl(1 / fl(fp32(S_b) * s_dec)), 0 for S_b = 0
__device__ __forceinline__ float encode_scale_of_byte(uint32_t byte, float s_dec) {
  uint32_t h2;
  asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"((uint16_t)byte));
  const float sf = __half2float(__ushort_as_half((unsigned short)(h2 & 0xffffu)));
  const float d = __fmul_rn(sf, s_dec);
  return (byte == 0u) ? 0.0f : fminf(__frcp_rn(d), kFltMax);
}

// max(m, |a|, |b|)
__device__ __forceinline__ float amax3(float m, float a, float b) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(m), "f"(fabsf(a)), "f"(fabsf(b)));
  return r;
}
__device__ __forceinline__ float amax16_3(const float (&f)[16]) {
  float m = 0.f;
#pragma unroll
  for (int i = 0; i < 16; i += 2) m = amax3(m, f[i], f[i + 1]);
  return m;
}

// Eq. 4 for sixteen values: v = fl(y * s_enc,b), two lanes per instruction; for stochastic rounding the result is
// then moved one binary32 towards zero, which is what e2m1x2_sr() expects.
template <bool SR>
__device__ __forceinline__ void scale16(const float (&f)[16], float s_enc_b, float (&v)[16]) {
#pragma unroll
  for (int i = 0; i < 16; i += 2) {
    float2 p = mul2(make_float2(f[i], f[i + 1]), make_float2(s_enc_b, s_enc_b));
    if (SR) p = mul2_rz(p, make_float2(kSrTowardsZero, kSrTowardsZero));
    v[i] = p.x;
    v[i + 1] = p.y;
  }
}

// 16 scaled values -> 16 E2M1 nibbles (element 0 in the lowest nibble of .x).  For stochastic rounding
// `draws.rbits(i, j)` returns the random word of e2m1x2_sr() for elements i (low) and j (high).
template <bool SR, class Draws>
__device__ __forceinline__ uint2 convert16(const float (&f)[16], float s_enc_b, Draws draws) {
  uint2 out;
  float v[16];
  scale16<SR>(f, s_enc_b, v);
  if (!SR) {
    const float(&lo)[8] = *reinterpret_cast<const float(*)[8]>(&v[0]);
    const float(&hi)[8] = *reinterpret_cast<const float(*)[8]>(&v[8]);
    out.x = e2m1x8_rne(lo);
    out.y = e2m1x8_rne(hi);
  } else {
    // nibbles 0 and 2 of each 16-bit half: elements (4k, 4k + 2) in `even`, (4k + 1, 4k + 3) in `odd`, k = 0, 1 | 2, 3
    const uint32_t even01 = e2m1x2_sr_pair(v[0], v[2], draws.rbits(0, 2), v[4], v[6], draws.rbits(4, 6));
    const uint32_t odd01 = e2m1x2_sr_pair(v[1], v[3], draws.rbits(1, 3), v[5], v[7], draws.rbits(5, 7));
    const uint32_t even23 = e2m1x2_sr_pair(v[8], v[10], draws.rbits(8, 10), v[12], v[14], draws.rbits(12, 14));
    const uint32_t odd23 = e2m1x2_sr_pair(v[9], v[11], draws.rbits(9, 11), v[13], v[15], draws.rbits(13, 15));
    out.x = even01 + odd01 * 16u;  // disjoint nibbles: the sum is the union
    out.y = even23 + odd23 * 16u;
  }
  return out;
}

// draws packed four to a word, byte i = element i (the row-wise copy: straight from the Philox output)
struct Nu14FromWords {
  const uint32_t (&rnd)[4];
  __device__ __forceinline__ uint32_t rbits(int i, int j) const {  // i, j in the same word, i even <=> j even
    return __byte_perm(~rnd[i >> 2], 0x80808080u, (i & 1) ? 0x3144u : 0x2044u);
  }
};
// draws of two adjacent columns, 16 bits per row (the transposed copy: read back from shared memory)
template <int COL>
struct Nu14FromPairs {
  const uint32_t (&two)[16];
  __device__ __forceinline__ uint32_t rbits(int i, int j) const {
    const uint32_t picked = __byte_perm(two[i], two[j], COL == 0 ? 0x4000u : 0x5100u);  // bytes 2, 3 = draws of i, j
    return (~picked & 0xFFFF0000u) | 0x8080u;
  }
};

// Two columns of sixteen rows at once (the transposed copy): y[r] = (row r of the first column, of the second), which is
// how the tile is read and transformed, so that a packed multiplication scales a row of both without moving registers.
template <bool SR>
__device__ __forceinline__ float2 scale_row_pair(float2 y, float2 enc) {  // Eq. 4 (see scale16)
  const float2 p = mul2(y, enc);
  return SR ? mul2_rz(p, make_float2(kSrTowardsZero, kSrTowardsZero)) : p;
}
// Stochastic rounding, element r of both columns in one conversion.  ntwo[r]: low byte = 255 - draw of (row r, first
// column), next byte = the same for the second one.
__device__ __forceinline__ void convert16x2_sr(const float2* y, float2 enc, const uint32_t (&ntwo)[16], uint2& out0,
                                               uint2& out1) {
  // rows (r, r + 1) of both columns: byte 0 = first column, byte 1 = second column; rows (r + 2, r + 3) in bytes 2, 3
  uint32_t e[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const int r = 4 * m;
    float2 v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = scale_row_pair<true>(y[r + k], enc);
    const uint32_t a = e2m1x2_sr_pair(v[0].x, v[0].y, __byte_perm(ntwo[r], 0x80808080u, 0x1044u), v[2].x, v[2].y,
                                      __byte_perm(ntwo[r + 2], 0x80808080u, 0x1044u));
    const uint32_t b = e2m1x2_sr_pair(v[1].x, v[1].y, __byte_perm(ntwo[r + 1], 0x80808080u, 0x1044u), v[3].x, v[3].y,
                                      __byte_perm(ntwo[r + 3], 0x80808080u, 0x1044u));
    e[m] = a + b * 16u;  // disjoint nibbles
  }
  out0 = make_uint2(__byte_perm(e[0], e[1], 0x6420u), __byte_perm(e[2], e[3], 0x6420u));
  out1 = make_uint2(__byte_perm(e[0], e[1], 0x7531u), __byte_perm(e[2], e[3], 0x7531u));
}
// Rounding to nearest even
__device__ __forceinline__ void convert16x2_rne(const float2* y, float2 enc, uint2& out0, uint2& out1) {
  uint32_t o0[2], o1[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float v0[8], v1[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float2 v = scale_row_pair<false>(y[8 * h + k], enc);
      v0[k] = v.x;
      v1[k] = v.y;
    }
    o0[h] = e2m1x8_rne(v0);
    o1[h] = e2m1x8_rne(v1);
  }
  out0 = make_uint2(o0[0], o0[1]);
  out1 = make_uint2(o1[0], o1[1]);
}
// block maxima of both columns
template <int ROWS>
__device__ __forceinline__ float2 amax_pairs(const float2 (&y)[ROWS]) {
  float2 m = make_float2(0.f, 0.f);
#pragma unroll
  for (int r = 0; r < ROWS; r += 2) {
    m.x = amax3(m.x, y[r].x, y[r + 1].x);
    m.y = amax3(m.y, y[r].y, y[r + 1].y);
  }
  return m;
}

__device__ __forceinline__ float amax16(const float (&f)[16]) {
  float m = 0.f;
#pragma unroll
  for (int i = 0; i < 16; ++i) m = fmaxf(m, fabsf(f[i]));
  return m;
}

// Row-by-row scale bytes of a tile of ROWS x KB blocks (staged row by row): as words where the row length keeps them aligned.
// Row lengths are any number; otherwise the bytes leave one by one, but neighbouring lanes write the bytes of a row: a warp's
// store touches four (eight) rows, not sixteen (four bytes of a row per thread made the stores a microsecond of the tile's
// five).
template <int ROWS, int KB>
__device__ __forceinline__ void store_linear_scales(const uint8_t* src, uint8_t* dst, int64_t R0, int64_t K0, int64_t Rn,
                                                    int64_t n_kb, bool full_tile) {
  if (full_tile && (n_kb & 3) == 0) {
    if (threadIdx.x < ROWS * KB / 4)
      *reinterpret_cast<uint32_t*>(dst + (R0 + threadIdx.x / (KB / 4)) * n_kb + K0 + threadIdx.x % (KB / 4) * 4) =
          *reinterpret_cast<const uint32_t*>(src + threadIdx.x * 4);
    return;
  }
  const int r = threadIdx.x / KB, kb = threadIdx.x % KB;
  uint8_t* d = dst + (R0 + r) * n_kb + K0 + kb;
#pragma unroll
  for (int p = 0; p < ROWS * KB / 256; ++p, d += 256 / KB * n_kb)
    if (full_tile || (R0 + r + 256 / KB * p < Rn && K0 + kb < n_kb)) *d = src[threadIdx.x + 256 * p];
}

// Eight rows of CL nibbles (a word each, columns from the low end) -> CL columns of eight nibbles (rows from the low end): 16-bit
// halves, then bytes, then nibbles.
template <int CL>
__device__ __forceinline__ void transpose_nibbles(const uint32_t (&w)[8], uint32_t (&col)[CL]) {
#pragma unroll
  for (int h = 0; h < CL / 4; ++h) {  // columns 4h .. 4h + 3
    uint32_t p[4];                     // [row k | row k + 4]
#pragma unroll
    for (int k = 0; k < 4; ++k) p[k] = __byte_perm(w[k], w[k + 4], h ? 0x7632 : 0x5410);
#pragma unroll
    for (int b = 0; b < 2; ++b) {  // the pair of columns in bytes b and b + 2
      const uint32_t even = __byte_perm(p[0], p[2], b ? 0x7351 : 0x6240);  // rows 0, 2, 4, 6
      const uint32_t odd = __byte_perm(p[1], p[3], b ? 0x7351 : 0x6240);   // rows 1, 3, 5, 7
      col[4 * h + 2 * b] = (even & 0x0F0F0F0Fu) | ((odd << 4) & 0xF0F0F0F0u);
      col[4 * h + 2 * b + 1] = ((even >> 4) & 0x0F0F0F0Fu) | (odd & 0xF0F0F0F0u);
    }
  }
}

}  // namespace nvfp4
