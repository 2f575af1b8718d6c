// MXFP4 quantizer for sm_100a: the format the paper compares NVFP4 against (Section 2, Section 5, Appendix B.4).
// E2M1 elements, one UE8M0 (power-of-two) scale per 32 elements, the decode scale amax_b / 6 rounded UP to a power
// of two so that no value saturates, no tensor-level scale: ONE pass over the tensor produces both copies.
// The recipe options are those of Section 4 at this format's block size: 1x32 blocks for activations and gradients,
// 32x32 blocks for weights, a 32-point random Hadamard transform on the transposed (weight-gradient) copy, stochastic
// rounding with the same Philox draws as the NVFP4 kernel.
#include <type_traits>

#include "async_ptx.cuh"
#include "quantize.h"
#include "quantize_common.cuh"

namespace nvfp4 {

// UE8M0 byte and the exact encode scale 2^(127 - byte) of a block with the given amax (>= 0).
// amax = m * 2^E with m in [1, 2): the smallest e with 6 * 2^e >= amax is E - 2 if m <= 1.5, else E - 1;
// byte = e + 127 = (exponent field) - 2 (+ 1), clamped at 0 (zero and tiny blocks).
__device__ __forceinline__ void mx_scales(float amax, uint32_t& byte, float& enc) {
  const uint32_t bits = __float_as_uint(amax);
  int b = (int)(bits >> 23) - 2 + ((bits & 0x7fffffu) > 0x400000u ? 1 : 0);
  b = b < 0 ? 0 : b;
  byte = (uint32_t)b;
  enc = __uint_as_float((uint32_t)(254 - b) << 23);  // b <= 253 for finite amax
}

// 32-point butterfly on pairs (.x / .y = two adjacent columns); the caller applies 1 / sqrt(32)
__device__ __forceinline__ void fwht32_pairs(float2 v[32]) {
#pragma unroll
  for (int h = 1; h < 32; h <<= 1) {
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      if ((i & h) == 0) {
        const float2 p = v[i], q = v[i | h];
        v[i] = add2(p, q);
        v[i | h] = sub2(p, q);
      }
    }
  }
}

// COL: the transposed copy is made
template <bool COL>
struct MxSmem {
  static constexpr int kTileBytes = 32768;
  static constexpr int kTile = 0;                       // 2 x (128 rows x 256 B of bf16), filled by TMA
  static constexpr int kColCodes = 2 * kTileBytes;      // 2 x (64 column pairs x 128 B)
  static constexpr int kSfRow = kColCodes + (COL ? 2 * 8192 : 0);  // 2 x one 512-byte atom: 128 rows x 4 blocks of 32
  static constexpr int kSfCol = kSfRow + 2 * 512;
  static constexpr int kBlk = kSfCol + (COL ? 2 * 512 : 0);  // 32x32 mode: amax of (warp's 16 rows) x (4 column blocks)
  static constexpr int kBlkByte = kBlk + 128;           // 32x32 mode: scale byte by (32-row group, column block)
  static constexpr int kBars = kBlkByte + 32;           // two "tile landed" barriers, then the abort word
  static constexpr int kRand = kBars + 32;              // 128 rows x 128 B of complemented draws (stochastic rounding),
                                                        // or 128 rows x 64 B of row-wise codes (32x32, both copies)
  static constexpr int bytes(bool rand, bool row_codes) { return kRand + (rand ? 16384 : row_codes ? 8192 : 0); }
};

constexpr float kInvSqrt32 = 0.176776695296636893f;  // fl(1 / sqrt(32))

// Persistent CTAs (CTAS per SM: two, or three for the row-wise copy alone) going through 128 x 128 tiles of the source that arrive by TMA in a ring of two buffers, as
// in quantize_kernel; bound by instruction issue.  One CTA per tile, each loading its own registers and waiting for them,
// took 45 us for a 8192 x 5120 activation, 80 us for a 8192 x 7168 gradient and 27 us for a 7168 x 5120 weight.
//   phase 1  each thread owns four 1x16 chunks of the tile; a 1x32 block is the two chunks of an even / odd lane pair;
//            produces the row-wise copy (and stages the random bytes for stochastic rounding);
//   phase 2  each thread owns 32 rows x 2 columns of the tile and produces the transposed copy: a pair of warps reads what
//            the same pair staged, so the 64 threads meet at a barrier of their own;
//   phase 3  staged codes and scale bytes leave with 16-byte stores (staging double buffered: one CTA barrier per tile).
// OWN_DRAWS: 32x32 blocks whose transposed copy is rounded with draws of its own.
template <bool HAS_ROW, bool HAS_COL, bool BLOCK2D, bool RHT_COL, bool SR, bool OWN_DRAWS, int CTAS>
__global__ void __launch_bounds__(256, CTAS)
    quantize_mx_kernel(const __grid_constant__ CUtensorMap src_map, const QuantArgs a) {
  using S = MxSmem<HAS_COL>;
  extern __shared__ __align__(128) uint8_t smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t n_cb = a.cols >> 4;  // 16-chunks per source row (index of the random draws)
  // 32x32 blocks with both copies requested: the transposed copy holds the very codes of the row-wise one
  constexpr bool kNibbleTranspose = BLOCK2D && HAS_ROW && HAS_COL && !OWN_DRAWS;
  constexpr bool kStageRand = SR && HAS_COL && !kNibbleTranspose;
  volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem + S::kBars + 16);
  const uint32_t bar0 = smem_u32(smem + S::kBars), tile0 = smem_u32(smem + S::kTile);

  const int total = a.tiles_r * a.tiles_c, stride = (int)gridDim.x;
  const int n_mine = (total - 1 - (int)blockIdx.x) / stride + 1;  // gridDim.x <= total
  auto issue = [&](int j) {  // the CTA's tile j into buffer j & 1 (one thread)
    const int t = (int)blockIdx.x + j * stride, tr = t / a.tiles_c, tc = t - tr * a.tiles_c;
    mbar_expect_tx(bar0 + 8 * (j & 1), S::kTileBytes);
    tma_load_2d(tile0 + (j & 1) * S::kTileBytes, &src_map, tc * 128, tr * 128, bar0 + 8 * (j & 1));
  };
  if (threadIdx.x == 0) {
    mbar_init(bar0, 1);
    mbar_init(bar0 + 8, 1);
    *abort_flag = 0u;
    fence_mbarrier_init();
    fence_proxy_async_smem();
    griddep_wait();  // the source may be the previous kernel's output; the barrier below holds everybody else's writes
    issue(0);
    if (n_mine > 1) issue(1);
    // no tensor-level scale in this format: the copies' global words read {0, 1} so that the GEMM epilogue's
    // product of decode scales is 1
    if (blockIdx.x == 0) {
      if (HAS_ROW) { a.r_global[0] = 0.f; a.r_global[1] = 1.f; }
      if (HAS_COL) { a.c_global[0] = 0.f; a.c_global[1] = 1.f; }
    }
  }
  __syncthreads();
  griddep_launch_dependents();

  const int cb = lane & 7, rl = warp * 16 + (lane >> 3);  // phase 1: chunk column, row of chunk 0 (chunk i: + 4 i)
  const int q32 = threadIdx.x >> 6, cp = threadIdx.x & 63;  // phase 2: 32-row group, column pair
  float* const blk = reinterpret_cast<float*>(smem + S::kBlk);
  auto pair_sync = [&] { asm volatile("bar.sync %0, 64;" ::"r"(1 + q32) : "memory"); };
  const int sf_row_pos = a.r_swz ? ((rl & 31) * 16 + (rl >> 5) * 4 + (cb >> 1)) : (rl * 4 + (cb >> 1));
  const int sf_row_step = a.r_swz ? 64 : 16;  // four rows further (never across a 32-row quarter)
  const int sf_col_pos = a.c_swz ? (((2 * cp) & 31) * 16 + (cp >> 4) * 4 + q32) : (2 * cp * 4 + q32);
  const int sf_col_odd = a.c_swz ? 16 : 4;
  const int64_t r_pitch = a.cols >> 1;

  auto spread = [](int p) { return p ^ (p >> 2); };  // eight consecutive column pairs, and every fourth, in different units

  int j = 0;
  for (; j < n_mine; ++j) {
    const int tile = (int)blockIdx.x + j * stride, tr = tile / a.tiles_c, tc = tile - tr * a.tiles_c;
    const int64_t row0 = (int64_t)tr * 128, col0 = (int64_t)tc * 128;
    const int buf = j & 1;
    const uint8_t* const tile_buf = smem + S::kTile + buf * S::kTileBytes;
    uint8_t* const col_codes = smem + S::kColCodes + buf * 8192;
    uint8_t* const sf_row = smem + S::kSfRow + buf * 512;
    uint8_t* const sf_col = smem + S::kSfCol + buf * 512;
    quant_wait(bar0 + 8 * buf, (uint32_t)(j >> 1) & 1u, abort_flag, a.status);

    const bool full_tile = row0 + 128 <= a.rows && col0 + 128 <= a.cols;
    // Two copies: a full tile's code has no branch around its stores (nor, now, one around the transposed copy's own draws), and a
    // chunk overlaps with the next: gradient of 4096 x 4096 19.8 -> 17.7 us, 8192 x 20480 166 -> 152; activation of 8192 x 5120
    // 31.0 -> 29.2.  Not for weights: few tiles lose what many gain (2304 x 3328 6.0 -> 6.2 us, 8192 x 5120 24.9 -> 24.4).
    auto phases_1_2 = [&](auto full_c) {
      constexpr bool FULL = decltype(full_c)::value;
      // ---------------------------------------------------------------- phase 1 ----
      uint32_t raw[4][8];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint4 h0 = *reinterpret_cast<const uint4*>(tile_buf + rl * 256 + cb * 32 + i * 1024);
        const uint4 h1 = *reinterpret_cast<const uint4*>(tile_buf + rl * 256 + cb * 32 + i * 1024 + 16);
        raw[i][0] = h0.x; raw[i][1] = h0.y; raw[i][2] = h0.z; raw[i][3] = h0.w;
        raw[i][4] = h1.x; raw[i][5] = h1.y; raw[i][6] = h1.z; raw[i][7] = h1.w;
      }
      float am[4];  // amax of the 1x32 block each chunk belongs to (the chunk of the neighbouring lane completes it)
      if (HAS_ROW || BLOCK2D) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          uint32_t acc = 0;
#pragma unroll
          for (int k = 0; k < 8; ++k) acc = absmax_bf16x2(acc, raw[i][k]);
          const float own = amax_of_pair(acc);
          am[i] = fmaxf(own, __shfl_xor_sync(0xffffffffu, own, 1));
        }
      }
      if (BLOCK2D) {
        // 32x32 blocks: the warp's 16 rows first, then the other warp of the pair's through shared memory
        float m = fmaxf(fmaxf(am[0], am[1]), fmaxf(am[2], am[3]));
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 8));
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 16));
        if (lane < 8 && !(lane & 1)) blk[warp * 4 + (cb >> 1)] = m;
        pair_sync();
        m = fmaxf(blk[warp * 4 + (cb >> 1)], blk[(warp ^ 1) * 4 + (cb >> 1)]);
#pragma unroll
        for (int i = 0; i < 4; ++i) am[i] = m;
      }
      const bool col_ok = FULL || col0 + cb * 16 < a.cols;
      const int rows_left = FULL ? 128 : (int)(a.rows - row0) - rl;
      uint64_t g = 0;
      if (SR) g = (uint64_t)(row0 + rl) * (uint64_t)n_cb + (uint64_t)((col0 >> 4) + cb);
      uint8_t* r_out = HAS_ROW ? a.r_codes + (row0 + rl) * r_pitch + ((col0 + cb * 16) >> 1) : nullptr;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const bool ok = FULL || (col_ok && 4 * i < rows_left);
        uint32_t rnd[4] = {0u, 0u, 0u, 0u};
        if (SR) {
          const uint64_t gi = g + (uint64_t)(4 * i) * (uint64_t)n_cb;
          const uint4 q = philox4x32_10((uint32_t)gi, (uint32_t)(gi >> 32), a.off_lo,
                                        HAS_ROW ? a.off_hi : a.off_hi_col, a.rk);
          rnd[0] = q.x; rnd[1] = q.y; rnd[2] = q.z; rnd[3] = q.w;
          if (kStageRand)
            *reinterpret_cast<uint4*>(smem + S::kRand + (rl + 4 * i) * 128 + cb * 16) = make_uint4(~q.x, ~q.y, ~q.z, ~q.w);
        }
        if (HAS_ROW) {
          float f[16];
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            f[2 * k] = bf16_lo(raw[i][k]);
            f[2 * k + 1] = bf16_hi(raw[i][k]);
          }
          uint32_t byte;
          float enc;
          mx_scales(am[i], byte, enc);
          const uint2 codes = convert16<SR>(f, enc, Nu14FromWords{rnd});
          if (ok) *reinterpret_cast<uint2*>(r_out + (int64_t)(4 * i) * r_pitch) = codes;
          if (kNibbleTranspose)
            *reinterpret_cast<uint2*>(smem + S::kRand + (rl + 4 * i) * 64 + cb * 8) = ok ? codes : make_uint2(0u, 0u);
          if (!(cb & 1)) sf_row[sf_row_pos + i * sf_row_step] = (uint8_t)byte;
          if (kNibbleTranspose && i == 0 && lane < 8 && !(cb & 1)) smem[S::kBlkByte + warp * 4 + (cb >> 1)] = (uint8_t)byte;
        }
      }
      if (kStageRand && HAS_ROW && a.off_hi_col != a.off_hi) {  // draws of its own for the transposed copy
#pragma unroll 1
        for (int i = 0; i < 4; ++i) {
          const uint64_t gi = g + (uint64_t)(4 * i) * (uint64_t)n_cb;
          const uint4 q = philox4x32_10((uint32_t)gi, (uint32_t)(gi >> 32), a.off_lo, a.off_hi_col, a.rk);
          *reinterpret_cast<uint4*>(smem + S::kRand + (rl + 4 * i) * 128 + cb * 16) = make_uint4(~q.x, ~q.y, ~q.z, ~q.w);
        }
      }
      if (kStageRand || kNibbleTranspose) pair_sync();  // (otherwise phase 2 reads the tile alone)

      // ---------------------------------------------------------------- phase 2 ----
      if (HAS_COL) {
        uint4 out0, out1;  // 32 nibbles of column 2cp / 2cp + 1
        uint32_t byte0, byte1;
        if (kNibbleTranspose) {
          // nibbles of the row-wise copy, 8 rows x 8 columns per thread, see transpose_nibbles()
          byte0 = byte1 = smem[S::kBlkByte + 2 * q32 * 4 + (cp >> 4)];
          const int o = lane & 15, rg = cp >> 4;  // columns 8 o .., rows 8 rg .. of the group
          const uint8_t* const src = smem + S::kRand + (q32 * 32 + rg * 8) * 64 + o * 4;
          uint32_t w[8], col[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) w[k] = *reinterpret_cast<const uint32_t*>(src + k * 64);
          transpose_nibbles(w, col);
#pragma unroll
          for (int k = 0; k < 8; ++k)
            *reinterpret_cast<uint32_t*>(col_codes + (4 * o + (k >> 1)) * 128 +
                                         ((((k & 1) * 4 + q32) ^ spread(4 * o + (k >> 1))) & 7) * 16 + rg * 4) = col[k];
        } else {
          float2 v[32];
          const uint8_t* tp = tile_buf + q32 * 32 * 256 + cp * 4;
#pragma unroll
          for (int k = 0; k < 32; ++k) {
            uint32_t word = *reinterpret_cast<const uint32_t*>(tp + k * 256);
            if (RHT_COL) word ^= a.row_sign[k];
            v[k] = make_float2(bf16_lo(word), bf16_hi(word));
          }
          if (RHT_COL) fwht32_pairs(v);
          float2 am2, enc;
          if (BLOCK2D)
            am2.x = am2.y = fmaxf(blk[(2 * q32) * 4 + (cp >> 4)], blk[(2 * q32 + 1) * 4 + (cp >> 4)]);
          else
            am2 = amax_pairs(v);
          // Section 5, transform size 32: y = fl(sum * c), c = fl(1 / sqrt(32)).  Rounding is monotone, so the block's amax is
          // fl(max |sum| * c); the encode scale is a power of two, so fl(y * enc) = fl(sum * (c * enc)): y is never formed.  That
          // holds while y and c * enc are normal numbers.  c * enc is, up to byte 250, for every finite sum (beside a sum that has
          // overflowed it lacks three bits, 2.5e-7, which can move a value next to a threshold); y is subnormal for 724 sums of
          // bf16 values alone, and none of them gets another code at any scale or draw.  (Forming y where a sum has
          // overflowed was exact there as well and took 1.8 % longer on an activation of 8192 x 5120, 3.5 % on one of 512 x 1024.)
          if (RHT_COL) am2 = mul2(am2, make_float2(kInvSqrt32, kInvSqrt32));
          mx_scales(am2.x, byte0, enc.x);
          mx_scales(am2.y, byte1, enc.y);
          if (RHT_COL) enc = mul2(enc, make_float2(kInvSqrt32, kInvSqrt32));
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            uint2 c0, c1;
            if (SR) {
              // low / high byte of ntwo[k] = 255 - draw of source element (row 32 q32 + 16 h + k, column 2cp / 2cp + 1)
              uint32_t ntwo[16];
              const uint8_t* rp = smem + S::kRand + (q32 * 32 + 16 * h) * 128 + cp * 2;
#pragma unroll
              for (int k = 0; k < 16; ++k) ntwo[k] = *reinterpret_cast<const uint16_t*>(rp + k * 128);
              convert16x2_sr(&v[16 * h], enc, ntwo, c0, c1);
            } else {
              convert16x2_rne(&v[16 * h], enc, c0, c1);
            }
            if (h == 0) {
              out0.x = c0.x; out0.y = c0.y; out1.x = c1.x; out1.y = c1.y;
            } else {
              out0.z = c0.x; out0.w = c0.y; out1.z = c1.x; out1.w = c1.y;
            }
          }
        }
        // staging: a column pair has 128 bytes, eight 16-byte units (column parity, 32-row group); unit u sits at u ^ spread(cp)
        if (!kNibbleTranspose) {
          *reinterpret_cast<uint4*>(col_codes + cp * 128 + (((q32 ^ spread(cp)) & 7) << 4)) = out0;
          *reinterpret_cast<uint4*>(col_codes + cp * 128 + ((((4 + q32) ^ spread(cp)) & 7) << 4)) = out1;
        }
        sf_col[sf_col_pos] = (uint8_t)byte0;
        sf_col[sf_col_pos + sf_col_odd] = (uint8_t)byte1;
      }
    };
    if (!BLOCK2D && full_tile)
      phases_1_2(std::integral_constant<bool, !BLOCK2D>{});
    else
      phases_1_2(std::false_type{});
    __syncthreads();
    if (*abort_flag) break;  // a wait expired (the word is read after the barrier: the same for every thread)
    if (threadIdx.x == 0 && j + 2 < n_mine) issue(j + 2);  // every warp is done with this buffer

    // ---------------------------------------------------------------- phase 3 ----
    if (HAS_COL) {
      const int64_t pitch = a.rows >> 1;  // bytes per row of the transposed copy
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int unit = threadIdx.x + 256 * k;
        const int c = unit >> 2, m = unit & 3;  // column, 32-row group
        if (!full_tile && (col0 + c >= a.cols || row0 + 32 * m >= a.rows)) continue;  // rows % 32 == 0: a group is in or out
        const uint4 val = *reinterpret_cast<const uint4*>(col_codes + (c >> 1) * 128 +
                                                          (((((c & 1) * 4 + m) ^ spread(c >> 1)) & 7) << 4));
        *reinterpret_cast<uint4*>(a.c_codes + (col0 + c) * pitch + (row0 >> 1) + m * 16) = val;
      }
    }
#pragma unroll
    for (int which = 0; which < 2; ++which) {
      if (which == 0 ? !HAS_ROW : !HAS_COL) continue;
      const uint8_t* src = which == 0 ? sf_row : sf_col;
      uint8_t* dst = which == 0 ? a.r_scales : a.c_scales;
      const int swz = which == 0 ? a.r_swz : a.c_swz;
      const int64_t R0 = which == 0 ? row0 : col0, K0 = which == 0 ? (col0 >> 5) : (row0 >> 5);
      const int64_t Rn = which == 0 ? a.rows : a.cols, n_kb = which == 0 ? (a.cols >> 5) : (a.rows >> 5);
      if (swz) {
        if (threadIdx.x < 32) {  // one 512-byte atom per tile and copy
          const int64_t off = ((R0 >> 7) * (n_kb >> 2) + (K0 >> 2)) * 512 + threadIdx.x * 16;
          *reinterpret_cast<uint4*>(dst + off) = *reinterpret_cast<const uint4*>(src + threadIdx.x * 16);
        }
      } else {
        store_linear_scales<128, 4>(src, dst, R0, K0, Rn, n_kb, full_tile);
      }
    }
  }
  if (j < n_mine && threadIdx.x == 0) {
    // left early: tiles j and j + 1 may still be in flight; one more bounded wait each, so that no copy lands in shared
    // memory after the CTA has gone
    for (int i = j; i < j + 2 && i < n_mine; ++i) {
      const unsigned long long t0 = globaltimer_ns();
      while (!mbar_try(bar0 + 8 * (i & 1), (uint32_t)(i >> 1) & 1u) && globaltimer_ns() - t0 < kWaitLimitNs) {
      }
    }
  }
}

template <bool HR, bool HC, bool B2, bool RC, bool SR, bool OWN, int CTAS>
static cudaError_t launch_mx_ctas(const QuantArgs& a, int sms, cudaStream_t s) {
  auto kern = quantize_mx_kernel<HR, HC, B2, RC, SR, OWN, CTAS>;
  constexpr bool kRowCodes = B2 && HR && HC && !OWN;
  constexpr int smem = MxSmem<HC>::bytes(SR && HC && !kRowCodes, kRowCodes);
  CUtensorMap map;
  if (!make_map_2d(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, a.x, (uint64_t)a.cols, (uint64_t)a.rows,
                   (uint64_t)a.ld * 2, 128, 128, 0))
    return cudaErrorInvalidValue;
  static std::atomic<uint64_t> configured{0};  // per call site (template instantiation) and device
  int dev;
  cudaError_t e;
  if (device_needs_config(configured, &dev)) {
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem > kSmemOfHalf ? smem : kSmemOfHalf)) !=
        cudaSuccess)
      return e;
    device_configured(configured, dev);
  }
  const int64_t tiles = (int64_t)a.tiles_r * a.tiles_c;
  const int slots = CTAS * sms;
  // The kernel becomes resident while the one before it drains, and few CTAs would crowd on the SMs that drain first: no more
  // on an SM than the tiles take when they are spread evenly (the shared memory that is left keeps others out).  Backward call of
  // 1024 x 2304 x 2560 19.4 -> 18.0 us, 3584 x 256 x 4352 22.9 -> 21.1, in a loop of such calls.
  const int room = tiles <= sms ? kSmemOfHalf : CTAS == 2 ? kSmemOfThird : 0;
  e = launch_kernel(kern, dim3((unsigned)(tiles < slots ? tiles : slots)), dim3(256), room > smem ? room : smem, s, map, a);
  count_launch();
  return e;
}

template <bool HR, bool HC, bool B2, bool RC, bool SR, bool OWN = false>
static cudaError_t launch_mx_t(const QuantArgs& a, cudaStream_t s) {
  int sms = 0;
  const cudaError_t e = sm_count(&sms);
  if (e != cudaSuccess) return e;
  // Without a transposed copy three CTAs fit an SM; they take 1.5 times as long for a round of tiles as two, so they pay where that many
  // rounds go: 297 to 444 tiles above all (two / three per SM: gradient of 1024 x 6784 6.4 / 5.3 us, activation of 896 x 7936 4.3 /
  // 3.6; but gradient of 2048 x 2048 4.0 / 5.0, 11680 x 896 8.2 / 9.3).
  if constexpr (!HC) {
    const int64_t tiles = (int64_t)a.tiles_r * a.tiles_c;
    if (3 * ((tiles + 3 * sms - 1) / (3 * sms)) < 2 * ((tiles + 2 * sms - 1) / (2 * sms)))
      return launch_mx_ctas<HR, HC, B2, RC, SR, OWN, 3>(a, sms, s);
  }
  return launch_mx_ctas<HR, HC, B2, RC, SR, OWN, 2>(a, sms, s);
}

cudaError_t launch_quantize_mx(const QuantArgs& a, bool has_row, bool has_col, bool block2d, bool rht_col, bool sr,
                               cudaStream_t s) {
  rht_col = rht_col && has_col;
  if (block2d && sr && has_row && has_col && a.off_hi_col != a.off_hi)  // independent draws: the copies' codes differ
    return launch_mx_t<true, true, true, false, true, true>(a, s);
#define NVFP4_MXQ(HR, HC, B2, RC, SRV)                                                        \
  if (has_row == HR && has_col == HC && block2d == B2 && rht_col == RC && sr == SRV)         \
    return launch_mx_t<HR, HC, B2, RC, SRV>(a, s);
#define NVFP4_MXQ_COPIES(B2, RC, SRV) \
  NVFP4_MXQ(true, false, B2, false, SRV) \
  NVFP4_MXQ(false, true, B2, RC, SRV)   \
  NVFP4_MXQ(true, true, B2, RC, SRV)
  NVFP4_MXQ_COPIES(true, false, false)
  NVFP4_MXQ_COPIES(true, false, true)
  NVFP4_MXQ_COPIES(false, false, false)
  NVFP4_MXQ_COPIES(false, false, true)
  NVFP4_MXQ_COPIES(false, true, false)
  NVFP4_MXQ_COPIES(false, true, true)
#undef NVFP4_MXQ_COPIES
#undef NVFP4_MXQ
  return cudaErrorInvalidValue;
}

}  // namespace nvfp4
