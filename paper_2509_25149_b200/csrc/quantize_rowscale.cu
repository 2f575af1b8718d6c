// Single-pass NVFP4 quantizer with the FP32 "global" scale taken per ROW instead of per tensor (the closing remark of
// Appendix B.1: a global scale spanning a row or a block of elements avoids the extra trip through device memory
// that the tensor amax costs).  Row-wise copy only: a scale per row of the copy is constant along the contraction
// dimension, so the GEMM can apply it in its epilogue as a vector; the transposed copy of the same tensor would need
// a statistic over all source rows, i.e. the pass this variant exists to remove.
//
// CTAs of four warps.  A row of up to 20480 elements is held in the registers of one, two or four warps between the amax
// step and the encoding (two, five or ten 16-element chunks per lane); the warps of a row exchange their partial maxima
// through shared memory: one read from HBM in every case.  Longer rows are read a second
// time (from L1 / L2).  Eq. 1 per row, Eq. 2-4 as in the main quantizer; stochastic-rounding draws are keyed by the
// element's position in the source, as everywhere.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "async_ptx.cuh"
#include "common.cuh"
#include "quantize.h"
#include "quantize_common.cuh"

namespace nvfp4 {

namespace {

// Coherent loads that allocate in L1.  They are no volatile statements, so that the compiler may take them ahead of the code before
// them; what keeps them behind griddep_wait() is their address, which behind_wait() makes known only there.  (Volatile ones: rows of 20608, 512
// of them 34.1 us by the side of 27.0, 4096 71.0 / 70.4; __ldg, which may be moved ahead of the wait, 28.8 / 69.0.)
__device__ __forceinline__ void ld256_cached(const void* p, uint32_t (&r)[8]) {
  asm("ld.global.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "l"(p));
  asm("ld.global.v4.b32 {%0,%1,%2,%3}, [%4 + 16];" : "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "l"(p));
}
__device__ __forceinline__ const uint16_t* behind_wait(const uint16_t* p) {
  asm volatile("" : "+l"(p)::"memory");
  return p;
}

// TABLE: encode scale by E4M3 byte, for a row whose s_enc is at most kPlainDivisionLimit; ok: the chunk exists
template <bool SR, bool TABLE = false>
__device__ __forceinline__ void encode_chunk(const QuantArgs& a, const uint32_t (&raw)[8], int64_t row, int64_t cb, int64_t n_cb,
                                             float s_enc, float s_dec, const float* table = nullptr, bool ok = true) {
  uint32_t acc = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) acc = absmax_bf16x2(acc, raw[k]);
  uint32_t byte;
  float enc;
  if (TABLE) {
    byte = block_scale_byte<false>(amax_of_pair(acc), s_enc);
    enc = table[byte];
  } else {
    block_scales(amax_of_pair(acc), s_enc, s_dec, byte, enc);
  }
  float f[16];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    f[2 * k] = bf16_lo(raw[k]);
    f[2 * k + 1] = bf16_hi(raw[k]);
  }
  uint32_t rnd[4] = {0u, 0u, 0u, 0u};
  if (SR) {
    const uint64_t g = (uint64_t)row * (uint64_t)n_cb + (uint64_t)cb;
    const uint4 q = philox4x32_10((uint32_t)g, (uint32_t)(g >> 32), a.off_lo, a.off_hi, a.rk);
    rnd[0] = q.x; rnd[1] = q.y; rnd[2] = q.z; rnd[3] = q.w;
  }
  const uint2 codes = convert16<SR>(f, enc, Nu14FromWords{rnd});
  if (!ok) return;
  *reinterpret_cast<uint2*>(a.r_codes + row * (a.cols >> 1) + cb * 8) = codes;
  a.r_scales[a.r_swz ? sf_swizzled_offset(row, cb, n_cb) : (row * n_cb + cb)] = (uint8_t)byte;
}

// CTAs resident per SM by what a lane keeps (registers).  Eight with five chunks: 64 registers, and with one or two warps a row 8 to 24
// bytes of a thread spill; six: 71 to 78 and none.  Six / eight, sources in turn that exceed L2: 16384 x 2064 16.7 / 16.0 us, 16384 x 5120
// 37.1 / 35.6, 16384 x 7168 54.7 / 52.1, 8192 x 10240 36.1 / 34.8, with stochastic rounding 25.7 / 25.5, 53.4 / 52.3, 80.9 / 76.3, 52.6 /
// 51.2.  Six would be faster where 1024 CTAs all fit at once but not evenly: 4096 x 2560 7.1 / 7.7, 1024 x 10240 6.8 / 7.5, with
// stochastic rounding 10.0 / 10.7 and 10.2 / 10.7, behind a product 16.4 / 16.6 and 19.4 / 19.9.
constexpr int ctas_per_sm(int keep) { return keep <= 5 ? 8 : 4; }

// WPR warps per row (1, 2 or 4): row (4 / WPR) * i + w / WPR of iteration i belongs to warp w, whose lanes take every WPR-th
// group of 32 chunks, so that a row of any length is spread evenly.
template <bool SR, int WPR, int kKeep>
__global__ void __launch_bounds__(128, ctas_per_sm(kKeep)) quantize_rowscale_kernel(const QuantArgs a) {
  __shared__ float part[2][4];  // partial maxima, double-buffered across iterations
  // A warp with ten chunks a lane (rows of more than 10240 elements) makes a table of the 127 encode scales of its row first: a
  // reciprocal for each of four entries a lane instead of each of its chunks, and the chunks' code has no branch (neither a
  // reciprocal's nor a division's), so that chunks overlap: 8192 x 20480 83.7 -> 74.0 us.  With five chunks a lane 16384 x 5120
  // stayed at 41 us and 1024 x 7168 went from 6.2 to 8.2; with stochastic rounding the registers do not suffice.
  constexpr bool kTable = kKeep >= 10 && !SR;
  __shared__ float tables[kTable ? 4 : 1][128];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int kRowsPerCta = 4 / WPR;
  const int seg = warp % WPR, sub = warp / WPR;
  const int64_t n_cb = a.cols >> 4;
  griddep_wait();
  griddep_launch_dependents();
  int it = 0;
  // every warp of a CTA runs the same number of iterations (rows are padded), so the barriers below are uniform
  for (int64_t base = (int64_t)blockIdx.x * kRowsPerCta; base < a.rows; base += (int64_t)gridDim.x * kRowsPerCta, ++it) {
    const int64_t row = base + sub;
    const bool live = row < a.rows;
    const uint16_t* src = a.x + (live ? row : 0) * a.ld;
    uint32_t keep[kKeep][8];
    uint32_t acc = 0;
#pragma unroll
    for (int i = 0; i < kKeep; ++i) {
      const int64_t cb = lane + 32 * (seg + WPR * i);
      if (live && cb < n_cb) {
        ldg256_stream(src + cb * 16, keep[i]);
      } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) keep[i][k] = 0u;
      }
    }
#pragma unroll
    for (int i = 0; i < kKeep; ++i)
#pragma unroll
      for (int k = 0; k < 8; ++k) acc = absmax_bf16x2(acc, keep[i][k]);
    float amax = warp_max(amax_of_pair(acc));
    if (WPR > 1) {
      if (lane == 0) part[it & 1][warp] = amax;
      __syncthreads();
#pragma unroll
      for (int w = 0; w < WPR; ++w) amax = fmaxf(amax, part[it & 1][sub * WPR + w]);
    }
    float s_enc, s_dec;
    global_scales(amax, s_enc, s_dec);  // Eq. 1 with the row's amax
    if (live && seg == 0 && lane == 0) {
      a.r_global[2 * row] = amax;
      a.r_global[2 * row + 1] = s_dec;
    }
    if (kTable && s_enc <= kPlainDivisionLimit) {
      float* const table = tables[kTable ? warp : 0];
      __syncwarp();  // (the row before is encoded)
#pragma unroll
      for (int k = 0; k < 4; ++k) table[lane + 32 * k] = encode_scale_of_byte(lane + 32 * k, s_dec);
      __syncwarp();
#pragma unroll
      for (int i = 0; i < kKeep; i += 2) {
        if (!live || 32 * (seg + WPR * i) >= n_cb) break;  // the same for the whole warp
#pragma unroll
        for (int k = i; k < i + 2 && k < kKeep; ++k) {
          const int64_t cb = lane + 32 * (seg + WPR * k);
          encode_chunk<SR, true>(a, keep[k], row, cb, n_cb, s_enc, s_dec, table, cb < n_cb);
        }
      }
    } else if (live) {
#pragma unroll
      for (int i = 0; i < kKeep; ++i) {
        const int64_t cb = lane + 32 * (seg + WPR * i);
        if (cb < n_cb) encode_chunk<SR>(a, keep[i], row, cb, n_cb, s_enc, s_dec);
      }
    }
  }
}

// rows longer than 4 * 5120 elements: one warp per row, two sweeps (the second one from L1 / L2)
template <bool SR>
__global__ void __launch_bounds__(256) quantize_rowscale_long_kernel(const QuantArgs a) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t n_cb = a.cols >> 4;
  griddep_wait();
  const uint16_t* const x = behind_wait(a.x);
  griddep_launch_dependents();
  for (int64_t row = (int64_t)blockIdx.x * 8 + warp; row < a.rows; row += (int64_t)gridDim.x * 8) {
    const uint16_t* src = x + row * a.ld;
    uint32_t acc = 0;
    for (int64_t cb0 = 0; cb0 < n_cb; cb0 += 128) {  // four independent loads per lane in flight
      uint32_t raw[4][8];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int64_t cb = cb0 + lane + 32 * u;
        if (cb < n_cb) {
          ld256_cached(src + cb * 16, raw[u]);  // allocate in L1: the second sweep comes back for it
        } else {
#pragma unroll
          for (int k = 0; k < 8; ++k) raw[u][k] = 0u;
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int k = 0; k < 8; ++k) acc = absmax_bf16x2(acc, raw[u][k]);
    }
    const float amax = warp_max(amax_of_pair(acc));
    float s_enc, s_dec;
    global_scales(amax, s_enc, s_dec);
    if (lane == 0) {
      a.r_global[2 * row] = amax;
      a.r_global[2 * row + 1] = s_dec;
    }
    for (int64_t cb0 = 0; cb0 < n_cb; cb0 += 64) {
      uint32_t raw[2][8];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int64_t cb = cb0 + lane + 32 * u;
        if (cb < n_cb) ld256_cached(src + cb * 16, raw[u]);
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int64_t cb = cb0 + lane + 32 * u;
        if (cb < n_cb) encode_chunk<SR>(a, raw[u], row, cb, n_cb, s_enc, s_dec);
      }
    }
  }
}

// Programmatic launch: behind an ordinary one the next kernel begins on a grid of 2.05 us.  Without an ordinary launch's pause, though, the
// SMs stay divided the way the kernel before wanted them, nearly all shared memory behind a product, and the loads in flight do not fit
// what is left as L1; so the kernel asks for 7 % of the SM as shared memory (15 % and more do not make an SM change, and with none at all
// rows of 20480, whose CTAs have 3 KB, lose 40 %).  Sources in turn that exceed L2, ordinary / programmatic / that with the division, all
// with eight CTAs: copies of 8192 x 1536 10.3 / 8.6 / 8.6 us, 16384 x 2560 20.5 / 18.8 / 18.8, 16384 x 5120 37.0 / 35.7 / 35.9; forward
// calls of 16384 x 1024 x 5120 82.2 to 84.2 / 94.8 to 97.9 / 80.5 to 82.6, 4096 x 4096 x 4096 47.1 / 49.0 / 45.2, 16384 x 5120 x 5120
// 231 / 251 / 230 (two runs of one build differ by 1 %).
//
// Few CTAs crowd that way: they become resident while a product still runs, as many as fit an SM on each that has none of its tiles.  So
// up to four CTAs per SM have a share of 16 KB each as shared memory, and no more of them fit an SM than an even spread puts there.  Behind
// a product of 64 tiles, ordinary / crowded / spread: 512 x 20608 39.6 / 51.2 / 36.7 us, 512 x 5120 14.4 / 15.1 / 12.5, with stochastic
// rounding 44.4 / 73.6 / 39.1 and 14.4 / 18.0 / 13.4; forward of 256 x 1024 x 24576 with a fresh weight 65.1 / 86.2 / 61.3, of 1024 x 2048
// x 2048 10.3 / 10.4 / 9.3.  For this the kernel asks for 5 %: CTAs of 3.5 KB and more then meet an SM divided at 16 KB; with 7 % most
// sizes meet 32 KB (seen by how many were resident: of 4 KB eight).  From five CTAs per SM on the even shares would be below that; there
// nothing lost against an ordinary launch of six (1024 x 7168 to 20480 x 5120, alone and behind a product 1.5 to 35 % faster).
constexpr int kSpreadCarveout = 5, kSpreadBytes = 16384, kSpreadCtas = 4;

template <typename Kernel>
cudaError_t launch_spread(Kernel kern, int64_t want, int64_t cap, int threads, int static_smem, const QuantArgs& a, int sms, cudaStream_t s) {
  const int64_t per_sm = (want + sms - 1) / sms;
  const bool few = per_sm <= kSpreadCtas;
  const size_t smem = few ? (size_t)((kSpreadBytes / per_sm) & ~127) - (size_t)static_smem - 1024 : 0;  // (1 KB a CTA is the system's)
  return launch_divided(few ? kSpreadCarveout : kStreamingCarveout, kern, dim3((unsigned)(want < cap ? want : cap)), dim3((unsigned)threads),
                        smem, s, a);
}

template <bool SR, int WPR, int KEEP>
cudaError_t launch_kept(const QuantArgs& a, int sms, cudaStream_t s) {
  const int64_t want = (a.rows * WPR + 3) / 4, cap = (int64_t)sms * ctas_per_sm(KEEP) * 4;  // up to four rounds of CTAs
  return launch_spread(quantize_rowscale_kernel<SR, WPR, KEEP>, want, cap, 128, KEEP >= 10 && !SR ? 2176 : 128, a, sms, s);
}

template <bool SR>
cudaError_t launch_t(const QuantArgs& a, int sms, cudaStream_t s) {
  // The fewest registers per lane that hold the row: more warps per SM are more bytes in flight.  Ten chunks per lane for
  // every row up to 5120 elements left rows of 1024 waiting (16384 rows: 18.7 -> 10.8 us); 2560 15.7 -> 12.0 us (8192 rows),
  // 5120 39.6 -> 37.9 us (16384 rows).  A row that fits one warp with five chunks does not gain from a second one (15.1 us).
  const int64_t chunks = a.cols >> 4;
  if (chunks <= 32 * 2) return launch_kept<SR, 1, 2>(a, sms, s);
  if (chunks <= 32 * 4) return launch_kept<SR, 2, 2>(a, sms, s);
  if (chunks <= 32 * 5) return launch_kept<SR, 1, 5>(a, sms, s);
  if (chunks <= 32 * 10) return launch_kept<SR, 2, 5>(a, sms, s);
  if (chunks <= 32 * 20) return launch_kept<SR, 4, 5>(a, sms, s);
  if (chunks <= 32 * 40) return launch_kept<SR, 4, 10>(a, sms, s);
  return launch_spread(quantize_rowscale_long_kernel<SR>, (a.rows + 7) / 8, (int64_t)sms * 6, 256, 0, a, sms, s);
}

}  // namespace

cudaError_t launch_quantize_rowscale(const QuantArgs& a, bool sr, cudaStream_t s) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  e = sr ? launch_t<true>(a, sms, s) : launch_t<false>(a, sms, s);
  count_launch();
  return e;
}

}  // namespace nvfp4
