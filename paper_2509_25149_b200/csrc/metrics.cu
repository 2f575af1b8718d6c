// Quantization-error reductions (Appendix E.2 of the paper: error metrics as a way to decide which linear layers
// stay in higher precision).  Two HBM-bound kernels:
//   quant_error_kernel : sum (x - decode(q))^2 and sum x^2 of a row-wise quantized copy against its bf16 source,
//                        decoding on the fly (2 + 0.5 + 1/16 bytes per element);
//   sq_error_kernel    : the same two sums between two dense tensors (bf16 or fp32 each), e.g. a weight gradient
//                        from the FP4 GEMM against the one from the BF16 GEMM.
// A thread sums 16 elements in FP32 and adds that into an FP64 partial; warps and CTAs are combined in FP64 and
// leave through one atomicAdd pair per CTA.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "async_ptx.cuh"
#include "common.cuh"
#include "quantize.h"
#include "quantize_common.cuh"

namespace nvfp4 {

namespace {

// CTAs of 16 warps, two per SM: a quarter of the FP64 atomics on the two sums that CTAs of eight at eight per SM took
constexpr int kWarps = 16, kThreads = 32 * kWarps;

__device__ __forceinline__ void block_reduce_add(double err, double ref, double* out) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    err += __shfl_xor_sync(0xffffffffu, err, o);
    ref += __shfl_xor_sync(0xffffffffu, ref, o);
  }
  __shared__ double red[2][kWarps];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    red[0][warp] = err;
    red[1][warp] = ref;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    griddep_wait();  // the sums are zero
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) s += red[threadIdx.x][w];
    atomicAdd(out + threadIdx.x, s);
  }
}

// Walks a thread through units first, first + step, ... of a [rows x n] array: coordinates move by additions (a division
// per 16 elements cost a sixth of the instructions).
struct Walk {
  int64_t r, dr, c, dc, n;
  __device__ __forceinline__ Walk(int64_t first, int64_t step, int64_t n_) : n(n_) {
    r = first / n;
    c = first - r * n;
    dr = step / n;
    dc = step - dr * n;
  }
  __device__ __forceinline__ void next() {
    r += dr;
    c += dc;
    if (c >= n) {
      c -= n;
      ++r;
    }
  }
};

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 r;
  asm("{.reg .b64 ra, rb, rc, rd; mov.b64 ra, {%2, %3}; mov.b64 rb, {%4, %5}; mov.b64 rc, {%6, %7}; "
      "fma.rn.f32x2 rd, ra, rb, rc; mov.b64 {%0, %1}, rd;}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return r;
}

// one byte of codes -> its two E2M1 values (low nibble first)
__device__ __forceinline__ float2 e2m1x2_values(uint32_t byte) {
  uint32_t h2;
  asm("{\n\t.reg .b8 lo, hi;\n\t"
      "mov.b16 {lo, hi}, %1;\n\t"
      "cvt.rn.f16x2.e2m1x2 %0, lo;\n\t}"
      : "=r"(h2)
      : "h"((uint16_t)byte));
  return __half22float2(*reinterpret_cast<__half2*>(&h2));
}

template <bool MX>
__global__ void __launch_bounds__(kThreads, 2) quant_error_kernel(const uint16_t* __restrict__ x, int64_t rows, int64_t cols,
                                                          int64_t ld, const uint8_t* __restrict__ codes,
                                                          const uint8_t* __restrict__ scales,
                                                          const float* __restrict__ global, int swz,
                                                          int per_row, double* __restrict__ out) {
  const int64_t n_cb = cols >> 4;                 // 16-element chunks per row
  const int64_t n_sb = MX ? (cols >> 5) : n_cb;   // scale blocks per row
  const float s_dec_t = MX ? 1.f : global[1];
  double err = 0.0, ref = 0.0;
  const int64_t first = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
  Walk w(first, step, n_cb);
  constexpr int kDepth = 2;  // chunks whose loads are in flight
  uint32_t raw[kDepth][8] = {};
  uint2 codes2[kDepth] = {};
  uint32_t byte[kDepth] = {};
  float s_dec[kDepth] = {};
  auto load = [&](int u) {
    if (w.r < rows) {
      const int64_t r = w.r, cb = w.c, sb = MX ? (cb >> 1) : cb;
      ldg256_stream(x + r * ld + cb * 16, raw[u]);
      codes2[u] = __ldg(reinterpret_cast<const uint2*>(codes + r * (cols >> 1) + cb * 8));
      byte[u] = __ldg(scales + (swz ? sf_swizzled_offset(r, sb, n_sb) : (r * n_sb + sb)));
      s_dec[u] = per_row ? __ldg(global + 2 * r + 1) : s_dec_t;  // per_row: {amax, s_dec} per row
    }
    w.next();
  };
  auto add = [&](int u) {
    float sf;
    if (MX) {
      sf = byte[u] == 0 ? __uint_as_float(0x00400000u) : __uint_as_float(byte[u] << 23);  // 2^(byte - 127)
    } else {
      uint32_t h2;
      asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"((uint16_t)byte[u]));
      sf = __half2float(__ushort_as_half((unsigned short)(h2 & 0xffffu)));
    }
    const float neg = -__fmul_rn(sf, s_dec[u]);
    float2 e = make_float2(0.f, 0.f), n = e;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float2 q = e2m1x2_values(((k < 4 ? codes2[u].x : codes2[u].y) >> (8 * (k & 3))) & 0xffu);
      const float2 xv = make_float2(bf16_lo(raw[u][k]), bf16_hi(raw[u][k]));
      const float2 d = fma2(q, make_float2(neg, neg), xv);
      e = fma2(d, d, e);
      n = fma2(xv, xv, n);
    }
    err += (double)(e.x + e.y);
    ref += (double)(n.x + n.y);
  };
  const int64_t units = rows * n_cb;
  int64_t left = first < units ? (units - first + step - 1) / step : 0;  // chunks of this thread
#pragma unroll
  for (int u = 0; u < kDepth; ++u) load(u);
  // Two chunks a turn without a branch between them, so that they overlap (three, each in a branch of its own: 8192 x 5120 20.5
  // us, now 19.3; 20480 x 5120 52.5, now 49.3)
  for (; left > 1; left -= 2) {
    add(0);
    load(0);  // the slot's next chunk, while the other's is worked on
    add(1);
    load(1);
  }
  if (left > 0) add(0);
  block_reduce_add(err, ref, out);
}

template <bool FP32>
__device__ __forceinline__ void load8(const void* base, int64_t elem, float (&v)[8]) {
  if (FP32) {
    const float4* p = reinterpret_cast<const float4*>(static_cast<const float*>(base) + elem);
    const float4 a = __ldg(p), b = __ldg(p + 1);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  } else {
    const uint4 a = ldg128_stream(static_cast<const uint16_t*>(base) + elem);
    v[0] = bf16_lo(a.x); v[1] = bf16_hi(a.x); v[2] = bf16_lo(a.y); v[3] = bf16_hi(a.y);
    v[4] = bf16_lo(a.z); v[5] = bf16_hi(a.z); v[6] = bf16_lo(a.w); v[7] = bf16_hi(a.w);
  }
}

template <bool REF32, bool TEST32>
__global__ void __launch_bounds__(kThreads, 2) sq_error_kernel(const void* __restrict__ refp, int64_t ld_ref,
                                                       const void* __restrict__ testp, int64_t ld_test, int64_t rows,
                                                       int64_t cols, double* __restrict__ out) {
  Walk w(blockIdx.x * (int64_t)blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x, cols >> 3);  // units of 8
  double err = 0.0, ref = 0.0;
  constexpr int kDepth = 2;  // units whose loads are in flight together
  float a[kDepth][8], b[kDepth][8];
  bool live[kDepth];
  while (w.r < rows) {
#pragma unroll
    for (int u = 0; u < kDepth; ++u) {
      live[u] = w.r < rows;
      if (live[u]) {
        load8<REF32>(refp, w.r * ld_ref + w.c * 8, a[u]);
        load8<TEST32>(testp, w.r * ld_test + w.c * 8, b[u]);
      }
      w.next();
    }
#pragma unroll
    for (int u = 0; u < kDepth; ++u) {
      if (!live[u]) continue;
      float e = 0.f, n = 0.f;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const float d = a[u][k] - b[u][k];
        e = fmaf(d, d, e);
        n = fmaf(a[u][k], a[u][k], n);
      }
      err += (double)e;
      ref += (double)n;
    }
  }
  block_reduce_add(err, ref, out);
}

cudaError_t grid_for(int64_t units, unsigned* grid) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int64_t want = (units + kThreads - 1) / kThreads, cap = (int64_t)sms * 2;  // resident CTAs
  *grid = (unsigned)(want < cap ? (want > 0 ? want : 1) : cap);
  return cudaSuccess;
}

cudaError_t zero_sums(double* out, cudaStream_t s) {  // the kernel behind it reads its tensors meanwhile
  float* w = reinterpret_cast<float*>(out);
  return launch_zero_words(w, w + 1, w + 2, w + 3, s);
}

}  // namespace

cudaError_t launch_quant_error(const void* x, int64_t rows, int64_t cols, int64_t ld, const nvfp4_tensor& q,
                               double* out, cudaStream_t s) {
  cudaError_t e = zero_sums(out, s);
  if (e != cudaSuccess) return e;
  unsigned grid;
  if ((e = grid_for(rows * (cols >> 4), &grid)) != cudaSuccess) return e;
  const int swz = q.sf_layout == NVFP4_SF_SWIZZLED;
  e = launch_kernel(q.format == NVFP4_FORMAT_MXFP4 ? quant_error_kernel<true> : quant_error_kernel<false>, dim3(grid),
                    dim3(kThreads), 0, s, static_cast<const uint16_t*>(x), rows, cols, ld, q.codes, q.scales, q.global, swz,
                    q.format == NVFP4_FORMAT_NVFP4_ROWSCALE, out);
  count_launch();
  return e;
}

cudaError_t launch_sq_error(const void* ref, bool ref_fp32, int64_t ld_ref, const void* test, bool test_fp32,
                            int64_t ld_test, int64_t rows, int64_t cols, double* out, cudaStream_t s) {
  cudaError_t e = zero_sums(out, s);
  if (e != cudaSuccess) return e;
  unsigned grid;
  if ((e = grid_for(rows * (cols >> 3), &grid)) != cudaSuccess) return e;
  auto kern = ref_fp32 ? (test_fp32 ? sq_error_kernel<true, true> : sq_error_kernel<true, false>)
                       : (test_fp32 ? sq_error_kernel<false, true> : sq_error_kernel<false, false>);
  e = launch_kernel(kern, dim3(grid), dim3(kThreads), 0, s, ref, ld_ref, test, ld_test, rows, cols, out);
  count_launch();
  return e;
}

}  // namespace nvfp4
