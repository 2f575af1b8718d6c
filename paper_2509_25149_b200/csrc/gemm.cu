// Block-scaled NVFP4 GEMM for sm_100a: D[M x N] = alpha * A[M x K] * B[N x K]^T  (Eq. 5 of the paper:
// per 16-element block partial dot products times the two E4M3 block scales, accumulated in FP32;
// alpha = s_dec^A * s_dec^B applied once on the result).
//
// Persistent, warp-specialised kernel, one CTA per SM:
//   warp 0   producer: TMA loads of the code tiles (128-byte swizzle) and bulk copies of the scale atoms
//   warp 1   MMA issuer: tcgen05.mma kind::mxf4nvf4.block_scale.scale_vec::4X (M 128, N = BN, K 64 per
//            instruction), accumulator in tensor memory
//   warp 2   scale-atom copier: tcgen05.cp of the E4M3 atoms shared -> tensor memory (its own warp because
//            instruction issue by a single thread, not the tensor pipe, was the bottleneck with both in one)
//   warps 3-6 epilogue: tcgen05.ld of the FP32 accumulator, alpha, conversion, global stores
// Every wait is bounded: when one expires the kernel records a code in a device status word, every role
// leaves its loop, tensor memory is released and the kernel returns.
//
// This file holds the one-CTA kernel (for odd multiples of 128, see one_cta_time, and on request), the tensor-map helpers and the
// launchers of all kernels; the CTA-pair kernels that take every shape are in gemm_2cta.cuh and gemm_wide.cuh.
#include <cuda.h>
#include <cuda_bf16.h>

#include "common.cuh"
#include <algorithm>
#include <vector>

#include "gemm.h"
#include "tc_ptx.cuh"
#include "tile_memo.h"
#include "gemm_2cta.cuh"
#include "gemm_wide.cuh"
#include "gemm_bf16.cuh"

namespace nvfp4 {

EncodeTiledFn tensor_map_encoder() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return nullptr;
    fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// Encoding a tensor map is pure host arithmetic in the driver (about a microsecond each, three to eight per GEMM
// launch): the result depends only on the arguments, so a small per-thread cache keyed by them returns repeats (the
// same buffers launch after launch, as in a training loop) without the call.
bool make_map_2d(CUtensorMap* map, CUtensorMapDataType dtype, int elem_bytes, const void* base, uint64_t inner_elems,
                 uint64_t rows, uint64_t row_pitch_bytes, uint32_t box_inner, uint32_t box_rows, int swizzle) {
  (void)elem_bytes;
  struct Entry {
    uint64_t key[6];
    bool valid;
    CUtensorMap map;
  };
  constexpr int kEntries = 64;
  static thread_local Entry cache[kEntries] = {};
  const uint64_t key[6] = {reinterpret_cast<uint64_t>(base), inner_elems, rows, row_pitch_bytes,
                           ((uint64_t)box_inner << 32) | box_rows, ((uint64_t)dtype << 2) | (uint64_t)(swizzle & 3)};
  uint64_t h = 0x9E3779B97F4A7C15ull;
  for (uint64_t k : key) h = (h ^ k) * 0xFF51AFD7ED558CCDull + (h >> 29);
  Entry& e = cache[(h >> 20) % kEntries];
  if (e.valid && std::equal(key, key + 6, e.key)) {
    *map = e.map;
    return true;
  }
  EncodeTiledFn fn = tensor_map_encoder();
  if (!fn) return false;
  cuuint64_t dims[2] = {inner_elems, rows};
  cuuint64_t strides[1] = {row_pitch_bytes};
  cuuint32_t box[2] = {box_inner, box_rows};
  cuuint32_t estr[2] = {1, 1};
  if (fn(map, dtype, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
         swizzle == 1 ? CU_TENSOR_MAP_SWIZZLE_128B : swizzle == 2 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_NONE,
         CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return false;
  std::copy(key, key + 6, e.key);
  e.map = *map;
  e.valid = true;
  return true;
}

cudaError_t sm_count(int* n) {
  static std::atomic<int> cache[64] = {};  // per device ordinal
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  int v = (dev >= 0 && dev < 64) ? cache[dev].load(std::memory_order_relaxed) : 0;
  if (!v) {
    e = cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) cache[dev].store(v, std::memory_order_relaxed);
  }
  *n = v;
  return cudaSuccess;
}

namespace {

constexpr int BM = 128;
constexpr int BK_BYTES = 128;           // bytes of codes per row per stage = 256 elements of K
constexpr int BK = 256;
constexpr int kThreads = 224;
constexpr uint32_t kTmemCols = 512;

template <int BN>
struct Cfg {
  static constexpr int kStages = (BN == 256) ? 4 : 6;
  static constexpr int kAccStages = (BN == 256) ? 1 : 2;
  static constexpr int kABytes = BM * BK_BYTES;             // 16 KB
  static constexpr int kBBytes = BN * BK_BYTES;             // 16 / 32 KB
  static constexpr int kSfaBytes = 4 * 512;                 // 4 K64-steps x one 128-row atom
  static constexpr int kSfbBytes = (BN / 128) * 4 * 512;
  static constexpr int kStageBytes = kABytes + kBBytes + kSfaBytes + kSfbBytes;
  static constexpr int kSmemBytes = kStages * kStageBytes + 1024 /*alignment slack*/ + 256 /*barriers*/;
  // tensor memory columns
  static constexpr int kAccCol = 0;
  static constexpr int kSfCol = kAccStages * BN;            // one slot of (SFA 16 + SFB 4*BN/32) columns per stage
  static constexpr int kSfaCols = 16;
  static constexpr int kSfbCols = 4 * (BN / 32);
  static constexpr int kSfBufCols = kSfaCols + kSfbCols;
  static_assert(kSfCol + kStages * kSfBufCols <= 512, "tensor memory budget");
};

// ------------------------------------------------------------------------------------ kernel ----
// MX = true: MXFP4 operands (UE8M0 scale per 32 elements): half the scale atoms per k-block, one atom serving two
// K = 64 steps through the scale-id field of the instruction descriptor (see gemm_2cta.cuh).
template <int BN, bool MX>
__global__ void __launch_bounds__(kThreads, 1)
    gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                const GemmArgs g) {
  using C = Cfg<BN>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - smem_u32(smem_raw));
  // barriers live after the stages
  const uint32_t bar_base = base + C::kStages * C::kStageBytes;
  auto full_bar = [&](int s) { return bar_base + 8u * s; };                      // operands + scale atoms landed
  auto sff_bar = [&](int s) { return bar_base + 8u * (C::kStages + s); };        // scale atoms are in tensor memory
  auto empty_bar = [&](int s) { return bar_base + 8u * (2 * C::kStages + s); };  // MMAs have consumed the stage
  auto accf_bar = [&](int s) { return bar_base + 8u * (3 * C::kStages + s); };
  auto acce_bar = [&](int s) { return bar_base + 8u * (3 * C::kStages + C::kAccStages + s); };
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(
      base_ptr + C::kStages * C::kStageBytes + 8 * (3 * C::kStages + 2 * C::kAccStages));
  volatile uint32_t* abort_flag = tmem_slot + 1;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tiles_m = g.M / BM, tiles_n = g.N / BN;
  const int n_tiles = tiles_m * tiles_n;
  const int k_blocks = g.K / BK;
  const int64_t sf_atoms_per_row_group = g.K / (MX ? 128 : 64);
  constexpr int kAtomsKb = MX ? 2 : 4;  // scale atoms per 256-deep k-block and 128-row group

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::kStages; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(sff_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int s = 0; s < C::kAccStages; ++s) {
      mbar_init(accf_bar(s), 1);
      mbar_init(acce_bar(s), 4);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32((const void*)tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  griddep_wait();  // the set-up above ran beside the previous kernel; from here on its output is touched
  griddep_launch_dependents();

  if (warp == 0) {
    // ------------------------------------------------------------------ producer ----
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x) {
        const int m_blk = tile % tiles_m, n_blk = tile / tiles_m;
        const uint8_t* sfa = g.sfa + (int64_t)m_blk * sf_atoms_per_row_group * 512;
        const uint8_t* sfb = g.sfb + (int64_t)n_blk * (BN / 128) * sf_atoms_per_row_group * 512;
        for (int kb = 0; kb < k_blocks; ++kb) {
          if (!(ok = mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, 0x100u + stage))) break;
          const uint32_t st = base + stage * C::kStageBytes;
          mbar_expect_tx(full_bar(stage), C::kABytes + C::kBBytes + (1 + BN / 128) * kAtomsKb * 512);
          tma_load_2d(st, &map_a, kb * BK_BYTES, m_blk * BM, full_bar(stage));
          tma_load_2d(st + C::kABytes, &map_b, kb * BK_BYTES, n_blk * BN, full_bar(stage));
          bulk_load(st + C::kABytes + C::kBBytes, sfa + (int64_t)kb * kAtomsKb * 512, kAtomsKb * 512, full_bar(stage));
#pragma unroll
          for (int grp = 0; grp < BN / 128; ++grp)
            bulk_load(st + C::kABytes + C::kBBytes + C::kSfaBytes + grp * 2048,
                      sfb + ((int64_t)grp * sf_atoms_per_row_group + (int64_t)kb * kAtomsKb) * 512, kAtomsKb * 512,
                      full_bar(stage));
          if (++stage == C::kStages) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
    }
  } else if (warp == 2) {
    // ------------------------------------------- scale atoms: shared -> tensor memory ----
    // SFA of K64-step j goes to columns [4j, 4j+4) of the stage's slot; SFB of step j to
    // [16 + j*BN/32, ...), 4 columns per 128 rows of B.  The slot of a stage is free again when the
    // stage's operands are (empty -> producer -> full), so no extra barrier guards it.
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      const uint32_t sf_lo0 = (base + C::kABytes + C::kBBytes) >> 4;
      for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x) {
        for (int kb = 0; kb < k_blocks; ++kb) {
          if (!(ok = mbar_wait(full_bar(stage), phase, abort_flag, 0x500u + stage))) break;
          tc_fence_after();
          const uint32_t lo = sf_lo0 + stage * (C::kStageBytes >> 4);
          const uint32_t sf_t = tmem + C::kSfCol + stage * C::kSfBufCols;
#pragma unroll
          for (int j = 0; j < kAtomsKb; ++j) {
            tc_cp_sf(sf_t + j * 4, make_desc(lo + j * 32, kDescHiSf));
#pragma unroll
            for (int grp = 0; grp < BN / 128; ++grp)
              tc_cp_sf(sf_t + C::kSfaCols + j * (BN / 32) + grp * 4,
                       make_desc(lo + (C::kSfaBytes >> 4) + grp * 128 + j * 32, kDescHiSf));
          }
          tc_commit(sff_bar(stage));
          if (++stage == C::kStages) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer ----
    if (lane == 0) {
      int stage = 0, acc = 0;
      uint32_t phase = 0, acc_phase = 0;
      bool ok = true;
      constexpr uint32_t idesc = instr_desc_nvf4(BM, BN);
      constexpr uint32_t idesc_mx[2] = {instr_desc_mxf4(BM, BN, 0), instr_desc_mxf4(BM, BN, 2)};
      const uint32_t a_lo0 = ((base >> 4) & 0x3fffu) | (1u << 16);
      const uint32_t b_lo0 = (((base + C::kABytes) >> 4) & 0x3fffu) | (1u << 16);
      for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x) {
        if (!(ok = mbar_wait(acce_bar(acc), acc_phase ^ 1u, abort_flag, 0x300u + acc))) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem + C::kAccCol + acc * BN;
        for (int kb = 0; kb < k_blocks; ++kb) {
          if (!(ok = mbar_wait(sff_bar(stage), phase, abort_flag, 0x200u + stage))) break;
          tc_fence_after();
          const uint32_t a_lo = a_lo0 + stage * (C::kStageBytes >> 4);
          const uint32_t b_lo = b_lo0 + stage * (C::kStageBytes >> 4);
          const uint32_t sf_t = tmem + C::kSfCol + stage * C::kSfBufCols;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            // advancing 64 elements of K = 32 bytes inside the 128-byte swizzle span: +2 in the address field
            if (MX)
              tc_mma_mxf4(d_tmem, make_desc(a_lo + 2 * j, kDescHiOperand), make_desc(b_lo + 2 * j, kDescHiOperand),
                          idesc_mx[j & 1], sf_t + (j >> 1) * 4, sf_t + C::kSfaCols + (j >> 1) * (BN / 32),
                          (kb > 0 || j > 0) ? 1u : 0u);
            else
              tc_mma_nvf4(d_tmem, make_desc(a_lo + 2 * j, kDescHiOperand), make_desc(b_lo + 2 * j, kDescHiOperand), idesc,
                          sf_t + j * 4, sf_t + C::kSfaCols + j * (BN / 32), (kb > 0 || j > 0) ? 1u : 0u);
          }
          tc_commit(empty_bar(stage));  // frees the stage once the MMAs above have read it
          if (++stage == C::kStages) {
            stage = 0;
            phase ^= 1u;
          }
        }
        if (!ok) break;
        tc_commit(accf_bar(acc));  // accumulator complete
        if (++acc == C::kAccStages) {
          acc = 0;
          acc_phase ^= 1u;
        }
      }
    }
  } else if (warp >= 3) {
    // ------------------------------------------------------------------ epilogue ----
    const int quad = warp & 3;  // the 32 tensor-memory lanes this warp may read
    int acc = 0;
    uint32_t acc_phase = 0;
    bool ok = true;
    const float alpha = __fmul_rn(g.a_global[1], g.b_global[1]);
    for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x) {
      const int m_blk = tile % tiles_m, n_blk = tile / tiles_m;
      ok = mbar_wait(accf_bar(acc), acc_phase, abort_flag, 0x400u + acc);
      ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
      if (!ok) break;
      tc_fence_after();
      const int64_t row = (int64_t)m_blk * BM + quad * 32 + lane;
      const uint32_t t_row = tmem + ((uint32_t)(quad * 32) << 16) + C::kAccCol + acc * BN;
#pragma unroll 1
      for (int c = 0; c < BN / 32; ++c) {
        uint32_t r[32];
        tc_ld32(t_row + c * 32, r);
        tc_wait_ld();
        const int64_t col = (int64_t)n_blk * BN + c * 32;
        if (g.d_is_fp32) {
          float* dst = reinterpret_cast<float*>(g.d) + row * g.ldd + col;
#pragma unroll
          for (int v = 0; v < 8; ++v) {
            float4 o = make_float4(__fmul_rn(__uint_as_float(r[4 * v]), alpha), __fmul_rn(__uint_as_float(r[4 * v + 1]), alpha),
                                   __fmul_rn(__uint_as_float(r[4 * v + 2]), alpha), __fmul_rn(__uint_as_float(r[4 * v + 3]), alpha));
            if (g.accumulate) {
              float4 old = *reinterpret_cast<const float4*>(dst + 4 * v);
              o.x += old.x; o.y += old.y; o.z += old.z; o.w += old.w;
            }
            *reinterpret_cast<float4*>(dst + 4 * v) = o;
          }
        } else {
          __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(g.d) + row * g.ldd + col;
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            uint32_t p[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(r[8 * v + 2 * e]) * alpha,
                                                       __uint_as_float(r[8 * v + 2 * e + 1]) * alpha);
              p[e] = *reinterpret_cast<uint32_t*>(&h);
            }
            *reinterpret_cast<uint4*>(dst + 8 * v) = make_uint4(p[0], p[1], p[2], p[3]);
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acce_bar(acc));
      if (++acc == C::kAccStages) {
        acc = 0;
        acc_phase ^= 1u;
      }
    }
  }

  // ------------------------------------------------------------------ teardown ----
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    // give copies that may still be in flight time to land before the shared memory is handed back
    for (int i = 0; i < 100; ++i) __nanosleep(1000);
  }
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

// ------------------------------------------------------------------------------- host side ----
// codes [rows][k_bytes] uint8, box = 128 bytes x box_rows, 128-byte swizzle
bool make_code_map(CUtensorMap* map, const void* codes, int64_t rows, int64_t k_bytes, int box_rows) {
  return make_map_2d(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, codes, (uint64_t)k_bytes, (uint64_t)rows, (uint64_t)k_bytes,
                     BK_BYTES, (uint32_t)box_rows, true);
}

template <int BN, bool MX>
cudaError_t launch_t(const GemmArgs& g, const void* a_codes, const void* b_codes, int num_sms, cudaStream_t s) {
  using C = Cfg<BN>;
  CUtensorMap map_a, map_b;
  if (!make_code_map(&map_a, a_codes, g.M, g.K / 2, BM) || !make_code_map(&map_b, b_codes, g.N, g.K / 2, BN))
    return cudaErrorInvalidValue;
  auto kern = gemm_kernel<BN, MX>;
  static std::atomic<uint64_t> configured{0};  // per call site (template instantiation) and device
  int dev;
  if (device_needs_config(configured, &dev)) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
    if (e != cudaSuccess) return e;
    device_configured(configured, dev);
  }
  const int n_tiles = (g.M / BM) * (g.N / BN);
  const int grid = n_tiles < num_sms ? n_tiles : num_sms;
  const cudaError_t le = launch_kernel(kern, dim3(grid), dim3(kThreads), C::kSmemBytes, s, map_a, map_b, g);
  count_launch();
  return le;
}

bool make_pair_maps(const GemmArgs& g, const void* a_codes, const void* b_codes, int bn, int store_cols, CUtensorMap* map_a,
                    CUtensorMap* map_b, CUtensorMap* map_d) {
  bool ok = make_code_map(map_a, a_codes, g.M, g.K / 2, 128) && make_code_map(map_b, b_codes, g.N, g.K / 2, bn / 2);
  if (g.d_is_fp32)
    ok = ok && make_map_2d(map_d, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, g.d, (uint64_t)g.N, (uint64_t)g.M,
                           (uint64_t)g.ldd * 4, 16, 128, 2);
  else
    ok = ok && make_map_2d(map_d, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, g.d, (uint64_t)g.N, (uint64_t)g.M,
                           (uint64_t)g.ldd * 2, store_cols < 64 ? 32 : 64, 128, store_cols < 64 ? 2 : 1);
  return ok;
}

// measurement aids of the CTA-pair kernel (set_gemm_experiment)
std::atomic<int> g_exp_mode{0}, g_exp_max_pairs{0};
std::atomic<unsigned long long*> g_exp_probe{nullptr};

pair::Problem pair_problem(const GemmArgs& g) {
  return pair::Problem{g.M,         g.N,          g.K,      g.sfa,    g.sfb,   g.a_global, g.b_global,
                       g.d_is_fp32, g.accumulate, g.a_rows, g.b_rows, g.shares == 4 ? 2 : g.shares == 2 ? 1 : 0};
}

bool has_row_scales(const GemmArgs& g0, const GemmArgs* g1) {
  return g0.a_rows || g0.b_rows || (g1 && (g1->a_rows || g1->b_rows));
}

// tiles of a problem on CTA pairs with BN columns; the last one in either direction may be half outside
inline int pair_tiles(const GemmArgs& g, int bn) { return ((g.M + 255) / 256) * ((g.N + bn - 1) / bn); }

// g1 == nullptr: one problem
template <bool MX, bool ROWS, int BN, int SPLIT = 1, bool SHARES = false>
cudaError_t launch_pair_t(const GemmArgs& g0, const void* a0, const void* b0, const GemmArgs* g1, const void* a1,
                          const void* b1, int num_sms, cudaStream_t s) {
  auto kern = pair::gemm_pair_kernel<MX, ROWS, BN, SPLIT, SHARES>;
  constexpr int smem = pair::Cfg<BN, SPLIT>::kSmemBytes, store_cols = SPLIT > 1 ? BN / SPLIT : 64;
  CUtensorMap m[6];
  if (!make_pair_maps(g0, a0, b0, BN, store_cols, &m[0], &m[1], &m[2])) return cudaErrorInvalidValue;
  if (g1) {
    if (!make_pair_maps(*g1, a1, b1, BN, store_cols, &m[3], &m[4], &m[5])) return cudaErrorInvalidValue;
  } else {
    m[3] = m[0]; m[4] = m[1]; m[5] = m[2];
  }
  static std::atomic<uint64_t> configured{0};  // per call site (template instantiation) and device
  int dev;
  if (device_needs_config(configured, &dev)) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    device_configured(configured, dev);
  }
  pair::Args a{};
  a.p[0] = pair_problem(g0);
  a.p[1] = pair_problem(g1 ? *g1 : g0);
  a.n_tiles0 = pair_tiles(g0, BN);
  a.n_tiles = a.n_tiles0 + (g1 ? pair_tiles(*g1, BN) : 0);
  int max_pairs = num_sms / 2;
  if (BN == 256) {  // measurement aids (0 / NULL normally) of the kernel with 256 x 256 tiles; no other launch may see them
    const int cap = g_exp_max_pairs.load(std::memory_order_relaxed);
    if (cap > 0 && cap < max_pairs) max_pairs = cap;
    a.exp = g_exp_mode.load(std::memory_order_relaxed);
    a.probe = g_exp_probe.load(std::memory_order_relaxed);
  }
  const int pairs = a.n_tiles < max_pairs || SPLIT > 1 ? a.n_tiles : max_pairs;  // SPLIT > 1: a cluster for each tile
  const cudaError_t e =
      launch_kernel(kern, dim3(2 * SPLIT * pairs), dim3(pair::kThreads), smem, s, m[0], m[1], m[2], m[3], m[4], m[5], a);
  count_launch();
  return e;
}

cudaError_t launch_pair(const GemmArgs& g0, const void* a0, const void* b0, const GemmArgs* g1, const void* a1,
                        const void* b1, int bn, int num_sms, cudaStream_t s) {
  if (g1 && g1->mx != g0.mx) return cudaErrorInvalidValue;
  if (has_row_scales(g0, g1)) {
    if (g0.mx) return cudaErrorInvalidValue;
    return bn == 128 ? launch_pair_t<false, true, 128>(g0, a0, b0, g1, a1, b1, num_sms, s)
                     : launch_pair_t<false, true, 256>(g0, a0, b0, g1, a1, b1, num_sms, s);
  }
  if (bn == 128)
    return g0.mx ? launch_pair_t<true, false, 128>(g0, a0, b0, g1, a1, b1, num_sms, s)
                 : launch_pair_t<false, false, 128>(g0, a0, b0, g1, a1, b1, num_sms, s);
  return g0.mx ? launch_pair_t<true, false, 256>(g0, a0, b0, g1, a1, b1, num_sms, s)
               : launch_pair_t<false, false, 256>(g0, a0, b0, g1, a1, b1, num_sms, s);
}

template <int SPLIT>
cudaError_t launch_split(const GemmArgs& g, const void* a, const void* b, int num_sms, cudaStream_t s) {
  if (has_row_scales(g, nullptr))
    return g.mx ? cudaErrorInvalidValue
                : launch_pair_t<false, true, 128, SPLIT>(g, a, b, nullptr, nullptr, nullptr, num_sms, s);
  return g.mx ? launch_pair_t<true, false, 128, SPLIT>(g, a, b, nullptr, nullptr, nullptr, num_sms, s)
              : launch_pair_t<false, false, 128, SPLIT>(g, a, b, nullptr, nullptr, nullptr, num_sms, s);
}

// N = 128 q = 384 a + 256 b with b in {0, 1, 2}: a wide column tiles, b narrow ones (q >= 2)
bool wide_split(int N, int* n_wide, int* n_narrow) {
  if (N % 128 != 0 || N < 256) return false;
  const int q = N / 128;
  const int b = (q % 3 == 0) ? 0 : (q % 3 == 1) ? 2 : 1;
  if (q - 2 * b < 0) return false;
  *n_wide = (q - 2 * b) / 3;
  *n_narrow = b;
  return true;
}

bool wide_eligible(const GemmArgs& g) {
  int a, b;
  return wide_split(g.N, &a, &b);
}

wide::WProblem wide_problem(const GemmArgs& g) {
  int a = 0, b = 0;
  wide_split(g.N, &a, &b);
  return wide::WProblem{g.M, g.N, g.K, g.sfa, g.sfb, g.a_global, g.b_global, g.d_is_fp32, g.accumulate, a, a + b, g.a_rows,
                        g.b_rows};
}

bool make_wide_maps(const GemmArgs& g, const void* a_codes, const void* b_codes, CUtensorMap* m) {
  // m[0] A (128-row boxes), m[1] B (128-row boxes), m[2] B (64-row boxes), m[3] D
  bool ok = make_code_map(&m[0], a_codes, g.M, g.K / 2, 128) && make_code_map(&m[1], b_codes, g.N, g.K / 2, 128) &&
            make_code_map(&m[2], b_codes, g.N, g.K / 2, 64);
  // D: the epilogue's store chunks, 128 rows x 64 bytes with the 64-byte swizzle (fp32) or x 128 bytes (bf16)
  if (g.d_is_fp32)
    ok = ok && make_map_2d(&m[3], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, g.d, (uint64_t)g.N, (uint64_t)g.M,
                           (uint64_t)g.ldd * 4, 16, 128, 2);
  else
    ok = ok && make_map_2d(&m[3], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, g.d, (uint64_t)g.N, (uint64_t)g.M,
                           (uint64_t)g.ldd * 2, 64, 128, 1);
  return ok;
}

// Estimated time (microseconds, without the launch) of the static round-robin schedule the pair kernels use, for one or
// two problems: round r hands tiles r * pairs .. to the pairs in order, odd rounds in reverse order.  A tile costs its
// k-blocks plus the accumulator hand-over, and no less than its output takes to store.  The constants are a fit to 90
// shapes drawn over M 128 .. 16384, N 256 .. 20480, K 512 .. 20480, both output types, timed with all three tiles (rms
// error 5 %); choosing by them loses 0.1 % on average against the best tile of each shape, always 256 x 256 loses 17 %.
double pair_makespan(const GemmArgs* const* gs, int n_problems, int tile, int pairs) {
  std::vector<double> load((size_t)pairs, 0.0);
  constexpr int kGroupM = 8;
  int64_t t = 0;
  for (int pi = 0; pi < n_problems; ++pi) {
    const GemmArgs& g = *gs[pi];
    int n_wide = 0, n_narrow = tile == kTilePair128 ? (g.N + 127) / 128 : (g.N + 255) / 256;
    if (tile == kTileWide) wide_split(g.N, &n_wide, &n_narrow);
    const int tiles_m = (g.M + 255) / 256, tiles_n = n_wide + n_narrow;
    const double kb = g.K / 256.0;
    const bool f = g.d_is_fp32;
    const double wide_cost = std::max(0.505 * kb + (f ? 3.56 : 2.03), f ? 4.9 : 0.0);
    const double narrow_cost = tile == kTilePair128 ? std::max(0.323 * kb + (f ? 0.97 : 0.64), f ? 1.8 : 1.4)
                               : tile == kTileWide  ? std::max(0.383 * kb + 2.0, f ? 3.3 : 0.0)
                                                    : std::max(0.383 * kb + (f ? 2.5 : 1.83), f ? 4.9 : 0.0);
    for (int m0 = 0; m0 < tiles_m; m0 += kGroupM) {
      const int gm = tiles_m - m0 < kGroupM ? tiles_m - m0 : kGroupM;
      for (int n_idx = 0; n_idx < tiles_n; ++n_idx) {
        const double cost = n_idx < n_wide ? wide_cost : narrow_cost;
        for (int i = 0; i < gm; ++i, ++t) {
          const int64_t rnd = t / pairs, p = t % pairs;
          load[(size_t)((rnd & 1) ? pairs - 1 - p : p)] += cost;  // odd rounds run through the pairs in reverse
        }
      }
    }
  }
  double worst = 0.0;
  for (double v : load) worst = v > worst ? v : worst;
  return worst;
}

// Clusters of 2 * SPLIT CTAs of this kernel that are resident at once on the current device (0: none)
template <auto KERN, int SPLIT>
int resident_clusters(int threads, int smem) {
  constexpr int kMaxDevices = 64;
  static std::atomic<int> known[kMaxDevices];  // the number + 1
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 0;
  if (const int n = known[dev].load(std::memory_order_relaxed)) return n - 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(2 * SPLIT);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  int n = 0;
  if (cudaFuncSetAttribute(KERN, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, KERN, &cfg) != cudaSuccess)
    n = 0;
  known[dev].store(n + 1, std::memory_order_relaxed);
  return n;
}
template <int SPLIT>
int split_clusters() {
  return resident_clusters<pair::gemm_pair_kernel<false, false, 128, SPLIT>, SPLIT>(pair::kThreads,
                                                                                   pair::Cfg<128, SPLIT>::kSmemBytes);
}

// The split of a product that has a launch to itself, or 0 (`least`: the estimate of the best tile).  A split pays where a
// tile's contraction is long and the clusters of all tiles are resident at once; its exchange costs 1.4 us (2.1 where most of
// the chip takes part) and it has to win by half a microsecond.  The two products of a backward call fill one launch
// together: with one of them split and the other behind it, 512 x 3584 x 768 took 22.6 us instead of 16.0.
// Time of a product, 256 x 128 tiles / two pairs / four pairs per tile: 256 x 512 x 5120 10.5 / 8.5 / 7.3 us, 256 x 512 x 20480
// 29.1 / 17.8 / 12.2, 512 x 1024 x 4096 9.5 / 8.1 / 14.1 (two rounds), 1024 x 1024 x 10240 17.6 / 12.9 / 27.6; 256 x 1024 x 2048
// 6.7 / 6.7 / 6.4, 256 x 2048 x 1024 5.5 / 6.2 / 12.1.
int split_tile(const GemmArgs& g, double least) {
  const int tiles = ((g.M + 255) / 256) * (g.N / 128), kb = g.K / 256;
  const double fixed = (g.d_is_fp32 ? 0.97 : 0.64) + (tiles > 16 ? 2.1 : 1.4);
  int best = 0;
  least -= 0.5;
  auto consider = [&](int split, int clusters, int tile) {
    const double v = 0.323 * ((kb + split - 1) / split) + fixed;
    if (kb < split || tiles > clusters || v >= least) return;
    best = tile;
    least = v;
  };
  consider(2, split_clusters<2>(), kTileSplit2);
  consider(4, split_clusters<4>(), kTileSplit4);
  return best;
}

// g1 == nullptr: one problem
template <bool MX, bool ROWS>
cudaError_t launch_wide_t(const GemmArgs& g0, const void* a0, const void* b0, const GemmArgs* g1, const void* a1,
                          const void* b1, int num_sms, cudaStream_t s) {
  auto kern = wide::gemm_wide_kernel<MX, ROWS>;
  CUtensorMap m[8];
  if (!make_wide_maps(g0, a0, b0, &m[0])) return cudaErrorInvalidValue;
  if (g1) {
    if (!make_wide_maps(*g1, a1, b1, &m[4])) return cudaErrorInvalidValue;
  } else {
    for (int i = 0; i < 4; ++i) m[4 + i] = m[i];
  }
  static std::atomic<uint64_t> configured{0};  // per call site (template instantiation) and device
  int dev;
  if (device_needs_config(configured, &dev)) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, wide::kWSmemBytes);
    if (e != cudaSuccess) return e;
    device_configured(configured, dev);
  }
  wide::WArgs a{};
  a.p[0] = wide_problem(g0);
  a.p[1] = wide_problem(g1 ? *g1 : g0);
  a.n_tiles0 = ((g0.M + 255) / 256) * a.p[0].tiles_n;
  a.n_tiles = a.n_tiles0 + (g1 ? ((g1->M + 255) / 256) * a.p[1].tiles_n : 0);
  const int max_pairs = num_sms / 2;
  const int pairs = a.n_tiles < max_pairs ? a.n_tiles : max_pairs;
  const cudaError_t le = launch_kernel(kern, dim3(2 * pairs), dim3(wide::kWThreads), wide::kWSmemBytes, s, m[0], m[1], m[2],
                                       m[3], m[4], m[5], m[6], m[7], a);
  count_launch();
  return le;
}

cudaError_t launch_wide(const GemmArgs& g0, const void* a0, const void* b0, const GemmArgs* g1, const void* a1,
                        const void* b1, int num_sms, cudaStream_t s) {
  if (g1 && g1->mx != g0.mx) return cudaErrorInvalidValue;
  if (has_row_scales(g0, g1))
    return g0.mx ? cudaErrorInvalidValue : launch_wide_t<false, true>(g0, a0, b0, g1, a1, b1, num_sms, s);
  return g0.mx ? launch_wide_t<true, false>(g0, a0, b0, g1, a1, b1, num_sms, s)
               : launch_wide_t<false, false>(g0, a0, b0, g1, a1, b1, num_sms, s);
}

}  // namespace

int split_of(const GemmArgs& g, int tile) {
  const int split = tile == kTileSplit2 ? 2 : tile == kTileSplit4 ? 4 : 1;
  return g.K / 256 >= split ? split : 1;  // a pair has a k-block at least
}

cudaError_t launch_gemm(const GemmArgs& g, const void* a_codes, const void* b_codes, int tile, cudaStream_t s) {
  int num_sms = 0;
  cudaError_t e = sm_count(&num_sms);
  if (e != cudaSuccess) return e;
  const bool rows = has_row_scales(g, nullptr);  // scale vectors: the pair kernels' epilogues only
  const int split = split_of(g, tile);
  if (split == 2) return launch_split<2>(g, a_codes, b_codes, num_sms, s);
  if (split == 4) return launch_split<4>(g, a_codes, b_codes, num_sms, s);
  if (tile == kTileSplit2 || tile == kTileSplit4) tile = kTilePair128;
  if (tile == kTileWide && wide_eligible(g)) return launch_wide(g, a_codes, b_codes, nullptr, nullptr, nullptr, num_sms, s);
  if (tile >= kTilePair256 || rows)
    return launch_pair(g, a_codes, b_codes, nullptr, nullptr, nullptr, tile == kTilePair128 ? 128 : 256, num_sms, s);
  if (tile == 256 && g.N % 256 == 0)
    return g.mx ? launch_t<256, true>(g, a_codes, b_codes, num_sms, s) : launch_t<256, false>(g, a_codes, b_codes, num_sms, s);
  return g.mx ? launch_t<128, true>(g, a_codes, b_codes, num_sms, s) : launch_t<128, false>(g, a_codes, b_codes, num_sms, s);
}

cudaError_t launch_gemm_two(const GemmArgs& g0, const void* a0, const void* b0, const GemmArgs& g1, const void* a1,
                            const void* b1, int tile, cudaStream_t s) {
  int num_sms = 0;
  cudaError_t e = sm_count(&num_sms);
  if (e != cudaSuccess) return e;
  if (g0.shares > 1 || g1.shares > 1) {
    if (g1.mx != g0.mx || has_row_scales(g0, &g1)) return cudaErrorInvalidValue;
    return g0.mx ? launch_pair_t<true, false, 128, 1, true>(g0, a0, b0, &g1, a1, b1, num_sms, s)
                 : launch_pair_t<false, false, 128, 1, true>(g0, a0, b0, &g1, a1, b1, num_sms, s);
  }
  if (tile == kTileWide && wide_eligible(g0) && wide_eligible(g1)) return launch_wide(g0, a0, b0, &g1, a1, b1, num_sms, s);
  return launch_pair(g0, a0, b0, &g1, a1, b1, tile == kTilePair256 || tile == kTileWide ? 256 : 128, num_sms, s);
}

// 128 x 128 tiles of one CTA each, for one product: its time, or 0 where they are no candidates.  They double the operand
// traffic of a pair, but where M is an odd multiple of 128 the pairs compute a row of half tiles: if that takes the narrow pair
// tiles over one round of the chip and the single ones fit it, those win.  Single / pair tiles: 1152 x 2048 x 2048 7.2 / 9.0
// us, x 5120 12.3 / 13.3, MXFP4 6.4 / 8.8 and 10.0 / 13.1; 1664 x 1408 x 5120 13.3 / 13.3, MXFP4 10.9 / 13.0, fp32 output 15.4 /
// 14.8 and 13.2 / 14.3.  (Not for an accumulated output: its read-modify-write in the epilogue costs 3 us.)
static double one_cta_time(const GemmArgs& g, int num_sms) {
  const int64_t tiles = (int64_t)(g.M / 128) * (g.N / 128);
  if (g.accumulate || g.a_rows || g.b_rows || tiles > num_sms || pair_tiles(g, 128) <= num_sms / 2) return 0.0;
  const double kb = g.K / 256.0;
  return (g.mx ? 0.29 : 0.40) * kb + (g.d_is_fp32 ? 3.7 : 1.4);
}

int best_tile(const GemmArgs& g0, const GemmArgs* g1) {
  int num_sms = 0;
  if (sm_count(&num_sms) != cudaSuccess) return kTilePair256;
  const bool wide_fits = wide_eligible(g0) && (!g1 || wide_eligible(*g1));
  int dev = 0, best = kTilePair256;
  if (cudaGetDevice(&dev) != cudaSuccess) return best;
  static TileMemo memo;
  const double single = g1 ? 0.0 : one_cta_time(g0, num_sms);
  // (the output type is part of the key: an fp32 output changes the hand-over cost and with it the choice)
  const int key[TileMemo::kKey] = {g0.M, g0.N, g0.K, g1 ? g1->M : 0, g1 ? g1->N : 0, g1 ? g1->K : 0,
                                   (g0.d_is_fp32 ? 1 : 0) | (g1 && g1->d_is_fp32 ? 2 : 0) | (single > 0.0 ? 4 : 0) | (g0.mx ? 8 : 0),
                                   dev};
  if (memo.find(key, &best)) return best;
  const GemmArgs* gs[2] = {&g0, g1};
  const int n = g1 ? 2 : 1, pairs = num_sms / 2;
  best = kTilePair256;
  double least = pair_makespan(gs, n, kTilePair256, pairs);
  for (int tile : {kTilePair128, kTileWide}) {
    if (tile == kTileWide && !wide_fits) continue;
    const double v = pair_makespan(gs, n, tile, pairs);
    if (v < least) {
      least = v;
      best = tile;
    }
  }
  if (!g1) {
    if (single > 0.0 && single + 0.2 < least) {
      least = single;
      best = kTileOne128;
    }
    if (const int tile = split_tile(g0, least)) best = tile;
  }
  memo.put(key, best);
  return best;
}

template <int BN, int SPLIT>
static bool make_bf16_maps(const DenseGemmArgs& g, CUtensorMap* m) {  // A, B, D
  const CUtensorMapDataType bf = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  bool ok = g.a_mn ? make_map_2d(&m[0], bf, 2, g.a, (uint64_t)g.M, (uint64_t)g.K, (uint64_t)g.lda * 2, 64, 64, true)
                   : make_map_2d(&m[0], bf, 2, g.a, (uint64_t)g.K, (uint64_t)g.M, (uint64_t)g.lda * 2, 64, 128, true);
  ok = ok && (g.b_mn ? make_map_2d(&m[1], bf, 2, g.b, (uint64_t)g.N, (uint64_t)g.K, (uint64_t)g.ldb * 2, 64, 64, true)
                     : make_map_2d(&m[1], bf, 2, g.b, (uint64_t)g.K, (uint64_t)g.N, (uint64_t)g.ldb * 2, 64,
                                   BN == 512 ? 128 : BN / 2, true));
  if (g.d_is_fp32)
    ok = ok && make_map_2d(&m[2], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, g.d, (uint64_t)g.N, (uint64_t)g.M,
                           (uint64_t)g.ldd * 4, 16, 128, 2);
  else
    ok = ok && make_map_2d(&m[2], bf, 2, g.d, (uint64_t)g.N, (uint64_t)g.M, (uint64_t)g.ldd * 2,
                           SPLIT == 4 ? 32 : 64, 128, SPLIT == 4 ? 2 : 1);
  return ok;
}

static int bf16_tiles(const DenseGemmArgs& g, int bn) { return ((g.M + 255) / 256) * ((g.N + bn - 1) / bn); }

template <int BN, int SPLIT, bool TWO>
static cudaError_t launch_bf16_problems(const DenseGemmArgs& g0, const DenseGemmArgs* g1, const Bf16Wide& wide_cols, int max_pairs,
                                        cudaStream_t s) {
  auto kern = dense::gemm_bf16_pair_kernel<BN, SPLIT, TWO>;
  constexpr int smem = dense::Cfg<BN, SPLIT>::kSmemBytes;
  CUtensorMap m[6];
  if (!make_bf16_maps<BN, SPLIT>(g0, m)) return cudaErrorInvalidValue;
  if (g1) {
    if (!make_bf16_maps<BN, SPLIT>(*g1, m + 3)) return cudaErrorInvalidValue;
  } else {
    for (int i = 0; i < 3; ++i) m[3 + i] = m[i];
  }
  static std::atomic<uint64_t> configured{0};  // per call site (template instantiation) and device
  int dev;
  if (device_needs_config(configured, &dev)) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    device_configured(configured, dev);
  }
  auto problem = [](const DenseGemmArgs& g) {
    return dense::Problem{g.M, g.N, g.K, g.a_mn, g.b_mn, g.d_is_fp32, g.accumulate};
  };
  dense::Args a{};
  a.p[0] = problem(g0);
  a.p[1] = problem(g1 ? *g1 : g0);
  if (BN == 512) {
    for (int i = 0; i < (g1 ? 2 : 1); ++i) {
      const DenseGemmArgs& g = i ? *g1 : g0;
      const int tiles_m = (g.M + 255) / 256, wide = std::min(wide_cols.n[i], (g.N + 255) / 512);
      a.wide_n[i] = wide;
      a.seg_end[i] = tiles_m * wide;
      a.seg_end[2 + i] = tiles_m * ((g.N + 255) / 256 - 2 * wide);
    }
    for (int i = 1; i < 4; ++i) a.seg_end[i] += a.seg_end[i - 1];
    a.n_tiles0 = a.n_tiles = a.seg_end[3];
  } else {
    a.n_tiles0 = bf16_tiles(g0, BN);
    a.n_tiles = a.n_tiles0 + (g1 ? bf16_tiles(*g1, BN) : 0);
  }
  const int pairs = a.n_tiles < max_pairs || SPLIT > 1 ? a.n_tiles : max_pairs;  // SPLIT > 1: a cluster for each tile
  const cudaError_t e = launch_kernel(kern, dim3(2 * SPLIT * pairs), dim3(dense::kThreads), smem, s, m[0], m[1], m[2],
                                      m[3], m[4], m[5], a);
  count_launch();
  return e;
}

// g1 == nullptr: one problem
template <int BN, int SPLIT = 1>
static cudaError_t launch_bf16_t(const DenseGemmArgs& g0, const DenseGemmArgs* g1, const Bf16Wide& wide_cols, int max_pairs,
                                 cudaStream_t s) {
  return g1 ? launch_bf16_problems<BN, SPLIT, true>(g0, g1, wide_cols, max_pairs, s)
            : launch_bf16_problems<BN, SPLIT, false>(g0, nullptr, wide_cols, max_pairs, s);
}

static Bf16Wide bf16_wide_tiles(const DenseGemmArgs& g0, const DenseGemmArgs* g1, int pairs) {
  Bf16Walk w[2];
  for (int i = 0; i < (g1 ? 2 : 1); ++i) {
    const DenseGemmArgs& g = i ? *g1 : g0;
    w[i] = bf16_walk(g.M, g.N, g.K, reinterpret_cast<uintptr_t>(g.a), g.lda, reinterpret_cast<uintptr_t>(g.b), g.ldb);
  }
  return bf16_wide_tiles(w, g1 ? 2 : 1, pairs);
}

int bf16_tile(const DenseGemmArgs& g0, const DenseGemmArgs* g1, int forced, Bf16Wide* wide) {
  int num_sms = 0;
  *wide = Bf16Wide{{0, 0}};
  if (sm_count(&num_sms) != cudaSuccess) return kTilePair256;
  // 256 x 128 tiles while every one of them has a pair to itself: less to load per k-block and half the epilogue (1000 x
  // 2000 x 3000 22.9 -> 19.0 us, 512 x 4096 x 4096 24.2 -> 23.2, 512 x 1024 x 1024 9.1 -> 8.1).  Beyond one round they lose:
  // an instruction 128 columns wide takes as long as one 256 wide (264 x 7168 x 5120 30 -> 50 us).
  const int64_t tiles128 = (int64_t)bf16_tiles(g0, 128) + (g1 ? bf16_tiles(*g1, 128) : 0);
  // Fewer tiles than clusters of several pairs: each tile's contraction is shared by two or four pairs, where what that saves
  // of the longest contraction (0.305 us per 64 deep) exceeds the exchange, 1.1 us (1.5 where most of the chip takes part) |
  // 1.6.  One / two / four pairs per tile: 264 x 512 x 512 6.4 / 6.0 / 6.2 us, 264 x 512 x 4096 23.6 / 14.8 / 10.4, 512 x 512 x
  // 16384 83 / 45 / 26, 1024 x 1024 x 512 6.5 / 6.6 / 18.5 (two rounds), 1024 x 1024 x 4096 24.9 / 16.2 / 31.5.
  auto clusters = [](auto split) {
    constexpr int kSplit = decltype(split)::value;
    return resident_clusters<dense::gemm_bf16_pair_kernel<128, kSplit>, kSplit>(dense::kThreads,
                                                                             dense::Cfg<128, kSplit>::kSmemBytes);
  };
  const int kb0 = (g0.K + 63) / 64, kb1 = g1 ? (g1->K + 63) / 64 : kb0, kb = std::max(kb0, kb1), least = std::min(kb0, kb1);
  if ((forced == kTileSplit2 && least >= 2) || (forced == kTileSplit4 && least >= 4)) return forced;
  auto gain = [&](int split) {
    return 0.305 * (kb - (kb + split - 1) / split) - (split == 4 ? 1.6 : tiles128 > 16 ? 1.5 : 1.1);
  };
  if (tiles128 <= 64 && least >= 4 && gain(2) > 0.2) {
    if (gain(4) > gain(2) && tiles128 <= clusters(std::integral_constant<int, 4>())) return kTileSplit4;
    if (tiles128 <= clusters(std::integral_constant<int, 2>())) return kTileSplit2;
  }
  if (tiles128 <= num_sms / 2) return kTilePair128;
  *wide = bf16_wide_tiles(g0, g1, num_sms / 2);
  return wide->n[0] + wide->n[1] ? kTileDouble : kTilePair256;
}

cudaError_t launch_gemm_bf16(const DenseGemmArgs& g0, const DenseGemmArgs* g1, int tile, const Bf16Wide& wide, cudaStream_t s) {
  int num_sms = 0;
  const cudaError_t e = sm_count(&num_sms);
  if (e != cudaSuccess) return e;
  const int pairs = num_sms / 2;
  if (tile == kTileSplit4) return launch_bf16_t<128, 4>(g0, g1, wide, pairs, s);
  if (tile == kTileSplit2) return launch_bf16_t<128, 2>(g0, g1, wide, pairs, s);
  if (tile == kTilePair128) return launch_bf16_t<128>(g0, g1, wide, pairs, s);
  return tile == kTileDouble ? launch_bf16_t<512>(g0, g1, wide, pairs, s) : launch_bf16_t<256>(g0, g1, wide, pairs, s);
}

// Test aid: one warp waits, with the given limit, on a barrier nobody arrives at.  The wait runs out, the code lands
// in the status word, the abort word stops the other lanes, and the kernel returns by itself.
__global__ void wait_probe_kernel(unsigned long long limit_ns) {
  __shared__ __align__(8) unsigned long long bar;
  __shared__ uint32_t abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    abort_flag = 0u;
  }
  __syncthreads();
  mbar_wait_limit(smem_u32(&bar), 0u, &abort_flag, kWaitProbeCode, limit_ns);
}

cudaError_t launch_wait_probe(unsigned long long limit_ns, cudaStream_t s) {
  wait_probe_kernel<<<1, 32, 0, s>>>(limit_ns);
  count_launch();
  return cudaGetLastError();
}

// Test aid: a cluster of eight whose first CTA has given up while the others arrive at the exit after k / 7 of the delay.
// times[2 k], [2 k + 1]: when CTA k got to the exit and when it was let go; times[16 + k]: its abort word then.
__global__ void __cluster_dims__(8, 1, 1) leave_probe_kernel(unsigned long long delay_ns, unsigned long long* times) {
  __shared__ __align__(8) unsigned long long bar;
  __shared__ uint32_t abort_flag;
  const uint32_t cta = pair::cluster_ctarank();
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 7);
    abort_flag = cta == 0 ? kLeaveProbeCode : 0u;
    fence_mbarrier_init();
  }
  __syncthreads();
  pair::cluster_sync_all();
  if (threadIdx.x == 0) {
    const unsigned long long t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < delay_ns / 7 * cta) __nanosleep(1000);
    times[2 * cta] = globaltimer_ns();
  }
  pair::leave_cluster<8>(smem_u32(&bar), cta, &abort_flag, 0x610u);
  if (threadIdx.x == 0) {
    times[2 * cta + 1] = globaltimer_ns();
    times[16 + cta] = abort_flag;
  }
}

cudaError_t launch_leave_probe(unsigned long long delay_ns, unsigned long long* times, cudaStream_t s) {
  leave_probe_kernel<<<8, 32, 0, s>>>(delay_ns, times);
  count_launch();
  return cudaGetLastError();
}

void set_gemm_experiment(int mode, int max_pairs, unsigned long long* probe) {
  g_exp_mode.store(mode, std::memory_order_relaxed);
  g_exp_max_pairs.store(max_pairs, std::memory_order_relaxed);
  g_exp_probe.store(probe, std::memory_order_relaxed);
}

cudaError_t device_status_word(unsigned int** word) {
  static std::atomic<unsigned int*> cache[64] = {};  // per device ordinal
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  unsigned int* p = (dev >= 0 && dev < 64) ? cache[dev].load(std::memory_order_acquire) : nullptr;
  if (!p) {
    e = cudaGetSymbolAddress(reinterpret_cast<void**>(&p), g_device_status);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) cache[dev].store(p, std::memory_order_release);
  }
  *word = p;
  return cudaSuccess;
}

cudaError_t read_device_status(cudaStream_t s, uint32_t* code) {
  cudaError_t e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return e;
  unsigned int v = 0;
  e = cudaMemcpyFromSymbol(&v, g_device_status, sizeof(v));
  if (e != cudaSuccess) return e;
  if (v) {
    unsigned int zero = 0;
    e = cudaMemcpyToSymbol(g_device_status, &zero, sizeof(zero));
  }
  *code = v;
  return e;
}

}  // namespace nvfp4
