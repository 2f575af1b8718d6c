// PTX wrappers for asynchronous copies (sm_100a): mbarrier and TMA loads, and the host-side tensor-map encoder.
// Used by the GEMM kernels and by the quantizer.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace nvfp4 {

constexpr unsigned long long kWaitLimitNs = 2000000000ull;  // 2 s per device-side wait

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

__device__ __forceinline__ void fence_mbarrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// orders this thread's earlier generic-proxy accesses to shared memory before later asynchronous-proxy ones (TMA)
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// ---- programmatic dependent launch: every kernel launched with `launch_divided` or `launch_kernel` may become resident while the previous
// kernel of the stream drains; it runs its set-up (barriers, tensor memory, descriptor prefetch) and then waits here for
// that kernel to finish with all its writes visible.  Behind a kernel that does not know the scheme (a caller's own) the
// launch is held until that kernel's CTAs have exited, and the wait covers its writes.  Rules that keep it transitive:
//   - every kernel waits before it finishes, so "kernel n has finished" implies "kernel n - 1 has finished";
//   - before its wait a kernel touches only what no kernel that may still run writes: the kernel that zeroes the words of
//     a call (zero_words_kernel) waits first and only then lets its dependent start, so the reductions behind it may read
//     their inputs at once and wait just before their first atomic (a reduction that is the first
//     kernel of its call waits and lets its dependent start in the same order).
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// lets the next kernel of the stream, if it was launched that way, become resident as CTAs of this grid retire
__device__ __forceinline__ void griddep_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

#ifdef __CUDACC__
// carveout: per cent of the SM that the kernel wants as shared memory, or -1 for whatever there is.  Between kernels launched this way
// an SM stays divided as the one before wanted it, nearly all shared memory behind a product or a quantizer's pass 2, and a kernel
// that streams with loads of its own finds little L1 for those in flight.
template <typename... Params, typename... Args>
inline cudaError_t launch_divided(int carveout, void (*kern)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                  Args&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
  attr[1].val.sharedMemCarveout = (unsigned)carveout;
  cfg.attrs = attr;
  cfg.numAttrs = carveout < 0 ? 1 : 2;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, static_cast<Params>(args)...);
  if (e != cudaSuccess) (void)cudaGetLastError();  // reported here, and not left for a later ordinary launch to find
  return e;
}
template <typename... Params, typename... Args>
inline cudaError_t launch_kernel(void (*kern)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                 Args&&... args) {
  return launch_divided(-1, kern, grid, block, smem, s, static_cast<Args&&>(args)...);
}
constexpr int kStreamingCarveout = 7;  // an SM then has 32 KB; with 15 per cent or more it was not divided again (see quantize_rowscale.cu)
#endif

// ---- host-side tensor-map encoder (driver entry point fetched through the runtime) ----
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn tensor_map_encoder();
// 2-D map over a row-major [rows][row_bytes / elem] array; box = box_inner elements x box_rows;
// swizzle: 0 = none, 1 = 128-byte (box rows of 128 bytes), 2 = 64-byte (box rows of 64 bytes)
bool make_map_2d(CUtensorMap* map, CUtensorMapDataType dtype, int elem_bytes, const void* base, uint64_t inner_elems,
                 uint64_t rows, uint64_t row_pitch_bytes, uint32_t box_inner, uint32_t box_rows, int swizzle);

}  // namespace nvfp4
