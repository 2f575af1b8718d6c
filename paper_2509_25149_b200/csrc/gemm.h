// Internal launch interface of the block-scaled GEMM kernel.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "bf16_schedule.h"

namespace nvfp4 {

struct GemmArgs {
  const uint8_t* sfa;     // swizzled scale atoms of A [M x K/16]
  const uint8_t* sfb;     // swizzled scale atoms of B [N x K/16]
  const float* a_global;  // {amax, s_dec}
  const float* b_global;
  void* d;                // [M x N], bf16 or fp32
  int64_t ldd;
  int M, N, K;
  int d_is_fp32, accumulate;
  int mx;                 // operands are MXFP4 (UE8M0 scale per 32 elements) instead of NVFP4
  const float* a_rows;    // per-row {amax, s_dec} pairs of A / B when their global scale is taken per row, else NULL
  const float* b_rows;    // (CTA-pair kernels only)
  int shares;             // launch_gemm_two: parts of the contraction that are summed apart (split_of; 1 otherwise)
};

// Tiles: 128 or 256 = one CTA per 128 x 128 / 128 x 256 tile (256 needs N % 256 == 0, otherwise 128 is used); the others
// run on CTA pairs and take any M and N that are multiples of 128 (a half beyond the edge is computed on zeros and clipped).
constexpr int kTileOne128 = 128;   // 128 x 128, one CTA
constexpr int kTilePair256 = 512;  // 256 x 256
constexpr int kTilePair128 = 640;  // 256 x 128
constexpr int kTileWide = 768;     // 256 x 384, needs N >= 256
constexpr int kTileDouble = 1024;  // BF16: 256 x 512, and 256 x 256 for the columns that are left (chosen by size alone)
constexpr int kTileSplit2 = 642;   // 256 x 128, a cluster of two pairs per tile shares its contraction (K >= 512)
constexpr int kTileSplit4 = 644;   // the same with four pairs (K >= 1024)
cudaError_t launch_gemm(const GemmArgs& g, const void* a_codes, const void* b_codes, int tile, cudaStream_t s);
// CTA pairs that share a tile's contraction when `tile` is asked for: 4, 2 or 1
int split_of(const GemmArgs& g, int tile);
// Two independent GEMMs in one launch of a CTA-pair kernel: the tiles of g0 are worked through first, then those of g1,
// on one persistent grid.  Where either is split when it has a launch to itself (GemmArgs::shares), the sums of both are taken
// in the same order here, on 256 x 128 tiles whatever `tile` says.
cudaError_t launch_gemm_two(const GemmArgs& g0, const void* a0, const void* b0, const GemmArgs& g1, const void* a1,
                            const void* b1, int tile, cudaStream_t s);
// Scheduling estimate: the tile for this problem (or for two problems in one launch, then a whole CTA-pair one)
int best_tile(const GemmArgs& g0, const GemmArgs* g1);
// Measurement aids of the CTA-pair kernel with 256 x 256 tiles (0, 0, NULL = normal operation): mode bit 0 = no MMAs,
// bit 1 = no operand loads, bit 2 = no scale loads / copies, bit 3 = accumulator handed back unread and nothing
// stored, bit 4 = the issuer does not wait for the accumulator (results meaningless with any bit set); max_pairs caps the
// persistent grid; probe = device array of eight 64-bit words per pair (SM cycles and nanoseconds of the issuer's main
// loop, k-blocks, tiles, cycles waiting for the accumulator hand-over; three unused).
void set_gemm_experiment(int mode, int max_pairs, unsigned long long* probe);
cudaError_t read_device_status(cudaStream_t s, uint32_t* code);
// test aid: a bounded wait that is made to run out (a barrier nobody arrives at); leaves kWaitProbeCode in the
// status word and returns by itself
constexpr uint32_t kWaitProbeCode = 0x7E570001u;
cudaError_t launch_wait_probe(unsigned long long limit_ns, cudaStream_t s);
// test aid: how a cluster in which one CTA has given up is left (times: device array of 24 words)
constexpr uint32_t kLeaveProbeCode = 0x7E570002u;
cudaError_t launch_leave_probe(unsigned long long delay_ns, unsigned long long* times, cudaStream_t s);
// device address of the status word on the current device (for kernels of other translation units)
cudaError_t device_status_word(unsigned int** word);

// BF16 GEMM D[M x N] = A B^T on CTA pairs (gemm_bf16.cuh) for layers kept in higher precision.
// a_mn / b_mn = 0: the operand is stored [M or N][K] (contraction contiguous); 1: stored [K][M or N].
// M, N, K multiples of 8 (tiles of 256 x 512, 256 x 256 or 256 x 128, 64 deep, with zero-filled / clipped edges); leading dimensions in
// elements.
struct DenseGemmArgs {
  const void* a;
  const void* b;
  void* d;
  int64_t lda, ldb, ldd;
  int M, N, K;
  int a_mn, b_mn;
  int d_is_fp32, accumulate;
};
// g1 (may be NULL): a second, independent product in the same launch, its tiles after those of g0 (kTileDouble: 512-wide ones of
// both, then 256-wide ones of both)
// The tile of such a launch: kTilePair256, kTilePair128, kTileDouble (*wide: how many column tiles of each product are 512 wide) or a
// split one (`forced`, where every share has a k-block, or by size)
int bf16_tile(const DenseGemmArgs& g0, const DenseGemmArgs* g1, int forced, Bf16Wide* wide);
cudaError_t launch_gemm_bf16(const DenseGemmArgs& g0, const DenseGemmArgs* g1, int tile, const Bf16Wide& wide, cudaStream_t s);

}  // namespace nvfp4
