// BF16 GEMM on CTA pairs (tcgen05 cta_group::2, kind::f16) for the linear layers the recipe leaves in higher
// precision (Section 4.1: the most sensitive layers stay in BF16; Appendix D: every layer late in training).
//   D[M x N] = A * B^T, FP32 accumulation in tensor memory, bf16 or fp32 output, optional accumulation into D.
// Same persistent structure as the block-scaled pair kernel (256 x 256 tiles, each CTA holding its 128 rows of A
// and half of the B tile) minus the scale path; the tensor-memory columns the scales would take hold a second
// accumulator, so a tile's epilogue runs entirely under the next tile's main loop.
//
// Operand layouts.  An operand is "K-major" when the contraction index is contiguous in memory (A stored [M][K],
// B stored [N][K]) and "MN-major" when the output index is (A stored [K][M], B stored [K][N]).  The three GEMMs of a
// layer with row-major X [M x K], W [N x K], dY [M x N] need no transposed copies:
//   Fprop  Y  = X  W^T : A = X  K-major,  B = W  K-major
//   Dgrad  dX = dY W   : A = dY K-major,  B = W  MN-major (contraction over N, W's rows)
//   Wgrad  dW = dY^T X : A = dY MN-major, B = X  MN-major (contraction over the tokens, the rows of both)
// Shared-memory tiles per stage (K = 64 elements): K-major  128 rows x 128 bytes, 128-byte swizzle, 8-row groups
// 1024 bytes apart; MN-major two boxes of 64 k-rows x 128 bytes (64 contiguous output indices each), 8 KB apart.
// One instruction covers K = 16: 32 bytes further along a K-major row, two 8-row groups further in an MN-major box.
// Included by gemm.cu only.
#pragma once

#include "gemm_2cta.cuh"

namespace nvfp4 {
namespace dense {

constexpr int kThreads = 320;       // producer, MMA issuer, 2 x 4 epilogue warps
constexpr int kOperandBytes = 128 * 128;           // 128 rows (or output indices) x 64 bf16
constexpr int kStagingBytes = 2 * 16384;
template <int BN, int SPLIT>
struct Cfg {
  static constexpr int kStages = BN == 512 ? 4 : 6;
  // A, this CTA's half of B.  (32 KB for the narrow tile as well: 24 KB apart, 1024 x 1280 x 4096 takes 24.3 us, not 23.9)
  static constexpr int kStageBytes =
      SPLIT > 1 ? kOperandBytes + BN / 2 * 128 : BN == 512 ? 3 * kOperandBytes : 2 * kOperandBytes;
  static constexpr int kRecvBytes = (SPLIT - 1) * 128 * (BN / SPLIT) * 4;
  static constexpr int kSmemBytes = kStages * kStageBytes + kStagingBytes + 1024 /*alignment*/ + 256 /*barriers*/ + kRecvBytes;
  static_assert(kSmemBytes <= 232448, "shared memory budget");
};
constexpr uint32_t kTmemCols = 512;                // two 256-column accumulators

struct Problem {
  int M, N, K;
  int a_mn, b_mn;  // 1 = the operand is stored with the output index contiguous
  int d_is_fp32, accumulate;
};
// One launch works through the tiles of up to two independent products: Dgrad and Wgrad of a layer fill each other's partial last
// round (4088 x 5128 x 5112: 5 + 6 rounds of 256-wide tiles on 74 pairs become 10).
struct Args {
  Problem p[2];
  int n_tiles0;  // tiles of problem 0, which come first (BN < 512)
  int n_tiles;   // tiles of both problems
  // BN = 512: tiles 512 columns wide of problem 0 and 1, then the tiles 256 wide of both, and where each of these four ends
  int wide_n[2];  // column tiles 512 wide of each problem
  int seg_end[4];
};

// kind::f16 instruction descriptor: FP32 accumulator (bit 4), BF16 x BF16 (format 1 at bits 7 and 10), operand
// major-ness at bits 15 / 16 (0 = K-major), N >> 3 at bit 17, M >> 4 at bit 24
__host__ __device__ constexpr uint32_t instr_desc_bf16(int m, int n, int a_mn, int b_mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) |
         ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ void tc2_mma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                             uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// BN: columns of a tile (512, 256 or 128).  BN = 512: two accumulators side by side share the loads of A, 48 KB per k-block and
// CTA instead of 64; what is left of the columns, and what balances the rounds better, is taken in tiles of 256 (bf16_wide_tiles).
// That is for operands whose rows do not all begin on 32 bytes: a 128-byte row of a box that does not takes 1.75 times as long on the
// SM's path to L2 (with rows an odd multiple of 16 bytes apart 1.375 on average), and 256-wide tiles wait for it.
// The two halves of such a tile begin and end apart (kLead): the epilogue drains one while the tensor pipe works on the other.
// SPLIT > 1 (BN = 128): a cluster of SPLIT pairs takes one tile, the only one of its life,
// each pair a share of the k-blocks (the exchange: pair::exchange_columns).
// TWO: the launch has two problems.
template <int BN, int SPLIT = 1, bool TWO = true>
__global__ void __cluster_dims__(2 * SPLIT, 1, 1) __launch_bounds__(kThreads, 1)
    gemm_bf16_pair_kernel(const __grid_constant__ CUtensorMap map_a0, const __grid_constant__ CUtensorMap map_b0,
                          const __grid_constant__ CUtensorMap map_d0, const __grid_constant__ CUtensorMap map_a1,
                          const __grid_constant__ CUtensorMap map_b1, const __grid_constant__ CUtensorMap map_d1,
                          const __grid_constant__ Args g) {
  using namespace pair;
  constexpr int S = dense::Cfg<BN, SPLIT>::kStages, kStageBytes = dense::Cfg<BN, SPLIT>::kStageBytes;
  constexpr bool kDouble = BN == 512;        // two 256-column halves
  constexpr int HN = kDouble ? 256 : BN;     // columns of an accumulator
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - smem_u32(smem_raw));
  const uint32_t staging = base + S * kStageBytes;
  const uint32_t bar_base = staging + dense::kStagingBytes;
  auto full_bar = [&](int s) { return bar_base + 8u * s; };              // leader only: both CTAs' operands landed
  auto empty_bar = [&](int s) { return bar_base + 8u * (S + s); };       // one per CTA
  auto accf_bar = [&](int b) { return bar_base + 8u * (2 * S + b); };    // one per CTA and accumulator
  auto acce_bar = [&](int b) { return bar_base + 8u * (2 * S + 2 + b); };  // leader only, 16 arrivals
  const uint32_t done_bar = bar_base + 8u * (2 * S + 4);
  const uint32_t recv_bar = done_bar + 16;                               // SPLIT > 1: all shares are here
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(
      base_ptr + S * kStageBytes + dense::kStagingBytes + 8 * (2 * S + 5));
  volatile uint32_t* abort_flag = tmem_slot + 1;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t cta = cluster_ctarank();
  const uint32_t rank = SPLIT > 1 ? cta & 1u : cta;          // in the pair, 0 = leader
  const uint32_t leader_cta = SPLIT > 1 ? cta & ~1u : 0u;    // the leader's rank in the cluster
  const uint16_t pair_mask = (uint16_t)(3u << leader_cta);   // both CTAs of the pair
  const int split = SPLIT > 1 ? (int)(cta >> 1) : 0;         // which share of the contraction
  const bool leader = rank == 0;
  const int pair_id = blockIdx.x / (2 * SPLIT), n_pairs = gridDim.x / (2 * SPLIT);  // (SPLIT > 1: clusters)
  // ragged edges: loads beyond the operands read zeros, stores beyond D are clipped (both by the tensor maps)
  const int n_tiles = g.n_tiles;
  auto prob_of = [&](int tile) {
    if (kDouble) return TWO ? ((tile >= g.seg_end[0] && tile < g.seg_end[1]) || tile >= g.seg_end[2] ? 1 : 0) : 0;
    return TWO && tile >= g.n_tiles0 ? 1 : 0;
  };
  auto halves_of = [&](int tile) { return kDouble && tile < g.seg_end[1] ? 2 : 1; };
  auto k_begin = [&](int tile, int s) {  // first k-block of share s
    const int n = (g.p[prob_of(tile)].K + 63) / 64;
    return SPLIT > 1 ? n * s / SPLIT : n * s;
  };
  // rounds of the pairs; kDouble: odd ones in reverse order, which evens out tiles of different cost
  auto next_tile = [&](int rnd) { return rnd * n_pairs + (kDouble && (rnd & 1) ? n_pairs - 1 - pair_id : pair_id); };
  // groups of eight row-blocks sweep all column-blocks before the next group starts (L2 reuse of A and B);
  // n_blk: the tile's first column in units of HN
  constexpr int kGroupM = 8;
  auto tile_coords = [&](int tile, int& prob, int& m_blk, int& n_blk) {
    prob = prob_of(tile);
    int tiles_n = (g.p[prob].N + HN - 1) / HN, n_first = 0, n_step = 1;
    if constexpr (kDouble) {
      const int seg = (tile >= g.seg_end[0]) + (tile >= g.seg_end[1]) + (tile >= g.seg_end[2]);
      if (seg) tile -= g.seg_end[seg - 1];
      if (seg < 2) {
        tiles_n = g.wide_n[prob];
        n_step = 2;
      } else {
        n_first = 2 * g.wide_n[prob];
        tiles_n -= n_first;
      }
    } else if (prob) {
      tile -= g.n_tiles0;
    }
    const int tiles_m = (g.p[prob].M + 255) / 256;
    const int per_group = kGroupM * tiles_n;
    const int grp = tile / per_group, in_grp = tile - grp * per_group;
    const int m0 = grp * kGroupM;
    const int gm = (tiles_m - m0 < kGroupM) ? (tiles_m - m0) : kGroupM;
    m_blk = m0 + in_grp % gm;
    n_blk = n_first + n_step * (in_grp / gm);
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(full_bar(s), 2);  // one arrive.expect_tx from each CTA's producer
      mbar_init(empty_bar(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(accf_bar(b), 1);
      mbar_init(acce_bar(b), 16);  // eight epilogue warps in each CTA
    }
    mbar_init(done_bar, 2 * SPLIT - 1);
    if (SPLIT > 1) mbar_init(recv_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (SPLIT > 1) mbar_expect_tx(recv_bar, dense::Cfg<BN, SPLIT>::kRecvBytes);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32((const void*)tmem_slot)),
                 "r"(dense::kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // both CTAs' barriers are initialised before any remote signal
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
      for (int rnd = 0, tile = pair_id; tile < n_tiles && ok; tile = next_tile(++rnd)) {
        int prob, m_blk, n_blk;
        tile_coords(tile, prob, m_blk, n_blk);
        const int row_a = m_blk * 256 + (int)rank * 128;  // this CTA's rows of A
        const int row_b = n_blk * HN + (int)rank * (HN / 2);  // this CTA's half of the B tile (of its first 256 columns)
        const int halves = halves_of(tile);
        const int k_end = k_begin(tile, split + 1);
        // One copy of the loop for each problem of the launch, with its tensor maps and layouts at fixed places of the parameter
        // bank: with the maps picked by pointer the loads of a stage were issued so late that a pair could not go faster even
        // when it had L2 to itself (last rounds): forward of 3632 x 1552 x 3136 41.0 us, now 35.4, backward 67.6, now 63.4.
        auto load_tile = [&](const CUtensorMap* map_a, const CUtensorMap* map_b, const Problem& pr) {
          for (int kb = k_begin(tile, split); kb < k_end; ++kb) {
            if (!(ok = mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, 0x900u + stage))) break;
            const uint32_t st = base + stage * kStageBytes;
            const uint32_t bar = map_to_cta(full_bar(stage), leader_cta);  // the leader's barrier counts both CTAs' operands
            mbar_expect_tx_cluster(bar, dense::kOperandBytes + (kDouble ? halves * dense::kOperandBytes : BN / 2 * 128));
            if (pr.a_mn) {
              tma_load_2d_pair(st, map_a, row_a, kb * 64, bar);
              tma_load_2d_pair(st + 8192, map_a, row_a + 64, kb * 64, bar);
            } else {
              tma_load_2d_pair(st, map_a, kb * 64, row_a, bar);
            }
#pragma unroll
            for (int h = 0; h < (kDouble ? 2 : 1); ++h) {
              if (h >= halves) break;
              const uint32_t st_b = st + (1 + h) * dense::kOperandBytes;
              if (pr.b_mn) {
                tma_load_2d_pair(st_b, map_b, row_b + 256 * h, kb * 64, bar);
                if (HN == 256) tma_load_2d_pair(st_b + 8192, map_b, row_b + 256 * h + 64, kb * 64, bar);
              } else {
                tma_load_2d_pair(st_b, map_b, kb * 64, row_b + 256 * h, bar);
              }
            }
            if (++stage == S) {
              stage = 0;
              phase ^= 1u;
            }
          }
        };
        if (!TWO || prob == 0)
          load_tile(&map_a0, &map_b0, g.p[0]);
        else
          load_tile(&map_a1, &map_b1, g.p[1]);
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer (leader) ----
    if (leader && lane == 0) {
      int stage = 0;
      uint32_t phase = 0, acc_phase = 0;  // bit b: phase of accumulator b's barrier
      bool ok = true;
      // descriptor halves: start address and leading byte offset (low word), stride byte offset / version /
      // 128-byte swizzle (high word).  K-major: 8-row groups 1024 bytes apart, leading offset unused.  MN-major:
      // 64-index boxes 8192 bytes apart (leading), 8-row k groups 1024 bytes apart (stride).
      const uint32_t a_lo_base = (base >> 4) & 0x3fffu, b_lo_base = ((base + dense::kOperandBytes) >> 4) & 0x3fffu;
      int buf = 0;
      auto acc_free = [&](int b) {
        return mbar_wait_cluster(acce_bar(b), ((acc_phase >> b) & 1u) ^ 1u, abort_flag, 0xB00u + b);
      };
      for (int rnd = 0, tile = pair_id; tile < n_tiles && ok; tile = next_tile(++rnd)) {
        const bool both = halves_of(tile) == 2;
        if (both) buf = 0;
        if (!(ok = acc_free(buf))) break;
        tc_fence_after();
        const int k_blocks = k_begin(tile, split + 1) - k_begin(tile, split);
        // (one copy of the loop for each problem, as in the producer)
        auto main_loop = [&](const Problem& pr) {
          const uint32_t idesc = instr_desc_bf16(256, HN, pr.a_mn, pr.b_mn);
          const uint32_t a_lo0 = a_lo_base | ((pr.a_mn ? (8192u >> 4) : 1u) << 16);
          const uint32_t b_lo0 = b_lo_base | ((pr.b_mn ? (8192u >> 4) : 1u) << 16);
          const uint32_t a_step = pr.a_mn ? (2048u >> 4) : (32u >> 4);  // one K = 16 instruction further
          const uint32_t b_step = pr.b_mn ? (2048u >> 4) : (32u >> 4);
          auto mma = [&](int st, int half, int acc, bool first) {  // a k-block of one half
            const uint32_t a_lo = a_lo0 + st * (kStageBytes >> 4);
            const uint32_t b_lo = b_lo0 + st * (kStageBytes >> 4) + half * (dense::kOperandBytes >> 4);
#pragma unroll
            for (int j = 0; j < 4; ++j)
              tc2_mma_bf16(tmem + acc * 256, make_desc(a_lo + j * a_step, kDescHiOperand),
                           make_desc(b_lo + j * b_step, kDescHiOperand), idesc, (!first || j > 0) ? 1u : 0u);
          };
          auto landed = [&](int st, uint32_t ph) {
            if (!(ok = mbar_wait_cluster(full_bar(st), ph, abort_flag, 0xA00u + st))) return false;
            tc_fence_after();
            return true;
          };
          auto release = [&] {
            tc2_commit_both(empty_bar(stage), pair_mask);  // both CTAs' stages are free once these MMAs have read them
            if (++stage == S) {
              stage = 0;
              phase ^= 1u;
            }
          };
          if constexpr (kDouble) {
            if (both) {
              // runs of up to kLead k-blocks of the first half and then of the second at either end of the tile, half by
              // half in between
              constexpr int kLead = 3;
              for (int kb = 0; kb < k_blocks;) {
                const int left = k_blocks - kb;
                const int run = kb == 0 || left <= kLead ? min(left, kLead) : 1;
                for (int i = 0; i < run; ++i) {
                  const int st = stage + i < S ? stage + i : stage + i - S;
                  if (!landed(st, phase ^ (stage + i < S ? 0u : 1u))) return;
                  mma(st, 0, 0, kb + i == 0);
                }
                if (kb + run == k_blocks) tc2_commit_both(accf_bar(0), pair_mask);  // the first accumulator is complete
                if (kb == 0) {
                  if (!(ok = acc_free(1))) return;
                  tc_fence_after();
                }
                for (int i = 0; i < run; ++i) {
                  mma(stage, 1, 1, kb + i == 0);
                  release();
                }
                kb += run;
              }
              return;
            }
          }
          for (int kb = 0; kb < k_blocks; ++kb) {
            if (!landed(stage, phase)) return;
            mma(stage, 0, buf, kb == 0);
            release();
          }
        };
        if (!TWO || prob_of(tile) == 0)
          main_loop(g.p[0]);
        else
          main_loop(g.p[1]);
        if (!ok) break;
        if (both) {
          tc2_commit_both(accf_bar(1), pair_mask);
          acc_phase ^= 3u;
        } else {
          tc2_commit_both(accf_bar(buf), pair_mask);  // this accumulator is complete in both CTAs
          acc_phase ^= 1u << buf;
          buf ^= 1;
        }
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue (warps 2-9) ----
    const int quad = warp & 3;              // tensor-memory lanes this warp may read
    const int half = (warp - 2) >> 2;       // column half / epilogue group
    const int et = (threadIdx.x - 64) & 127;  // 0..127 inside the group
    const int bar_id = 1 + half;
    uint32_t acc_phase = 0;
    const int row_in_tile = quad * 32 + lane;
    const uint32_t stage_buf = staging + half * 16384;
    int buf = 0, last_prob = 0, halves = 1;
    // (kDouble: a tile comes up once for each of its halves, the second time without a step of the walk)
    for (int rnd = 0, half_no = 0, tile = pair_id; tile < n_tiles; tile = half_no ? tile : next_tile(++rnd)) {
      int prob, m_blk, n_blk;
      tile_coords(tile, prob, m_blk, n_blk);
      if constexpr (kDouble) {
        halves = halves_of(tile);
        if (halves == 2) {
          buf = half_no;
          n_blk += half_no;
        }
      }
      const CUtensorMap* map_d = prob ? &map_d1 : &map_d0;
      const bool drain = prob != last_prob;  // the problems of a launch may have different output types
      last_prob = prob;
      mbar_wait_cluster(accf_bar(buf), (acc_phase >> buf) & 1u, abort_flag, 0xC00u + buf);
      // agree on giving up: a warp that timed out still joins this barrier, and all 128 threads take ONE decision
      if (group_gave_up(abort_flag, bar_id, 128)) break;
      tc_fence_after();
      const int row0 = m_blk * 256 + (int)rank * 128;
      const uint32_t t_row = tmem + ((uint32_t)(quad * 32) << 16) + buf * 256 + half * (HN / 2);
      uint32_t r[HN / 2];
#pragma unroll
      for (int q = 0; q < HN / 32; ++q) tc_ld16(t_row + q * 16, *reinterpret_cast<uint32_t(*)[16]>(&r[q * 16]));
      tc_wait_ld();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(map_to_cta(acce_bar(buf), leader_cta));
      if constexpr (SPLIT > 1) {
        constexpr int kCols = BN / SPLIT;
        uint32_t v[kCols];
        if (!exchange_columns<SPLIT>(r, v, half, split, rank, staging + dense::kStagingBytes + 256, recv_bar, row_in_tile,
                                     abort_flag, bar_id))
          break;
        const int xs = n_blk * BN + split * kCols;
        if (g.p[prob].d_is_fp32)
          store_half<true, false, kCols>(v, 1.0f, et, bar_id, row_in_tile, stage_buf, map_d, xs, row0, g.p[prob].accumulate, drain);
        else
          store_half<false, false, kCols>(v, 1.0f, et, bar_id, row_in_tile, stage_buf, map_d, xs, row0, g.p[prob].accumulate, drain);
      } else if (g.p[prob].d_is_fp32)
        store_half<true, false, HN / 2>(r, 1.0f, et, bar_id, row_in_tile, stage_buf, map_d, n_blk * HN + half * (HN / 2),
                                        row0, g.p[prob].accumulate, drain);
      else
        store_half<false, false, HN / 2>(r, 1.0f, et, bar_id, row_in_tile, stage_buf, map_d, n_blk * HN + half * (HN / 2),
                                         row0, g.p[prob].accumulate, drain);
      acc_phase ^= 1u << buf;
      buf = halves == 2 ? 0 : buf ^ 1;
      if (kDouble) half_no = halves == 2 ? half_no ^ 1 : 0;
    }
    if (et == 0) bulk_wait_all<0>();  // all stores have left shared memory and are visible
  }

  // ------------------------------------------------------------------ teardown ----
  tc_fence_before();
  leave_cluster<2 * SPLIT>(done_bar, cta, abort_flag, 0xD00u);
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(dense::kTmemCols) : "memory");
  }
}

}  // namespace dense
}  // namespace nvfp4
