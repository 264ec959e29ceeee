// Stand-alone linear layer of many tokens: the tile of two SMs.
//
// A pair of CTAs (one per SM, a cluster) works on 256 tokens x up to 256 features with tcgen05.mma.cta_group::2: each CTA
// stages its own 128 tokens and its own half of the weight rows, the leader issues MMAs that read both SMs' shared memory, and
// each CTA's tensor memory receives its own tokens' rows.  An SM so loads 32 KB per 256 x 256 x 64 block where two separate
// 128 x 256 tiles load 48 KB, and the L2-to-shared-memory path is what bounds the layer.  Two accumulators of 256 columns: the
// eight epilogue warps store one tile while the MMAs of the next run (or two to four accumulators that take a part of K each, where the
// sums of an fp32 result are kept short).  Persistent, one CTA per SM.  4096 x 4096 x 4096 114 -> 96 us
// (1.43 PFLOP/s), 8192 x 3072 x 768 with GELU 47.7 -> 42.2 called from Python on new inputs: 700 cycles a k-block of 512 cycles of MMA,
// since a lone CTA gets 47 B/clk from L2 whichever warps ask (two of them loading one operand each changed nothing).
#pragma once
#include "op_linear.cuh"

namespace vla {

constexpr int LINP_TMEM_COLS = 512;            // all there is

__device__ __forceinline__ void tmem_alloc_pair(uint32_t* smem_dst, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_dst)), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
// A load into this CTA's shared memory that reports to a barrier of the pair's leader (`bar`: cluster address).
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const void* tmap, uint32_t bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(tmap), "r"(bar), "r"(x), "r"(y)
      : "memory");
}
__device__ __forceinline__ void umma_bf16_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}
// Arrives at the barriers of this offset in both CTAs when the MMAs issued so far are complete.
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"((unsigned short)3) : "memory");
}

// PARTS: accumulators that take a part of K each (a kernel of its own for 1: worked out at run time, 8192 x 3072 x 768 42.2 -> 44.2 us).
template <int VEC, bool PARTS>
__global__ void __launch_bounds__(LIN_THREADS, 1) vla_op_linear_pair_kernel(const __grid_constant__ LinearArgs g, const __grid_constant__ OpMaps maps,
                                                                            OpFault fault) {
  extern __shared__ __align__(1024) char smem_raw[];
  __shared__ uint32_t tmem_base_s;
  __shared__ __align__(8) uint64_t bars[2 * LIN_MAX_STAGES + 4];       // full (the leader's count), empty; accumulators full (2), empty (2, the leader's)
  __shared__ unsigned failed_s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rank = (int)blockIdx.x & 1;
  const int S = g.stages, first_tile = (int)blockIdx.x >> 1, step = (int)gridDim.x >> 1, nkb = g.kp / GEMM_BK;
  const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8u * LIN_MAX_STAGES, accf0 = empty0 + 8u * LIN_MAX_STAGES, acce0 = accf0 + 16u;
  const uint32_t a_bytes = (uint32_t)(g.bm * GEMM_BK * 2), stage_bytes = a_bytes + (uint32_t)(g.bn / 2 * GEMM_BK * 2);
  const uint32_t stage0 = smem_u32(smem_raw);
  if (warp == 0) {
    if (lane < 2 * LIN_MAX_STAGES + 4) {
      mbar_init(full0 + 8u * lane, lane < 2 * LIN_MAX_STAGES + 2 ? 1 : 2 * LIN_EPI_WARPS);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (lane == 0) failed_s = 0;
  } else if (warp == 1) {
    tmem_alloc_pair(&tmem_base_s, LINP_TMEM_COLS);
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();                              // both CTAs' barriers and tensor memory are there
  tc_fence_after();
  op_wait_previous(maps, 2);
  if (threadIdx.x == 0 && blockIdx.x == 0) *g.err = 0u;
  TileCtx c;                                   // (what the bounded waits look at)
  c.error = &failed_s;
  c.deadline = gtimer() + fault.wait_limit_ns;
  op_let_next_start();
  const uint32_t tmem = tmem_base_s;
  // An accumulator for each of the parts K is summed in, and where there is room two sets of them.
  const int parts = PARTS ? g.ks : 1;
  const uint32_t sets = !PARTS || 2 * parts * g.bn <= LINP_TMEM_COLS ? 2u : 1u, part_cols = LINP_TMEM_COLS / (sets * (uint32_t)parts), set_cols = part_cols * (uint32_t)parts;
  bool ok = true;
  if (warp == 0) {
    if (lane == 0 && !fault.drop_loads) {
      uint32_t s = 0, ph = 1u;
      const uint32_t full_leader = cluster_addr(full0, 0u);
      for (int t = first_tile; t < g.tiles && ok; t += step) {
        const int tm = t % g.tiles_m, row0 = (2 * tm + rank) * g.bm, n0 = t / g.tiles_m * g.bn + rank * (g.bn / 2);
#pragma unroll 1
        for (int kb = 0; kb < nkb; ++kb) {
          const uint32_t dst = stage0 + s * stage_bytes;
          if (!(ok = mbar_wait(c, empty0 + 8u * s, ph))) break;
          if (rank == 0) mbar_expect_tx(full0 + 8u * s, 2u * stage_bytes);
          tma_load_2d_pair(dst + a_bytes, &maps.m[0], full_leader + 8u * s, kb * GEMM_BK, n0);
          tma_load_2d_pair(dst, &maps.m[1], full_leader + 8u * s, kb * GEMM_BK, row0);
          // weights come from HBM once: the first token tile's CTAs ask for them ahead, so that a stage waits for L2 only
          if (tm == 0 && kb + LIN_AHEAD < nkb) tma_prefetch_2d(&maps.m[0], (kb + LIN_AHEAD) * GEMM_BK, n0);
          if (++s == (uint32_t)S) { s = 0; ph ^= 1u; }
        }
      }
      if (!ok) for (int i = 0; i < 100; ++i) __nanosleep(1000);      // gave up: the copies in flight land before the pair ends
    }
    __syncwarp();
  } else if (warp == 1) {
    if (rank == 0) {
      const uint32_t idesc = umma_idesc_bf16(g.bn, 256);
      const uint64_t desc0 = umma_desc_sw128(stage0);
      uint32_t s = 0, ph = 0u, buf = 0, bph = 1u;
      // A stage is released where a later k-block is loaded into it (in both CTAs, whose producers wait for that): an arrival that
      // nobody waits for could come when the other CTA has ended and its shared memory is somebody else's.
      int left = first_tile < g.tiles ? ((g.tiles - 1 - first_tile) / step + 1) * nkb : 0;
      for (int t = first_tile; t < g.tiles && ok; t += step) {
        if (!(ok = mbar_wait(c, acce0 + 8u * buf, bph))) break;
        tc_fence_after();
        int part = 0, from = 0, to = nkb / parts;                     // k-blocks of this part
#pragma unroll 1
        for (int kb = 0; kb < nkb; ++kb, --left) {
          if (PARTS && kb == to) { ++part; from = to; to = nkb * (part + 1) / parts; }
          if (!(ok = mbar_wait(c, full0 + 8u * s, ph))) break;
          tc_fence_after();
          const uint64_t ad = desc0 + s * (stage_bytes >> 4), wd = ad + (a_bytes >> 4);
          const uint32_t acc = tmem + set_cols * buf + part_cols * (uint32_t)part;
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < GEMM_BK / 16; ++k) umma_bf16_pair(acc, ad + 2u * k, wd + 2u * k, idesc, kb != from || k != 0 ? 1u : 0u);
            if (left > S) umma_commit_pair(empty0 + 8u * s);
            if (kb == nkb - 1) umma_commit_pair(accf0 + 8u * buf);
          }
          __syncwarp();
          if (++s == (uint32_t)S) { s = 0; ph ^= 1u; }
        }
        if (++buf == sets) { buf = 0; bph ^= 1u; }
      }
    }
  } else {
    const int quarter = warp & 3, half = warp >= 6 ? 1 : 0;           // (epilogue warps 2..9: a quarter of the lanes is fixed by warp % 4)
    const uint32_t lanes = (uint32_t)(quarter * 32) << 16, acce_leader = cluster_addr(acce0, 0u);
    const int groups = (g.bn + 31) / 32, mid = (groups + 1) / 2, lo = half ? mid : 0, hi = half ? groups : mid;
    uint32_t buf = 0, bph = 0u;
    for (int t = first_tile; t < g.tiles; t += step) {
      const uint32_t acc = tmem + set_cols * buf + lanes;
      if (!mbar_wait(c, accf0 + 8u * buf, bph)) break;
      __syncwarp();
      tc_fence_after();
      const int cta_row = (2 * (t % g.tiles_m) + rank) * g.bm, row0 = cta_row + 32 * quarter, rows = min(g.bm, g.m - cta_row) - 32 * quarter;
      const int n0 = t / g.tiles_m * g.bn;
      LinearArgs gg = g;
      gg.m = row0 + max(rows, 0);                                     // (this tile's rows and features only)
      gg.n_end = min(g.n, n0 + g.bn);
      if (g.act == ACT_GELU) linear_rows<ACT_GELU, VEC>(gg, acc, lane, row0, rows, n0, lo, hi, nullptr, 0, 0, PARTS ? parts : 1, part_cols);
      else if (g.act == ACT_SILU) linear_rows<ACT_SILU, VEC>(gg, acc, lane, row0, rows, n0, lo, hi, nullptr, 0, 0, PARTS ? parts : 1, part_cols);
      else linear_rows<ACT_NONE, VEC>(gg, acc, lane, row0, rows, n0, lo, hi, nullptr, 0, 0, PARTS ? parts : 1, part_cols);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(acce_leader + 8u * buf) : "memory");
      if (++buf == sets) { buf = 0; bph ^= 1u; }
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();                              // nobody reads or signals the other CTA any more
  if (warp == 1) tmem_dealloc_pair(tmem, LINP_TMEM_COLS);
  if (threadIdx.x == 0 && *reinterpret_cast<volatile unsigned*>(&failed_s) != 0u) *g.err = (unsigned)DEV_ERR_WAIT_MBAR;
  cluster_sync();                              // (both have given their columns back)
}

}  // namespace vla
