// Stand-alone linear layer: y = act(a w^T) as a kernel of its own, persistent and warp-specialised (the engine's GEMM tile
// is built to share an SM with two strangers; a call that has the GPU to itself can do better).
//
// CTA: 192 threads -- a TMA warp, an MMA warp, four epilogue warps -- and half an SM's shared and tensor memory, two CTAs
// per SM: one CTA's loads alone do not saturate the L2-to-shared-memory path (47 of 70 B/clk), and one CTA's epilogue runs
// beside the other's main loop.  Tile: up to 128 tokens (MMA M, a TMEM lane each) x bn features (MMA N), K in 64-element
// stages with both operands K-major.  Where there are few tokens the activation box is only as high as they need, and the
// MMA's further rows read whatever lies behind it (lanes nobody looks at).
//
// What bounds it: large shapes the L2-to-shared-memory path (48 KB per 512 tensor-core cycles at bn = 256), small ones the
// chain launch -> operand round trip -> 50 cycles per MMA -> stores; so bn is as wide as still gives every SM work
// (linear_plan).
#pragma once
#include "dispatch.cuh"

namespace vla {

constexpr int LIN_THREADS = 192;
constexpr int LIN_MAX_STAGES = 12;
constexpr int LIN_SMEM = 112 * 1024;          // half an SM
constexpr int LIN_TMEM_COLS = 256;            // half an SM: two accumulators of up to 128 columns, or one of 256

struct LinearArgs {
  int m, n, kp, bm, bn, tiles_m, tiles, stages, act;
  int vec16;                                  // rows of the results allow 16-byte stores, n whole chunks of 16
  float* out32;
  unsigned short* out16;
  unsigned* err;                              // gets `call` when a wait runs out
  unsigned call;
};

// Tile shape of a call.  Tokens: as few tiles as hold them, of equal height.  Features: the widest tile that still gives
// about two tiles to every SM's pair of CTAs; below that narrower tiles win as long as SMs would idle (16 is the MMA's
// narrowest step and costs as much time per k-step as 64, so the work grows with the tile count while the chain shortens).
inline void linear_plan(LinearArgs& g, int sms) {
  g.tiles_m = (g.m + 127) / 128;
  g.bm = (int)(((g.m + g.tiles_m - 1) / g.tiles_m + 15) / 16 * 16);
  g.bn = 256;
  while (g.bn > 16 && (long long)g.tiles_m * ((g.n + g.bn - 1) / g.bn) < (g.bn > 64 ? 2 * sms : sms)) g.bn >>= 1;
  if (g.bn < 64 && (long long)g.tiles_m * ((g.n + g.bn - 1) / g.bn) > 2 * sms) g.bn <<= 1;
  g.tiles = g.tiles_m * ((g.n + g.bn - 1) / g.bn);
  const int stage = (g.bm + g.bn) * GEMM_BK * 2, tail = stage < 16384 ? 16384 - stage : 0;    // the MMA always reads 128 rows
  const int nkb = g.kp / GEMM_BK;
  g.stages = (LIN_SMEM - tail) / stage;
  if (g.stages > LIN_MAX_STAGES) g.stages = LIN_MAX_STAGES;
}
inline int linear_smem(const LinearArgs& g) {
  const int stage = (g.bm + g.bn) * GEMM_BK * 2;
  return g.stages * stage + (stage < 16384 ? 16384 - stage : 0);
}

template <int ACT>
__device__ __forceinline__ void linear_rows(const LinearArgs& g, uint32_t tmem, int row, bool live, int n0, int cols) {
  float* const o32 = g.out32 ? g.out32 + (size_t)row * g.n + n0 : nullptr;
  unsigned short* const o16 = g.out16 ? g.out16 + (size_t)row * g.n + n0 : nullptr;
  epi_chunks(tmem, 0, (cols + EPI - 1) / EPI * EPI, 1.0f, [&](int c0, float* v) {
    activate<ACT, EPI>(v);
    if (!live) return;
    if (g.vec16) {
      if (o32) {
#pragma unroll
        for (int j = 0; j < EPI; j += 4) *reinterpret_cast<float4*>(o32 + c0 + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
      }
      if (o16) put16(o16 + c0, v);
    } else {
#pragma unroll
      for (int j = 0; j < EPI; ++j)
        if (c0 + j < cols) {
          if (o32) o32[c0 + j] = v[j];
          if (o16) o16[c0 + j] = f32_to_bf16_bits(v[j]);
        }
    }
  });
}

__global__ void __launch_bounds__(LIN_THREADS, 2) vla_op_linear_kernel(const __grid_constant__ LinearArgs g, const __grid_constant__ OpMaps maps,
                                                                       OpFault fault) {
  extern __shared__ __align__(1024) char smem_raw[];
  __shared__ uint32_t tmem_base_s;
  __shared__ __align__(8) uint64_t bars[2 * LIN_MAX_STAGES + 4];       // full, empty; accumulators full (2), empty (2)
  __shared__ unsigned failed_s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int S = g.stages, nkb = g.kp / GEMM_BK, n_acc = g.bn <= 128 ? 2 : 1;
  const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8u * LIN_MAX_STAGES, accf0 = empty0 + 8u * LIN_MAX_STAGES, acce0 = accf0 + 16u;
  const uint32_t a_bytes = (uint32_t)(g.bm * GEMM_BK * 2), stage_bytes = (uint32_t)((g.bm + g.bn) * GEMM_BK * 2);
  const uint32_t stage0 = smem_u32(smem_raw);
  if (warp == 0) {
    if (lane < 2 * LIN_MAX_STAGES + 4) {
      mbar_init(full0 + 8u * lane, lane < 2 * LIN_MAX_STAGES + 2 ? 1 : 4);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (lane == 0) failed_s = 0;
  } else if (warp == 1) {
    tmem_alloc(&tmem_base_s, LIN_TMEM_COLS);
  }
  TileCtx c;                                   // (what the bounded waits look at)
  c.error = &failed_s;
  c.deadline = gtimer() + fault.wait_limit_ns;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_s;
  bool ok = true;
  if (warp == 0) {
    if (lane == 0 && !fault.drop_loads) {
      uint32_t s = 0, ph = 1u;
      for (int t = blockIdx.x; t < g.tiles && ok; t += gridDim.x) {
        const int row0 = t % g.tiles_m * g.bm, n0 = t / g.tiles_m * g.bn;
#pragma unroll 1
        for (int kb = 0; kb < nkb; ++kb) {
          const uint32_t full = full0 + 8u * s, dst = stage0 + s * stage_bytes;
          if (!(ok = mbar_wait(c, empty0 + 8u * s, ph))) break;
          mbar_expect_tx(full, stage_bytes);
          tma_load_2d(dst + a_bytes, &maps.m[0], full, kb * GEMM_BK, n0);
          tma_load_2d(dst, &maps.m[1], full, kb * GEMM_BK, row0);
          if (++s == (uint32_t)S) { s = 0; ph ^= 1u; }
        }
      }
      if (!ok) for (int i = 0; i < 100; ++i) __nanosleep(1000);      // gave up: the copies in flight land before the CTA ends
    }
    __syncwarp();
  } else if (warp == 1) {
    const uint32_t idesc = umma_idesc_bf16(g.bn);
    const uint64_t desc0 = umma_desc_sw128(stage0);
    uint32_t s = 0, ph = 0u, i = 0;
    for (int t = blockIdx.x; t < g.tiles && ok; t += gridDim.x, ++i) {
      const uint32_t buf = n_acc == 2 ? i & 1u : 0u, use = n_acc == 2 ? i >> 1 : i;
      if (!(ok = mbar_wait(c, acce0 + 8u * buf, (use & 1u) ^ 1u))) break;
      tc_fence_after();
#pragma unroll 1
      for (int kb = 0; kb < nkb; ++kb) {
        if (!(ok = mbar_wait(c, full0 + 8u * s, ph))) break;
        tc_fence_after();
        const uint64_t ad = desc0 + s * (stage_bytes >> 4), wd = ad + (a_bytes >> 4);
        if (elect_one()) {
#pragma unroll
          for (int k = 0; k < GEMM_BK / 16; ++k) umma_bf16(tmem + 128u * buf, ad + 2u * k, wd + 2u * k, idesc, (kb | k) != 0 ? 1u : 0u);
          umma_commit(empty0 + 8u * s);
          if (kb == nkb - 1) umma_commit(accf0 + 8u * buf);
        }
        __syncwarp();
        if (++s == (uint32_t)S) { s = 0; ph ^= 1u; }
      }
    }
  } else {
    uint32_t i = 0;
    const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16;
    for (int t = blockIdx.x; t < g.tiles; t += gridDim.x, ++i) {
      const uint32_t buf = n_acc == 2 ? i & 1u : 0u, use = n_acc == 2 ? i >> 1 : i;
      if (!mbar_wait(c, accf0 + 8u * buf, use & 1u)) break;
      __syncwarp();
      tc_fence_after();
      const int row0 = t % g.tiles_m * g.bm, n0 = t / g.tiles_m * g.bn, r = (warp & 3) * 32 + lane;
      const int rows = min(g.bm, g.m - row0), cols = min(g.bn, g.n - n0);
      if ((warp & 3) * 32 < rows) {
        const int row = row0 + min(r, rows - 1);
        if (g.act == ACT_GELU) linear_rows<ACT_GELU>(g, tmem + lanes + 128u * buf, row, r < rows, n0, cols);
        else if (g.act == ACT_SILU) linear_rows<ACT_SILU>(g, tmem + lanes + 128u * buf, row, r < rows, n0, cols);
        else linear_rows<ACT_NONE>(g, tmem + lanes + 128u * buf, row, r < rows, n0, cols);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(acce0 + 8u * buf) : "memory");
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, LIN_TMEM_COLS);
  if (threadIdx.x == 0 && *reinterpret_cast<volatile unsigned*>(&failed_s) != 0u) *g.err = g.call;
}

}  // namespace vla
