// Stand-alone linear layer: y = act(a w^T) as a kernel of its own, persistent and warp-specialised (the engine's GEMM tile
// is built to share an SM with two strangers; a call that has the GPU to itself can do better).
//
// CTA: 320 threads -- a TMA warp, an MMA warp, eight epilogue warps (two per quarter of the lanes, each half of the columns)
// -- and half an SM's shared and tensor memory, two CTAs per SM: one CTA's loads alone do not saturate the
// L2-to-shared-memory path (47 of 70 B/clk), and one CTA's epilogue runs beside the other's main loop.  Tile: up to 128
// tokens (MMA M, a TMEM lane each) x bn features (MMA N), K in 64-element stages with both operands K-major.  Where there
// are few tokens the activation box is only as high as they need, and the MMA's further rows read whatever lies behind it
// (lanes nobody looks at).  Where there are few tiles a cluster of `ks` CTAs shares the K range of one and adds up in
// distributed shared memory, each CTA its share of the columns.
#pragma once
#include "dispatch.cuh"
#include "linear_plan.h"

namespace vla {

constexpr int LIN_EPI_WARPS = 8;
constexpr int LIN_THREADS = 64 + 32 * LIN_EPI_WARPS;
constexpr int LIN_AHEAD = 8;                  // k-blocks
constexpr int LIN_TMEM_COLS = 256;            // half an SM: two accumulators of up to 128 columns, or one of 256

struct LinearArgs {
  int m, n, n_end, kp, bm, bn, ks, tiles_m, tiles, stages, act;
  float* out32;
  unsigned short* out16;
  unsigned* err;                              // 0, or why a wait ran out
};

// Features a store may cover: what every row's start and the width allow.  Eight go out as 16 bytes of bf16 or four pairs of
// fp32, two as a pair, and an odd width (or address) leaves single elements.  8192 tokens, K = 768, GELU, bf16: 3072 features 40 us,
// 3076 in pairs 47 (96 in single elements), 3073 105; K = 64 without GELU 13.7, 24 (71), 87.  A kernel for each: chosen at run time
// inside one, the branches cost the wide rows 3 %.
inline int linear_vec(int n, const float* out32, const void* out16) {
  const uintptr_t a32 = reinterpret_cast<uintptr_t>(out32), a16 = reinterpret_cast<uintptr_t>(out16);
  if (n % 8 == 0 && ((a32 | a16) & 15) == 0) return 8;
  return n % 2 == 0 && (a32 & 7) == 0 && (a16 & 3) == 0 ? 2 : 1;
}
inline int linear_smem(const LinearArgs& g) {
  const int stage = (g.bm + g.bn) * GEMM_BK * 2;
  return g.stages * stage + (stage < 16384 ? 16384 - stage : 0);
}

// 4 x 4 transposition of one register each over a quad: lane q gets the four lanes' w[q], in lane order.
__device__ __forceinline__ void quad_transpose(uint32_t* w, int q) {
  const bool o1 = (q & 1) != 0, o2 = (q & 2) != 0;
#pragma unroll
  for (int b = 0; b < 4; b += 2) {
    const uint32_t got = __shfl_xor_sync(0xffffffffu, o1 ? w[b] : w[b + 1], 1);
    if (o1) w[b] = got; else w[b + 1] = got;
  }
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    const uint32_t got = __shfl_xor_sync(0xffffffffu, o2 ? w[b] : w[b + 2], 2);
    if (o2) w[b] = got; else w[b + 2] = got;
  }
}
// One fragment (see tmem_ld_frag) of finished values: rows `row` and `row` + 8 of the output, 32 features from `f`.
// VEC: features a store may cover (linear_vec).
template <int VEC>
__device__ __forceinline__ void linear_store(const LinearArgs& g, float* v, int row, int f, int q) {
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const bool live = row + 8 * r < g.m;
    const size_t at = (size_t)(row + 8 * r) * g.n + f;
    if (VEC == 8) {
      if (g.out32) {
#pragma unroll
        for (int b = 0; b < 4; ++b)
          if (live && f + 8 * b < g.n_end) *reinterpret_cast<float2*>(g.out32 + at + 8 * b + 2 * q) = make_float2(v[4 * b + 2 * r], v[4 * b + 2 * r + 1]);
      }
      if (g.out16) {
        uint32_t w[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) w[b] = pack_bf16(v[4 * b + 2 * r], v[4 * b + 2 * r + 1]);
        quad_transpose(w, q);
        if (live && f + 8 * q < g.n_end) *reinterpret_cast<uint4*>(g.out16 + at + 8 * q) = make_uint4(w[0], w[1], w[2], w[3]);
      }
    } else if (VEC == 2) {
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const int c = 8 * b + 2 * q;
        if (!live || f + c >= g.n_end) continue;
        if (g.out32) *reinterpret_cast<float2*>(g.out32 + at + c) = make_float2(v[4 * b + 2 * r], v[4 * b + 2 * r + 1]);
        if (g.out16) *reinterpret_cast<uint32_t*>(g.out16 + at + c) = pack_bf16(v[4 * b + 2 * r], v[4 * b + 2 * r + 1]);
      }
    } else {
#pragma unroll
      for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int c = 8 * b + 2 * q + e;
          if (!live || f + c >= g.n_end) continue;
          if (g.out32) g.out32[at + c] = v[4 * b + 2 * r + e];
          if (g.out16) g.out16[at + c] = f32_to_bf16_bits(v[4 * b + 2 * r + e]);
        }
    }
  }
}
// This warp's share of a tile's columns: groups of 32, [lo, hi), for its 32 lanes.  `part` (split K): the other CTAs'
// fragments of the same group, written by the threads that hold the same place.  `n_acc`: accumulators of the same columns,
// `acc_stride` apart, that add up to the result.
template <int ACT, int VEC>
__device__ __forceinline__ void linear_rows(const LinearArgs& g, uint32_t tmem, int lane, int row0, int rows, int n0, int lo, int hi, const float4* part,
                                            int n_part, int part_stride, int n_acc = 1, uint32_t acc_stride = 0) {
  const int q = lane & 3;
#pragma unroll 1
  for (int h = 0; h < 2 && 16 * h < rows; ++h) {
    if (lo >= hi) break;
    const uint32_t th = tmem + ((uint32_t)(16 * h) << 16);
    uint32_t nx[EPI];
    tmem_ld_frag(th + 32u * (uint32_t)lo, nx);
#pragma unroll 1
    for (int c = lo; c < hi; ++c) {
      float v[EPI];
      tmem_ld_wait();
#pragma unroll
      for (int j = 0; j < EPI; ++j) v[j] = __uint_as_float(nx[j]);
      tmem_ld_frag(th + 32u * (uint32_t)(c + 1 < hi ? c + 1 : c), nx);
#pragma unroll 1
      for (int r = 1; r < n_acc; ++r) {
        uint32_t t[EPI];
        tmem_ld_frag(th + (uint32_t)r * acc_stride + 32u * (uint32_t)c, t);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < EPI; ++j) v[j] += __uint_as_float(t[j]);
      }
#pragma unroll 1
      for (int r = 0; r < n_part; ++r) {
        const float4* p = part + (size_t)r * part_stride + ((c - lo) * 2 + h) * (4 * 128);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float4 t = p[j * 128];
          v[4 * j] += t.x; v[4 * j + 1] += t.y; v[4 * j + 2] += t.z; v[4 * j + 3] += t.w;
        }
      }
      activate<ACT, EPI>(v);
      linear_store<VEC>(g, v, row0 + 16 * h + (lane >> 2), n0 + 32 * c, q);
    }
    tmem_ld_wait();
  }
}

template <int VEC>
__global__ void __launch_bounds__(LIN_THREADS, 2) vla_op_linear_kernel(const __grid_constant__ LinearArgs g, const __grid_constant__ OpMaps maps,
                                                                       OpFault fault) {
  extern __shared__ __align__(1024) char smem_raw[];
  __shared__ uint32_t tmem_base_s;
  __shared__ __align__(8) uint64_t bars[2 * LIN_MAX_STAGES + 4];       // full, empty; accumulators full (2), empty (2)
  __shared__ unsigned failed_s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int S = g.stages, n_acc = g.bn <= 128 ? 2 : 1, rank = (int)blockIdx.x % g.ks;
  const int first_tile = (int)blockIdx.x / g.ks, step = g.ks > 1 ? g.tiles : (int)gridDim.x;       // (a cluster does one tile)
  const int nkb_all = g.kp / GEMM_BK, kb0 = nkb_all * rank / g.ks, nkb = nkb_all * (rank + 1) / g.ks - kb0;
  const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8u * LIN_MAX_STAGES, accf0 = empty0 + 8u * LIN_MAX_STAGES, acce0 = accf0 + 16u;
  const uint32_t a_bytes = (uint32_t)(g.bm * GEMM_BK * 2), stage_bytes = (uint32_t)((g.bm + g.bn) * GEMM_BK * 2);
  const uint32_t stage0 = smem_u32(smem_raw);
  if (warp == 0) {
    if (lane < 2 * LIN_MAX_STAGES + 4) {
      mbar_init(full0 + 8u * lane, lane < 2 * LIN_MAX_STAGES + 2 ? 1 : LIN_EPI_WARPS);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (lane == 0) failed_s = 0;
  } else if (warp == 1) {
    tmem_alloc(&tmem_base_s, LIN_TMEM_COLS);
  }
  op_wait_previous(maps, 2);
  if (threadIdx.x == 0 && blockIdx.x == 0) *g.err = 0u;
  TileCtx c;                                   // (what the bounded waits look at)
  c.error = &failed_s;
  c.deadline = gtimer() + fault.wait_limit_ns;
  tc_fence_before();
  __syncthreads();
  op_let_next_start();
  tc_fence_after();
  const uint32_t tmem = tmem_base_s;
  bool ok = true;
  if (warp == 0) {
    if (lane == 0 && !fault.drop_loads) {
      uint32_t s = 0, ph = 1u;
      for (int t = first_tile; t < g.tiles && ok; t += step) {
        const int row0 = t % g.tiles_m * g.bm, n0 = t / g.tiles_m * g.bn;
#pragma unroll 1
        for (int kb = 0; kb < nkb; ++kb) {
          const uint32_t full = full0 + 8u * s, dst = stage0 + s * stage_bytes;
          if (!(ok = mbar_wait(c, empty0 + 8u * s, ph))) break;
          mbar_expect_tx(full, stage_bytes);
          tma_load_2d(dst + a_bytes, &maps.m[0], full, (kb0 + kb) * GEMM_BK, n0);
          tma_load_2d(dst, &maps.m[1], full, (kb0 + kb) * GEMM_BK, row0);
          // weights come from HBM once: the first token tile's CTA asks for them ahead, so that a stage waits for L2 only
          if (row0 == 0 && kb + LIN_AHEAD < nkb) tma_prefetch_2d(&maps.m[0], (kb0 + kb + LIN_AHEAD) * GEMM_BK, n0);
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
    for (int t = first_tile; t < g.tiles && ok; t += step, ++i) {
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
  }
  const int quarter = warp & 3, half = warp >= 6 ? 1 : 0;             // (epilogue warps 2..9: a quarter of the lanes is fixed by warp % 4)
  const uint32_t lanes = (uint32_t)(quarter * 32) << 16;
  const int groups = (g.bn + 31) / 32;
  auto rows_of = [&](uint32_t acc, int t, int lo, int hi, const float4* part, int n_part, int part_stride) {
    const int row0 = t % g.tiles_m * g.bm + 32 * quarter, rows = min(g.bm, g.m - t % g.tiles_m * g.bm) - 32 * quarter, n0 = t / g.tiles_m * g.bn;
    LinearArgs gg = g;
    gg.m = row0 + max(rows, 0);                                       // (this tile's rows and features only)
    gg.n_end = min(g.n, n0 + g.bn);
    if (g.act == ACT_GELU) linear_rows<ACT_GELU, VEC>(gg, acc + lanes, lane, row0, rows, n0, lo, hi, part, n_part, part_stride);
    else if (g.act == ACT_SILU) linear_rows<ACT_SILU, VEC>(gg, acc + lanes, lane, row0, rows, n0, lo, hi, part, n_part, part_stride);
    else linear_rows<ACT_NONE, VEC>(gg, acc + lanes, lane, row0, rows, n0, lo, hi, part, n_part, part_stride);
  };
  if (g.ks == 1) {
    if (warp >= 2) {
      uint32_t i = 0;
      for (int t = first_tile; t < g.tiles; t += step, ++i) {
        const uint32_t buf = n_acc == 2 ? i & 1u : 0u, use = n_acc == 2 ? i >> 1 : i;
        if (!mbar_wait(c, accf0 + 8u * buf, use & 1u)) break;
        __syncwarp();
        tc_fence_after();
        const int mid = (groups + 1) / 2;
        rows_of(tmem + 128u * buf, t, half ? mid : 0, half ? groups : mid, nullptr, 0, 0);
        tc_fence_before();
        arrive_warp(acce0 + 8u * buf, lane);
      }
    }
  } else {
    // ---------------- split K: every CTA sends the columns of the others away, then finishes its own
    const int own = groups / g.ks, thread = 32 * quarter + lane, stride = own * 2 * 4 * 128;          // float4 of one source CTA
    cluster_sync();                                                   // every CTA of the cluster has started
    if (warp >= 2) {
      mbar_wait(c, accf0, 0u);
      __syncwarp();
      tc_fence_after();
    }
    __syncthreads();
    cluster_sync();                                                   // ... and has done its last load and MMA: stages are free
    if (warp >= 2) {
#pragma unroll 1
      for (int c0 = half; c0 < groups; c0 += 2) {
        const int to = c0 / own;
        if (to == rank) continue;
        const int from = rank < to ? rank : rank - 1;                 // this CTA among the others of `to`
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
          uint32_t v[EPI];
          tmem_ld_frag(tmem + lanes + ((uint32_t)(16 * h) << 16) + 32u * (uint32_t)c0, v);
          tmem_ld_wait();
          const uint32_t at = cluster_addr(stage0 + (uint32_t)(from * stride + ((c0 % own) * 2 + h) * (4 * 128) + thread) * 16u, (uint32_t)to);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float w[4] = {__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]), __uint_as_float(v[4 * j + 2]), __uint_as_float(v[4 * j + 3])};
            st_cluster_f4(at + (uint32_t)(j * 128 * 16), w);
          }
        }
      }
    }
    cluster_sync();
    if (warp >= 2) {
      // the two warps of a quarter share the owned groups
      const int lo = rank * own, mid = lo + (own + 1) / 2, hi = lo + own, b = half ? mid : lo;
      rows_of(tmem, first_tile, b, half ? hi : mid, reinterpret_cast<const float4*>(smem_raw) + (b - lo) * 2 * (4 * 128) + thread, g.ks - 1, stride);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, LIN_TMEM_COLS);
  if (threadIdx.x == 0 && *reinterpret_cast<volatile unsigned*>(&failed_s) != 0u) *g.err = (unsigned)DEV_ERR_WAIT_MBAR;
}

}  // namespace vla
