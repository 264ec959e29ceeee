// Stand-alone fused attention as a kernel of its own: softmax(Q K^T / sqrt(hd)) V on tensors as the caller has them.
//
// A tile is one query head x 128 queries (or several query heads of one KV head side by side where there are few queries,
// see attn_fold).  A cluster of `split` CTAs shares a tile: each takes a contiguous part of the keys, and the partial
// results meet in distributed shared memory -- a call of few tiles (96 heads x query blocks, or the action head's 4) is
// bound by the length of a tile's chain of key blocks, not by throughput, and this cuts the chain.
//
// Inside a CTA: a TMA warp, an MMA warp and four softmax warps (a query row per thread).  S has two tensor-memory buffers, so
// the scores of block i + 1 are computed under the softmax of block i; the probabilities go back into the front of their
// scores' buffer and are the first operand of P V.  V is read as it lies, [key, head dim] (MN-major second operand), so
// nothing is transposed in front of the kernel.
#pragma once
#include "dispatch.cuh"

namespace vla {

constexpr int OPA_THREADS = 192;
constexpr int OPA_MAX_STAGES = 4;

struct OpAttnLaunch { int split, stages, smem, tmem_cols; };

inline int opa_smem(int hs, int stages) {
  const int nbox = (hs + 63) / 64;
  return nbox * (128 * 128 + stages * 2 * 64 * 128);
}
// Two CTAs share an SM up to a head width of 128 (tensor memory 128 + hs columns of 512); the keys are split while that
// still gives every CTA a slot of its own and at least one block of 64 keys.
inline OpAttnLaunch opa_plan(int tiles, int tkv, int hs, int sms) {
  OpAttnLaunch p;
  const int per_sm = hs <= 128 ? 2 : 1, budget = per_sm == 2 ? 112 * 1024 : 224 * 1024, blocks = (tkv + 63) / 64, chunks = hs / 16;
  p.stages = OPA_MAX_STAGES;
  while (p.stages > 2 && opa_smem(hs, p.stages) > budget) --p.stages;
  p.smem = opa_smem(hs, p.stages);
  p.split = 1;
  while (p.split < 8 && tiles * p.split * 2 <= per_sm * sms && blocks >= p.split * 2 &&
         ((chunks + 2 * p.split - 1) / (2 * p.split)) * 2 * p.split * 8192 <= p.smem)
    p.split *= 2;
  p.tmem_cols = hs <= 128 ? 256 : 512;
  return p;
}

// second operand [key, head dim] as it lies: MN-major, 128-byte swizzle -- 64-wide columns of boxes `box` bytes apart, groups
// of eight keys 1024 bytes apart
__device__ __forceinline__ uint64_t umma_desc_mn_sw128(uint32_t saddr, uint32_t box) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)(box >> 4) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
__device__ __forceinline__ uint32_t cluster_addr(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
__device__ __forceinline__ float2 ld_cluster_f2(uint32_t a) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void st_cluster_f4(uint32_t a, const float* v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]) : "memory");
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// maps: 0 Q [tq, hq*hd], 1 K, 2 V [tkv, hkv*hd].  a.out is an absolute address; a.t0 keys, no second segment.
__global__ void __launch_bounds__(OPA_THREADS) vla_op_attention_kernel(const __grid_constant__ AttnArgs a, const __grid_constant__ OpMaps maps,
                                                                       const __grid_constant__ OpAttnLaunch p, unsigned* err, OpFault fault) {
  extern __shared__ __align__(1024) char smem_raw[];
  __shared__ uint32_t tmem_base_s;
  __shared__ __align__(8) uint64_t bars[4 * OPA_MAX_STAGES + 6];
  __shared__ __align__(8) float2 row_ml[ATTN_BQ];
  __shared__ unsigned failed_s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int split = p.split, rank = (int)blockIdx.x % split, tile = (int)blockIdx.x / split, NS = p.stages;
  const AttnPlace at = attn_place(a, tile);
  const int g = (at.head * a.hkv) / a.hq, hs = a.hs, nbox = (hs + 63) / 64;
  int nb = (a.t0 + ATTN_BN - 1) / ATTN_BN;
  if (a.causal) nb = min(nb, (at.q0 + ATTN_BQ - 1) / ATTN_BN + 1);
  const int b0 = nb * rank / split, n = nb * (rank + 1) / split - b0;          // this CTA's key blocks
  const uint32_t bar0 = smem_u32(bars);
  const uint32_t kfull = bar0, kempty = bar0 + 8 * OPA_MAX_STAGES, vfull = kempty + 8 * OPA_MAX_STAGES, vempty = vfull + 8 * OPA_MAX_STAGES;
  const uint32_t bar_s = vempty + 8 * OPA_MAX_STAGES, bar_p = bar_s + 16, bar_o = bar_p + 16, bar_q = bar_o + 8;
  const uint32_t kv_bytes = (uint32_t)nbox * (ATTN_BN * 128);
  const uint32_t Qs = smem_u32(smem_raw), Ks = Qs + (uint32_t)nbox * (ATTN_BQ * 128), Vs = Ks + (uint32_t)NS * kv_bytes;
  if (warp == 4) {
    if (lane < 4 * OPA_MAX_STAGES + 6) {
      const bool is_p = lane == 4 * OPA_MAX_STAGES + 2 || lane == 4 * OPA_MAX_STAGES + 3;
      mbar_init(bar0 + 8u * lane, is_p ? 4 : 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (lane == 0) failed_s = 0;
  } else if (warp == 5) {
    tmem_alloc(&tmem_base_s, (uint32_t)p.tmem_cols);
  }
  op_wait_previous(maps, 3);
  if (threadIdx.x == 0 && blockIdx.x == 0) *err = 0u;
  TileCtx c;                                    // (what the bounded waits look at)
  c.error = &failed_s;
  c.deadline = gtimer() + fault.wait_limit_ns;
  tc_fence_before();
  __syncthreads();
  op_let_next_start();
  tc_fence_after();
  const uint32_t tmem = tmem_base_s, tmem_o = tmem + 2u * ATTN_BN;     // two score buffers, then O

  if (warp == 4) {
    // ---------------- loads
    if (lane == 0 && !fault.drop_loads && n > 0) {
      if (a.hpt <= 1) {
        mbar_expect_tx(bar_q, (uint32_t)nbox * (ATTN_BQ * 128));
#pragma unroll 1
        for (int b = 0; b < nbox; ++b) tma_load_2d(Qs + (uint32_t)b * (ATTN_BQ * 128), &maps.m[0], bar_q, at.head * hs + b * 64, at.q0);
      } else {
        mbar_expect_tx(bar_q, (uint32_t)(at.nh * nbox * a.rph * 128));
#pragma unroll 1
        for (int i = 0; i < at.nh; ++i)
#pragma unroll 1
          for (int b = 0; b < nbox; ++b)
            tma_load_2d(Qs + (uint32_t)b * (ATTN_BQ * 128) + (uint32_t)(i * a.rph * 128), &maps.m[0], bar_q, (at.head + i) * hs + b * 64, 0);
      }
      uint32_t s = 0, ph = 1u;
      bool ok = true;
#pragma unroll 1
      for (int i = 0; i < n && ok; ++i) {
        const int kv0 = (b0 + i) * ATTN_BN;
        for (int which = 0; which < 2 && ok; ++which) {
          const uint32_t full = (which ? vfull : kfull) + 8u * s, dst = (which ? Vs : Ks) + s * kv_bytes;
          if (!(ok = mbar_wait(c, (which ? vempty : kempty) + 8u * s, ph))) break;
          mbar_expect_tx(full, kv_bytes);
#pragma unroll 1
          for (int b = 0; b < nbox; ++b) tma_load_2d(dst + (uint32_t)b * (ATTN_BN * 128), &maps.m[1 + which], full, g * hs + b * 64, kv0);
        }
        if (++s == (uint32_t)NS) { s = 0; ph ^= 1u; }
      }
      if (!ok) for (int i = 0; i < 100; ++i) __nanosleep(1000);        // gave up: the copies in flight land before the CTA ends
    }
    __syncwarp();
  } else if (warp == 5) {
    // ---------------- MMAs
    const uint32_t idesc_s = umma_idesc_bf16(ATTN_BN), idesc_o = umma_idesc_bf16(hs) | (1u << 16);       // second operand MN-major
    const uint64_t qdesc = umma_desc_sw128(Qs);
    uint32_t ks = 0, kph = 0u, vs = 0, vph = 0u;
    auto issue_s = [&](int i) -> bool {
      if (!mbar_wait(c, kfull + 8u * ks, kph)) return false;
      tc_fence_after();
      uint64_t qd = qdesc, kd = umma_desc_sw128(Ks + ks * kv_bytes);
      if (elect_one()) {
        int kc = 0;
#pragma unroll 1
        for (; kc + 4 <= hs / 16; kc += 4) {
#pragma unroll
          for (int k = 0; k < 4; ++k) umma_bf16(tmem + ATTN_BN * (uint32_t)(i & 1), qd + 2u * k, kd + 2u * k, idesc_s, (kc | k) != 0 ? 1u : 0u);
          qd += (ATTN_BQ * 128) >> 4; kd += (ATTN_BN * 128) >> 4;
        }
#pragma unroll 1
        for (int k = 0; kc < hs / 16; ++kc, ++k) umma_bf16(tmem + ATTN_BN * (uint32_t)(i & 1), qd + 2u * k, kd + 2u * k, idesc_s, kc != 0 ? 1u : 0u);
        umma_commit(kempty + 8u * ks);
        umma_commit(bar_s + 8u * (uint32_t)(i & 1));
      }
      __syncwarp();
      if (++ks == (uint32_t)NS) { ks = 0; kph ^= 1u; }
      return true;
    };
    bool ok = n > 0 && mbar_wait(c, bar_q, 0u) && issue_s(0);
    if (ok && n > 1) ok = issue_s(1);
#pragma unroll 1
    for (int i = 0; i < n && ok; ++i) {
      if (!(ok = mbar_wait(c, bar_p + 8u * (uint32_t)(i & 1), ((uint32_t)i >> 1) & 1u) && mbar_wait(c, vfull + 8u * vs, vph))) break;
      tc_fence_after();
      const uint64_t vd = umma_desc_mn_sw128(Vs + vs * kv_bytes, ATTN_BN * 128);
      if (elect_one()) {
#pragma unroll
        for (int k = 0; k < ATTN_BN / 16; ++k)      // 16 keys = 16 rows of 128 bytes = 32 words of P pairs / 4
          umma_bf16_ta(tmem_o, tmem + ATTN_BN * (uint32_t)(i & 1) + 8u * k, vd + (uint64_t)(k * (16 * 128 >> 4)), idesc_o, (i | k) != 0 ? 1u : 0u);
        umma_commit(vempty + 8u * vs);
        umma_commit(bar_o);
      }
      __syncwarp();
      if (++vs == (uint32_t)NS) { vs = 0; vph ^= 1u; }
      if (i + 2 < n) ok = mbar_wait(c, bar_o, (uint32_t)i & 1u) && issue_s(i + 2);     // (its scores go where P(i) was read from)
    }
  }
  float m_run = -INFINITY, l_run = 0.f;
  const uint32_t my_lanes = (uint32_t)((warp & 3) * 32) << 16;
  const int row = a.hpt > 1 ? (int)threadIdx.x % a.rph : at.q0 + (int)threadIdx.x;            // this thread's query (softmax warps)
  const float sl2 = a.scale_log2e;
  if (warp < 4) {
    // ---------------- softmax: one thread per query row
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
      const uint32_t buf = tmem + my_lanes + ATTN_BN * (uint32_t)(i & 1);
      if (!mbar_wait(c, bar_s + 8u * (uint32_t)(i & 1), ((uint32_t)i >> 1) & 1u)) break;
      __syncwarp();
      tc_fence_after();
      uint32_t sr[ATTN_BN];
      tmem_ld16_nowait(buf + 0u, sr + 0);
      tmem_ld16_nowait(buf + 16u, sr + 16);
      tmem_ld16_nowait(buf + 32u, sr + 32);
      tmem_ld16_nowait(buf + 48u, sr + 48);
      tmem_ld_wait();
      {
        const int kv0 = (b0 + i) * ATTN_BN;
        const int lim = a.causal ? min(a.t0 - kv0, row - kv0 + 1) : a.t0 - kv0;
        if (a.causal || a.t0 - kv0 < ATTN_BN) attn_mask(sr, lim);
      }
      float alpha;
      attn_softmax_block(sr, sl2, m_run, l_run, alpha);
      // O follows a moved maximum (rarely); everything before has been added by then.  The last block waits for P V of the one
      // before it in any case: the wait behind the loop tells phases apart by parity, and this warp may be a whole block ahead
      // of another one, whose part of that P V is still to come.  (P V of this block cannot start before this warp arrives.)
      const bool moved = __any_sync(0xffffffffu, alpha != 1.0f);
      if (i > 0 && (moved || i == n - 1)) {
        mbar_wait(c, bar_o, (uint32_t)(i - 1) & 1u);
        __syncwarp();
        tc_fence_after();
        if (moved) attn_rescale(tmem_o + my_lanes, hs, alpha);
      }
      tmem_st16u(buf, sr);
      tmem_st16u(buf + 16u, sr + 16);
      tmem_st_wait();
      tc_fence_before();
      arrive_warp(bar_p + 8u * (uint32_t)(i & 1), lane);
    }
    if (n > 0) mbar_wait(c, bar_o, (uint32_t)(n - 1) & 1u);
    __syncwarp();
    tc_fence_after();
  }
  const int fold_h = a.hpt > 1 ? (int)threadIdx.x / a.rph : 0;
  const bool row_ok = warp < 4 && row < a.tq && fold_h < at.nh;
  unsigned short* const O = reinterpret_cast<unsigned short*>(a.out) + (size_t)row * a.ldo + (at.head + fold_h) * a.hd;
  if (split == 1) {
    if (warp < 4) {
      const float inv = l_run > 0.f ? 1.0f / l_run : 0.f;
#pragma unroll 1
      for (int c0 = 0; c0 < hs; c0 += 16) {
        float o[16];
        tmem_ld16(tmem_o + my_lanes + (uint32_t)c0, o);
#pragma unroll
        for (int j = 0; j < 16; ++j) o[j] *= inv;
        if (row_ok) put16(O + c0, o);
      }
    }
  } else {
    // ---------------- the cluster's partial rows: maxima and sums first, then each CTA adds up its share of the columns
    if (warp < 4) row_ml[threadIdx.x] = make_float2(m_run, l_run);
    cluster_sync();                       // (and: every CTA has done its last load and MMA, so shared memory is free)
    const uint32_t slab = smem_u32(smem_raw);
    if (warp < 4) {
      float M = -INFINITY, L = 0.f;
      float2 ml[8];
#pragma unroll
      for (int r = 0; r < 8; ++r)
        if (r < split) { ml[r] = ld_cluster_f2(cluster_addr(smem_u32(&row_ml[threadIdx.x]), (uint32_t)r)); M = fmaxf(M, ml[r].x); }
#pragma unroll
      for (int r = 0; r < 8; ++r)
        if (r < split && ml[r].x != -INFINITY) L = fmaf(ml[r].y, exp2_fast((ml[r].x - M) * sl2), L);
      const float f = (m_run == -INFINITY || L == 0.f) ? 0.f : exp2_fast((m_run - M) * sl2) / L;
#pragma unroll 1
      for (int ch = 0; ch < hs / 16; ++ch) {
        float o[16];
        tmem_ld16(tmem_o + my_lanes + 16u * (uint32_t)ch, o);
#pragma unroll
        for (int j = 0; j < 16; ++j) o[j] = f != 0.f ? o[j] * f : 0.f;
        // [owned chunk][source CTA][quarter][row] of four floats
        const uint32_t at_ = cluster_addr(slab + (uint32_t)(((ch / split) * split + rank) * 4 * ATTN_BQ + (int)threadIdx.x) * 16u, (uint32_t)(ch % split));
#pragma unroll
        for (int q = 0; q < 4; ++q) st_cluster_f4(at_ + (uint32_t)(q * ATTN_BQ * 16), o + 4 * q);
      }
    }
    cluster_sync();
    if (row_ok) {
      const float4* part = reinterpret_cast<const float4*>(smem_raw);
#pragma unroll 1
      for (int ch = rank; ch < hs / 16; ch += split) {
        float o[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) o[j] = 0.f;
#pragma unroll 1
        for (int r = 0; r < split; ++r) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const float4 v = part[(((ch / split) * split + r) * 4 + q) * ATTN_BQ + (int)threadIdx.x];
            o[4 * q] += v.x; o[4 * q + 1] += v.y; o[4 * q + 2] += v.z; o[4 * q + 3] += v.w;
          }
        }
        put16(O + 16 * ch, o);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 5) tmem_dealloc(tmem, (uint32_t)p.tmem_cols);
  if (threadIdx.x == 0 && *reinterpret_cast<volatile unsigned*>(&failed_s) != 0u) *err = (unsigned)DEV_ERR_WAIT_MBAR;
}

}  // namespace vla
