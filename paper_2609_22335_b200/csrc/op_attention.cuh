// Stand-alone fused attention as a kernel of its own: softmax(Q K^T / sqrt(hd)) V on tensors as the caller has them.
//
// A tile is one query head x 128 queries (or several query heads of one KV head side by side where there are few queries,
// see attn_fold).  A cluster of `split` CTAs shares a tile: each takes a contiguous part of the keys, and the partial
// results meet in distributed shared memory -- a call of few tiles (96 heads x query blocks, or the action head's 4) is
// bound by the length of a tile's chain of key blocks, not by throughput, and this cuts the chain.
//
// Inside a CTA: a TMA warp, a warp that issues Q K^T, one that issues P V, and four softmax warps (a query row per thread).  S
// has three tensor-memory buffers where the output leaves room for them (two elsewhere), so scores are computed up to two blocks ahead
// of the softmax; the probabilities go back into the front of their scores' buffer and are the first operand of P V.  V is read as it lies,
// [key, head dim] (MN-major second operand), so nothing is transposed in front of the kernel.  Where the keys are in few parts (opa_plan) a
// probability is the sum of two bf16 numbers, the second in the back of the buffer, and P V takes two products: rel-L2 to 64 bits 1.65e-3
// where one number gives 2.0e-3 to 2.3e-3.
#pragma once
#include "attention_plan.h"
#include "dispatch.cuh"

namespace vla {

constexpr int OPA_THREADS = 224;

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
__device__ __forceinline__ void st_cluster_f2(uint32_t a, float x, float y) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(x), "f"(y) : "memory");
}
__device__ __forceinline__ void st_cluster_f4(uint32_t a, const float* v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]) : "memory");
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// maps: 0 Q [tq, hq*hd], 1 K, 2 V [tkv, hkv*hd].  a.out is an absolute address; a.t0 keys, no second segment.  TERMS: bf16 numbers of a
// probability.  (Two of its CTAs share an SM only up to 128 registers a thread -- 14 warps put four on one scheduler -- which the form of
// two terms exceeds unless it is told: 1024 x 1024 of 12 heads of 64 22.6 instead of 15.7 us.)
template <int TERMS>
__global__ void __launch_bounds__(OPA_THREADS, TERMS) vla_op_attention_kernel(const __grid_constant__ AttnArgs a, const __grid_constant__ OpMaps maps,
                                                                       const __grid_constant__ OpAttnLaunch p, unsigned* err, OpFault fault) {
  extern __shared__ __align__(1024) char smem_raw[];
  __shared__ uint32_t tmem_base_s;
  __shared__ __align__(8) uint64_t bars[4 * OPA_MAX_STAGES + 3 * OPA_MAX_S + 1];
  __shared__ __align__(8) float2 row_ml[OPA_MAX_SPLIT][ATTN_BQ];       // each CTA's maximum and sum of a row
  __shared__ unsigned failed_s;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int split = p.split, rank = (int)blockIdx.x % split, tile = (int)blockIdx.x / split, NS = p.stages, NB = p.s_bufs;
  const AttnPlace at = attn_place(a, tile);
  const int g = (at.head * a.hkv) / a.hq, hs = a.hs, nbox = (hs + 63) / 64;
  int nb = (a.t0 + ATTN_BN - 1) / ATTN_BN;
  if (a.causal) nb = min(nb, (at.q0 + ATTN_BQ - 1) / ATTN_BN + 1);
  const int b0 = nb * rank / split, n = nb * (rank + 1) / split - b0;          // this CTA's key blocks
  const uint32_t bar0 = smem_u32(bars);
  const uint32_t kfull = bar0, kempty = bar0 + 8 * OPA_MAX_STAGES, vfull = kempty + 8 * OPA_MAX_STAGES, vempty = vfull + 8 * OPA_MAX_STAGES;
  const uint32_t bar_s = vempty + 8 * OPA_MAX_STAGES, bar_p = bar_s + 8 * OPA_MAX_S, bar_o = bar_p + 8 * OPA_MAX_S, bar_q = bar_o + 8 * OPA_MAX_S;   // (s, p, o: one per score buffer)
  const uint32_t kv_bytes = (uint32_t)nbox * (ATTN_BN * 128);
  const uint32_t Qs = smem_u32(smem_raw), Ks = Qs + (uint32_t)nbox * (ATTN_BQ * 128), Vs = Ks + (uint32_t)NS * kv_bytes;
  if (warp == 4) {
    if (lane < 4 * OPA_MAX_STAGES + 3 * OPA_MAX_S + 1) {
      const bool is_p = lane >= 4 * OPA_MAX_STAGES + OPA_MAX_S && lane < 4 * OPA_MAX_STAGES + 2 * OPA_MAX_S;
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
  const uint32_t tmem = tmem_base_s, tmem_o = tmem + (uint32_t)(NB * ATTN_BN);     // score buffers, then O

  if (warp == 4) {
    // ---------------- loads
    if (lane == 0 && !fault.drop_loads && n > 0) {
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
    // ---------------- S = Q K^T, into a buffer as soon as P V has read the probabilities that were in it.  (The commit that somebody
    // waits for goes first: each costs its thread 150 cycles.  A stage that no later block is loaded into is not released: nobody would
    // wait for that arrival, and it could come after the CTA's end.)
    const uint32_t idesc_s = umma_idesc_bf16(ATTN_BN);
    const uint64_t qdesc = umma_desc_sw128(Qs);
    uint32_t s = 0, ph = 0u, buf = 0, bph = 1u;
    bool ok = n > 0 && mbar_wait(c, bar_q, 0u);
#pragma unroll 1
    for (int i = 0; i < n && ok; ++i) {
      if (i >= NB && !(ok = mbar_wait(c, bar_o + 8u * buf, bph))) break;
      if (!(ok = mbar_wait(c, kfull + 8u * s, ph))) break;
      tc_fence_after();
      uint64_t qd = qdesc, kd = umma_desc_sw128(Ks + s * kv_bytes);
      const uint32_t ts = tmem + ATTN_BN * buf;
      if (elect_one()) {
        int kc = 0;
#pragma unroll 1
        for (; kc + 4 <= hs / 16; kc += 4) {
#pragma unroll
          for (int k = 0; k < 4; ++k) umma_bf16(ts, qd + 2u * k, kd + 2u * k, idesc_s, (kc | k) != 0 ? 1u : 0u);
          qd += (ATTN_BQ * 128) >> 4; kd += (ATTN_BN * 128) >> 4;
        }
#pragma unroll 1
        for (int k = 0; kc < hs / 16; ++kc, ++k) umma_bf16(ts, qd + 2u * k, kd + 2u * k, idesc_s, kc != 0 ? 1u : 0u);
        umma_commit(bar_s + 8u * buf);
        if (i + NS < n) umma_commit(kempty + 8u * s);
      }
      __syncwarp();
      if (++s == (uint32_t)NS) { s = 0; ph ^= 1u; }
      if (++buf == (uint32_t)NB) { buf = 0; bph ^= 1u; }
    }
  } else if (warp == 6) {
    // ---------------- the queries (beside the first keys, which warp 4 asks for), then O += P V
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
    }
    __syncwarp();
    const uint32_t idesc_o = umma_idesc_bf16(hs) | (1u << 16);       // second operand MN-major
    uint32_t s = 0, ph = 0u, buf = 0, bph = 0u;
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
      if (!mbar_wait(c, vfull + 8u * s, ph) || !mbar_wait(c, bar_p + 8u * buf, bph)) break;
      tc_fence_after();
      const uint64_t vd = umma_desc_mn_sw128(Vs + s * kv_bytes, ATTN_BN * 128);
      const uint32_t tp = tmem + ATTN_BN * buf;
      if (elect_one()) {
#pragma unroll
        for (int k = 0; k < TERMS * (ATTN_BN / 16); ++k)      // 16 keys = 16 rows of 128 bytes = 32 words of P pairs / 4
          umma_bf16_ta(tmem_o, tp + 8u * k, vd + (uint64_t)(k % (ATTN_BN / 16) * (16 * 128 >> 4)), idesc_o, (i | k) != 0 ? 1u : 0u);
        umma_commit(bar_o + 8u * buf);
        if (i + NS < n) umma_commit(vempty + 8u * s);
      }
      __syncwarp();
      if (++s == (uint32_t)NS) { s = 0; ph ^= 1u; }
      if (++buf == (uint32_t)NB) { buf = 0; bph ^= 1u; }
    }
  }
  float m_run = -INFINITY, l_run = 0.f;
  const uint32_t my_lanes = (uint32_t)((warp & 3) * 32) << 16;
  const int row = a.hpt > 1 ? (int)threadIdx.x % a.rph : at.q0 + (int)threadIdx.x;            // this thread's query (softmax warps)
  const float sl2 = a.scale_log2e;
  if (warp < 4) {
    // ---------------- softmax: one thread per query row.  A wait on a buffer's barriers never sees one more than a phase behind: S(i)
    // was issued after P V of the block that had the buffer before.
    uint32_t b = 0, bph = 0u, last = 0, lph = 0u;           // this block's score buffer and its phase; those of the block before
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
      const uint32_t buf = tmem + my_lanes + ATTN_BN * b;
      if (!mbar_wait(c, bar_s + 8u * b, bph)) break;
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
      attn_softmax_block<TERMS>(sr, sl2, m_run, l_run, alpha);
      // O follows a moved maximum (rarely); everything before has been added by then.  (P V of this block cannot start before this
      // warp arrives.)
      if (i > 0 && __any_sync(0xffffffffu, alpha != 1.0f)) {
        mbar_wait(c, bar_o + 8u * last, lph);
        __syncwarp();
        tc_fence_after();
        attn_rescale(tmem_o + my_lanes, hs, alpha);
      }
      tmem_st16u(buf, sr);
      tmem_st16u(buf + 16u, sr + 16);
      if (TERMS == 2) {
        tmem_st16u(buf + 32u, sr + 32);
        tmem_st16u(buf + 48u, sr + 48);
      }
      tmem_st_wait();
      tc_fence_before();
      arrive_warp(bar_p + 8u * b, lane);
      last = b; lph = bph;
      if (++b == (uint32_t)NB) { b = 0; bph ^= 1u; }
    }
    if (n > 0) mbar_wait(c, bar_o + 8u * last, lph);
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
    // ---------------- the cluster's partial rows go to the CTA that finishes their columns as they are, with every CTA's maxima and
    // sums, so that they are weighted there and one exchange does
    cluster_sync();                       // every CTA has done its last load and MMA, so shared memory is free
    if (warp < 4) {
      const uint32_t ml = smem_u32(&row_ml[rank][threadIdx.x]);
#pragma unroll 1
      for (int r = 0; r < split; ++r) st_cluster_f2(cluster_addr(ml, (uint32_t)r), m_run, l_run);
    }
    const uint32_t slab = smem_u32(smem_raw);
    if (warp < 4 && n > 0) {
      int to = 0, own = 0;                // chunk ch = own * split + to
      uint32_t nx[16];
      tmem_ld16_nowait(tmem_o + my_lanes, nx);
#pragma unroll 1
      for (int ch = 0; ch < hs / 16; ++ch) {
        float o[16];
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 16; ++j) o[j] = __uint_as_float(nx[j]);
        tmem_ld16_nowait(tmem_o + my_lanes + 16u * (uint32_t)min(ch + 1, hs / 16 - 1), nx);
        // [owned chunk][source CTA][quarter][row] of four floats
        const uint32_t at_ = cluster_addr(slab + (uint32_t)((own * split + rank) * 4 * ATTN_BQ + (int)threadIdx.x) * 16u, (uint32_t)to);
        if (row_ok) {                     // (rows that nobody stores are not sent: the exchange is most of a short call of wide heads)
#pragma unroll
          for (int q = 0; q < 4; ++q) st_cluster_f4(at_ + (uint32_t)(q * ATTN_BQ * 16), o + 4 * q);
        }
        if (++to == split) { to = 0; ++own; }
      }
      tmem_ld_wait();
    }
    cluster_sync();
    if (row_ok) {
      float M = -INFINITY, L = 0.f, f[OPA_MAX_SPLIT];
#pragma unroll
      for (int r = 0; r < OPA_MAX_SPLIT; ++r)
        if (r < split) M = fmaxf(M, row_ml[r][threadIdx.x].x);
#pragma unroll
      for (int r = 0; r < OPA_MAX_SPLIT; ++r) {
        const float2 v = r < split ? row_ml[r][threadIdx.x] : make_float2(-INFINITY, 0.f);
        // (no maximum: a part without keys of this row, or one whose scores are all NaN -- its sum is then, and the row is as it would be unsplit)
        f[r] = v.x == -INFINITY ? (v.y == 0.f ? 0.f : v.y) : exp2_fast((v.x - M) * sl2);
        if (f[r] != 0.f) L = fmaf(v.y, f[r], L);
      }
      const float inv = L == 0.f ? 0.f : 1.0f / L;
      const float4* part = reinterpret_cast<const float4*>(smem_raw) + threadIdx.x;
#pragma unroll 1
      for (int ch = rank; ch < hs / 16; ch += split, part += split * 4 * ATTN_BQ) {
        float o[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) o[j] = 0.f;
#pragma unroll
        for (int r = 0; r < OPA_MAX_SPLIT; ++r) {
          if (f[r] == 0.f) continue;      // (a CTA without keys of this row: whatever lies there)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const float4 v = part[(r * 4 + q) * ATTN_BQ];
            o[4 * q] = fmaf(f[r], v.x, o[4 * q]); o[4 * q + 1] = fmaf(f[r], v.y, o[4 * q + 1]);
            o[4 * q + 2] = fmaf(f[r], v.z, o[4 * q + 2]); o[4 * q + 3] = fmaf(f[r], v.w, o[4 * q + 3]);
          }
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) o[j] *= inv;
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
