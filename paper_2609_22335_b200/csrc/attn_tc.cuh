// Fused attention tile on tcgen05 / tensor memory.
//
// One tile = one query head x 128 queries -- or, where few queries meet grouped KV heads (the action head's 9..51
// tokens), several query heads of one KV head side by side in the 128 rows.  Per block of 64 keys:
//   S = Q K^T          tcgen05.mma, Q and K tiles K-major (head dim contiguous), S in TMEM
//   online softmax     one thread per query row holds its 64 scores in registers (no shuffles) and leaves the
//                      probabilities as bf16 in TMEM
//   O += P V           tcgen05.mma with P read from TMEM, V consumed from its transposed copy V^T
//                      [head dim, tokens], K-major; O in TMEM, rescaled in place when a row maximum moves
// Keys come from up to two segments (cached prefix K/V, then the head's own K/V); blocks
// never straddle segments.  Head dims are handled in 16-wide K steps, so a head padded to
// a multiple of 16 (72 -> 80) costs only its padding.  All waits are bounded.
//
// What bounds it: one tile alone is a chain of barrier tests, MMA issue and tensor-memory round trips around 800 cycles of
// softmax per block.  So S of block b+1 is issued as soon as the scores of block b are in registers (warp 0), and the loads run
// two blocks (K) and one block (V) ahead on warps 2 and 3: 3560 -> 3010 cycles per block of a tile alone on its SM, 52 -> 40 us
// for a 16-block tile among three.  Warp 1 issues P V of block b-1 behind its reading of S, where it no longer delays S of the
// next block, and warps 2 and 3, which issue nothing, wait for K and V on the issuers' behalf (a test of a barrier that is
// ready costs 160-190 cycles): single frame 12.07 -> 11.98 ms, 4 x 2 pi0 streams 77.9 -> 77.3.
#pragma once
#include "attention_plan.h"
#include "gemm_tc.cuh"

namespace vla {

constexpr float ATTN_RESCALE_LOG2 = 8.0f;   // the running row maximum may lag the true one by this much (log2 units)

// Every warp of the tile arrives (after its lanes are together), one warp waits: an mbarrier of count four, so that a wait
// that ran out somewhere can never leave warps at different numbers of hardware barriers.
__device__ __forceinline__ void arrive_warp(uint32_t bar, int lane) {
  __syncwarp();
  if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void umma_bf16_ta(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(tmem_d), "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate));
}
__device__ __forceinline__ void tmem_st16u(uint32_t taddr, const uint32_t* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]),
        "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
      : "memory");
}

__device__ __forceinline__ float exp2_fast(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// two fp32 values in one 64-bit register pair
__device__ __forceinline__ uint64_t pack2(float x, float y) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& x, float& y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v)); }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float max3(float x, float y, float z) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(x), "f"(y), "f"(z));
  return r;
}

// Scores of the keys a row must not see, [lim, 64), become -inf.
__device__ __forceinline__ void attn_mask(uint32_t* sr, int lim) {
  if (!__any_sync(0xffffffffu, lim < ATTN_BN)) return;
#pragma unroll
  for (int j = 0; j < ATTN_BN; ++j)
    if (j >= lim) sr[j] = 0xFF800000u;
}
// One block of a row's online softmax: 64 scores in, 32 bf16 probability pairs out (front half of the registers).  TERMS 2: the pairs'
// rounding errors, in bf16 themselves, in the other half.
template <int TERMS = 1>
__device__ __forceinline__ void attn_softmax_block(uint32_t* sr, float sl2, float& m_run, float& l_run, float& alpha) {
  float m4[4] = {m_run, __uint_as_float(sr[0]), __uint_as_float(sr[1]), __uint_as_float(sr[2])};
#pragma unroll
  for (int j = 3; j < ATTN_BN - 1; j += 2) m4[(j >> 1) & 3] = max3(m4[(j >> 1) & 3], __uint_as_float(sr[j]), __uint_as_float(sr[j + 1]));
  float mx = fmaxf(max3(m4[0], m4[1], m4[2]), fmaxf(m4[3], __uint_as_float(sr[ATTN_BN - 1])));
  // The running maximum only has to keep the exponentials in range, not to be exact: softmax does not depend on
  // the shift, and l and O are accumulated with the same one.  It follows the true maximum only when that has
  // moved by more than 8 in the exponent (p then stays below 2^8), so O is rescaled on few blocks instead of
  // on nearly every one (with 32 rows per warp some row's maximum moves in almost every block).
  if (m_run == -INFINITY) alpha = 0.f;
  else if ((mx - m_run) * sl2 <= ATTN_RESCALE_LOG2) { mx = m_run; alpha = 1.0f; }
  else alpha = exp2_fast((m_run - mx) * sl2);
  const float mb = mx == -INFINITY ? 0.f : -mx * sl2;
  const uint64_t sl2_2 = pack2(sl2, sl2), mb_2 = pack2(mb, mb);
  uint64_t s2[2] = {0ull, 0ull};
  uint32_t lo[ATTN_BN / 2];
#pragma unroll
  for (int j = 0; j < ATTN_BN; j += 2) {
    const uint64_t e2 = fma2(pack2(__uint_as_float(sr[j]), __uint_as_float(sr[j + 1])), sl2_2, mb_2);
    float p0, p1;
    unpack2(e2, p0, p1);
    p0 = exp2_fast(p0); p1 = exp2_fast(p1);
    s2[(j >> 1) & 1] = add2(s2[(j >> 1) & 1], pack2(p0, p1));
    sr[j >> 1] = pack_bf16(p0, p1);
    if (TERMS == 2) lo[j >> 1] = pack_bf16(p0 - __uint_as_float(sr[j >> 1] << 16), p1 - __uint_as_float(sr[j >> 1] & 0xFFFF0000u));
  }
  if (TERMS == 2) {
#pragma unroll
    for (int j = 0; j < ATTN_BN / 2; ++j) sr[ATTN_BN / 2 + j] = lo[j];
  }
  float x0, x1;
  unpack2(add2(s2[0], s2[1]), x0, x1);
  l_run = l_run * alpha + (x0 + x1);
  m_run = mx;
}
__device__ __forceinline__ void attn_rescale(uint32_t tmem, int hs, float alpha) {
#pragma unroll 1
  for (int c0 = 0; c0 < hs; c0 += 16) {
    float o[16];
    tmem_ld16(tmem + (uint32_t)c0, o);
#pragma unroll
    for (int j = 0; j < 16; ++j) o[j] *= alpha;
    tmem_st16(tmem + (uint32_t)c0, o);
  }
}

// Key blocks of a tile: segment 0 (cached prefix) then segment 1 (the head's own keys), 64 keys each,
// never straddling a segment; with a causal mask the walk stops at the diagonal.
struct KvWalk {
  int n0, n;            // blocks of segment 0, blocks in all
  __device__ __forceinline__ int seg(int b) const { return b >= n0 ? 1 : 0; }
  __device__ __forceinline__ int kv0(int b) const { return (b >= n0 ? b - n0 : b) * ATTN_BN; }
};

// Where a tile lies.  Folded: tile -> (KV head, first query head, heads in this tile); else tile -> (head, query block).
struct AttnPlace { int head, q0, nh; };
__device__ __forceinline__ AttnPlace attn_place(const AttnArgs& a, int tile) {
  AttnPlace p;
  if (a.hpt > 1) {
    const int group = a.hq / a.hkv, per_group = (group + a.hpt - 1) / a.hpt, i = tile % per_group * a.hpt;
    p.head = tile / per_group * group + i; p.q0 = 0; p.nh = min(a.hpt, group - i);
  } else {
    p.head = tile / a.q_blocks; p.q0 = tile % a.q_blocks * ATTN_BQ; p.nh = 1;
  }
  return p;
}

// Shared-memory carve-up (all tile bases 1024-byte aligned): Q, two K blocks, two V^T blocks.
struct AttnSmem { uint32_t q, k, v, k_bytes, v_bytes; int nbox; };
__device__ __forceinline__ AttnSmem attn_smem(const TileCtx& c, const AttnArgs& a) {
  AttnSmem m;
  m.nbox = (a.hs + 63) / 64;                // 64-column boxes covering one head
  m.k_bytes = (uint32_t)m.nbox * (ATTN_BN * 128); m.v_bytes = (uint32_t)(a.hs * 128);
  m.q = smem_u32(c.smem); m.k = m.q + (uint32_t)m.nbox * (ATTN_BQ * 128); m.v = m.k + 2u * m.k_bytes;
  return m;
}
__device__ __forceinline__ void attn_load_k(const TileCtx& c, const AttnArgs& a, KvWalk kv, int g, int b) {
  const AttnSmem m = attn_smem(c, a);
  const uint32_t buf = (uint32_t)b & 1u, bar = smem_u32(c.ctl) + 8u + 8u * buf;
  const char* map = reinterpret_cast<const char*>(c.tmaps) + (size_t)(c.amap_base + (kv.seg(b) ? a.k1map : a.k0map)) * 128;
  mbar_expect_tx(bar, m.k_bytes);
#pragma unroll 1
  for (int i = 0; i < m.nbox; ++i) tma_load_2d(m.k + buf * m.k_bytes + (uint32_t)i * (ATTN_BN * 128), map, bar, g * a.hs + i * 64, kv.kv0(b));
}
__device__ __forceinline__ void attn_load_v(const TileCtx& c, const AttnArgs& a, KvWalk kv, int g, int b) {
  const AttnSmem m = attn_smem(c, a);
  const uint32_t buf = (uint32_t)b & 1u, bar = smem_u32(c.ctl) + 24u + 8u * buf;
  mbar_expect_tx(bar, m.v_bytes);
  tma_load_2d(m.v + buf * m.v_bytes, reinterpret_cast<const char*>(c.tmaps) + (size_t)(c.amap_base + (kv.seg(b) ? a.v1map : a.v0map)) * 128, bar,
              kv.kv0(b), g * a.hs);
}

// The arguments are read where they are used (they lie in shared memory): what stays live through the block loop is little
// more than a row's 64 scores.
__device__ __forceinline__ void tile_attention(const TileCtx& c, const AttnArgs& a, int tile) {
  const int warp = worker_tid() >> 5, lane = worker_tid() & 31;
  const AttnPlace at = attn_place(a, tile);
  const int g = (at.head * a.hkv) / a.hq, q0 = at.q0;
  const uint32_t bar_q = smem_u32(c.ctl), bar_k = bar_q + 8, bar_v = bar_q + 24, bar_s = bar_q + 40, bar_o = bar_q + 48;   // (K, V: two each)
  const uint32_t met_s = bar_q + 56, met_p = bar_q + 64;     // every warp has read its scores; has written its probabilities
  const bool loads_on = !c.drop_loads;          // (test hook: with the loads off, the waits below run out)
  KvWalk kv;                                    // a tile always has at least one key block
  kv.n0 = (a.t0 + ATTN_BN - 1) / ATTN_BN;
  kv.n = kv.n0 + (a.t1 + ATTN_BN - 1) / ATTN_BN;
  if (a.causal) kv.n = min(kv.n, (q0 + ATTN_BQ - 1) / ATTN_BN + 1);

  if (warp == 0) {
    if (lane < 9) {
      mbar_init(bar_q + 8u * lane, lane < 7 ? 1 : WORKER_THREADS / 32);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    if (lane == 0 && loads_on) {
      asm volatile("fence.proxy.async;" ::: "memory");
      const AttnSmem m = attn_smem(c, a);
      const int nbox = m.nbox, hs = a.hs;
      const uint32_t Qs = m.q;
      const char* qmap = reinterpret_cast<const char*>(c.tmaps) + (size_t)(c.amap_base + a.qmap) * 128;
      if (a.hpt <= 1) {
        mbar_expect_tx(bar_q, (uint32_t)nbox * (ATTN_BQ * 128));
#pragma unroll 1
        for (int b = 0; b < nbox; ++b) tma_load_2d(Qs + (uint32_t)b * (ATTN_BQ * 128), qmap, bar_q, at.head * hs + b * 64, q0);
      } else {
        // head i of the tile: a box of rph rows (rows past tq are outside the tensor and arrive as zeros) at row i * rph
        // (a multiple of 8 rows = of one 1024-byte swizzle group); rows past the last head keep whatever the slab held --
        // every output row depends on its own query row only, and those rows are never stored
        const int rph = a.rph;
        mbar_expect_tx(bar_q, (uint32_t)(at.nh * nbox * rph * 128));
#pragma unroll 1
        for (int i = 0; i < at.nh; ++i)
#pragma unroll 1
          for (int b = 0; b < nbox; ++b)
            tma_load_2d(Qs + (uint32_t)b * (ATTN_BQ * 128) + (uint32_t)(i * rph * 128), qmap, bar_q, (at.head + i) * hs + b * 64, 0);
      }
      attn_load_k(c, a, kv, g, 0);
      attn_load_v(c, a, kv, g, 0);
      if (kv.n > 1) attn_load_k(c, a, kv, g, 1);
    }
    __syncwarp();
  }
  worker_sync(c);

  const uint32_t lane_off = (uint32_t)(warp * 32) << 16;
  const uint32_t tmem_s = c.tmem;                            // S: columns [0, 64)
  const uint32_t tmem_p = c.tmem + (uint32_t)ATTN_BN;        // P: 32 columns of bf16 pairs
  const uint32_t tmem_o = tmem_p + (uint32_t)ATTN_BN / 2;    // O: hs columns
  // Low words of the descriptors a warp issues from, worked out once: warp 0 Q and K, warp 1 V^T.
  const uint64_t desc_hi = umma_desc_sw128(0u);
  uint32_t lo_k, lo_q, step;
  {
    const AttnSmem m = attn_smem(c, a);
    lo_q = m.q >> 4; lo_k = (warp == 1 ? m.v : m.k) >> 4; step = (warp == 1 ? m.v_bytes : m.k_bytes) >> 4;
  }
  const int hs16 = a.hs / 16;
  auto issue_s = [&](uint32_t buf) {                         // warp 0, converged: S of the K block in `buf`
    tc_fence_after();
    const uint32_t idesc_s = umma_idesc_bf16(ATTN_BN);
    uint64_t qd = desc_hi + lo_q, kd = desc_hi + (lo_k + buf * step);
    if (elect_one()) {
      int kc = 0;
#pragma unroll 1
      for (; kc + 4 <= hs16; kc += 4) {                      // one 64-column box
#pragma unroll
        for (int k = 0; k < 4; ++k) umma_bf16(tmem_s, qd + 2u * k, kd + 2u * k, idesc_s, (kc | k) != 0 ? 1u : 0u);
        qd += (ATTN_BQ * 128) >> 4; kd += (ATTN_BN * 128) >> 4;
      }
#pragma unroll 1
      for (int k = 0; kc < hs16; ++kc, ++k) umma_bf16(tmem_s, qd + 2u * k, kd + 2u * k, idesc_s, kc != 0 ? 1u : 0u);
      umma_commit(bar_s);
    }
    __syncwarp();
  };
  auto issue_pv = [&](int blk) {                             // warp 1: O += P V of block blk, once every warp has its rows of P (and O) in place
    const uint32_t ph = (uint32_t)blk & 1u;
    if (!mbar_wait(c, met_p, ph)) return;
    tc_fence_after();
    const uint32_t idesc_o = umma_idesc_bf16(16) + ((uint32_t)(hs16 - 1) << 18);         // N = hs
    const uint64_t vd = desc_hi + (lo_k + ph * step);
    if (elect_one()) {
#pragma unroll
      for (int k = 0; k < ATTN_BN / 16; ++k) umma_bf16_ta(tmem_o, tmem_p + 8u * k, vd + 2u * k, idesc_o, (blk | k) != 0 ? 1u : 0u);
      umma_commit(bar_o);
    }
    __syncwarp();
  };
  if (warp == 0 && mbar_wait(c, bar_q, 0u) && mbar_wait(c, bar_k, 0u)) issue_s(0u);

  const int row = a.hpt > 1 ? worker_tid() % a.rph : q0 + worker_tid();   // this thread's query
  float m_run = -INFINITY, l_run = 0.f;
  // A wait that runs out records the error and the loop goes on (the rest passes quickly).
  for (int blk = 0;; ++blk) {
    const uint32_t ph = (uint32_t)blk & 1u;
    const bool more = blk + 1 < kv.n;
    mbar_wait(c, bar_s, ph);                            // S(blk) complete: its K buffer is free
    __syncwarp();
    tc_fence_after();
    if (warp == 2 && lane == 0 && blk + 2 < kv.n && loads_on) attn_load_k(c, a, kv, g, blk + 2);
    __syncwarp();
    uint32_t sr[ATTN_BN];
    tmem_ld16_nowait(tmem_s + lane_off + 0u, sr + 0);
    tmem_ld16_nowait(tmem_s + lane_off + 16u, sr + 16);
    tmem_ld16_nowait(tmem_s + lane_off + 32u, sr + 32);
    tmem_ld16_nowait(tmem_s + lane_off + 48u, sr + 48);
    if (warp == 2 && more) mbar_wait(c, bar_k + 8u * (ph ^ 1u), ((uint32_t)(blk + 1) >> 1) & 1u);   // (its arrival tells warp 0)
    tmem_ld_wait();
    if (more) {                                         // the scores are in registers: the next block's go on their way
      tc_fence_before();
      arrive_warp(met_s, lane);
      if (warp == 0 && mbar_wait(c, met_s, ph)) issue_s(ph ^ 1u);
    }
    if (warp == 1 && blk > 0) issue_pv(blk - 1);        // (only now: it runs under this softmax, and no other warp waited for warp 1)
    // ---- softmax of this block: one thread per query row.  Keys a row must not see get a score of -inf first (ragged,
    // diagonal and suffix blocks only), then every block runs the same straight code: three-input maxima, two-wide
    // multiply-adds and sums (660 -> 300 instructions per warp and block), which leaves the 64 exponentials as the bulk
    {
      const int kv0 = kv.kv0(blk), seg = kv.seg(blk), valid = (seg == 0 ? a.t0 : a.t1) - kv0;
      bool ragged = valid < ATTN_BN;
      int lim = valid;                                  // keys [0, lim) of the block are visible to this row
      if (a.causal) { lim = min(lim, row - kv0 + 1); ragged = true; }
      if (a.sfx > 0 && seg == 1) {                      // blocked suffix: the leading own tokens see only one another
        ragged = true;
        if (row < a.sfx) lim = min(lim, a.sfx - kv0);
      }
      if (ragged) attn_mask(sr, lim);
    }
    float alpha;
    attn_softmax_block(sr, a.scale_log2e, m_run, l_run, alpha);
    if (blk > 0) {
      mbar_wait(c, bar_o, ph ^ 1u);                     // P V (blk-1) complete: P, O and its V^T buffer are free
      __syncwarp();
      tc_fence_after();
      // rescale O where a row maximum moved (warp-uniform decision: the TMEM accesses are warp-wide)
      if (__any_sync(0xffffffffu, alpha != 1.0f)) attn_rescale(tmem_o + lane_off, a.hs, alpha);
    }
    tmem_st16u(tmem_p + lane_off, sr);
    tmem_st16u(tmem_p + lane_off + 16u, sr + 16);
    if (warp == 3) {
      if (lane == 0 && more && loads_on) attn_load_v(c, a, kv, g, blk + 1);
      __syncwarp();
      mbar_wait(c, bar_v + 8u * ph, ((uint32_t)blk >> 1) & 1u);                                      // (its arrival tells warp 1)
    }
    tmem_st_wait();
    tc_fence_before();
    arrive_warp(met_p, lane);
    if (!more) {
      if (warp == 1) issue_pv(blk);
      mbar_wait(c, bar_o, ph);
      break;
    }
  }
  // ---- epilogue: O / l -> bf16
  __syncwarp();
  tc_fence_after();
  {
    int again = tile;                                   // (worked out anew: nothing of it stays live through the loop)
    asm volatile("" : "+r"(again));
    const AttnPlace p = attn_place(a, again);
    const int fold_h = a.hpt > 1 ? worker_tid() / a.rph : 0, q = a.hpt > 1 ? worker_tid() - fold_h * a.rph : p.q0 + worker_tid();
    const bool row_ok = q < a.tq && fold_h < p.nh;
    const int hd = a.hd;
    const float inv = l_run > 0.f ? 1.0f / l_run : 0.f;
    unsigned short* O = resolve<unsigned short>(c, a.out) + (size_t)q * a.ldo + (p.head + fold_h) * hd;
#pragma unroll 1
    for (int c0 = 0; c0 < a.hs; c0 += 16) {
      float o[16];
      tmem_ld16(tmem_o + lane_off + (uint32_t)c0, o);
      if (row_ok) {
        uint32_t pk[8];
#pragma unroll
        for (int j = 0; j < 16; j += 2) {
          __nv_bfloat162 v = __floats2bfloat162_rn(o[j] * inv, o[j + 1] * inv);
          pk[j >> 1] = *reinterpret_cast<uint32_t*>(&v);
        }
        unsigned short* dst = O + c0;
        if (c0 + 16 <= hd) {
          *reinterpret_cast<uint4*>(dst) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
          *reinterpret_cast<uint4*>(dst + 8) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
        } else {
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if (c0 + j < hd) dst[j] = (unsigned short)((j & 1) ? (pk[j >> 1] >> 16) : (pk[j >> 1] & 0xFFFFu));
        }
      }
    }
  }
  tc_fence_before();
  worker_sync(c);
  if (worker_tid() < 9) mbar_inval(bar_q + 8u * worker_tid());
}

}  // namespace vla
