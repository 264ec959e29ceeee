// GEMM tile on the 5th-generation tensor cores: operands staged by TMA into
// 128-byte-swizzled shared memory, tcgen05.mma accumulating in tensor memory,
// epilogue read back with tcgen05.ld.
//
// Tile: up to 128 tokens (MMA M, one TMEM lane each) x 128 weight rows (MMA N, one
// TMEM column each), K walked in 64-element stages, both operands K-major.  Where a node
// has few tokens (the action head's 9..51) the activation box is only as high as they
// need; the MMA reads on into the weight tile behind it and leaves lanes nobody looks at.
// A gated MLP tile covers 64 output features: gate and up rows alternate in its weight
// matrix, so it is one MMA stream and one accumulator like any other tile; the epilogue
// multiplies act(gate) by up.
//
// Roles inside the 128-thread worker: thread 0 of warp 0 issues TMA loads,
// warp 1 issues MMAs, all four warps run the epilogue (warp w reads
// TMEM lanes 32w..32w+31, a token per thread).  Every mbarrier wait is bounded; on expiry
// the worker records an error and leaves the tile.
#pragma once
#include "tiles_common.cuh"

namespace vla {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_inval(uint32_t bar) {
  asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// Suspended by the hardware until the phase completes or about `hint_ns` have passed: a waiting warp takes no issue slots
// from the warps that share its scheduler.
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity, uint32_t hint_ns) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(hint_ns)
      : "memory");
  return ok != 0;
}
// Bounded wait: false when the deadline passed or another worker already reported an error.
__device__ __forceinline__ bool mbar_wait(const TileCtx& c, uint32_t bar, uint32_t parity) {
  while (!mbar_try_wait(bar, parity, 20000u)) {
    if (*reinterpret_cast<volatile unsigned*>(c.error) != 0u) return false;
    uint64_t now;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
    if (now > c.deadline) {
      atomicCAS(c.error, 0u, (unsigned)DEV_ERR_WAIT_MBAR);
      return false;
    }
  }
  return true;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const void* tmap, uint32_t bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(tmap), "r"(bar), "r"(x), "r"(y)
      : "memory");
}

__device__ __forceinline__ void tma_prefetch_2d(const void* tmap, int x, int y) {
  asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(tmap), "r"(x), "r"(y) : "memory");
}

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, rows of 128 bytes,
// 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)1 << 16;                 // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;       // stride byte offset between 8-row groups
  d |= (uint64_t)1 << 46;                 // descriptor version
  d |= (uint64_t)2 << 61;                 // SWIZZLE_128B
  return d;
}
// Instruction descriptor: bf16 x bf16 -> fp32, both operands K-major, M = 128, N = n.
__device__ __forceinline__ uint32_t umma_idesc_bf16(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(GEMM_BM >> 4) << 24);
}
__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));   // no memory clobber: the waits, fences and
                                                                           // commits around a batch of MMAs order it
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
        "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])),
        "r"(__float_as_uint(v[7])), "r"(__float_as_uint(v[8])), "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])),
        "r"(__float_as_uint(v[11])), "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])),
        "r"(__float_as_uint(v[15]))
      : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// One lane of a converged warp (warp-uniform control flow around the asynchronous instructions it guards lets their
// descriptors live in uniform registers: 200 instead of 230 cycles per four-MMA k-block at N <= 64).
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.b32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}

// ------------------------------------------------------------------ epilogue
// Straight from tensor memory to global memory, sixteen columns at a time; nothing is staged.  A thread owns one token, so
// its row scale, its sum of squares, gate and up values, rotary pairs and sixteen-byte stores all lie in its own registers.
// A lone warp per scheduler pays for instructions (one every three or four cycles) and above all for branches (about 30
// cycles each, taken or skipped over): the five common kinds of result have straight loops of their own, everything else
// goes through one general loop.  (With every kind unrolled for every activation the kernel had 160 KB of epilogues and 30 %
// of its instruction fetches missed the cache; with the general loop alone a chunk cost 600 cycles.)
constexpr int EPI = 16;

template <int ACT, int N>
__device__ __forceinline__ void activate(float* v) {
#pragma unroll
  for (int j = 0; j < N; ++j) v[j] = apply_act_t<ACT>(v[j]);
}
__device__ __forceinline__ uint32_t pack_bf16(float x, float y) {
  __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  return *reinterpret_cast<uint32_t*>(&h);
}
__device__ __forceinline__ void put16(unsigned short* p, const float* v) {
#pragma unroll
  for (int j = 0; j < EPI; j += 8)
    *reinterpret_cast<uint4*>(p + j) = make_uint4(pack_bf16(v[j], v[j + 1]), pack_bf16(v[j + 2], v[j + 3]), pack_bf16(v[j + 4], v[j + 5]), pack_bf16(v[j + 6], v[j + 7]));
}
// v[j] += scale * p[j], j < n (n = EPI: four 16-byte loads, else element by element)
__device__ __forceinline__ void add_row(float* v, const float* p, int n, float scale) {
  if (n == EPI) {
#pragma unroll
    for (int j = 0; j < EPI; j += 4) {
      const float4 t = __ldcg(reinterpret_cast<const float4*>(p + j));
      v[j] = fmaf(scale, t.x, v[j]); v[j + 1] = fmaf(scale, t.y, v[j + 1]);
      v[j + 2] = fmaf(scale, t.z, v[j + 2]); v[j + 3] = fmaf(scale, t.w, v[j + 3]);
    }
  } else {
#pragma unroll
    for (int j = 0; j < EPI; ++j)
      if (j < n) v[j] = fmaf(scale, ld_act(p + j), v[j]);
  }
}

// Calls body(c0, v) for the accumulator columns [lo, hi) of this thread's token, scaled by rs; the next chunk is on its way
// from tensor memory meanwhile.
template <typename F>
__device__ __forceinline__ void epi_chunks(uint32_t tmem, int lo, int hi, float rs, F body) {
  if (lo >= hi) return;
  uint32_t nx[EPI];
  tmem_ld16_nowait(tmem + (uint32_t)lo, nx);
#pragma unroll 1
  for (int c0 = lo; c0 < hi; c0 += EPI) {
    float v[EPI];
    tmem_ld_wait();
#pragma unroll
    for (int j = 0; j < EPI; ++j) v[j] = __uint_as_float(nx[j]) * rs;
    tmem_ld16_nowait(tmem + (uint32_t)min(c0 + EPI, hi - EPI), nx);          // (the last chunk again after the last one)
    body(c0, v);
  }
  tmem_ld_wait();
}
template <int ACT>
__device__ __forceinline__ void epi_gated(uint32_t tmem, int cols, float rs, float c_acc, unsigned short* out, bool live) {
  epi_chunks(tmem, 0, cols, rs, [&](int c0, float* v) {      // columns 2i, 2i + 1: gate and up value of output feature i
    float o[EPI / 2];
#pragma unroll
    for (int j = 0; j < EPI / 2; ++j) o[j] = v[2 * j];
    activate<ACT, EPI / 2>(o);
#pragma unroll
    for (int j = 0; j < EPI / 2; ++j) o[j] *= v[2 * j + 1] * c_acc;
    if (live) *reinterpret_cast<uint4*>(out + (c0 >> 1)) = make_uint4(pack_bf16(o[0], o[1]), pack_bf16(o[2], o[3]), pack_bf16(o[4], o[5]), pack_bf16(o[6], o[7]));
  });
}

// One token's row of the tile.  `tok` is the token's index in the node (a lane past the last token repeats it, `live` false,
// and stores nothing), `r0` the tile's first weight row, `rs` the token's row scale, `under` says that the accumulators
// already hold X.
__device__ __forceinline__ void gemm_epilogue(const TileCtx& c, const GemmArgs& g, uint32_t tmem, int tok, bool live, int r0, float rs, bool under,
                                              int ft) {
  const int act = g.act, N = g.N;
  const float c_acc = g.c_acc;
  const GemmPtrs ptrs = gemm_ptrs(c, g);
  float* const ssq_out = resolve<float>(c, g.ss_out);
  float* const out32 = ptrs.out32 ? ptrs.out32 + (size_t)tok * g.ldo32 + r0 : nullptr;
  unsigned short* const out16 = ptrs.out16 ? ptrs.out16 + (size_t)tok * g.ldo16 + (g.dual ? r0 / 2 : r0) : nullptr;
  const int cols = min(GEMM_BM, (g.dual ? 2 * N : N) - r0);
  if (g.vec16) {
    if (g.dual) {
      if (act == ACT_SILU) epi_gated<ACT_SILU>(tmem, cols, rs, c_acc, out16, live);
      else if (act == ACT_GELU) epi_gated<ACT_GELU>(tmem, cols, rs, c_acc, out16, live);
      else epi_gated<ACT_NONE>(tmem, cols, rs, c_acc, out16, live);
      return;
    }
    const bool plain = !ptrs.bias && !ptrs.vec && !ptrs.tab && !ptrs.tab2 && (!ptrs.X || under) && c_acc == 1.0f;
    if (plain && !ssq_out && !ptrs.out32 && act != ACT_SILU) {            // bf16 only (q|k|v, MLP up, cross projections)
      int split = cols;                                                     // columns from here on are V features
      if (ptrs.outT) split = max(0, min(cols, g.t_col0 - r0));
      if (act == ACT_GELU)
        epi_chunks(tmem, 0, split, rs, [&](int c0, float* v) { activate<ACT_GELU, EPI>(v); if (live) put16(out16 + c0, v); });
      else if (g.rope_cols > 0) {       // q and k columns: rotary pairs are neighbours; the table holds (cos, sin) per pair
        const float* t0 = resolve<const float>(c, g.rope_tab) + (size_t)tok * g.rope_hd;
        epi_chunks(tmem, 0, split, rs, [&](int c0, float* v) {
          const float4* t = reinterpret_cast<const float4*>(t0 + (r0 + c0) % g.rope_hd);
#pragma unroll
          for (int j = 0; j < EPI; j += 4) {
            const float4 cs = __ldg(t + (j >> 2));
            const float x0 = v[j], x1 = v[j + 1], x2 = v[j + 2], x3 = v[j + 3];
            v[j] = fmaf(x0, cs.x, -x1 * cs.y); v[j + 1] = fmaf(x1, cs.x, x0 * cs.y);
            v[j + 2] = fmaf(x2, cs.z, -x3 * cs.w); v[j + 3] = fmaf(x3, cs.z, x2 * cs.w);
          }
          if (live) put16(out16 + c0, v);
        });
      } else
        epi_chunks(tmem, 0, split, rs, [&](int c0, float* v) { if (live) put16(out16 + c0, v); });
      if (split < cols) {               // rows of V^T, a warp's tokens side by side
        unsigned short* const base = ptrs.outT + (ptrdiff_t)(r0 - g.t_col0) * g.ldoT + tok;
        epi_chunks(tmem, split, cols, rs, [&](int c0, float* v) {
          unsigned short* op = base + (ptrdiff_t)c0 * g.ldoT;
          if (live) {
#pragma unroll
            for (int j = 0; j < EPI; ++j) { *op = f32_to_bf16_bits(v[j]); op += g.ldoT; }
          }
        });
      }
      return;
    }
    if (plain && act == ACT_NONE && out32 && out16 && ssq_out) {            // residual stream
      float sq = 0.f;
      epi_chunks(tmem, 0, cols, rs, [&](int c0, float* v) {
#pragma unroll
        for (int j = 0; j < EPI; ++j) sq = fmaf(v[j], v[j], sq);
        if (live) {
#pragma unroll
          for (int j = 0; j < EPI; j += 4) *reinterpret_cast<float4*>(out32 + c0 + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
          put16(out16 + c0, v);
        }
      });
      if (live) ssq_out[(size_t)tok * g.ss_out_ld + ft] = sq;
      return;
    }
  }
  // ---- anything else: biases, tables, addends, solver coefficients, odd widths
  float sq = 0.f;
#pragma unroll 1
  for (int c0 = 0; c0 < cols; c0 += EPI) {
    const int f = r0 + c0, n = g.vec16 ? EPI : min(EPI, (g.dual ? 2 * N : N) - f);
    float v[EPI];
    tmem_ld16(tmem + (uint32_t)c0, v);
#pragma unroll
    for (int j = 0; j < EPI; ++j) v[j] *= rs;
    if (g.dual) {
#pragma unroll
      for (int j = 0; j < EPI / 2; ++j)
        if (live && 2 * j < n) out16[(c0 >> 1) + j] = f32_to_bf16_bits(apply_act(act, v[2 * j]) * v[2 * j + 1] * c_acc);
      continue;
    }
    if (ptrs.bias) add_row(v, ptrs.bias + f, n, 1.0f);
    if (act == ACT_GELU) activate<ACT_GELU, EPI>(v);
    else if (act == ACT_SILU) activate<ACT_SILU, EPI>(v);
#pragma unroll
    for (int j = 0; j < EPI; ++j) v[j] *= c_acc;
    if (ptrs.X && !under) add_row(v, ptrs.X + (size_t)tok * g.ldx + f, n, g.c_x);
    if (ptrs.vec) add_row(v, ptrs.vec + f, n, 1.0f);
    if (ptrs.tab) add_row(v, ptrs.tab + (size_t)tok * g.ldtab + f, n, 1.0f);
    if (ptrs.tab2) add_row(v, ptrs.tab2 + (size_t)tok * g.ldtab2 + f, n, 1.0f);
#pragma unroll
    for (int j = 0; j < EPI; ++j)
      if (j < n) sq = fmaf(v[j], v[j], sq);
    if (!live) continue;
    if (ptrs.outT && f >= g.t_col0) {
      unsigned short* op = ptrs.outT + (size_t)(f - g.t_col0) * g.ldoT + tok;
#pragma unroll
      for (int j = 0; j < EPI; ++j) { *op = f32_to_bf16_bits(v[j]); op += g.ldoT; }
    } else if (g.vec16) {
      if (out32) {
#pragma unroll
        for (int j = 0; j < EPI; j += 4) *reinterpret_cast<float4*>(out32 + c0 + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
      }
      if (out16) put16(out16 + c0, v);
    } else {
#pragma unroll
      for (int j = 0; j < EPI; ++j) {
        if (j < n && out32) out32[c0 + j] = v[j];
        if (j < n && out16) out16[c0 + j] = f32_to_bf16_bits(v[j]);
      }
    }
  }
  if (ssq_out && live) ssq_out[(size_t)tok * g.ss_out_ld + ft] = sq;
}

constexpr int GEMM_W_STAGE_BYTES = GEMM_BM * GEMM_BK * 2;

// The producer lane's look at the worker's next tile (see tile_gemm).  Not while another worker of the SM waits for room (this
// one would keep its own), and not past a waiting action-head tile, which goes first and needs the memory.
__device__ __forceinline__ void prime_next(const TileCtx& c, int bt, int S, int s, uint32_t ph, uint32_t acc_ph, uint32_t bar0, uint32_t stage0,
                                           uint32_t a_bytes, uint32_t stage_bytes) {
  WorkerSlot* const w = c.slot;
  if (w->held_tail == w->held_head || w->prio_tail != w->prio_head || *w->room_wait != 0u) return;
  __threadfence_block();
  const TileJob& j = w->job[w->held_head & 1u];
  const GemmArgs& g = j.desc.u.gemm;
  if (j.desc.op != OP_GEMM || j.early || g.bt != bt || j.smem_units > w->smem_units) return;
  const int nkb = g.Kp / GEMM_BK, n = min(S, nkb);
  w->ring_stages = S; w->ring_s = s; w->ring_ph = ph; w->ring_acc = acc_ph ^ 1u; w->ring_n = n;
  w->primed = 1;
  const char* tm = reinterpret_cast<const char*>(c.tmaps);
  const void* wmap = tm + (size_t)g.wmap * 128;
  const void* amap = tm + (size_t)(c.n_weight_tmaps + (int)j.inst * c.n_act_tmaps + g.amap) * 128;
  const int r0 = (int)j.tile / g.tiles_t * GEMM_BM, t0 = (int)j.tile % g.tiles_t * bt;
  asm volatile("fence.proxy.async;" ::: "memory");
#pragma unroll 1
  for (int kb = 0; kb < n; ++kb) {
    const uint32_t bar = bar0 + 8u * (uint32_t)s, dst = stage0 + (uint32_t)s * stage_bytes;
    mbar_wait(c, bar + 8u * (uint32_t)S, ph ^ 1u);     // (after a wait that ran out the tile only has to end)
    mbar_expect_tx(bar, stage_bytes);
    tma_load_2d(dst + a_bytes, wmap, bar, kb * GEMM_BK, r0);
    tma_load_2d(dst, amap, bar, kb * GEMM_BK, t0);
    if (++s == S) { s = 0; ph ^= 1u; }
  }
}

// What bounds it: with one tile per SM, the issuing lanes (per k-block one barrier test, two loads, four MMAs) and the
// round trip of a stage; with three, instruction fetch and the L2-to-shared-memory path.  Stage and phase run along instead
// of being divided out of the k-block index (a runtime division per role cost as much as the four MMAs).
__device__ __forceinline__ void tile_gemm(const TileCtx& c, const GemmArgs& g, int tile) {
  const int bt = g.bt;
  const int ft = tile / g.tiles_t, t0 = tile % g.tiles_t * bt, r0 = ft * GEMM_BM;   // first token and first weight row of the tile
  const int nt = min(bt, g.M - t0);
  const int warp = worker_tid() >> 5, lane = worker_tid() & 31;
  const int nkb = g.Kp / GEMM_BK;
  const uint32_t a_bytes = (uint32_t)(bt * GEMM_BK * 2), stage_bytes = a_bytes + GEMM_W_STAGE_BYTES;   // activations, then weights
  // The operand ring starts afresh, or goes on where the tile before left it (its producer has requested this tile's first
  // k-blocks already).  s0, ph0: stage and full-barrier parity of the first k-block; pre: k-blocks on their way.
  int S, s0 = 0, pre;
  uint32_t ph0 = 0u, acc_ph = 0u;
  const bool cont = c.cont != 0;
  if (cont) { S = c.slot->ring_stages; s0 = c.slot->ring_s; ph0 = c.slot->ring_ph; acc_ph = c.slot->ring_acc; pre = c.slot->ring_n; }
  else { S = gemm_stages_in(c.smem_bytes, bt, g.Kp, g.stages); pre = S; }

  const uint32_t bar0 = smem_u32(c.ctl);               // full[S], empty[S], accum (the worker's control block)
  const uint32_t stage0 = smem_u32(c.smem);
  const uint32_t accum_bar = bar0 + 16u * (uint32_t)S;
  if (warp == 0 && !cont) {
    if (lane <= 2 * S) {                               // (2 S + 1 <= 25 barriers: one lane each)
      mbar_init(bar0 + 8u * lane, 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
  }
  const char* tm = reinterpret_cast<const char*>(c.tmaps);
  const void* wmap = tm + (size_t)g.wmap * 128;
  const void* amap = tm + (size_t)(c.amap_base + g.amap) * 128;
  auto load_w = [&](int kb, uint32_t bar, uint32_t dst) {
    mbar_expect_tx(bar, stage_bytes);
    tma_load_2d(dst + a_bytes, wmap, bar, kb * GEMM_BK, r0);
  };
  auto load_a = [&](int kb, uint32_t bar, uint32_t dst) { tma_load_2d(dst, amap, bar, kb * GEMM_BK, t0); };
  if (warp == 0) {
    if (lane == 0 && !c.drop_loads && !cont) {         // the first stages are on their way before anything else happens
      // The weights do not depend on anything: they fill the stages (and, where the tile was taken before its operands
      // exist, the L2 beyond those) while the predecessors still run; the activations follow the release.
#pragma unroll 1
      for (int kb = 0; kb < S; ++kb) load_w(kb, bar0 + 8u * (uint32_t)kb, stage0 + (uint32_t)kb * stage_bytes);
      if (c.wait_word) {
#pragma unroll 1
        for (int kb = S; kb < nkb; ++kb) tma_prefetch_2d(wmap, kb * GEMM_BK, r0);
        asm volatile("prefetch.tensormap [%0];" ::"l"(amap) : "memory");
        wait_release(c);
      }
      asm volatile("fence.proxy.async;" ::: "memory");   // operands were written by generic stores on other SMs
#pragma unroll 1
      for (int kb = 0; kb < S; ++kb) load_a(kb, bar0 + 8u * (uint32_t)kb, stage0 + (uint32_t)kb * stage_bytes);
    }
    __syncwarp();
  }
  if (c.wait_word) worker_sync(c);                     // nobody reads an operand before the release

  const int tok = t0 + min(worker_tid(), nt - 1);      // this thread's token (lanes past the last one repeat it)
  const bool warp_live = warp * 32 < nt;
  const uint32_t my_tmem = c.tmem + ((uint32_t)(warp * 32) << 16);
  // Residual rows go into the accumulators before the first MMA: their round trip then lies beside that of the first
  // operand stages, and the epilogue neither reads nor adds anything.
  const bool under = g.X != 0 && g.vec16 && g.c_acc == 1.0f && g.c_x == 1.0f && g.rs_d == 0 && g.act == ACT_NONE;
  if (under) {
    if (warp_live) {
      const float* x = resolve<const float>(c, g.X) + (size_t)tok * g.ldx + r0;
      const int cols = min(GEMM_BM, g.N - r0);
#pragma unroll 1
      for (int c0 = 0; c0 < cols; c0 += 16) {
        float v[16];
#pragma unroll
        for (int j = 0; j < 16; j += 4) *reinterpret_cast<float4*>(v + j) = __ldcg(reinterpret_cast<const float4*>(x + c0 + j));
        tmem_st16(my_tmem + (uint32_t)c0, v);
      }
      tmem_st_wait();
    }
    tc_fence_before();
  }
  // Folded RMSNorm: the token's row scale from the stream's partial sums of squares, added in a fixed order.
  float rs = 1.0f;
  if (g.rs_d > 0 && warp_live) {
    const float* sp = resolve<const float>(c, g.ss_in) + (size_t)tok * g.ss_nft;
    float ssq = 0.f;
#pragma unroll 4
    for (int q = 0; q < g.ss_nft; ++q) ssq += ld_act(sp + q);
    rs = 1.0f / sqrtf(ssq / (float)g.rs_d + 1e-6f);
  }
  worker_sync(c);

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA producer
      uint32_t ph = ph0;
      int s = s0 + pre;
      if (s >= S) { s -= S; ph ^= 1u; }
      bool go = !c.drop_loads;
#pragma unroll 1
      for (int kb = pre; kb < nkb && go; ++kb) {
        const uint32_t bar = bar0 + 8u * (uint32_t)s, dst = stage0 + (uint32_t)s * stage_bytes;
        if (!(go = mbar_wait(c, bar + 8u * (uint32_t)S, ph ^ 1u))) break;
        load_w(kb, bar, dst);
        load_a(kb, bar, dst);
        if (++s == S) { s = 0; ph ^= 1u; }
      }
      // While this tile's last MMAs and its epilogue run, the stages would stand empty: if the tile this worker runs next is
      // already here and has the same shape, its first k-blocks go into them now.  It then keeps this tile's memory and
      // barriers.  (Operand loads cover about half a worker's time otherwise, and the L2-to-shared-memory path is what
      // three workers share.)
      if (go && c.slot) prime_next(c, bt, S, s, ph, acc_ph, bar0, stage0, a_bytes, stage_bytes);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- MMA issuer (the whole warp walks the loop, one elected lane issues)
    const uint32_t idesc = umma_idesc_bf16(GEMM_BM);
    const uint64_t desc0 = umma_desc_sw128(stage0);
    uint32_t ph = ph0;
    int s = s0;
#pragma unroll 1
    for (int kb = 0; kb < nkb; ++kb) {
      const uint32_t bar = bar0 + 8u * (uint32_t)s;
      if (!mbar_wait(c, bar, ph)) break;
      tc_fence_after();
      const uint64_t ad = desc0 + (uint32_t)s * (stage_bytes >> 4), wd = ad + (a_bytes >> 4);
      if (elect_one()) {
#pragma unroll
        for (int k = 0; k < GEMM_BK / 16; ++k)
          umma_bf16(c.tmem, ad + 2u * k, wd + 2u * k, idesc, (kb | k) != 0 || under ? 1u : 0u);   // 16 bf16 = 32 bytes per K step
        umma_commit(bar + 8u * (uint32_t)S);     // stage reusable once these MMAs have read it
        if (kb == nkb - 1) umma_commit(accum_bar);   // accumulators complete
      }
      __syncwarp();
      if (++s == S) { s = 0; ph ^= 1u; }
    }
  }

  const bool ready = mbar_wait(c, accum_bar, acc_ph);
  __syncwarp();
  tc_fence_after();
  if (ready && warp_live) gemm_epilogue(c, g, my_tmem, tok, worker_tid() < nt, r0, rs, under, ft);
  tc_fence_before();
  worker_sync(c);
  if (!(c.slot && c.slot->primed) && worker_tid() <= 2 * S) mbar_inval(bar0 + 8u * worker_tid());
}

}  // namespace vla
