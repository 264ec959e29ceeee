// GEMM tile on the 5th-generation tensor cores: operands staged by TMA into
// 128-byte-swizzled shared memory, tcgen05.mma accumulating in tensor memory,
// epilogue read back with tcgen05.ld.
//
// Tile: up to 128 tokens (MMA M, one TMEM lane each) x 128 weight rows (MMA N, one
// TMEM column each), K walked in 64-element stages, both operands K-major.  Where a node
// has few tokens (the action head's 9..51) the activation box is only as high as they
// need; the MMA (M = 64 there) reads on into the weight tile behind it and leaves lanes
// nobody looks at.
// A gated MLP tile covers 64 output features: gate and up rows alternate in its weight
// matrix, so it is one MMA stream and one accumulator like any other tile; the epilogue
// multiplies act(gate) by up.
//
// Roles inside the 128-thread worker: thread 0 of warp 0 issues TMA loads,
// warp 1 issues MMAs, all four warps run the epilogue (warp w reads TMEM lanes
// 32w..32w+31 in 16x256b fragments: a quad of lanes holds 32 features of a token).  Every
// mbarrier wait is bounded; on expiry the worker records an error and leaves the tile.
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
// Instruction descriptor: bf16 x bf16 -> fp32, both operands K-major, M = m (128, or 64: 16 rows per 32 tensor-memory lanes), N = n.
__device__ __forceinline__ uint32_t umma_idesc_bf16(int n, int m = 128) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
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
// Straight from tensor memory to global memory; nothing is staged.  The accumulators are read in the 16x256b fragment layout
// (a quad of lanes per token, two columns of every eight per lane), and the weight rows were reordered at load so that a
// lane's eight columns of a 32-column group are eight consecutive features: a quad writes a whole 128-byte line of fp32 (or
// 64 bytes of bf16), eight lines per instruction.  With a token per lane -- 32 lines per instruction -- the load/store unit
// was what three workers of an SM waited for (28 cycles a store; epilogues and residual rows cost 31 % of a full-load step).
// Gate and up values, rotary pairs and a token's partial sum of squares still meet in one lane or quad.
// A lone warp per scheduler pays for every branch (about 30 cycles), so the common kinds of result have straight loops of
// their own and everything else goes through one general loop; more variants than that and the instruction cache pays.
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
// One 16-lane half of a warp's tensor memory x 32 columns: v[4 b + 2 r + e] = token (lane / 4) + 8 r, column 8 b + 2 (lane % 4) + e.
__device__ __forceinline__ void tmem_ld_frag(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_st_frag(uint32_t taddr, const float* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x256b.x4.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "f"(v[8]), "f"(v[9]),
        "f"(v[10]), "f"(v[11]), "f"(v[12]), "f"(v[13]), "f"(v[14]), "f"(v[15])
      : "memory");
}
// Calls body(c0, v) for the accumulator columns [lo, hi) of this thread's token (one TMEM lane), scaled by rs; the next
// chunk is on its way from tensor memory meanwhile.
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
// Calls body(c0, v) for 32-column groups [0, cols) of one half, v in the order of tmem_ld_frag, the two tokens scaled.
template <typename F>
__device__ __forceinline__ void epi_frags(uint32_t tmem, int cols, float ra, float rb, F body) {
  uint32_t nx[EPI];
  tmem_ld_frag(tmem, nx);
#pragma unroll 1
  for (int c0 = 0; c0 < cols; c0 += 32) {
    float v[EPI];
    tmem_ld_wait();
#pragma unroll
    for (int j = 0; j < EPI; ++j) v[j] = __uint_as_float(nx[j]) * ((j & 2) ? rb : ra);
    tmem_ld_frag(tmem + (uint32_t)(c0 + 32 < cols ? c0 + 32 : c0), nx);
    body(c0, v);
  }
  tmem_ld_wait();
}
__device__ __forceinline__ void st_row8(float* p, const float* v) {     // v: one token's values of a fragment, at 0, 1, 4, 5, 8, 9, 12, 13
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
               ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[4]), "f"(v[5]), "f"(v[8]), "f"(v[9]), "f"(v[12]), "f"(v[13]) : "memory");
}
__device__ __forceinline__ void st_row8(unsigned short* p, const float* v) {
  *reinterpret_cast<uint4*>(p) = make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[4], v[5]), pack_bf16(v[8], v[9]), pack_bf16(v[12], v[13]));
}
// (cos, sin) per pair: the lane's four pairs of one token
__device__ __forceinline__ void rotate8(float* v, const float* tab) {
  const float4 lo = __ldg(reinterpret_cast<const float4*>(tab)), hi = __ldg(reinterpret_cast<const float4*>(tab) + 1);
  const float cs[4] = {lo.x, lo.z, hi.x, hi.z}, sn[4] = {lo.y, lo.w, hi.y, hi.w};
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const float x = v[4 * b], y = v[4 * b + 1];
    v[4 * b] = fmaf(x, cs[b], -y * sn[b]); v[4 * b + 1] = fmaf(y, cs[b], x * sn[b]);
  }
}

// What a straight epilogue needs beside the tile's place: `live` tokens of this warp exist, `tok` is the warp's first token.
struct EpiPlace { uint32_t tmem; int tok, live, lane, r0, cols; float rs; };

// Walks the two halves of the warp: fn(row, tmem, ra, rb) with this lane's tokens `row` and `row` + 8 of the warp.
template <typename F>
__device__ __forceinline__ void epi_halves(const EpiPlace& e, F fn) {
#pragma unroll 1
  for (int h = 0; h < 2 && 16 * h < e.live; ++h) {
    const int row = 16 * h + (e.lane >> 2);
    fn(row, e.tmem + ((uint32_t)(16 * h) << 16), __shfl_sync(0xffffffffu, e.rs, row), __shfl_sync(0xffffffffu, e.rs, row + 8));
  }
}
template <int ACT>
__device__ __forceinline__ void epi_gated(const EpiPlace& e, const GemmArgs& g, unsigned short* out16) {
  const int q = e.lane & 3;
  const float c_acc = g.c_acc;
  epi_halves(e, [&](int row, uint32_t tmem, float ra, float rb) {
    unsigned short* pa = out16 + (size_t)(e.tok + row) * g.ldo16 + e.r0 / 2 + 4 * q;
    unsigned short* pb = pa + (size_t)8 * g.ldo16;
    epi_frags(tmem, e.cols, ra, rb, [&](int c0, float* v) {       // a lane's columns 2 i, 2 i + 1: gate and up value of one feature
      float o[8];
#pragma unroll
      for (int b = 0; b < 4; ++b) { o[b] = v[4 * b]; o[4 + b] = v[4 * b + 2]; }
      activate<ACT, 8>(o);
#pragma unroll
      for (int b = 0; b < 4; ++b) { o[b] *= v[4 * b + 1] * c_acc; o[4 + b] *= v[4 * b + 3] * c_acc; }
      const bool fok = c0 + 8 * q < e.cols;
      if (fok && row < e.live) *reinterpret_cast<uint2*>(pa + c0 / 2) = make_uint2(pack_bf16(o[0], o[1]), pack_bf16(o[2], o[3]));
      if (fok && row + 8 < e.live) *reinterpret_cast<uint2*>(pb + c0 / 2) = make_uint2(pack_bf16(o[4], o[5]), pack_bf16(o[6], o[7]));
    });
  });
}
template <int ACT, bool ROPE>
__device__ __forceinline__ void epi_bf16(const EpiPlace& e, const GemmArgs& g, unsigned short* out16, const float* rope) {
  const int q = e.lane & 3;
  epi_halves(e, [&](int row, uint32_t tmem, float ra, float rb) {
    unsigned short* pa = out16 + (size_t)(e.tok + row) * g.ldo16 + e.r0 + 8 * q;
    unsigned short* pb = pa + (size_t)8 * g.ldo16;
    const int last = e.live - 1;
    const float* ta = ROPE ? rope + (size_t)(e.tok + min(row, last)) * g.rope_hd : nullptr;
    const float* tb = ROPE ? rope + (size_t)(e.tok + min(row + 8, last)) * g.rope_hd : nullptr;
    epi_frags(tmem, e.cols, ra, rb, [&](int c0, float* v) {
      activate<ACT, EPI>(v);
      if (ROPE) {
        const int i = (e.r0 + c0 + 8 * q) % g.rope_hd;
        rotate8(v, ta + i);
        rotate8(v + 2, tb + i);
      }
      const bool fok = c0 + 8 * q < e.cols;
      if (fok && row < e.live) st_row8(pa + c0, v);
      if (fok && row + 8 < e.live) st_row8(pb + c0, v + 2);
    });
  });
}
// fp32 rows with, optionally, their bf16 mirror and the tile's share of each token's sum of squares (residual streams).
// POST: the solver update, out = c_acc * v + c_x * X + tab, whose addends cannot lie under a product that gets scaled.
template <bool MIRROR, bool POST>
__device__ __forceinline__ void epi_stream(const TileCtx& c, const EpiPlace& e, const GemmArgs& g, float* out32, unsigned short* out16, float* ssq, int ft) {
  const int q = e.lane & 3;
  epi_halves(e, [&](int row, uint32_t tmem, float ra, float rb) {
    float* pa = out32 + (size_t)(e.tok + row) * g.ldo32 + e.r0 + 8 * q;
    float* pb = pa + (size_t)8 * g.ldo32;
    unsigned short* ha = MIRROR ? out16 + (size_t)(e.tok + row) * g.ldo16 + e.r0 + 8 * q : nullptr;
    unsigned short* hb = MIRROR ? ha + (size_t)8 * g.ldo16 : nullptr;
    float sa = 0.f, sb = 0.f;
    epi_frags(tmem, e.cols, ra, rb, [&](int c0, float* v) {
      const bool fok = c0 + 8 * q < e.cols;
      if (POST && fok) {
#pragma unroll
        for (int j = 0; j < EPI; ++j) v[j] *= g.c_acc;
        auto add = [&](Ref ref, int ld, float scale) {
          const float* p = resolve<const float>(c, ref) + e.r0 + c0 + 8 * q;
          float4 t[2][2];
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const float4* x = reinterpret_cast<const float4*>(p + (size_t)(e.tok + min(row + 8 * k, e.live - 1)) * ld);
            t[k][0] = __ldcg(x); t[k][1] = __ldcg(x + 1);
          }
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            float* u = v + 2 * k;
            u[0] = fmaf(scale, t[k][0].x, u[0]); u[1] = fmaf(scale, t[k][0].y, u[1]); u[4] = fmaf(scale, t[k][0].z, u[4]); u[5] = fmaf(scale, t[k][0].w, u[5]);
            u[8] = fmaf(scale, t[k][1].x, u[8]); u[9] = fmaf(scale, t[k][1].y, u[9]); u[12] = fmaf(scale, t[k][1].z, u[12]); u[13] = fmaf(scale, t[k][1].w, u[13]);
          }
        };
        if (g.X) add(g.X, g.ldx, g.c_x);
        if (g.tab) add(g.tab, g.ldtab, 1.0f);
      }
      if (MIRROR && fok) {
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          sa = fmaf(v[4 * b], v[4 * b], sa); sa = fmaf(v[4 * b + 1], v[4 * b + 1], sa);
          sb = fmaf(v[4 * b + 2], v[4 * b + 2], sb); sb = fmaf(v[4 * b + 3], v[4 * b + 3], sb);
        }
      }
      if (fok && row < e.live) { st_row8(pa + c0, v); if (MIRROR) st_row8(ha + c0, v); }
      if (fok && row + 8 < e.live) { st_row8(pb + c0, v + 2); if (MIRROR) st_row8(hb + c0, v + 2); }
    });
    if (MIRROR && ssq) {
      sa += __shfl_xor_sync(0xffffffffu, sa, 1); sb += __shfl_xor_sync(0xffffffffu, sb, 1);
      sa += __shfl_xor_sync(0xffffffffu, sa, 2); sb += __shfl_xor_sync(0xffffffffu, sb, 2);
      float* sp = ssq + (size_t)(e.tok + row) * g.ss_out_ld + ft;
      if (q == 0 && row < e.live) sp[0] = sa;
      if (q == 0 && row + 8 < e.live) sp[(size_t)8 * g.ss_out_ld] = sb;
    }
  });
}
// Residual rows, fp32, in the fragment layout: this lane's two tokens of a half, eight features of each, of two groups of 32
// columns.  The first two groups are asked for in front of the main loop, each later one in the place of a group just added: half
// the round trips lie under the loop, where laying the rows under the accumulators had all four of a 128-token tile in front of it,
// and the sum is rounded once, not once per MMA (CogACT 18.74 -> 18.57 ms; the other workloads 0.4 to 1.4 %, which is what their runs differ by).
// Two groups in flight cost 44 bytes of spills in the persistent kernel, one group 16 and 1 % of CogACT, GR00T and 4 x 3 (18.53 -> 18.76,
// 36.06 -> 36.43, 40.28 -> 40.71 ms); four groups 440 bytes.
struct ResidRows { float4 v[2][2][2]; };
__device__ __forceinline__ void resid_load(const float* x, int ldx, int tok, int live, int half, int lane, int cols, int c, float4 (&v)[2][2]) {
  const int q = lane & 3;
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const float4* p = reinterpret_cast<const float4*>(x + (size_t)(tok + min(16 * half + 8 * k + (lane >> 2), live - 1)) * ldx + min(32 * c + 8 * q, cols - 8));
    v[k][0] = __ldcg(p); v[k][1] = __ldcg(p + 1);
  }
}
// epi_stream with such rows (x: the tile's columns of them).
template <bool MIRROR>
__device__ __forceinline__ void epi_resid(const EpiPlace& e, const GemmArgs& g, const float* x, ResidRows& r, float* out32, unsigned short* out16, float* ssq, int ft) {
  const int q = e.lane & 3;
#pragma unroll 1
  for (int h = 0; h < 2 && 16 * h < e.live; ++h) {
    const int row = 16 * h + (e.lane >> 2);
    const uint32_t tmem = e.tmem + ((uint32_t)(16 * h) << 16);
    float* pa = out32 + (size_t)(e.tok + row) * g.ldo32 + e.r0 + 8 * q;
    float* pb = pa + (size_t)8 * g.ldo32;
    unsigned short* ha = MIRROR ? out16 + (size_t)(e.tok + row) * g.ldo16 + e.r0 + 8 * q : nullptr;
    unsigned short* hb = MIRROR ? ha + (size_t)8 * g.ldo16 : nullptr;
    float sa = 0.f, sb = 0.f;
    uint32_t nx[EPI];
#pragma unroll 1
    for (int c2 = 0; c2 < GEMM_BM / 32; c2 += 2) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int c = c2 + i;
        float v[EPI];
        tmem_ld_frag(tmem + 32u * (uint32_t)c, nx);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < EPI; ++j) v[j] = __uint_as_float(nx[j]);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const float4 lo = r.v[i][k][0], hi = r.v[i][k][1];
          float* u = v + 2 * k;
          u[0] += lo.x; u[1] += lo.y; u[4] += lo.z; u[5] += lo.w;
          u[8] += hi.x; u[9] += hi.y; u[12] += hi.z; u[13] += hi.w;
        }
        if (c2 == 0 || 16 * (h + 1) < e.live) resid_load(x, g.ldx, e.tok, e.live, c2 == 0 ? h : h + 1, e.lane, e.cols, c2 == 0 ? c + 2 : c - 2, r.v[i]);
        const bool fok = 32 * c + 8 * q < e.cols;
        if (MIRROR && fok) {
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            sa = fmaf(v[4 * b], v[4 * b], sa); sa = fmaf(v[4 * b + 1], v[4 * b + 1], sa);
            sb = fmaf(v[4 * b + 2], v[4 * b + 2], sb); sb = fmaf(v[4 * b + 3], v[4 * b + 3], sb);
          }
        }
        if (fok && row < e.live) { st_row8(pa + 32 * c, v); if (MIRROR) st_row8(ha + 32 * c, v); }
        if (fok && row + 8 < e.live) { st_row8(pb + 32 * c, v + 2); if (MIRROR) st_row8(hb + 32 * c, v + 2); }
      }
    }
    tmem_ld_wait();
    if (MIRROR && ssq) {
      sa += __shfl_xor_sync(0xffffffffu, sa, 1); sb += __shfl_xor_sync(0xffffffffu, sb, 1);
      sa += __shfl_xor_sync(0xffffffffu, sa, 2); sb += __shfl_xor_sync(0xffffffffu, sb, 2);
      float* sp = ssq + (size_t)(e.tok + row) * g.ss_out_ld + ft;
      if (q == 0 && row < e.live) sp[0] = sa;
      if (q == 0 && row + 8 < e.live) sp[(size_t)8 * g.ss_out_ld] = sb;
    }
  }
}
// Rows of V^T: a token per lane, so that a warp writes 32 consecutive tokens of a feature.
__device__ __forceinline__ void epi_vt(const EpiPlace& e, const GemmArgs& g, unsigned short* outT, int split) {
  unsigned short* const base = outT + e.tok + e.lane;
  const size_t ld = (size_t)g.ldoT;
  epi_chunks(e.tmem, split, e.cols, e.rs, [&](int c0, float* v) {
    unsigned short* op = base + (size_t)(e.r0 + (c0 & ~31) + ((c0 & 16) >> 2) - g.t_col0) * ld;
    if (e.lane < e.live) {
#pragma unroll
      for (int j = 0; j < EPI; ++j) op[(size_t)perm_feature(j) * ld] = f32_to_bf16_bits(v[j]);
    }
  });
}

// Anything else -- solver coefficients, norms with addends, odd widths and offsets: a token per lane, element by element.
__device__ __forceinline__ void epi_general(const TileCtx& c, const GemmArgs& g, const EpiPlace& e, int ft) {
  const GemmPtrs ptrs = gemm_ptrs(c, g);
  const int N = g.dual ? 2 * g.N : g.N, act = g.act;
  const int cols = g.perm ? (e.cols + 31) & ~31 : (e.cols + 1) & ~1;     // a reordered last group spreads over all its columns
  const bool live = e.lane < e.live;
  const size_t tok = (size_t)(e.tok + min(e.lane, e.live - 1));
  float* const ssq = resolve<float>(c, g.ss_out);
  float sq = 0.f;
#pragma unroll 1
  for (int c0 = 0; c0 < cols; c0 += 2) {                 // (rolled: few nodes come here, and the code would crowd the others out)
    const int f = e.r0 + (g.perm ? (c0 & ~31) + perm_feature(c0 & 31) : c0);         // a pair of features
    uint32_t acc[2];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=r"(acc[0]), "=r"(acc[1]) : "r"(e.tmem + (uint32_t)c0) : "memory");
    tmem_ld_wait();
    float x0 = __uint_as_float(acc[0]) * e.rs, x1 = __uint_as_float(acc[1]) * e.rs;
    if (g.dual) {
      if (live && f < N) ptrs.out16[tok * g.ldo16 + f / 2] = f32_to_bf16_bits(apply_act(act, x0) * x1 * g.c_acc);
      continue;
    }
    if (f < g.rope_cols) {
      const float2 cs = __ldg(reinterpret_cast<const float2*>(resolve<const float>(c, g.rope_tab) + tok * g.rope_hd + f % g.rope_hd));
      const float r = fmaf(x0, cs.x, -x1 * cs.y);
      x1 = fmaf(x1, cs.x, x0 * cs.y);
      x0 = r;
    }
    if (f >= N) continue;
    const int f1 = min(f + 1, N - 1);                     // (the pair's loads go out together)
    const bool two = f + 1 < N;
    if (ptrs.bias) { x0 += __ldg(ptrs.bias + f); x1 += __ldg(ptrs.bias + f1); }
    x0 = apply_act(act, x0) * g.c_acc; x1 = apply_act(act, x1) * g.c_acc;
    auto add = [&](const float* p, size_t ld, float scale) {
      const float a0 = ld_act(p + tok * ld + f), a1 = ld_act(p + tok * ld + f1);
      x0 = fmaf(scale, a0, x0); x1 = fmaf(scale, a1, x1);
    };
    if (ptrs.X) add(ptrs.X, g.ldx, g.c_x);
    if (ptrs.vec) add(ptrs.vec, 0, 1.0f);
    if (ptrs.tab) add(ptrs.tab, g.ldtab, 1.0f);
    if (ptrs.tab2) add(ptrs.tab2, g.ldtab2, 1.0f);
    sq = fmaf(x0, x0, sq);
    if (two) sq = fmaf(x1, x1, sq);
    if (!live) continue;
    const bool t0_ = ptrs.outT && f >= g.t_col0, t1_ = ptrs.outT && f1 >= g.t_col0;
    if (t0_) ptrs.outT[(size_t)(f - g.t_col0) * g.ldoT + tok] = f32_to_bf16_bits(x0);
    if (two && t1_) ptrs.outT[(size_t)(f1 - g.t_col0) * g.ldoT + tok] = f32_to_bf16_bits(x1);
    if (ptrs.out32 && !t0_) ptrs.out32[tok * g.ldo32 + f] = x0;
    if (ptrs.out32 && !t1_ && two) ptrs.out32[tok * g.ldo32 + f1] = x1;
    if (ptrs.out16 && !t0_) ptrs.out16[tok * g.ldo16 + f] = f32_to_bf16_bits(x0);
    if (ptrs.out16 && !t1_ && two) ptrs.out16[tok * g.ldo16 + f1] = f32_to_bf16_bits(x1);
  }
  if (ssq && live) ssq[tok * g.ss_out_ld + ft] = sq;
}

// This warp's tokens of the tile: `live` of them from `tok` on.  r0: the tile's first weight row, rs: row scale of the token
// in this lane.
__device__ __forceinline__ void gemm_epilogue(const TileCtx& c, const GemmArgs& g, uint32_t tmem, int tok, int live, int lane, int r0, float rs, int ft, ResidRows& resid) {
  EpiPlace e;
  e.tmem = tmem; e.tok = tok; e.live = live; e.lane = lane; e.r0 = r0; e.rs = rs;
  e.cols = min(GEMM_BM, (g.dual ? 2 * g.N : g.N) - r0);
  if (!g.fast) { epi_general(c, g, e, ft); return; }
  unsigned short* const out16 = resolve<unsigned short>(c, g.out16);
  if (g.dual) {
    if (g.act == ACT_SILU) epi_gated<ACT_SILU>(e, g, out16);
    else if (g.act == ACT_GELU) epi_gated<ACT_GELU>(e, g, out16);
    else epi_gated<ACT_NONE>(e, g, out16);
  } else if (g.out32 != 0) {
    float* const out32 = resolve<float>(c, g.out32);
    if (g.resid) {
      const float* const x = resolve<const float>(c, g.X) + r0;
      if (out16) epi_resid<true>(e, g, x, resid, out32, out16, resolve<float>(c, g.ss_out), ft);
      else epi_resid<false>(e, g, x, resid, out32, nullptr, nullptr, ft);
    } else if (g.fast == 2) {
      if (out16) epi_stream<true, true>(c, e, g, out32, out16, nullptr, ft);
      else epi_stream<false, true>(c, e, g, out32, nullptr, nullptr, ft);
    } else if (out16) epi_stream<true, false>(c, e, g, out32, out16, resolve<float>(c, g.ss_out), ft);
    else epi_stream<false, false>(c, e, g, out32, nullptr, nullptr, ft);
  } else {
    const int all = e.cols;
    if (g.outT != 0) e.cols = max(0, min(all, g.t_col0 - r0));              // columns from here on are V features
    if (e.cols > 0) {
      if (g.act == ACT_GELU) epi_bf16<ACT_GELU, false>(e, g, out16, nullptr);
      else if (g.rope_cols > 0) epi_bf16<ACT_NONE, true>(e, g, out16, resolve<const float>(c, g.rope_tab));
      else epi_bf16<ACT_NONE, false>(e, g, out16, nullptr);
    }
    if (e.cols < all) {
      const int split = e.cols;
      e.cols = all;
      epi_vt(e, g, resolve<unsigned short>(c, g.outT), split);
    }
  }
}

// Biases, broadcast vectors and tables of the warp's tokens (`live` from `tok` on) into the accumulators (fragment layout; columns
// past the last feature get zero).  The tensor core then sums from them, in fp32 but without the rounding that an addition behind
// the product has; residual rows are added behind it (epi_resid).  Two fragments at a time, all loads of an addend before the first
// use: 32 tokens x 32 columns, or with up to 64 tokens in the tile (16 per warp) 16 x 64.
__device__ __forceinline__ void preload_rows(const TileCtx& c, const GemmArgs& g, uint32_t tmem, int tok, int live, int tpw, int lane, int r0) {
  const int q = lane & 3, cols = min(GEMM_BM, g.N - r0), under = g.under;
  const int dcol = tpw == 16 ? 32 : 0;                 // second fragment: that many columns on, or (0) 16 tokens on
  int row[4];                                          // (lanes past the last token read that one)
#pragma unroll
  for (int k = 0; k < 4; ++k) row[k] = tok + min(((8 * k) & (tpw - 1)) + (lane >> 2), live - 1);
#pragma unroll 1
  for (int c0 = 0; c0 < cols; c0 += 32 + dcol) {
    float v[4][8];
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int j = 0; j < 8; ++j) v[k][j] = 0.f;
    const int f = r0 + c0 + 8 * q;
    if (c0 + 8 * q < cols) {
      const bool in2 = c0 + dcol + 8 * q < cols;
      const int f2 = in2 ? f + dcol : f;
      auto add = [&](Ref ref, int ld) {                // ld 0: the same row for every token
        const float* p = resolve<const float>(c, ref);
        float4 t[4][2];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float4* x = reinterpret_cast<const float4*>(p + (size_t)row[k] * ld + (k < 2 ? f : f2));
          t[k][0] = __ldcg(x); t[k][1] = __ldcg(x + 1);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          v[k][0] += t[k][0].x; v[k][1] += t[k][0].y; v[k][2] += t[k][0].z; v[k][3] += t[k][0].w;
          v[k][4] += t[k][1].x; v[k][5] += t[k][1].y; v[k][6] += t[k][1].z; v[k][7] += t[k][1].w;
        }
      };
#pragma unroll 1
      for (int m = under; m != 0; m &= m - 1) {
        const int which = m & -m;
        add(which == 1 ? g.bias : (which == 2 ? g.vec : (which == 8 ? g.tab : g.tab2)), which == 8 ? g.ldtab : (which == 16 ? g.ldtab2 : 0));
      }
      if (!in2) {
#pragma unroll
        for (int j = 0; j < 8; ++j) v[2][j] = v[3][j] = 0.f;
      }
    }
    const uint32_t t0 = tmem + (uint32_t)c0, dt = dcol ? 32u : (16u << 16);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float* a = v[2 * h];
      const float* b = v[2 * h + 1];
      const float w[EPI] = {a[0], a[1], b[0], b[1], a[2], a[3], b[2], b[3], a[4], a[5], b[4], b[5], a[6], a[7], b[6], b[7]};
      tmem_st_frag(t0 + h * dt, w);
    }
  }
  tmem_st_wait();
}

// The producer of a node's first token tile asks the L2 for weights this many k-blocks ahead: they come from HBM once per
// frame, and two to four stages do not cover that latency.
constexpr int GEMM_AHEAD = 6;
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

  // Tokens per warp.  A tile of at most 64 tokens uses M = 64, whose rows lie 16 to each warp's 32 TMEM lanes: all four warps
  // share its addends and its epilogue, where M = 128 left them to the first two (50-token head tiles: 6.5k cycles after the
  // main loop -> 4.5k; single frame 12.63 -> 12.08 ms, 32 streams x 2 cameras 191.7 -> 186.0 ms).
  const int tpw = bt <= 64 ? 16 : 32;
  const bool warp_live = warp * tpw < nt;
  const uint32_t my_tmem = c.tmem + ((uint32_t)(warp * 32) << 16);
  // Biases and tables go into the accumulators before the first MMA, beside the round trip of the first operand stages; residual
  // rows are asked for now and added in the epilogue.
  const bool under = g.under != 0;
  if (under) {
    if (warp_live) preload_rows(c, g, my_tmem, t0 + tpw * warp, min(tpw, nt - tpw * warp), tpw, lane, r0);
    tc_fence_before();
  }
  ResidRows resid;                                     // (set in every case: left open where there are none, 120 more bytes are spilled)
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int k = 0; k < 2; ++k) resid.v[j][k][0] = resid.v[j][k][1] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (g.resid && warp_live) {
    const float* const x = resolve<const float>(c, g.X) + r0;
#pragma unroll
    for (int j = 0; j < 2; ++j) resid_load(x, g.ldx, t0 + tpw * warp, min(tpw, nt - tpw * warp), 0, lane, min(GEMM_BM, g.N - r0), j, resid.v[j]);
  }
  // Folded RMSNorm: the partial sums of squares of this lane's token are requested now and added after the main loop, in a
  // fixed order (streams wider than 1024: the rest at once).
  float part[8], ssq = 0.f;
  const bool scaled = g.rs_d > 0 && warp_live;
#pragma unroll
  for (int j = 0; j < 8; ++j) part[j] = 0.f;
  if (scaled) {
    const float* sp = resolve<const float>(c, g.ss_in) + (size_t)(t0 + min(tpw * warp + lane, nt - 1)) * g.ss_nft;
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (j < g.ss_nft) part[j] = ld_act(sp + j);
#pragma unroll 4
    for (int j = 8; j < g.ss_nft; ++j) ssq += ld_act(sp + j);
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
        if (t0 == 0 && !c.wait_word && kb + GEMM_AHEAD < nkb) tma_prefetch_2d(wmap, (kb + GEMM_AHEAD) * GEMM_BK, r0);
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
    const uint32_t idesc = umma_idesc_bf16(GEMM_BM, bt <= 64 ? 64 : 128);
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
  float rs = 1.0f;
  if (scaled) {
#pragma unroll
    for (int j = 0; j < 8; ++j) ssq += part[j];
    rs = 1.0f / sqrtf(ssq / (float)g.rs_d + 1e-6f);
  }
  if (ready && warp_live) gemm_epilogue(c, g, my_tmem, t0 + tpw * warp, min(tpw, nt - tpw * warp), lane, r0, rs, ft, resid);
  tc_fence_before();
  worker_sync(c);
  if (!(c.slot && c.slot->primed) && worker_tid() <= 2 * S) mbar_inval(bar0 + 8u * worker_tid());
}

}  // namespace vla
