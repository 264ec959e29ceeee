// Tile bodies other than the GEMM (see gemm_tc.cuh): RMSNorm, fused attention, and the
// elementwise / gather tiles, plus the dispatch switch.
#pragma once
#include "attn_tc.cuh"
#include "gemm_tc.cuh"
#include "tiles_common.cuh"

namespace vla {

// ------------------------------------------------------------------ RMSNorm / LayerNorm tile (one warp per row)
// The row is read once per pass (mean of a LayerNorm, sum of squares, output) in steps of four float4 per lane, all in
// flight together; the later passes find it in L2.  Rolled loops instead of a row held in registers: the tile is a small
// part of any workload, and its unrolled code (55 KB) pushed the GEMM and attention bodies out of the instruction cache.
__device__ __forceinline__ void tile_rmsnorm(const TileCtx& c, const NormArgs& a, int tile) {
  const int warp = worker_tid() >> 5, lane = worker_tid() & 31;
  const float4* g4 = reinterpret_cast<const float4*>(resolve<const float>(c, a.g));
  const float4* b4 = reinterpret_cast<const float4*>(resolve<const float>(c, a.beta));
  const float4* m4 = reinterpret_cast<const float4*>(resolve<const float>(c, a.mod));
  const int d4 = a.d >> 2;                      // widths are multiples of 4
  const int row_hi = min((tile + 1) * a.rows_per_tile, a.M);
#pragma unroll 1
  for (int r = tile * a.rows_per_tile + warp; r < row_hi; r += WORKER_THREADS / 32) {
    const float4* x4 = reinterpret_cast<const float4*>(resolve<const float>(c, a.x) + (size_t)r * a.ldx);
    float mu = 0.f, ss = 0.f;
#pragma unroll 1
    for (int pass = a.ln ? 0 : 1; pass < 2; ++pass) {
      float acc = 0.f;
#pragma unroll 1
      for (int i0 = lane; i0 < d4; i0 += 128) {
        float4 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = __ldcg(x4 + min(i0 + 32 * k, d4 - 1));
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (i0 + 32 * k >= d4) continue;
          const float x = v[k].x - mu, y = v[k].y - mu, z = v[k].z - mu, w = v[k].w - mu;
          acc += pass == 0 ? (x + y) + (z + w) : fmaf(x, x, y * y) + fmaf(z, z, w * w);
        }
      }
      acc = warp_sum(acc) / (float)a.d;
      if (pass == 0) mu = acc; else ss = acc;
    }
    const float inv = 1.0f / sqrtf(ss + 1e-6f);
    size_t orow = r, ocol0 = 0;
    if (a.shuffle > 1) {
      const int y = r / a.grid, xx = r % a.grid, s = a.shuffle;
      orow = (size_t)(y / s) * (a.grid / s) + (xx / s);
      ocol0 = (size_t)((y % s) * s + (xx % s)) * a.d;
    }
    uint2* o2 = reinterpret_cast<uint2*>(resolve<unsigned short>(c, a.out) + orow * a.ldo + ocol0);
#pragma unroll 1
    for (int i0 = lane; i0 < d4; i0 += 64) {
      float4 v[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int i = min(i0 + 32 * k, d4 - 1);
        const float4 t = __ldcg(x4 + i), gg = __ldg(g4 + i);
        v[k] = make_float4((t.x - mu) * inv * gg.x, (t.y - mu) * inv * gg.y, (t.z - mu) * inv * gg.z, (t.w - mu) * inv * gg.w);
        if (b4) {
          const float4 bb = __ldg(b4 + i);
          v[k].x += bb.x; v[k].y += bb.y; v[k].z += bb.z; v[k].w += bb.w;
        }
        if (m4) {
          const float4 ga = __ldg(m4 + i), be = __ldg(m4 + d4 + i);
          v[k].x = fmaf(v[k].x, 1.0f + ga.x, be.x); v[k].y = fmaf(v[k].y, 1.0f + ga.y, be.y);
          v[k].z = fmaf(v[k].z, 1.0f + ga.z, be.z); v[k].w = fmaf(v[k].w, 1.0f + ga.w, be.w);
        }
      }
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        if (i0 + 32 * k >= d4) continue;
        __nv_bfloat162 lo = __floats2bfloat162_rn(v[k].x, v[k].y), hi = __floats2bfloat162_rn(v[k].z, v[k].w);
        o2[i0 + 32 * k] = make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
      }
    }
  }
}

// ------------------------------------------------------------------ elementwise tiles
// One warp per patch.  Each lane gathers eight pixel pairs before it stores any (the loads' latency, not bandwidth, bounds
// a tile); sides and buffers that do not allow 8-byte pairs go pixel by pixel.
__device__ void tile_patchify(const TileCtx& c, const PatchArgs& a_in, int tile) {
  const PatchArgs a = a_in;
  const int warp = worker_tid() >> 5, lane = worker_tid() & 31;
  const float* img = resolve<const float>(c, a.img);
  unsigned short* obase = resolve<unsigned short>(c, a.out);
  const int P = a.patch, pk = 3 * P * P;
  const bool pairs = P % 2 == 0 && (reinterpret_cast<uintptr_t>(img) & 7) == 0;
#pragma unroll 1
  for (int rr = warp; rr < a.rows_per_tile; rr += WORKER_THREADS / 32) {
    const int p = tile * a.rows_per_tile + rr;
    if (p >= a.grid * a.grid) break;
    unsigned short* out = obase + (size_t)p * a.ldo;
    const float* corner = img + (size_t)(p / a.grid * P) * a.img_side + p % a.grid * P;
    if (pairs) {
#pragma unroll 1
      for (int e0 = 2 * lane; e0 < pk; e0 += 64 * 8) {
        float2 v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int e = e0 + 64 * j, ch = e / (P * P), rem = e % (P * P);
          if (e < pk) v[j] = __ldcg(reinterpret_cast<const float2*>(corner + ((size_t)ch * a.img_side + rem / P) * a.img_side + rem % P));
        }
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (e0 + 64 * j < pk) *reinterpret_cast<__nv_bfloat162*>(out + e0 + 64 * j) = __floats2bfloat162_rn(v[j].x, v[j].y);
      }
    } else {
#pragma unroll 1
      for (int e = lane; e < pk; e += 32) {
        const int ch = e / (P * P), rem = e % (P * P);
        out[e] = f32_to_bf16_bits(ld_act(corner + ((size_t)ch * a.img_side + rem / P) * a.img_side + rem % P));
      }
    }
  }
}

// A warp's unit is one row x one 128-column block (four columns per lane, all loads in flight together), so that even a
// single row of the residual stream spreads over the tile's warps.
__device__ void tile_embed(const TileCtx& c, const EmbedArgs& a_in, int tile) {
  const EmbedArgs a = a_in;
  const int warp = worker_tid() >> 5, lane = worker_tid() & 31;
  const int* ids = resolve<const int>(c, a.ids);
  const unsigned short* table = resolve<const unsigned short>(c, a.table);
  const float* pos = resolve<const float>(c, a.pos);
  float* obase = resolve<float>(c, a.out);
  unsigned short* o16 = resolve<unsigned short>(c, a.out16);
  float* ss = resolve<float>(c, a.ss_out);
  const int nb = (a.d + 127) / 128, r0 = tile * a.rows_per_tile, nr = min(a.rows_per_tile, a.n - r0);
#pragma unroll 1
  for (int u = warp; u < nr * nb; u += WORKER_THREADS / 32) {
    const int r = r0 + u / nb, b0 = u % nb * 128;
    const int id = min(max(ld_act(ids + r), 0), a.vocab - 1);
    float v[4], sq = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int i = b0 + lane + 32 * j;
      v[j] = i < a.d ? bf16_bits_to_f32(__ldg(table + (size_t)id * a.ldt + i)) : 0.f;
      if (pos && i < a.d) v[j] += __ldg(pos + (size_t)r * a.d + i);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int i = b0 + lane + 32 * j;
      if (i < a.d) {
        obase[(size_t)r * a.ldo + i] = v[j];
        if (o16) o16[(size_t)r * a.ldo16 + i] = f32_to_bf16_bits(v[j]);
      }
      sq = fmaf(v[j], v[j], sq);
    }
    sq = warp_sum(sq);
    if (ss && lane == 0) ss[(size_t)r * a.ss_ld + (b0 >> 7)] = sq;
  }
}

__device__ void tile_addrows(const TileCtx& c, const AddRowsArgs& a_in, int) {
  const AddRowsArgs a = a_in;
  const int warp = worker_tid() >> 5, lane = worker_tid() & 31;
  const float* in = resolve<const float>(c, a.in);
  const float* vec = resolve<const float>(c, a.vec);
  const float* tab = resolve<const float>(c, a.tab);
  float* out = resolve<float>(c, a.out);
  unsigned short* out16 = resolve<unsigned short>(c, a.out16);
  float* ss = resolve<float>(c, a.ss_out);
  const int nb = (a.N + 127) / 128;
#pragma unroll 1
  for (int u = warp; u < a.M * nb; u += WORKER_THREADS / 32) {     // (row, 128 columns) per warp, as in tile_embed
    const int r = u / nb, b0 = u % nb * 128;
    float v[4], sq = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int col = b0 + lane + 32 * j;
      v[j] = 0.f;
      if (col < a.N) {
        v[j] = ld_act(in + (size_t)r * a.ldi + col);
        if (vec) v[j] += __ldg(vec + col);
        if (tab) v[j] += __ldg(tab + (size_t)r * a.ldt + col);
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int col = b0 + lane + 32 * j;
      if (col < a.N) {
        if (out) out[(size_t)r * a.ldo + col] = v[j];
        if (out16) out16[(size_t)r * a.ldo16 + col] = f32_to_bf16_bits(v[j]);
      }
      sq = fmaf(v[j], v[j], sq);
    }
    if (ss) {
      sq = warp_sum(sq);
      if (lane == 0) ss[(size_t)r * a.ss_ld + (b0 >> 7)] = sq;
    }
  }
}

__device__ void tile_timeemb(const TileCtx& c, const TimeEmbArgs& a, int) {
  const float* args = resolve<const float>(c, a.args);
  unsigned short* out = resolve<unsigned short>(c, a.out);
  const int half = a.width / 2;
  const float lnb = 9.210340371976184f;
#pragma unroll 1
  for (int e = worker_tid(); e < a.M * half; e += WORKER_THREADS) {
    int m = e / half, i = e % half;
    float om = expf(-lnb * (float)i / (float)half);
    float sn, cs;
    sincosf(args[m] * om, &sn, &cs);
    out[(size_t)m * a.ldo + i] = f32_to_bf16_bits(sn);
    out[(size_t)m * a.ldo + half + i] = f32_to_bf16_bits(cs);
  }
}

// Copies the chunk to the host-visible ring, then publishes the frame id (system-scope fence between).  After a wait that
// ran out nothing is published any more: a tile of this very frame may have gone on with operands that were not there (it set
// the error word before its end released anything, so it shows here).
__device__ void tile_emit(const TileCtx& c, const EmitArgs& a, float* chunk_host, DoneRec* done, uint64_t frame, bool last) {
  const float* x = resolve<const float>(c, a.x);
  chunk_host += a.chunk_off;
#pragma unroll 1
  for (int e = worker_tid(); e < a.H * a.A; e += WORKER_THREADS) {
    int r = e / a.A, col = e % a.A;
    chunk_host[e] = ld_act(x + (size_t)r * a.ldx + col);
  }
  __threadfence_system();
  worker_sync(c);
  if (worker_tid() == 0 && last && *reinterpret_cast<volatile unsigned*>(c.error) == 0u) {
    done->frame_plus1 = frame + 1;
    __threadfence_system();
  }
}

}  // namespace vla

#include "run_tile.cuh"
