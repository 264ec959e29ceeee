// Test hooks: the engine's GEMM and attention tile bodies on caller-owned device tensors, operator by operator.
//
// A hook puts together one node as program.cc would, uploads it with its tensor maps and runs it as the stream modes run any
// node (vla_node_kernel, one block per tile).  It allocates, waits and frees: nothing here is meant to be fast.
#pragma once
#include "ops_api.cuh"

namespace vla {

struct TileHookBlock {            // what the node kernel reads from device memory, in one allocation
  alignas(64) CUtensorMap maps[5];
  NodeDesc node;
  Control control;
  unsigned error_mirror;
};

inline int run_tile_hook(TileHookBlock& h, int n_maps) {
  int dev = 0, optin = 0;
  cudaFuncAttributes fa;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaFuncGetAttributes(&fa, vla_node_kernel) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
      cudaFuncSetAttribute(vla_node_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes) != cudaSuccess)
    return VLA_ERR_CUDA;
  TileHookBlock* d = nullptr;
  if (cudaMalloc(&d, sizeof h) != cudaSuccess) return VLA_ERR_NOMEM;
  DeviceCtx ctx;
  memset(&ctx, 0, sizeof ctx);    // (no arena: the Refs of a hook are absolute device addresses)
  ctx.nodes = &d->node; ctx.control = &d->control; ctx.error_host = &d->error_mirror;
  ctx.tmaps = d->maps; ctx.n_weight_tmaps = h.node.op == OP_GEMM ? 1 : 0; ctx.n_act_tmaps = n_maps - ctx.n_weight_tmaps;
  ctx.wait_limit_ns = op_fault().wait_limit_ns; ctx.drop_loads = op_fault().drop_loads;
  cudaError_t e = cudaDeviceSynchronize();          // the caller's tensors are complete
  if (e == cudaSuccess) e = cudaMemcpy(d, &h, sizeof h, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    vla_node_kernel<<<h.node.n_tiles, WORKER_THREADS, h.node.smem_bytes>>>(ctx, ctx.nodes, 0, -1);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e == cudaSuccess) e = cudaMemcpy(&h, d, sizeof h, cudaMemcpyDeviceToHost);
  cudaFree(d);
  if (e != cudaSuccess) return VLA_ERR_CUDA;
  return h.control.error == 0u && h.error_mirror == 0u ? VLA_OK : VLA_ERR_TIMEOUT;
}

inline bool hook_aligned(const void* p, uintptr_t bytes) { return (reinterpret_cast<uintptr_t>(p) & (bytes - 1)) == 0; }

// The GEMM node of a hook; `bias` .. `tab2` and `ss` with the straight epilogue only.
struct TileLinear {
  const void *a, *w;
  const float *x, *bias, *vec, *tab, *tab2;
  float* out32;
  void* out16;
  float* ss;
  int m, n, k, act, gated, fast;
};
inline int run_tile_linear(const TileLinear& t) {
  const bool under = t.bias || t.vec || t.tab || t.tab2, adds = t.x || t.vec || t.tab || t.tab2;
  if (!t.a || !t.w || (!t.out32 && !t.out16) || t.m < 1 || t.n < 1 || t.k < 8 || t.k % 8 || t.act < 0 || t.act > 2) return VLA_ERR_INVALID;
  if (t.gated && (t.x || under || t.out32)) return VLA_ERR_INVALID;
  if ((under || t.ss) && !t.fast) return VLA_ERR_INVALID;
  if (t.ss && (!t.out32 || !t.out16)) return VLA_ERR_INVALID;
  // what the straight epilogue takes (see the rule in program.cc): whole vectors, and no activation behind an addend or in fp32 rows
  if (t.fast && (t.n % (t.gated ? 4 : 8) || !hook_aligned(t.x, 16) || !hook_aligned(t.bias, 16) || !hook_aligned(t.vec, 16) || !hook_aligned(t.tab, 16) ||
                 !hook_aligned(t.tab2, 16) || !hook_aligned(t.out32, 32) || !hook_aligned(t.out16, 16) ||
                 (!t.gated && t.act != ACT_NONE && (t.act != ACT_GELU || t.out32 || adds)) || (t.x && !t.out32)))
    return VLA_ERR_INVALID;
  TileHookBlock h;
  memset(&h, 0, sizeof h);
  NodeDesc& nd = h.node;
  GemmArgs& g = nd.u.gemm;
  nd.op = OP_GEMM;
  g.M = t.m; g.N = t.n; g.Kp = (int)op_pad(t.k, GEMM_BK);
  g.X = reinterpret_cast<Ref>(t.x); g.ldx = t.n;
  g.bias = reinterpret_cast<Ref>(t.bias); g.vec = reinterpret_cast<Ref>(t.vec);
  g.tab = reinterpret_cast<Ref>(t.tab); g.ldtab = t.n;
  g.tab2 = reinterpret_cast<Ref>(t.tab2); g.ldtab2 = t.n;
  g.out32 = reinterpret_cast<Ref>(t.out32); g.ldo32 = t.n;
  g.out16 = reinterpret_cast<Ref>(t.out16); g.ldo16 = t.n;
  g.act = t.act; g.dual = t.gated ? 1 : 0; g.c_acc = 1.f; g.c_x = 1.f;
  g.tiles_t = (t.m + GEMM_MAX_BT - 1) / GEMM_MAX_BT;
  g.bt = (int)op_pad((t.m + g.tiles_t - 1) / g.tiles_t, 16);
  g.stages = gemm_stages(g.bt, g.Kp);
  g.fast = g.perm = t.fast ? 1 : 0;
  g.resid = t.fast && t.x ? 1 : 0;
  g.under = (t.bias ? 1 : 0) | (t.vec ? 2 : 0) | (t.tab ? 8 : 0) | (t.tab2 ? 16 : 0);
  nd.smem_bytes = gemm_smem_bytes(g.bt, g.stages);
  nd.tmem_cols = GEMM_BM;
  const int rows = t.gated ? 2 * t.n : t.n, per_tile = t.gated ? GEMM_BM / 2 : GEMM_BM, tiles_n = (t.n + per_tile - 1) / per_tile;
  g.ss_out = reinterpret_cast<Ref>(t.ss); g.ss_out_ld = tiles_n;
  nd.n_tiles = tiles_n * g.tiles_t;
  if (!op_encode(h.maps, t.w, t.fast ? op_pad(rows, 32) : rows, t.k, t.k, GEMM_BM) || !op_encode(h.maps + 1, t.a, t.m, t.k, t.k, g.bt)) return VLA_ERR_CUDA;
  return run_tile_hook(h, 2);
}

}  // namespace vla

extern "C" {

int vla_debug_tile_linear(const void* a, const void* w, const float* x, float* out32, void* out16, int32_t m, int32_t n, int32_t k,
                          int32_t act, int32_t gated, int32_t fast) {
  return vla::run_tile_linear({a, w, x, nullptr, nullptr, nullptr, nullptr, out32, out16, nullptr, m, n, k, act, gated, fast});
}

int vla_debug_tile_addends(const void* a, const void* w, const float* x, const float* bias, const float* vec, const float* tab,
                           const float* tab_b, float* out32, void* out16, float* ss, int32_t m, int32_t n, int32_t k, int32_t act) {
  return vla::run_tile_linear({a, w, x, bias, vec, tab, tab_b, out32, out16, ss, m, n, k, act, 0, 1});
}

int vla_debug_tile_attention(const void* q, const void* k0, const void* vt0, const void* k1, const void* vt1, void* out, int32_t tq,
                             int32_t t0, int32_t t1, int32_t hq, int32_t hkv, int32_t hd, int32_t causal, int32_t sfx) {
  using namespace vla;
  if (!q || !k0 || !vt0 || !out || t1 < 0 || (t1 > 0 && (!k1 || !vt1)) || !op_attention_shape_ok(tq, t0, hq, hkv, hd)) return VLA_ERR_INVALID;
  if ((causal && (tq != t0 || t1)) || sfx < 0 || sfx > t1 || !hook_aligned(out, 16)) return VLA_ERR_INVALID;
  TileHookBlock h;
  memset(&h, 0, sizeof h);
  NodeDesc& nd = h.node;
  AttnArgs& a = nd.u.attn;
  nd.op = OP_ATTN;
  a.out = reinterpret_cast<Ref>(out); a.ldo = hq * hd;
  a.tq = tq; a.t0 = t0; a.t1 = t1;
  a.hq = hq; a.hkv = hkv; a.hd = a.hs = hd; a.causal = causal ? 1 : 0; a.sfx = sfx;
  a.bn = ATTN_BN;
  a.q_blocks = (tq + ATTN_BQ - 1) / ATTN_BQ;
  a.hpt = attn_fold(tq, hq, hkv, &a.rph);
  a.scale_log2e = 1.4426950408889634f / sqrtf((float)hd);
  a.k0map = 1; a.v0map = 2; a.k1map = 3; a.v1map = 4;
  nd.smem_bytes = attn_smem_bytes(hd);
  nd.tmem_cols = (int)op_pad(attn_tmem_cols(hd), TMEM_UNIT);
  nd.n_tiles = a.hpt > 1 ? hkv * ((hq / hkv + a.hpt - 1) / a.hpt) : hq * a.q_blocks;
  CUtensorMap* m = h.maps;
  const int64_t kv = (int64_t)hkv * hd;
  if (!op_encode(m, q, tq, (int64_t)hq * hd, (int64_t)hq * hd, a.hpt > 1 ? a.rph : ATTN_BQ) || !op_encode(m + 1, k0, t0, kv, kv, ATTN_BN) ||
      !op_encode(m + 2, vt0, kv, t0, op_pad(t0, 64), hd))
    return VLA_ERR_CUDA;
  if (t1 > 0 && (!op_encode(m + 3, k1, t1, kv, kv, ATTN_BN) || !op_encode(m + 4, vt1, kv, t1, op_pad(t1, 64), hd))) return VLA_ERR_CUDA;
  return run_tile_hook(h, t1 > 0 ? 5 : 3);
}

}  // extern "C"
