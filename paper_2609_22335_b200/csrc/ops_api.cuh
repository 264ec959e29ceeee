// Stand-alone operator entry points: a linear layer and fused attention on caller-owned device tensors, for callers that
// want the kernels without the frame pipeline.  They are kernels of their own (op_linear.cuh, op_attention.cuh); the engine's
// tile bodies are reached one by one through tile_hooks.cuh.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include "../../include/vla.h"
#include "dispatch.cuh"
#include "per_device.h"

namespace vla {

struct OpMaps {
  alignas(64) CUtensorMap m[4];
};

typedef CUresult (*OpEncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                               const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                               CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline OpEncodeFn op_encoder() {
  static OpEncodeFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<OpEncodeFn>(p);
  }
  return fn;
}

// 2-D bf16 row-major tensor, 64-column boxes, 128-byte swizzle, zero fill outside.
inline bool op_encode(CUtensorMap* out, const void* base, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
  OpEncodeFn enc = op_encoder();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {(cuuint32_t)GEMM_BK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return enc(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Bound of the operators' device-side waits, and the test hook that makes one run out (vla_debug_op_fault).
struct OpFault {
  unsigned long long wait_limit_ns;
  int drop_loads;
};
inline OpFault& op_fault() {
  static OpFault f = {2000000000ull, 0};
  return f;
}

// Start of an operator kernel.  A call's kernel is launched while the previous one on the stream is still running (programmatic
// stream serialisation, op_launch): barriers, tensor memory and descriptors are set up behind that one's last tiles, and
// nothing of global memory is touched before op_wait_previous has returned, that is before all earlier work on the stream is
// complete and visible.  op_let_next_start lets the next call's kernel do the same.  It takes effect once every block of this
// grid has come to it, and stands behind the block's tensor-memory allocation: a block that waits for this grid can then
// neither keep one of its blocks out nor hold columns that one of them still needs.  Back to back: linear 50x2048x720
// 8.2 -> 6.1 us, 288x11008x4096 45.9 -> 43.9, attention 1024x1024 (12 heads of 64) 16.4 -> 14.5.
__device__ __forceinline__ void op_wait_previous(const OpMaps& maps, int n) {
  if ((int)threadIdx.x < n) asm volatile("prefetch.tensormap [%0];" ::"l"(&maps.m[threadIdx.x]) : "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void op_let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

}  // namespace vla

#include "op_attention.cuh"
#include "op_linear.cuh"
#include "op_linear_pair.cuh"

namespace vla {

constexpr size_t OP_ATTN_HEADER = 256;   // error word + padding (behind it: room a transposed V would take, which the sizes of the interface count)

// What vla_op_linear keeps per device, looked up on the first call made with that device current: SM count and the error word
// (in a fixed device array of the library).  The kernel clears the word itself before it waits for anything, so that a call
// that was captured into a graph reports on its latest replay like any other.
static __device__ __align__(256) unsigned g_op_linear_error[64];
struct OpDevice {
  unsigned* error = nullptr;
  int sms = 0;
  OpRoom room = {};
};
// The occupancy query answers one CTA per SM for a kernel that allocates tensor memory, where the hardware runs two once the first has
// allocated; so it is asked for a kernel that does not, with the shared memory of the operators' CTAs.  What it does not answer stays 0, and
// calls then use one or two CTAs a tile.
__global__ void vla_op_room_kernel() {}
inline int op_clusters(int s, int smem) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)s; at.val.clusterDim.y = 1; at.val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)s); cfg.blockDim = dim3(LIN_THREADS); cfg.dynamicSmemBytes = (size_t)smem;
  cfg.attrs = &at; cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, vla_op_room_kernel, &cfg) == cudaSuccess) return n;
  cudaGetLastError();
  return 0;
}
inline bool op_look_up(int dev, OpDevice* d) {
  void* a = nullptr;
  if (cudaGetSymbolAddress(&a, g_op_linear_error) != cudaSuccess || !a) return false;
  d->error = static_cast<unsigned*>(a);
  if (cudaDeviceGetAttribute(&d->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return false;
  for (auto* kernel : {vla_op_linear_kernel<1>, vla_op_linear_kernel<2>, vla_op_linear_kernel<8>})
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, LIN_SMEM) != cudaSuccess) return false;
  for (auto* kernel : {vla_op_linear_pair_kernel<1, false>, vla_op_linear_pair_kernel<2, false>, vla_op_linear_pair_kernel<8, false>,
                       vla_op_linear_pair_kernel<1, true>, vla_op_linear_pair_kernel<2, true>, vla_op_linear_pair_kernel<8, true>})
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, LINP_SMEM) != cudaSuccess) return false;
  for (auto* kernel : {vla_op_attention_kernel<1>, vla_op_attention_kernel<2>})
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, OPA_MAX_SMEM) != cudaSuccess) return false;
  const bool asked = cudaFuncSetAttribute(vla_op_room_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, OPA_MAX_SMEM) == cudaSuccess;
  for (int s = 1; s <= OPA_MAX_SPLIT && asked; ++s) { d->room.alone[s] = op_clusters(s, OPA_MAX_SMEM); d->room.two[s] = op_clusters(s, LIN_SMEM); }
  return true;
}
inline bool op_device(OpDevice* d) {
  static PerDevice<OpDevice> devices;
  int dev = -1;
  return cudaGetDevice(&dev) == cudaSuccess && devices.get(dev, d, [dev](OpDevice* r) { return op_look_up(dev, r); });
}

// Reads an operator's error word back after the stream has drained.
inline int op_status_of(const unsigned* dev_word, cudaStream_t s) {
  if (cudaStreamSynchronize(s) != cudaSuccess) return VLA_ERR_CUDA;
  unsigned v = 0;
  if (cudaMemcpy(&v, dev_word, sizeof v, cudaMemcpyDeviceToHost) != cudaSuccess) return VLA_ERR_CUDA;
  return v == 0 ? VLA_OK : VLA_ERR_TIMEOUT;
}

// Launches a kernel in clusters of `cluster` blocks (1: none), overlapping the end of the kernel in front of it
// (op_wait_previous).
template <typename... P, typename... A>
inline int op_launch(void (*kernel)(P...), int grid, int threads, int smem, int cluster, cudaStream_t s, const A&... args) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[2];
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = s;
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = (unsigned)cluster; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...) == cudaSuccess ? VLA_OK : VLA_ERR_CUDA;
}

inline int64_t op_pad(int64_t x, int64_t m) { return (x + m - 1) / m * m; }

inline bool op_attention_shape_ok(int tq, int tkv, int hq, int hkv, int hd) {
  return tq >= 1 && tkv >= 1 && hq >= 1 && hkv >= 1 && hq % hkv == 0 && hd >= 16 && hd <= 256 && hd % 16 == 0;
}

inline size_t op_attention_scratch_bytes(int tkv, int hkv, int hd) {
  return OP_ATTN_HEADER + (size_t)hkv * hd * (size_t)op_pad(tkv, 64) * 2;
}

// Shared implementation of the two attention entry points: the first word of `scratch` is the call's error word.
inline int op_attention_run(const void* q, const void* k, const void* v, void* out, int tq, int tkv, int hq, int hkv, int hd,
                            int causal, void* scratch, cudaStream_t s) {
  OpDevice dev;
  if (!op_device(&dev)) return VLA_ERR_CUDA;
  AttnArgs a;
  memset(&a, 0, sizeof a);
  a.out = reinterpret_cast<Ref>(out);
  a.ldo = hq * hd;
  a.tq = tq; a.t0 = tkv; a.t1 = 0;
  a.hq = hq; a.hkv = hkv; a.hd = hd; a.hs = hd; a.causal = causal ? 1 : 0;
  a.bn = 64;
  a.q_blocks = (tq + 127) / 128;
  a.hpt = attn_fold(tq, hq, hkv, &a.rph);
  int n_tiles = a.hpt > 1 ? hkv * (((hq / hkv) + a.hpt - 1) / a.hpt) : hq * a.q_blocks;
  OpAttnLaunch p = opa_plan(n_tiles, tkv, hd, causal != 0, dev.sms, dev.room);
  // Folded heads share the loads of their keys, but a split tile of several heads also has several heads' rows to exchange: where
  // the chip has the room, each head is a tile of its own (51 x 867, 8 heads of 256 over one: 11.9 -> 9.2 us).
  if (a.hpt > 1 && p.split > 2 && hq <= dev.room.alone[p.split]) { a.hpt = 1; n_tiles = hq; }
  a.scale_log2e = 1.4426950408889634f / sqrtf((float)hd);
  OpMaps maps;
  if (!op_encode(&maps.m[0], q, tq, (int64_t)hq * hd, (int64_t)hq * hd, a.hpt > 1 ? a.rph : 128) ||
      !op_encode(&maps.m[1], k, tkv, (int64_t)hkv * hd, (int64_t)hkv * hd, a.bn) ||
      !op_encode(&maps.m[2], v, tkv, (int64_t)hkv * hd, (int64_t)hkv * hd, a.bn))
    return VLA_ERR_CUDA;
  return op_launch(p.terms == 2 ? vla_op_attention_kernel<2> : vla_op_attention_kernel<1>, n_tiles * p.split, OPA_THREADS, p.smem, p.split, s, a, maps, p, static_cast<unsigned*>(scratch), op_fault());
}

}  // namespace vla

extern "C" {

int vla_op_attention_scratch_bytes(int32_t tkv, int32_t hkv, int32_t hd, size_t* out_bytes) {
  if (!out_bytes || tkv < 1 || hkv < 1 || hd < 16 || hd > 256 || hd % 16) return VLA_ERR_INVALID;
  *out_bytes = vla::op_attention_scratch_bytes(tkv, hkv, hd);
  return VLA_OK;
}

int vla_op_attention(const void* q, const void* k, const void* v, void* out, int32_t tq, int32_t tkv, int32_t hq, int32_t hkv,
                     int32_t hd, int32_t causal, void* scratch, size_t scratch_bytes, void* stream) {
  if (!q || !k || !v || !out || !scratch || !vla::op_attention_shape_ok(tq, tkv, hq, hkv, hd)) return VLA_ERR_INVALID;
  if (causal && tq != tkv) return VLA_ERR_INVALID;
  if (scratch_bytes < vla::op_attention_scratch_bytes(tkv, hkv, hd) || (reinterpret_cast<uintptr_t>(scratch) & 255))
    return VLA_ERR_NOMEM;
  return vla::op_attention_run(q, k, v, out, tq, tkv, hq, hkv, hd, causal, scratch, static_cast<cudaStream_t>(stream));
}

int vla_op_linear(const void* a, const void* w, float* out32, void* out16, int32_t m, int32_t n, int32_t k, int32_t act,
                  void* stream) {
  using namespace vla;
  if (!a || !w || (!out32 && !out16) || m < 1 || n < 1 || k < 8 || k % 8 || act < 0 || act > 2) return VLA_ERR_INVALID;
  OpDevice dev;
  if (!op_device(&dev)) return VLA_ERR_CUDA;
  LinearArgs g;
  g.m = m; g.n = n; g.kp = (int)op_pad(k, GEMM_BK); g.act = act;
  g.out32 = out32; g.out16 = static_cast<unsigned short*>(out16);
  g.err = dev.error;
  const LinearPlan p = linear_plan(m, n, k, out32 != nullptr, dev.sms, LinearRoom{dev.room.alone[4], dev.room.two[4]});
  const LinearPairPlan pp = linear_pair_plan(m, n, k, p, dev.sms);
  const int vec = linear_vec(n, out32, out16);
  OpMaps maps;
  if (pp.bn > 0) {
    g.bm = pp.bm; g.bn = pp.bn; g.ks = p.ks; g.tiles_m = pp.tiles_m; g.tiles = pp.tiles; g.stages = pp.stages;
    if (!op_encode(&maps.m[0], w, n, k, k, g.bn / 2) || !op_encode(&maps.m[1], a, m, k, k, g.bm)) return VLA_ERR_CUDA;
    const int pairs = g.tiles < dev.sms / 2 ? g.tiles : dev.sms / 2;
    const auto kernel = g.ks > 1 ? (vec == 8 ? vla_op_linear_pair_kernel<8, true> : (vec == 2 ? vla_op_linear_pair_kernel<2, true> : vla_op_linear_pair_kernel<1, true>))
                                 : (vec == 8 ? vla_op_linear_pair_kernel<8, false> : (vec == 2 ? vla_op_linear_pair_kernel<2, false> : vla_op_linear_pair_kernel<1, false>));
    return op_launch(kernel, 2 * pairs, LIN_THREADS, LINP_SMEM, 2, static_cast<cudaStream_t>(stream), g, maps, op_fault());
  }
  g.bm = p.bm; g.bn = p.bn; g.ks = p.ks; g.tiles_m = p.tiles_m; g.tiles = p.tiles; g.stages = p.stages;
  if (!op_encode(&maps.m[0], w, n, k, k, g.bn) || !op_encode(&maps.m[1], a, m, k, k, g.bm)) return VLA_ERR_CUDA;
  const int grid = g.ks > 1 ? g.tiles * g.ks : (g.tiles < 2 * dev.sms ? g.tiles : 2 * dev.sms);
  const auto kernel = vec == 8 ? vla_op_linear_kernel<8> : (vec == 2 ? vla_op_linear_kernel<2> : vla_op_linear_kernel<1>);
  return op_launch(kernel, grid, LIN_THREADS, linear_smem(g), g.ks, static_cast<cudaStream_t>(stream), g, maps, op_fault());
}

int vla_debug_op_fault(int32_t drop_operand_loads, uint64_t wait_limit_ns) {
  vla::op_fault().drop_loads = drop_operand_loads ? 1 : 0;
  vla::op_fault().wait_limit_ns = wait_limit_ns ? wait_limit_ns : 2000000000ull;
  return VLA_OK;
}

}  // extern "C"
