// Shared pieces of the tile bodies.  Each body is executed by one worker group of WORKER_THREADS
// threads: either a whole CTA of an ordinary kernel or one worker group inside
// the persistent co-scheduling kernel.  Bodies synchronise with the worker's
// named barrier only (never __syncthreads) and use the shared-memory slab they
// are handed, so the same code, tile shapes and reduction orders run in every
// mode -- which is what makes the modes bit-identical.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "vla_types.h"

namespace vla {

// A claimed tile with everything its worker needs to start it, put together by the claim warp while the worker still runs
// the tile before.
struct TileJob {
  uint32_t inst, node, tile;
  int cls, smem_units, tmem_units;
  int early;                     // queued before its node's release
  unsigned gen;                  // the frame's number in its slot
  int promised_s, promised_t;    // room promised to the tile when it was claimed
  unsigned held_at_claim;        // held_tail when it was claimed: tiles its worker had been given before it
  uint64_t frame, slot_base;
  alignas(16) NodeDesc desc;
};
constexpr int N_JOBS = 4;        // held tiles use jobs 0 and 1 in turn, priority tiles 2 and 3: one running, one waiting

// A finished tile on its way to the retire warp.
struct DoneTile {
  uint32_t inst, node, tile;
  int cls, succ_begin, succ_count, op;
  unsigned gen;
  uint64_t t0, t1, frame;
};

// Mailboxes between one worker group and the SM's service warps, and what the worker keeps from one tile to the next (all in
// shared memory).
struct WorkerSlot {
  volatile unsigned held_tail;   // claimed tiles pushed by the claim warp (single producer)
  volatile unsigned held_head;   // claimed tiles taken by the worker (single consumer)
  volatile unsigned prio_tail, prio_head;   // one-deep slot for an action-head tile that goes ahead of the held VLM tiles
  volatile int leave;            // claim warp -> worker: go home
  volatile int done_state;       // 0 empty, 1 finished tile posted for the retire warp
  volatile int busy;             // the worker is running a tile (set and cleared by the worker)
  volatile int cls;              // class of the running tile
  volatile unsigned long long t_busy;       // when the running tile was taken (worker), for the claim warp's estimate of its end
  volatile int start_state;      // 1: the worker took the last tile of (start_inst, start_node): its successors may be queued early
  uint32_t start_inst, start_node;
  uint32_t bell_parity;
  int run;                       // job of the running tile
  int verdict;                   // 1 run, 2 skip (error), 0 leave
  int smem_unit0, smem_units, tmem_unit0, tmem_units;      // what the running tile occupies
  uint64_t t_start, t_wait;                                // (t_wait: end of a wait for the release without memory, not kept)
  // GEMM operand ring carried over to the next tile: it is the held one, its first loads are in flight (see tile_gemm)
  volatile int primed;
  int ring_stages, ring_s, ring_n;          // stages; the next tile's first stage; its k-blocks already requested
  uint32_t ring_ph, ring_acc;               // parity of that stage's full barrier; of the accumulator barrier
  const volatile unsigned* room_wait;       // the SM's note of a worker waiting for room
  DoneTile done;
  TileJob job[N_JOBS];
};

// What a tile body needs to know beside its node's arguments.  The persistent kernel keeps one per worker in shared memory:
// the bodies have use for every register, and values that are the same in all threads are read from there when needed.
struct TileCtx {
  char* arena;
  uint64_t slot_base;   // arena offset of this frame slot's buffers
  char* smem;           // this tile's shared-memory slab (1024-byte aligned): operand stages, staging tiles
  int smem_bytes;       // size of the slab handed over (at least the node's smem_bytes)
  char* ctl;            // this worker's 1 KB control block (mbarriers, row scales): outside the slab, so tile
                        // slabs are whole powers-of-two-friendly sizes (64 KB, 72 KB, 48 KB)
  uint32_t tmem;        // this worker's tensor-memory column base
  int bar_id;           // named barrier of this worker
  uint64_t deadline;    // %globaltimer value after which bounded waits give up
  unsigned int* error;  // sticky device error word
  const uint64_t* inputs;  // this frame slot's input pointer table
  const void* tmaps;    // tensor-map table (128 bytes per entry)
  int amap_base;        // index of this frame slot's first activation map
  int n_weight_tmaps, n_act_tmaps;      // weight maps; activation maps per frame slot
  const unsigned long long* wait_word;   // not null: the tile was taken early and waits for its node's release, the moment this
  unsigned long long wait_count;         // word counts so many finished predecessor tiles; GEMM tiles fetch weights meanwhile
  uint64_t* t_start;                     // where the time of that moment goes
  WorkerSlot* slot;     // the persistent kernel's worker, null elsewhere
  int cont;             // this tile's operand ring was primed by the tile before
  int drop_loads;       // test hook (tile_hooks.cuh): the TMA producer issues nothing, so the consumers' bounded waits run out
                        // (0 in the persistent kernel)
};

// 0 .. WORKER_THREADS-1 (a kernel's workers are consecutive groups of WORKER_THREADS threads)
__device__ __forceinline__ int worker_tid() { return (int)(threadIdx.x % WORKER_THREADS); }

template <typename T>
__device__ __forceinline__ T* resolve(const TileCtx& c, Ref r) {
  if (r == 0) return nullptr;
  if (r & REF_INPUT) {
    const unsigned long long p = __ldcg(reinterpret_cast<const unsigned long long*>(c.inputs) + ((r >> 56) & 0xF));
    return reinterpret_cast<T*>(p + (r & ((1ull << 56) - 1)));
  }
  return reinterpret_cast<T*>(c.arena + (r & ~REF_SLOT) + ((r & REF_SLOT) ? c.slot_base : 0ull));
}

__device__ __forceinline__ void worker_sync(const TileCtx& c) {
  asm volatile("bar.sync %0, %1;" ::"r"(c.bar_id), "r"(WORKER_THREADS) : "memory");
}

__device__ __forceinline__ bool released(const unsigned long long* word, unsigned long long count) {
  unsigned long long w;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(word) : "memory");
  return (w & ((1ull << 62) - 1ull)) >= count;
}
// One thread: waits (bounded) until the tile's node is released.  After a time-out the error is recorded and the tile runs
// on whatever its operands hold, so that everything it has in flight ends in the ordinary way.  No pause between the looks:
// each is a trip to L2 (60 ns of sleep in between, where the tile waits empty-handed, changed none of five workloads).
__device__ __forceinline__ void wait_release(const TileCtx& c) {
  unsigned spins = 0;
  for (;;) {
    uint64_t now;
    if (released(c.wait_word, c.wait_count)) {
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
      *c.t_start = now;
      return;
    }
    if ((++spins & 63u) == 0) {
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
      if (now > c.deadline) atomicCAS(c.error, 0u, (unsigned)DEV_ERR_WAIT_DEP);
      if (*reinterpret_cast<volatile unsigned*>(c.error) != 0u) { *c.t_start = now; return; }
    }
  }
}

__device__ __forceinline__ void set_error(const DeviceCtx& ctx, unsigned code, unsigned info) {
  if (atomicCAS(&ctx.control->error, 0u, code) == 0u) {
    ctx.control->error_info = info;
    *ctx.error_host = code;
    __threadfence_system();
  }
}

// Activations are produced by other SMs during the same kernel: read them through L2.
__device__ __forceinline__ float ld_act(const float* p) { return __ldcg(p); }
__device__ __forceinline__ uint4 ld_act(const uint4* p) { return __ldcg(p); }
__device__ __forceinline__ unsigned short ld_act(const unsigned short* p) { return __ldcg(p); }
__device__ __forceinline__ int ld_act(const int* p) { return __ldcg(p); }

__device__ __forceinline__ float bf16_bits_to_f32(unsigned short b) { return __uint_as_float(((unsigned int)b) << 16); }
__device__ __forceinline__ unsigned short f32_to_bf16_bits(float f) {
  return __bfloat16_as_ushort(__float2bfloat16_rn(f));
}
__device__ __forceinline__ void unpack8(const uint4& v, float* f) {
  f[0] = __uint_as_float(v.x << 16); f[1] = __uint_as_float(v.x & 0xFFFF0000u);
  f[2] = __uint_as_float(v.y << 16); f[3] = __uint_as_float(v.y & 0xFFFF0000u);
  f[4] = __uint_as_float(v.z << 16); f[5] = __uint_as_float(v.z & 0xFFFF0000u);
  f[6] = __uint_as_float(v.w << 16); f[7] = __uint_as_float(v.w & 0xFFFF0000u);
}

// Activations use the hardware approximations (tanh.approx, ex2.approx): their error (~2^-11 relative)
// is below the bf16 rounding of the values they produce.
__device__ __forceinline__ float tanh_fast(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float gelu_tanh_f(float x) {     // 0.5 x (1 + tanh(c x + c 0.044715 x^3))
  const float c = 0.7978845608028654f, h = 0.5f * x;
  return fmaf(h, tanh_fast(x * fmaf(x * x, c * 0.044715f, c)), h);
}
// x / (1 + 2^(-x log2 e)) in five instructions.  The .ftz forms only differ where it does not show: 1 + e is never subnormal,
// a subnormal e adds nothing to 1, and past 2^126 the quotient is 0 either way (the plain forms spend ten instructions more
// on those: a 8192 x 3072 linear layer with SiLU 24.4 -> 21.9 us at K = 64, 46.2 -> 43.2 at K = 768).
__device__ __forceinline__ float silu_f(float x) {
  float e, r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(x * -1.44269504f));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(1.0f + e));
  return x * r;
}
template <int ACT>
__device__ __forceinline__ float apply_act_t(float v) {
  return ACT == ACT_GELU ? gelu_tanh_f(v) : (ACT == ACT_SILU ? silu_f(v) : v);
}
__device__ __forceinline__ float apply_act(int act, float v) {
  return act == ACT_GELU ? gelu_tanh_f(v) : (act == ACT_SILU ? silu_f(v) : v);
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// ------------------------------------------------------------------ GEMM epilogue (one output element)
struct GemmPtrs {
  const float* X; const float* vec; const float* tab; const float* tab2; const float* bias;
  float* out32; unsigned short* out16; unsigned short* outT;
};
__device__ __forceinline__ GemmPtrs gemm_ptrs(const TileCtx& c, const GemmArgs& g) {
  GemmPtrs p;
  p.X = resolve<const float>(c, g.X); p.vec = resolve<const float>(c, g.vec);
  p.tab = resolve<const float>(c, g.tab); p.tab2 = resolve<const float>(c, g.tab2);
  p.bias = resolve<const float>(c, g.bias);
  p.out32 = resolve<float>(c, g.out32); p.out16 = resolve<unsigned short>(c, g.out16);
  p.outT = resolve<unsigned short>(c, g.outT);
  return p;
}
}  // namespace vla
