// Device side of the dispatcher: tile queues, dependency counters, the persistent
// co-scheduling kernel, and the ordinary-kernel wrapper used by the stream modes.
#pragma once
#include "pick.cuh"
#include "tiles.cuh"

namespace vla {

constexpr unsigned CTRL_EXITING = 0x80000000u;
constexpr uint32_t TRACE_ADMIT_NODE = 0xFFFFFFFFu;   // node id of the trace record that marks a frame's admission
constexpr int MAX_WORKERS = 3;
constexpr int SM_CTL_BYTES = 1024;       // per-worker control block (mbarriers, row scales) handed to the tile bodies
constexpr int SM_STATE_BASE = 8192;      // dispatcher state of the SM
constexpr int SM_STATE_BYTES = SM_STATE_BASE + MAX_WORKERS * SM_CTL_BYTES;   // then the tile slab, 1024-byte aligned

__device__ __forceinline__ uint64_t gtimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ unsigned smid() {
  unsigned s;
  asm volatile("mov.u32 %0, %%smid;" : "=r"(s));
  return s;
}
__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned ld_volatile_u32(const unsigned* p) { return *reinterpret_cast<const volatile unsigned*>(p); }
__device__ __forceinline__ unsigned long long ld_volatile_u64(const unsigned long long* p) {
  return *reinterpret_cast<const volatile unsigned long long*>(p);
}
__device__ __forceinline__ long long ld_volatile_s64(const long long* p) { return *reinterpret_cast<const volatile long long*>(p); }

// Shows the host the error word, whichever wait has set it.
__device__ __forceinline__ void mirror_error(const DeviceCtx& ctx) {
  *reinterpret_cast<volatile unsigned*>(ctx.error_host) = ld_volatile_u32(&ctx.control->error);
  __threadfence_system();
}

// ------------------------------------------------------------------ doorbells inside an SM
// The service warps and idle workers must not spin: every instruction they issue is taken from the worker warps that
// share their scheduler (a claim loop polling flat out cost the tile bodies 10-40 % of their speed).  They wait on
// an mbarrier instead -- suspended by the hardware, no issue slots -- which whoever has news for them rings; the
// wait is bounded by a time hint, so a lost ring (two rings inside one phase look like none) only delays, never hangs.
__device__ __forceinline__ void bell_ring(const void* bell) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bell)) : "memory");
}
// Returns when the bell was rung since the last successful wait or, at the latest, after about `hint_ns`.
__device__ __forceinline__ bool bell_wait(const void* bell, uint32_t& parity, uint32_t hint_ns) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bell)), "r"(parity), "r"(hint_ns)
      : "memory");
  if (ok) parity ^= 1u;
  return ok != 0;
}

// ------------------------------------------------------------------ tensor memory (whole-warp calls)
__device__ __forceinline__ void tmem_alloc(uint32_t* smem_dst, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_dst)), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}

// ------------------------------------------------------------------ tile queues
// Pushing tiles is split in three so a whole warp can fill the entries in parallel:
// reserve (one thread), fill (any threads, entry i of the range), commit (one thread, after a barrier).
// The ring is sized for every tile of every frame slot, so a reservation can never overrun the head.
// One entry = one 64-bit word: generation (11 bits, never 0 for a written entry of the current lap... the lap count + 1)
// | node (20) | frame slot (9) | tile (12) | the node's per-tile resource need in units so that a claim needs no
// second load: shared memory (6) and tensor memory (5) | and whether the tile was queued before its node's release (1).
constexpr int QW_NODE_BITS = 20, QW_INST_BITS = 9, QW_TILE_BITS = 12, QW_SMEM_BITS = 6, QW_TMEM_BITS = 5, QW_GEN_BITS = 11;
static_assert(QW_NODE_BITS + QW_INST_BITS + QW_TILE_BITS + QW_SMEM_BITS + QW_TMEM_BITS + 1 + QW_GEN_BITS == 64, "queue word layout");
constexpr uint32_t RES_EARLY = 1u << (QW_SMEM_BITS + QW_TMEM_BITS);      // in the resource field of an entry being written
__device__ __forceinline__ unsigned long long queue_gen(const DeviceCtx& ctx, unsigned long long ticket) {
  return ((ticket >> ctx.q_shift) + 1ull) & ((1ull << QW_GEN_BITS) - 1ull);
}
__device__ __forceinline__ unsigned long long queue_word(const DeviceCtx& ctx, unsigned long long ticket, uint32_t inst,
                                                         uint32_t node, uint32_t tile, uint32_t res_units) {
  // res_units = smem units | tmem units << QW_SMEM_BITS (| RES_EARLY)
  return (queue_gen(ctx, ticket) << (64 - QW_GEN_BITS)) | ((unsigned long long)res_units << (QW_NODE_BITS + QW_INST_BITS + QW_TILE_BITS)) |
         ((unsigned long long)tile << (QW_NODE_BITS + QW_INST_BITS)) | ((unsigned long long)inst << QW_NODE_BITS) | (unsigned long long)node;
}
__device__ inline unsigned long long queue_reserve(const DeviceCtx& ctx, int cls, int n) {
  return atomicAdd(&ctx.queues[cls].tail, (unsigned long long)n);
}
// Ordering: a consumer may pop a ticket before that ticket's own commit (`avail` counts anybody's commits) and then
// waits for the entry's generation tag with an acquire load.  So the entry store itself must publish everything the
// producer has observed: every filling thread issues a device-scope fence before its (relaxed) entry stores
// -- queue_fill_fence() -- and the thread that watched the dependency counter reach zero fences after that atomic.
// The commit carries no ordering duty of its own.
__device__ __forceinline__ void queue_fill_fence() { __threadfence(); }
__device__ inline void queue_fill(const DeviceCtx& ctx, int cls, unsigned long long base, uint32_t inst, uint32_t node,
                                  uint32_t res_units, int first, int count, int stride) {
  const unsigned long long mask = (unsigned long long)ctx.q_capacity - 1;
  QueueEntry* ent = ctx.q_entries + (size_t)cls * ctx.q_capacity;
#pragma unroll 1
  for (int i = first; i < count; i += stride)
    *reinterpret_cast<volatile unsigned long long*>(ent + ((base + i) & mask)) = queue_word(ctx, base + i, inst, node, (uint32_t)i, res_units);
}
__device__ inline void queue_commit(const DeviceCtx& ctx, int cls, int n) {
  atomicAdd(reinterpret_cast<unsigned long long*>(&ctx.queues[cls].avail), (unsigned long long)n);
}
// One thread pushes everything (admission of a frame's root tiles).
__device__ __forceinline__ uint32_t node_res_units(const NodeDesc& nd) {
  return (uint32_t)((__ldg(&nd.smem_bytes) + SMEM_UNIT - 1) / SMEM_UNIT) |
         ((uint32_t)((__ldg(&nd.tmem_cols) + TMEM_UNIT - 1) / TMEM_UNIT) << QW_SMEM_BITS);
}
__device__ inline void queue_push(const DeviceCtx& ctx, int cls, uint32_t inst, uint32_t node, int n) {
  const unsigned long long base = queue_reserve(ctx, cls, n);
  queue_fill_fence();
  queue_fill(ctx, cls, base, inst, node, node_res_units(ctx.nodes[node]), 0, n, 1);
  queue_commit(ctx, cls, n);
}

// The entry of a claimed ticket.  Bounded wait for it to land.
__device__ __forceinline__ bool queue_entry(const DeviceCtx& ctx, int cls, unsigned long long t, QueueEntry& e, uint64_t deadline) {
  const unsigned long long want = queue_gen(ctx, t);
  const unsigned long long* slot = ctx.q_entries + (size_t)cls * ctx.q_capacity + (t & ((unsigned long long)ctx.q_capacity - 1));
  unsigned spins = 0;
  while (((e = ld_acquire_u64(slot)) >> (64 - QW_GEN_BITS)) != want) {
    if ((++spins & 63u) == 0 && gtimer() > deadline) {
      set_error(ctx, DEV_ERR_WAIT_QUEUE, cls);
      return false;
    }
  }
  return true;
}

// ------------------------------------------------------------------ per-SM state of the persistent kernel
constexpr int DISPATCH_THREADS = 128;    // a warpgroup with the two service warps of the SM (claim, retire), after the worker groups
// Registers a thread, after the split: the launch gives every thread 128 (four warps on each scheduler), and a tile body wants
// more: what it spilled came back from L2, since the slab leaves L1 next to nothing.  The service warpgroup hands back what it
// does not use: n * 144 + 80 <= (n + 1) * 128 for one, two and three workers.  120 -> 16 bytes of spills; single frame
// 11.97 -> 11.58 ms, 32 streams x 4 184.2 -> 181.4.
constexpr int WORKER_REGS = 144, DISPATCH_REGS = 80;
static_assert(MAX_WORKERS * WORKER_REGS + DISPATCH_REGS <= (MAX_WORKERS + 1) * 128, "the split must not exceed what the block was launched with");
constexpr long long PRIO_WINDOW_NS = 8000;   // an action-head tile may be claimed for a worker this close to the end of its tile
constexpr int PREFETCH_MIN_TOTAL = 300;   // tiles are claimed ahead of need only while this many VLM tiles are queued in all
                                          // (32 streams x 4: 181.5 ms at 600, 178.9 at 300, no better at 150)
constexpr int PREFETCH_MIN_AVAIL = 8;     // ... and only from queues at least this deep
constexpr int HELD_DEPTH = 1;            // claimed tiles a worker may have waiting
constexpr unsigned CLAIM_NAP_NS = 60, CLAIM_NAP_MAX_NS = 240;   // claim warp, while a worker of its SM has nothing to run
constexpr unsigned CLAIM_SLEEP_NS = 2000;    // claim warp, every worker busy: longest sleep without a ring
constexpr unsigned RETIRE_SLEEP_NS = 4000;   // retire warp: longest sleep without a ring
// With no more tiles queued or running than the GPU has SMs, tiles are spread one per SM (two per SM up to twice as many) and
// take the pipeline depth that leaves room for; an SM that has its share leaves the queue to the others for about a tile's
// length: the SM where the next tile ends is the better place, a second tile beside a first makes both of them late.  1, 4, 8,
// 16 us: 4 streams x 3 43.4, 41.7, 40.3, 39.5 ms; 8 x 3 GR00T 40.1, 38.6, 37.1, 36.3; 64 us brings nothing more.
constexpr unsigned long long SPREAD_WAIT_NS = 16000;
constexpr unsigned long long HEAD_WAIT_NS = 1500;   // an action-head tile nobody took for this long may go to a running worker

static_assert(sizeof(NodeDesc) % 16 == 0 && sizeof(NodeDesc) <= 512, "a node's description is copied by one warp, 16 bytes a lane");
struct __align__(16) SmState {
  unsigned long long smem_mask;    // bit i set = shared-memory unit i in use
  unsigned tmem_mask;              // bit i set = tensor-memory unit i in use
  int n_smem_units, n_tmem_units;
  PickState pick;
  unsigned tmem_base;
  volatile int quit;               // claim warp -> retire warp: everyone is leaving
  int smem_promised, tmem_promised;  // units of tiles handed to free workers that have not allocated them yet
  unsigned room_wait;              // a worker waiting for room right now: smem units | tmem units << 8 | (worker + 1) << 16, else 0
                                   // (the latest one when two wait); the claim warp keeps that room out of its offers
  volatile int outstanding;        // tiles queued or running on the whole GPU when the claim warp last looked
  volatile int ema_ns[N_CLASSES];  // running mean of tile durations per class on this SM (retire warp)
  // per class: intensity tags, pick group, tiles queued (-G score), largest need of a tile in units, R_k of the -R score
  int tau_tab[N_CLASSES * 3];
  unsigned group_mask[N_CLASSES];
  int grid[N_CLASSES], smem_units[N_CLASSES], tmem_units[N_CLASSES], res[N_CLASSES];
  unsigned long long bell_claim;   // rung by a worker that took a claimed tile or ran out of work
  unsigned long long bell_retire;  // rung by a worker that posted a finished tile
  unsigned long long bell_worker[MAX_WORKERS];   // rung by the claim warp when it hands worker w a tile or sends it home
  TileCtx tc[MAX_WORKERS];         // context of each worker's running tile
  WorkerSlot slot[MAX_WORKERS];
};
static_assert(sizeof(SmState) <= SM_STATE_BASE, "SM state too large");

__device__ __forceinline__ unsigned long long unit_bits(int n) { return n >= 64 ? ~0ull : ((1ull << n) - 1ull); }
// Lowest position of `need` consecutive free units among the first `total` (bit set = in use), or -1.
// run keeps the positions where k consecutive free units start; k doubles until it reaches `need`.
__device__ __forceinline__ int find_free(unsigned long long mask, int need, int total) {
  if (need == 0) return 0;
  if (need > total) return -1;
  unsigned long long run = ~mask & unit_bits(total);
#pragma unroll 1
  for (int k = 1; k < need;) {
    const int step = min(k, need - k);
    run &= run >> step;
    k += step;
  }
  return run ? __ffsll((long long)run) - 1 : -1;
}

__device__ inline void write_trace(const DeviceCtx& ctx, uint32_t inst, uint32_t node, uint32_t tile, int worker, int cls,
                                   uint64_t frame, uint64_t t0, uint64_t t1) {
  if (ctx.trace_capacity == 0) return;
  unsigned long long idx = atomicAdd(&ctx.control->trace_count, 1ull);
  if (idx >= ctx.trace_capacity) return;
  TraceRec r;
  r.inst = inst; r.node = node; r.tile = tile; r.sm = (uint16_t)smid(); r.worker = (uint8_t)worker; r.cls = (uint8_t)cls;
  r.frame = frame; r.t_start = t0; r.t_end = t1;
  ctx.trace[idx] = r;
}

// A frame became ready (its inputs are in HBM): take its admission record and queue its root tiles.
__device__ inline void try_admit(const DeviceCtx& ctx) {
  Control* ctl = ctx.control;
  const unsigned long long head = ld_volatile_u64(&ctl->admit_head);
  const unsigned long long tail = ld_volatile_u64(&ctl->admit_tail);
  if (head >= tail) return;
  unsigned old = ld_volatile_u32(&ctl->ctrl);
#pragma unroll 1
  for (int tries = 0; tries < 8; ++tries) {
    if (old & CTRL_EXITING) return;
    unsigned prev = atomicCAS(&ctl->ctrl, old, old + 1u);
    if (prev == old) { old = 0xffffffffu; break; }
    old = prev;
  }
  if (old != 0xffffffffu) return;
  if (atomicCAS(&ctl->admit_head, head, head + 1ull) != head) {
    atomicSub(&ctl->ctrl, 1u);
    return;
  }
  const volatile AdmitRec* rec = ctx.admit_ring + (head & (unsigned long long)(ctx.admit_capacity - 1));
  const uint32_t inst = rec->inst;
  const uint64_t frame = rec->frame;
  *reinterpret_cast<volatile uint64_t*>(ctx.inst_frame + inst) = frame;
  *reinterpret_cast<volatile uint32_t*>(ctx.inst_gen + inst) = rec->gen;
  {   // the frame's admission is a trace record of its own (node = TRACE_ADMIT_NODE): no tile of the frame may start earlier
    const uint64_t now = gtimer();
    write_trace(ctx, inst, TRACE_ADMIT_NODE, 0, 0, 0xFF, frame, now, now);
  }
  __threadfence();
#pragma unroll 1
  for (int i = 0; i < ctx.n_roots; ++i) {
    int r = ctx.roots[i];
    queue_push(ctx, ctx.nodes[r].cls, inst, (uint32_t)r, ctx.nodes[r].n_tiles);
  }
}

__device__ __forceinline__ SuccInfo load_succ(const DeviceCtx& ctx, int i) {
  const int4 v = __ldg(reinterpret_cast<const int4*>(ctx.succ + i));
  return SuccInfo{v.x, v.y, v.z, v.w};
}

// Queues the node each `ready` lane holds (whole warp): the lanes reserve their ranges at once, the warp writes the entries.
__device__ __forceinline__ void push_nodes(const DeviceCtx& ctx, bool ready, uint32_t inst, const SuccInfo& si, uint32_t early, int lane) {
  unsigned m = __ballot_sync(0xffffffffu, ready);
  if (m == 0u) return;
  const int cls = si.cls_res & 0xFF;
  const uint32_t res = (((uint32_t)si.cls_res >> 8) & (RES_EARLY - 1u)) | early;
  const unsigned long long base = ready ? queue_reserve(ctx, cls, si.n_tiles) : 0ull;
  queue_fill_fence();
#pragma unroll 1
  for (; m != 0u; m &= m - 1u) {
    const int src = __ffs((int)m) - 1;
    queue_fill(ctx, __shfl_sync(0xffffffffu, cls, src), __shfl_sync(0xffffffffu, base, src), __shfl_sync(0xffffffffu, inst, src),
               (uint32_t)__shfl_sync(0xffffffffu, si.node, src), __shfl_sync(0xffffffffu, res, src), lane,
               __shfl_sync(0xffffffffu, si.n_tiles, src), 32);
  }
  __syncwarp();
  if (ready) queue_commit(ctx, cls, si.n_tiles);
}

// ------------------------------------------------------------------ the two service warps of an SM
// Workers never touch global queues or counters.  Two extra warps per SM do it for them, so those
// round trips overlap tile execution instead of sitting between tiles:
//   * the CLAIM warp (lane w serves worker w) claims tiles under the pick policy -- for a busy worker one
//     tile ahead -- and hands a claimed tile over as soon as its worker is free and its exact
//     shared/tensor-memory need fits;
//   * the RETIRE warp (eight lanes serve one worker) takes a finished tile and does the global bookkeeping
//     (successors' dependency counters, queue pushes; the whole warp fills the released successors' entries).
// Per-SM state is shared-memory words updated with shared-memory atomics by these two warps only.
// Eight lanes serve one worker, a successor of its tile's node each, so the counter round trips of all workers and
// successors run at the same time.
constexpr int RETIRE_LANES = 8;
static_assert(RETIRE_LANES * MAX_WORKERS <= 32, "the retire warp has lanes for every worker");
__device__ __forceinline__ void retire_loop(const DeviceCtx& ctx, SmState* sm, int n_workers) {
  const int lane = threadIdx.x & 31, w = lane / RETIRE_LANES, sub = lane % RETIRE_LANES;
  const bool serving = w < n_workers;
  WorkerSlot* slot = sm->slot + (serving ? w : 0);
  uint32_t bell_parity = 0;
  for (;;) {
    // (the flags are read in this order and handled in the other: a tile's start is announced before its end is)
    const bool ended = serving && slot->done_state == 1;
    __threadfence_block();
    const bool started = serving && slot->start_state == 1;
    __syncwarp();
    if (!__any_sync(0xffffffffu, ended || started)) {
      if (sm->quit) break;
      bell_wait(&sm->bell_retire, bell_parity, RETIRE_SLEEP_NS);
      continue;
    }
    // ---- starts.  The last tile of a node has been taken by a worker: tiles of a class are claimed in queue order, so all of
    // them have been claimed.  Where that was the last predecessor of a successor, and everything queued or running still fits
    // one tile per SM (up to two per SM: 4 x 3 cfg2 43.3 -> 42.0 ms, but CogACT 18.8 -> 19.7), the successor is queued now: its
    // tiles are taken, fetch their weights and wait for the release, instead of going through the queues after it (hand-over 3 us
    // instead of 9).  No cycle can arise: a waiting tile waits only for tiles claimed before it, a worker takes tiles that may
    // have to wait in the order of their claims (see priority_goes_first), and such a tile holds shared memory while it waits
    // only on an SM where nothing claimed before it still needs some (see the worker's allocation).
    if (__any_sync(0xffffffffu, started)) {
      uint32_t inst = 0;
      int succ0 = 0, n_succ = 0;
      if (started) {
        inst = slot->start_inst;
        const int4 d = __ldg(reinterpret_cast<const int4*>(ctx.nodes + slot->start_node) + 1);     // succ_begin, succ_count, phase, step
        succ0 = d.x; n_succ = d.y;
      }
      __syncwarp();
      if (started && sub == 0) { __threadfence_block(); slot->start_state = 0; }
#pragma unroll 1
      for (int i = sub; __any_sync(0xffffffffu, i < n_succ); i += RETIRE_LANES) {
        SuccInfo si = {0, 0, 0, 0};
        bool early = false;
        if (i < n_succ) {
          si = load_succ(ctx, succ0 + i);
          const size_t at = (size_t)inst * ctx.n_nodes + si.node;
          if (atomicSub(ctx.start_count + at, 1) == 1) {
            ctx.start_count[at] = (int)((uint32_t)si.cls_res >> 20);
            early = sm->outstanding + si.n_tiles <= (int)gridDim.x;
            // marked before this SM reports the tile finished, so whoever releases the node sees the mark
            if (early) atomicOr(ctx.dep_word + at, 1ull << 63);
          }
        }
        push_nodes(ctx, early, inst, si, RES_EARLY, lane);
      }
    }
    // ---- ends.  Every successor's word counts one more finished predecessor tile; reaching the frame's total is the release,
    // which early-taken tiles of that node wait for; if the node was not queued early, it is now.
    if (__any_sync(0xffffffffu, ended)) {
      uint32_t inst = 0;
      int succ0 = 0, n_succ = 0;
      unsigned gen = 0;
      if (ended) {
        const DoneTile& f = slot->done;
        inst = f.inst; gen = f.gen; succ0 = f.succ_begin; n_succ = f.succ_count;
        if (sub == 0) {
          sm->ema_ns[f.cls] = (3 * sm->ema_ns[f.cls] + (int)(f.t1 - f.t0)) >> 2;
          write_trace(ctx, f.inst, f.node, f.tile, w, f.cls, f.frame, f.t0, f.t1);
        }
      }
      __threadfence();        // the tile's writes, seen through the mailbox, go ahead of the counters below
#pragma unroll 1
      for (int i = sub; __any_sync(0xffffffffu, i < n_succ); i += RETIRE_LANES) {
        SuccInfo si = {0, 0, 0, 0};
        bool release = false;
        if (i < n_succ) {
          si = load_succ(ctx, succ0 + i);
          unsigned long long* word = ctx.dep_word + (size_t)inst * ctx.n_nodes + si.node;
          const unsigned long long old = atomicAdd(word, 1ull);
          if ((old & ((1ull << 62) - 1ull)) + 1ull == DEP_BIAS + (unsigned long long)(unsigned)si.n_pred * gen) {
            if (old >> 63) atomicAnd(word, ~(1ull << 63));
            else release = true;
          }
        }
        push_nodes(ctx, release, inst, si, 0u, lane);
      }
      if (ended && sub == 0) {
        atomicAdd(&ctx.queues[slot->done.cls].done, 1ull);
        if (slot->done.op == OP_EMIT) atomicSub(&ctx.control->ctrl, 1u);
        __threadfence_block();
        slot->done_state = 0;
      }
      __syncwarp();
    }
  }
}

__device__ inline void claim_loop(const DeviceCtx& ctx, SmState* sm, int n_workers) {
  const int lane = threadIdx.x & 31;
  const bool serving = lane < n_workers;
  Control* ctl = ctx.control;
  WorkerSlot* slot = sm->slot + (serving ? lane : 0);
  // (Class tables are read from shared memory, and the loops below stay rolled: this code runs on every hand-over of the SM,
  // between tile bodies that need the instruction cache.)
  uint64_t idle_start = 0, last_progress = gtimer();
  unsigned iter = 0, nap = CLAIM_NAP_NS, lost = 0;
  uint32_t bell_parity = 0;
  uint64_t pending_since = 0;     // lane c: since when class c has had committed tiles without a break (0: it has none)
  bool leaving = false;

  // What this warp polls is one 16-byte word per lane, so that a round costs one trip to L2: lanes 0..7 a class's claimable
  // tiles, lanes 8..15 its tail and done, lane 16 the control words, lane 17 the admission ring.
  const void* poll_at = ctx.queues;
  if (lane < N_CLASSES) poll_at = &ctx.queues[lane].avail;
  else if (lane < 2 * N_CLASSES) poll_at = &ctx.queues[lane - N_CLASSES].tail;
  else if (lane == 16) poll_at = &ctl->ctrl;
  else if (lane == 17) poll_at = &ctl->admit_head;
  for (;;) {
    ++iter;
    bool progressed = false;
    unsigned long long px, py;
    asm volatile("ld.volatile.global.v2.u64 {%0, %1}, [%2];" : "=l"(px), "=l"(py) : "l"(poll_at) : "memory");
    const uint64_t now = gtimer();
    const long long av = lane < N_CLASSES ? (long long)px : 0;
    const unsigned pending = __ballot_sync(0xffffffffu, av > 0) & ((1u << N_CLASSES) - 1u);
    // Tiles are claimed ahead of need only while the VLM backlog as a whole exceeds what the GPU's workers can hold
    // (a held tile is a tile no idle worker elsewhere can take), and then from every VLM queue that is not nearly empty.
    long long vlm_total = (lane < N_KINDS && av > 0) ? av : 0;
    vlm_total += __shfl_xor_sync(0xffffffffu, vlm_total, 1);
    vlm_total += __shfl_xor_sync(0xffffffffu, vlm_total, 2);
    vlm_total = __shfl_sync(0xffffffffu, vlm_total, 0);
    const unsigned deep = __ballot_sync(0xffffffffu, vlm_total >= PREFETCH_MIN_TOTAL && av >= PREFETCH_MIN_AVAIL) &
                          ((1u << N_CLASSES) - 1u);
    // classes whose tiles free workers elsewhere did not drain within head_wait_ns (by the clock, not by polling
    // rounds: how fast this loop spins must not change what it decides)
    if (av > 0) { if (pending_since == 0) pending_since = now; } else pending_since = 0;
    const unsigned waiting = __ballot_sync(0xffffffffu, pending_since != 0 && now - pending_since >= HEAD_WAIT_NS) &
                             ((1u << N_CLASSES) - 1u);
    int outstanding = lane >= N_CLASSES && lane < 2 * N_CLASSES ? (int)min(px - py, 1ull << 20) : 0;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) outstanding += __shfl_xor_sync(0xffffffffu, outstanding, o);
    outstanding = __shfl_sync(0xffffffffu, outstanding, N_CLASSES);
    if (lane == 0) sm->outstanding = outstanding;
    const int n_sms = (int)gridDim.x;
    const int share = outstanding <= n_sms ? 1 : (outstanding <= 2 * n_sms ? 2 : MAX_WORKERS);
    unsigned spread = 0xffffffffu;
    int running = 0;
    if (share < MAX_WORKERS) {
      spread = __ballot_sync(0xffffffffu, pending_since != 0 && now - pending_since >= SPREAD_WAIT_NS) & ((1u << N_CLASSES) - 1u);
      running = __popc(__ballot_sync(0xffffffffu, serving && (slot->busy != 0 || slot->held_tail != slot->held_head || slot->prio_tail != slot->prio_head)));
    }
    if (lane < N_CLASSES) sm->grid[lane] = (int)(av < 0 ? 0 : (av > (1 << 20) ? (1 << 20) : av));   // G_k of the -G score: tiles still to place
    // ---- choose, lane by lane, which class each worker claims from
    int want = -1, promised_s = 0, promised_t = 0;
    bool to_prio = false;
    const unsigned avoid = lost;      // the class this lane just lost a race for: other SMs drained it
    lost = 0;
#pragma unroll 1
    for (int w = 0; w < n_workers; ++w) {
      const unsigned queued = serving ? slot->held_tail - slot->held_head : 0u;
      const unsigned pq = serving ? slot->prio_tail - slot->prio_head : 0u;
      if (lane == w && !leaving && (queued < (unsigned)HELD_DEPTH || pq == 0u)) {
        // A free worker serves the action head first.  A running worker gets VLM tiles claimed ahead of need (from
        // deep queues only), and an action-head tile when that tile has been waiting for more than a round (no
        // free worker anywhere took it) and the running tile is within PRIO_WINDOW_NS of its expected end (this
        // SM's running mean for the class): it goes into the priority slot, ahead of the held VLM tiles, so a
        // short action-head tile is never stuck behind more than the tail of one tile.
        const unsigned act_mask = ((1u << N_KINDS) - 1u) << N_KINDS;
        const bool busy = slot->busy != 0 || queued > 0 || pq > 0;
        const bool head_pending = pick_is_two_phase(ctx.policy) && (pending & act_mask & ~avoid) != 0u;
        unsigned cand;
        if (!busy) cand = head_pending ? (pending & act_mask) : pending;
        else if (pq == 0u && head_pending && (waiting & act_mask & ~avoid) != 0u && slot->busy != 0 && slot->primed == 0 &&
                 (long long)(now - slot->t_busy) + PRIO_WINDOW_NS >= (long long)sm->ema_ns[slot->cls]) {
          cand = waiting & act_mask; to_prio = true;
        }
        else if (queued < (unsigned)HELD_DEPTH) cand = deep & ((1u << N_KINDS) - 1u);
        else cand = 0u;
        cand &= ~avoid;
        if (running >= share) cand &= spread;
        const unsigned long long smask = *reinterpret_cast<volatile unsigned long long*>(&sm->smem_mask);
        const unsigned tmask = *reinterpret_cast<volatile unsigned*>(&sm->tmem_mask);
        // room: a free run of units now, and enough units left after what was promised to tiles already handed
        // to free workers of this SM (they allocate a moment later)
        int smem_left = sm->n_smem_units - __popcll(smask) - *reinterpret_cast<volatile int*>(&sm->smem_promised);
        int tmem_left = sm->n_tmem_units - __popc(tmask) - *reinterpret_cast<volatile int*>(&sm->tmem_promised);
        {   // a worker of this SM that waits for room is served first: what it needs is not offered to the others
          const unsigned rw = *reinterpret_cast<volatile unsigned*>(&sm->room_wait);
          if (rw != 0u && (int)(rw >> 16) != w + 1) { smem_left -= (int)(rw & 0xFFu); tmem_left -= (int)((rw >> 8) & 0xFFu); }
        }
        unsigned feasible = 0;
        if (busy) feasible = (1u << N_CLASSES) - 1u;   // a tile claimed ahead waits for room when its worker takes it
        else
#pragma unroll 1
          for (unsigned m = cand; m != 0u; m &= m - 1u) {                // only the candidate classes are looked at
            const int c = __ffs((int)m) - 1;
            const int su = sm->smem_units[c], tu = sm->tmem_units[c];
            if (su <= smem_left && tu <= tmem_left && find_free(smask, su, sm->n_smem_units) >= 0 &&
                find_free((unsigned long long)tmask, tu, sm->n_tmem_units) >= 0)
              feasible |= 1u << c;
          }
        if ((cand & feasible) != 0u) {
          int phase;
          want = pick_choose(N_CLASSES, sm->tau_tab, sm->group_mask, cand, feasible, sm->pick, sm->pick.rr, ctx.policy, ctx.u_max, &phase,
                             sm->grid, sm->res);
        }
        if (want >= 0) {
          if (!busy) {                                   // promised until the worker has allocated (or the pop is lost)
            promised_s = sm->smem_units[want]; promised_t = sm->tmem_units[want];
            atomicAdd(&sm->smem_promised, promised_s); atomicAdd(&sm->tmem_promised, promised_t);
          }
          atomicAdd(&sm->pick.cta_count[want], 1);     // counted from the claim on, so the next lane sees it
          for (int x = 0; x < 3; ++x) atomicAdd(&sm->pick.u[x], sm->tau_tab[want * 3 + x]);
          sm->pick.rr = (want + 1) % N_CLASSES;
        }
      }
      if (__shfl_sync(0xffffffffu, want, w) >= 0) ++running;
    }
    // ---- the claims themselves run in parallel across lanes (global atomics); the warp then brings the claimed tiles' node
    // descriptions into their jobs, so that a worker finds all it needs in shared memory
    bool popped = false;
    int ji = 0;
    uint32_t node = 0;
    const unsigned same = __match_any_sync(0xffffffffu, want);      // lanes that want the same class claim together
    const int rank = __popc(same & ((1u << lane) - 1u)), first = __ffs((int)same) - 1;
    int got = 0;
    unsigned long long ticket = 0;
    if (want >= 0 && rank == 0) {
      // (a compare-and-swap on the head alone, one trip instead of two, collapses when many SMs want the same few tiles)
      const int n = __popc(same);
      TileQueue* q = ctx.queues + want;
      const long long old = (long long)atomicAdd(reinterpret_cast<unsigned long long*>(&q->avail), (unsigned long long)(-(long long)n));
      got = old <= 0 ? 0 : (int)min(old, (long long)n);
      if (got < n) atomicAdd(reinterpret_cast<unsigned long long*>(&q->avail), (unsigned long long)(n - got));
      if (got > 0) ticket = atomicAdd(&q->head, (unsigned long long)got);
    }
    got = __shfl_sync(0xffffffffu, got, first);
    ticket = __shfl_sync(0xffffffffu, ticket, first) + (unsigned long long)rank;
    if (want >= 0) {
      QueueEntry e;
      if (rank < got && queue_entry(ctx, want, ticket, e, now + ctx.wait_limit_ns)) {
        popped = true;
        ji = to_prio ? 2 + (int)(slot->prio_tail & 1u) : (int)(slot->held_tail & 1u);
        TileJob& h = slot->job[ji];
        node = (uint32_t)e & ((1u << QW_NODE_BITS) - 1u);
        h.node = node;
        const uint32_t inst = (uint32_t)(e >> QW_NODE_BITS) & ((1u << QW_INST_BITS) - 1u);
        h.inst = inst;
        h.tile = (uint32_t)(e >> (QW_NODE_BITS + QW_INST_BITS)) & ((1u << QW_TILE_BITS) - 1u);
        h.smem_units = (int)((e >> (QW_NODE_BITS + QW_INST_BITS + QW_TILE_BITS)) & ((1u << QW_SMEM_BITS) - 1u));
        h.tmem_units = (int)((e >> (QW_NODE_BITS + QW_INST_BITS + QW_TILE_BITS + QW_SMEM_BITS)) & ((1u << QW_TMEM_BITS) - 1u));
        h.cls = want;
        h.early = (int)((e >> (64 - QW_GEN_BITS - 1)) & 1u);
        h.promised_s = promised_s; h.promised_t = promised_t;
        h.held_at_claim = slot->held_tail;
        h.slot_base = __ldg(ctx.slot_base + inst);
        h.frame = ld_volatile_u64(reinterpret_cast<const unsigned long long*>(ctx.inst_frame + inst));
        h.gen = ld_volatile_u32(ctx.inst_gen + inst);
      } else {                                         // lost the race: undo the count
        atomicSub(&sm->pick.cta_count[want], 1);
        for (int x = 0; x < 3; ++x) atomicSub(&sm->pick.u[x], sm->tau_tab[want * 3 + x]);
        if (promised_s | promised_t) { atomicSub(&sm->smem_promised, promised_s); atomicSub(&sm->tmem_promised, promised_t); }
        lost = 1u << want;                             // look elsewhere in the next round, which follows at once
      }
    }
#pragma unroll 1
    for (unsigned m = __ballot_sync(0xffffffffu, popped); m != 0u; m &= m - 1u) {
      const int w = __ffs((int)m) - 1;
      const int4* src = reinterpret_cast<const int4*>(ctx.nodes + __shfl_sync(0xffffffffu, node, w));
      int4* dst = reinterpret_cast<int4*>(&sm->slot[w].job[__shfl_sync(0xffffffffu, ji, w)].desc);
      if (lane < (int)(sizeof(NodeDesc) / 16)) dst[lane] = __ldg(src + lane);
    }
    __syncwarp();
    if (popped) {
      __threadfence_block();
      if (to_prio) slot->prio_tail = slot->prio_tail + 1;
      else slot->held_tail = slot->held_tail + 1;      // the worker takes it as soon as it is free
      bell_ring(&sm->bell_worker[lane]);
      progressed = true;
    }
    // ---- admission, exit and watchdog (lane 0 decides)
    int verdict = 0;   // 1 = leave
    const unsigned cw = (unsigned)__shfl_sync(0xffffffffu, px, 16), err = (unsigned)(__shfl_sync(0xffffffffu, px, 16) >> 32);
    const unsigned stop = (unsigned)(__shfl_sync(0xffffffffu, py, 16) >> 32);
    const bool admissions = __shfl_sync(0xffffffffu, px, 17) < __shfl_sync(0xffffffffu, py, 17);
    if (err != 0u || stop != 0u || (cw & CTRL_EXITING)) verdict = 1;
    else if (lane == 0) {
      if (admissions) try_admit(ctx);
      if (cw == 0u && !admissions) {
        if (idle_start == 0) idle_start = now;
        else if (now - idle_start > ctx.idle_exit_ns) atomicCAS(&ctl->ctrl, 0u, CTRL_EXITING);
      } else {
        idle_start = 0;
      }
    }
    const bool any_progress = __any_sync(0xffffffffu, progressed || (serving && slot->busy != 0));
    if (any_progress) last_progress = now;
    else if (lane == 0 && !verdict && (iter & 63u) == 0 && now - last_progress > ctx.wait_limit_ns && cw != 0u) {
      set_error(ctx, DEV_ERR_IDLE_LIMIT, (unsigned)blockIdx.x);   // frames in flight, nothing moved for too long
      verdict = 1;
    }
    verdict = __shfl_sync(0xffffffffu, verdict, 0);
    if (verdict) leaving = true;
    if (leaving) {
      // stop claiming; once every worker is idle and nothing is posted, send them home
      const bool quiet = !serving || (slot->busy == 0 && slot->done_state == 0 && slot->held_tail == slot->held_head &&
                                      slot->prio_tail == slot->prio_head);
      if (__all_sync(0xffffffffu, quiet)) {
        if (serving) { __threadfence_block(); slot->leave = 1; bell_ring(&sm->bell_worker[lane]); }
        __syncwarp();
        if (lane == 0) { __threadfence_block(); sm->quit = 1; bell_ring(&sm->bell_retire); }
        break;
      }
    }
    if (!__any_sync(0xffffffffu, progressed || lost != 0u)) {
      // A free worker with nothing to run: poll the queues at short intervals (its scheduler slots are idle anyway).
      // Every worker busy: sleep until one of them rings (it took its claimed tile, or ran dry) or the hint runs out.
      const bool hungry = serving && slot->busy == 0 && slot->held_tail == slot->held_head && slot->prio_tail == slot->prio_head;
      if (__any_sync(0xffffffffu, hungry)) { __nanosleep(nap); if (nap < CLAIM_NAP_MAX_NS) nap += CLAIM_NAP_NS; }
      else { bell_wait(&sm->bell_claim, bell_parity, CLAIM_SLEEP_NS); nap = CLAIM_NAP_NS; }
    } else nap = CLAIM_NAP_NS;
  }
}

// The worker's threads after a tile body.
__device__ __forceinline__ void end_of_tile(const DeviceCtx& ctx, SmState* sm, WorkerSlot* slot) {
  unsigned tid;
  asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid));
  const int worker = (int)tid / WORKER_THREADS, wt = (int)tid % WORKER_THREADS;
  DoneTile d;
  if (wt == 32) {              // (read before the barrier: afterwards the leader moves on)
    const TileJob& j = slot->job[slot->run];
    d.inst = j.inst; d.node = j.node; d.tile = j.tile; d.cls = j.cls; d.gen = j.gen; d.frame = j.frame; d.t0 = slot->t_start;
    d.succ_begin = j.desc.succ_begin; d.succ_count = j.desc.succ_count; d.op = j.desc.op;
  }
  asm volatile("bar.sync %0, %1;" ::"r"(worker + 1), "r"(WORKER_THREADS) : "memory");
  // Two lanes share the end of a tile: lane 0 frees the tile's memory and goes straight on to take the next
  // tile, the first lane of warp 1 posts the finished one to the retire warp meanwhile (both meet again at the
  // barrier that opens the next tile).
  if (wt == 0) {
    atomicAdd(&ctx.control->tiles_done, 1ull);
    if (!slot->primed) {
      if (slot->verdict == 1) {
        if (slot->smem_units) atomicAnd(&sm->smem_mask, ~(unit_bits(slot->smem_units) << slot->smem_unit0));
        if (slot->tmem_units) atomicAnd(&sm->tmem_mask, ~(unsigned)(unit_bits(slot->tmem_units) << slot->tmem_unit0));
      }
      slot->busy = 0;
      if (slot->held_tail == slot->held_head && slot->prio_tail == slot->prio_head) bell_ring(&sm->bell_claim);   // out of work
    }
  } else if (wt == 32) {
    d.t1 = gtimer();
    unsigned naps = 0;
    while (slot->done_state != 0) {
      __nanosleep(40);
      if ((++naps & 0xFFFFu) == 0 && gtimer() - d.t1 > 2 * ctx.wait_limit_ns) break;   // retire warp gone: give up posting
    }
    slot->done = d;
    // The tile's writes (all threads, ordered by the barrier above) must be visible device-wide before any
    // successor is released.  That fence is the retire warp's (after it has read this flag): fences are cumulative, and
    // barrier -> block-scope fence -> flag -> device-scope fence
    // keeps the writes ahead of the counter atomics without a device-scope round trip on the worker's path.
    __threadfence_block();
    slot->done_state = 1;
    bell_ring(&sm->bell_retire);
    atomicSub(&sm->pick.cta_count[d.cls], 1);    // the pick's view of this SM, after the completion is on its way
    for (int x = 0; x < 3; ++x) atomicSub(&sm->pick.u[x], sm->tau_tab[d.cls * 3 + x]);
  }
}

// What an early tile of `job` waits for: its node's dependency word and the count that releases it in this frame.
__device__ __forceinline__ const unsigned long long* release_word(const DeviceCtx& ctx, const TileJob& job) {
  return ctx.dep_word + (size_t)job.inst * ctx.n_nodes + job.node;
}
__device__ __forceinline__ unsigned long long release_count(const TileJob& job) {
  return DEP_BIAS + (unsigned long long)(unsigned)job.desc.n_pred * job.gen;
}

// The worker's leader: waits for a tile the claim warp has put together, gives it its memory and fills in its context.
__device__ __forceinline__ void take_tile(const DeviceCtx& ctx, SmState* sm, WorkerSlot* slot, char* slab, int worker, int n_workers) {
  Control* ctl = ctx.control;
  TileCtx& tc = sm->tc[worker];
  bool prio = false;
  unsigned naps = 0;
  if (!slot->primed) {
    uint32_t bell_parity = slot->bell_parity;
    for (;;) {
      if (slot->prio_tail != slot->prio_head) {
        __threadfence_block();
        const TileJob& j = slot->job[2 + (int)(slot->prio_head & 1u)];
        if (priority_goes_first(j.early != 0, slot->held_head, j.held_at_claim) || released(release_word(ctx, j), release_count(j))) { prio = true; break; }
      }
      if (slot->held_tail != slot->held_head) break;
      if (slot->leave) { slot->verdict = 0; return; }
      if (naps < 8) __nanosleep(20);                               // a claimed tile is usually a moment away
      else bell_wait(&sm->bell_worker[worker], bell_parity, 2000u);
      ++naps;
    }
    slot->bell_parity = bell_parity;
  }
  __threadfence_block();
  const int ji = prio ? 2 + (int)(slot->prio_head & 1u) : (int)(slot->held_head & 1u);
  TileJob& job = slot->job[ji];
  const uint64_t now = gtimer(), lim = now + ctx.wait_limit_ns;
  slot->run = ji;
  slot->t_busy = now;
  slot->cls = job.cls;
  slot->busy = 1;
  __threadfence_block();
  if (prio) slot->prio_head = slot->prio_head + 1;
  else slot->held_head = slot->held_head + 1;   // the claim warp may fill the other job of the pair
  bell_ring(&sm->bell_claim);
  int early = job.early;
  bool ok = true;
  tc.cont = slot->primed;
  if (slot->primed) slot->primed = 0;           // memory and operand ring stay with the worker
  else {
    ok = false;
    if (early) {
      // A tile taken before its node's release may hold memory while it waits only where no tile taken earlier can
      // still need some, that is, where it is the only one this SM has taken.  Elsewhere it waits empty-handed.
      int taken = 0;
#pragma unroll 1
      for (int k = 0; k < N_CLASSES; ++k) taken += *reinterpret_cast<volatile int*>(&sm->pick.cta_count[k]);
      if (taken != 1) {
        tc.wait_word = release_word(ctx, job);
        tc.wait_count = release_count(job);
        tc.t_start = &slot->t_wait;
        tc.deadline = lim;
        wait_release(tc);
        early = 0;
      }
    }
    const int need_units = job.smem_units, tmem_units = job.tmem_units;
    int deep_units = 0;
    if (sm->outstanding <= 2 * (int)gridDim.x) {
      // Few tiles on the whole GPU: a GEMM tile takes the pipeline depth its K has use for, up to its share of the
      // SM.  A k-block then costs its share of many loads in flight instead of half or a quarter of a round trip.
      const int third = sm->n_smem_units / MAX_WORKERS;
      const int share = sm->outstanding <= (int)gridDim.x / 2 ? sm->n_smem_units : (sm->outstanding <= (int)gridDim.x ? 2 * third : sm->n_smem_units / 2);
      deep_units = min((job.desc.smem_deep + SMEM_UNIT - 1) / SMEM_UNIT, share);
    }
    // every worker has a home region (a third of the slab, a third of the columns): a tile that fits it goes
    // there whenever it is free, so tiles of the common shapes never fragment the slab; larger tiles and a
    // home occupied by one of them fall back to the first free run
    const int third_s = sm->n_smem_units / n_workers, third_t = sm->n_tmem_units / n_workers;
#pragma unroll 1
    for (unsigned spin = 0;; ++spin) {
      const unsigned long long sm_old = *reinterpret_cast<volatile unsigned long long*>(&sm->smem_mask);
      int units = need_units, s0 = -1;
      if (deep_units > need_units && (s0 = find_free(sm_old, deep_units, sm->n_smem_units)) >= 0) units = deep_units;
      else if (units <= third_s && ((sm_old >> (worker * third_s)) & unit_bits(units)) == 0ull) s0 = worker * third_s;
      else s0 = find_free(sm_old, units, sm->n_smem_units);
      if (s0 >= 0) {
        const unsigned long long sbits = unit_bits(units) << s0;
        if (units == 0 || atomicCAS(&sm->smem_mask, sm_old, sm_old | sbits) == sm_old) {
          const unsigned tm_old = *reinterpret_cast<volatile unsigned*>(&sm->tmem_mask);
          int t0 = -1;
          if (tmem_units <= third_t && ((tm_old >> (worker * third_t)) & (unsigned)unit_bits(tmem_units)) == 0u) t0 = worker * third_t;
          else t0 = find_free((unsigned long long)tm_old, tmem_units, sm->n_tmem_units);
          const unsigned tbits = (unsigned)(unit_bits(tmem_units) << (t0 < 0 ? 0 : t0));
          if (t0 >= 0 && (tmem_units == 0 || atomicCAS(&sm->tmem_mask, tm_old, tm_old | tbits) == tm_old)) {
            slot->smem_unit0 = s0; slot->smem_units = units; slot->tmem_unit0 = t0; slot->tmem_units = tmem_units;
            ok = true;
            break;
          }
          if (units) atomicAnd(&sm->smem_mask, ~sbits);   // no tensor memory yet: give the shared memory back
        }
      }
      if (spin == 0)        // waiting for room
        *reinterpret_cast<volatile unsigned*>(&sm->room_wait) =
            (unsigned)need_units | ((unsigned)tmem_units << 8) | ((unsigned)(worker + 1) << 16);
      __nanosleep(100);
      if ((spin & 255u) == 255u && (gtimer() > lim || ld_volatile_u32(&ctl->error) != 0u)) break;
    }
    if ((*reinterpret_cast<volatile unsigned*>(&sm->room_wait) >> 16) == (unsigned)(worker + 1))
      *reinterpret_cast<volatile unsigned*>(&sm->room_wait) = 0u;
    if (job.promised_s | job.promised_t) {     // the claim warp's promise of room is settled either way
      atomicSub(&sm->smem_promised, job.promised_s); atomicSub(&sm->tmem_promised, job.promised_t);
    }
    if (!ok) set_error(ctx, DEV_ERR_IDLE_LIMIT, 0x2000u + (unsigned)blockIdx.x);
    tc.smem = slab + (size_t)slot->smem_unit0 * SMEM_UNIT;
    tc.smem_bytes = slot->smem_units * SMEM_UNIT;
    tc.tmem = sm->tmem_base + (unsigned)slot->tmem_unit0 * TMEM_UNIT;
  }
  if (ok && (int)job.tile + 1 == job.desc.n_tiles) {   // the node's last tile: its successors may be queued
    while (slot->start_state != 0 && gtimer() < lim) __nanosleep(20);
    slot->start_inst = job.inst; slot->start_node = job.node;
    __threadfence_block();
    slot->start_state = 1;
    bell_ring(&sm->bell_retire);
  }
  slot->verdict = ok ? 1 : 2;
  job.early = early;
  tc.slot_base = job.slot_base;
  tc.inputs = ctx.input_ptrs + (size_t)job.inst * N_FRAME_INPUTS;
  tc.amap_base = ctx.n_weight_tmaps + (int)job.inst * ctx.n_act_tmaps;
  tc.deadline = lim;
  tc.wait_word = early ? release_word(ctx, job) : nullptr;
  tc.wait_count = release_count(job);
  tc.t_start = &slot->t_start;
}

// ------------------------------------------------------------------ the persistent co-scheduling kernel
// One CTA per SM: `workers` worker groups of WORKER_THREADS threads run tiles; of one more warpgroup two warps are the
// dispatcher (claim, retire), two only bring their registers.  Every wait is bounded by ctx.wait_limit_ns.
__global__ void __launch_bounds__(MAX_WORKERS* WORKER_THREADS + DISPATCH_THREADS, 1)
    vla_cosched_kernel(DeviceCtx ctx, int dyn_smem_bytes) {
  extern __shared__ __align__(1024) char smem_raw[];
  SmState* sm = reinterpret_cast<SmState*>(smem_raw);
  char* slab = smem_raw + SM_STATE_BYTES;
  const int n_workers = (blockDim.x - DISPATCH_THREADS) / WORKER_THREADS;
  const bool is_dispatcher = threadIdx.x >= n_workers * WORKER_THREADS;
  if (threadIdx.x == 0) {
    sm->smem_mask = 0;
    sm->tmem_mask = 0;
    int units = (dyn_smem_bytes - SM_STATE_BYTES) / SMEM_UNIT;
    sm->n_smem_units = units > 64 ? 64 : units;
    sm->n_tmem_units = 512 / TMEM_UNIT;
    for (int c = 0; c < PICK_MAX_CLASSES; ++c) sm->pick.cta_count[c] = 0;
    sm->pick.u[0] = sm->pick.u[1] = sm->pick.u[2] = 0;
    sm->pick.rr = (int)(blockIdx.x % N_CLASSES);
    sm->tmem_base = 0;
    sm->quit = 0;
    sm->smem_promised = 0; sm->tmem_promised = 0;
    sm->room_wait = 0u; sm->outstanding = 0;
    mbar_init(smem_u32(&sm->bell_claim), 1); mbar_init(smem_u32(&sm->bell_retire), 1);
    for (int w = 0; w < MAX_WORKERS; ++w) mbar_init(smem_u32(&sm->bell_worker[w]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    for (int c = 0; c < N_CLASSES; ++c) sm->ema_ns[c] = 30000;
    for (int c = 0; c < N_CLASSES; ++c)
    {
      for (int x = 0; x < 3; ++x) sm->tau_tab[c * 3 + x] = ctx.classes[c].tau[x];
      sm->smem_units[c] = ctx.classes[c].smem_units; sm->tmem_units[c] = ctx.classes[c].tmem_units; sm->grid[c] = 0;
      sm->res[c] = sm->smem_units[c] > 0 ? sm->smem_units[c] : 1;
      unsigned m = 0;
      for (int j = 0; j < N_CLASSES; ++j) m |= (ctx.classes[j].group == ctx.classes[c].group ? 1u : 0u) << j;
      sm->group_mask[c] = m;
    }
    for (int w = 0; w < MAX_WORKERS; ++w) {
      sm->slot[w].held_tail = 0; sm->slot[w].held_head = 0; sm->slot[w].leave = 0; sm->slot[w].done_state = 0;
      sm->slot[w].prio_tail = 0; sm->slot[w].prio_head = 0; sm->slot[w].t_busy = 0; sm->slot[w].start_state = 0;
      sm->slot[w].bell_parity = 0; sm->slot[w].busy = 0; sm->slot[w].primed = 0; sm->slot[w].room_wait = &sm->room_wait;
      TileCtx& tc = sm->tc[w];                           // what never changes
      tc.arena = ctx.arena; tc.ctl = smem_raw + SM_STATE_BASE + w * SM_CTL_BYTES; tc.bar_id = w + 1; tc.error = &ctx.control->error;
      tc.tmaps = ctx.tmaps; tc.n_weight_tmaps = ctx.n_weight_tmaps; tc.n_act_tmaps = ctx.n_act_tmaps;
      tc.slot = &sm->slot[w]; tc.drop_loads = 0;
    }
  }
  __syncthreads();
  if (threadIdx.x < 32) tmem_alloc(&sm->tmem_base, 512);   // the whole tensor memory of this SM, sub-allocated per tile
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (is_dispatcher) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(DISPATCH_REGS));
    const int warp = (int)(threadIdx.x - n_workers * WORKER_THREADS) >> 5;
    if (warp == 0) claim_loop(ctx, sm, n_workers);
    else if (warp == 1) retire_loop(ctx, sm, n_workers);
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(WORKER_REGS));
    // Nothing is carried in registers through a tile body (it has use for all of them): a pass of this loop derives its
    // place from the thread index again and keeps its few counters in the worker's slot.
    for (;;) {
      unsigned tid;
      asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid));
      const int worker = (int)tid / WORKER_THREADS, wt = (int)tid % WORKER_THREADS, bar_id = worker + 1;
      WorkerSlot* slot = sm->slot + worker;
      if (wt == 0) take_tile(ctx, sm, slot, slab, worker, n_workers);
      asm volatile("bar.sync %0, %1;" ::"r"(bar_id), "r"(WORKER_THREADS) : "memory");
      if (slot->verdict == 0) break;
      {
        const TileJob& job = slot->job[slot->run];
        const TileCtx& tc = sm->tc[worker];
        if (job.early && job.desc.op != OP_GEMM) {
          if (wt == 0) wait_release(tc);
          asm volatile("bar.sync %0, %1;" ::"r"(bar_id), "r"(WORKER_THREADS) : "memory");
        }
        if (wt == 32) {     // the retire warp will need the tile's successor records when it ends: into L1 now
          if (!job.early) slot->t_start = gtimer();
          asm volatile("prefetch.global.L1 [%0];" ::"l"(reinterpret_cast<const char*>(ctx.succ + job.desc.succ_begin)));
        }
        if (slot->verdict == 1) run_tile<false>(ctx, tc, job.desc, (int)job.tile, (int)job.inst, job.frame);
      }
      // Outputs written here by ordinary stores are read by TMA on other SMs.  The proxy fence that must lie between
      // the two in causality order is the consumer's (first statement of its TMA-issuing thread, after the
      // dependency was observed); a second one here cost 2 % of the throughput and is not needed.
      end_of_tile(ctx, sm, slot);
    }
  }
  // After a wait that ran out, copies may still be in flight: they land before the block's memory goes.  The host reads the
  // mirror of the error word; the waits inside tile bodies set the word only (registers are short there).
  if (ld_volatile_u32(&ctx.control->error) != 0u) {
    if (threadIdx.x == 0) mirror_error(ctx);
    for (int i = 0; i < 200; ++i) __nanosleep(1000);
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x < 32) tmem_dealloc(sm->tmem_base, 512);
}

// ------------------------------------------------------------------ one node as an ordinary kernel (CTA = tile)
__global__ void __launch_bounds__(WORKER_THREADS) vla_node_kernel(DeviceCtx ctx, const NodeDesc* nodes, int node_idx, int inst) {
  extern __shared__ __align__(1024) char smem_raw[];
  __shared__ uint32_t tmem_base_s;
  __shared__ __align__(16) char ctl_block[1024];
  const NodeDesc& n = nodes[node_idx];
  uint32_t tmem_cols = 0;
  if (n.tmem_cols > 0) {
    tmem_cols = 32;
    while ((int)tmem_cols < n.tmem_cols) tmem_cols <<= 1;
    if (threadIdx.x < 32) tmem_alloc(&tmem_base_s, tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
  }
  TileCtx tc;
  tc.arena = ctx.arena;
  tc.slot_base = inst >= 0 ? ctx.slot_base[inst] : 0;
  tc.smem = smem_raw;
  tc.smem_bytes = n.smem_bytes;
  tc.ctl = ctl_block;
  tc.tmem = tmem_cols ? tmem_base_s : 0;
  tc.bar_id = 1;
  tc.error = &ctx.control->error;
  tc.tmaps = ctx.tmaps;
  tc.inputs = ctx.input_ptrs + (size_t)(inst >= 0 ? inst : 0) * N_FRAME_INPUTS;
  tc.amap_base = ctx.n_weight_tmaps + (inst >= 0 ? inst : 0) * ctx.n_act_tmaps;
  tc.drop_loads = ctx.drop_loads;
  tc.wait_word = nullptr;
  tc.slot = nullptr;
  tc.cont = 0;
  const uint64_t t0 = gtimer();
  tc.deadline = t0 + ctx.wait_limit_ns;
  const uint64_t frame = inst >= 0 ? ctx.inst_frame[inst] : 0;
  run_tile<true>(ctx, tc, n, (int)blockIdx.x, inst, frame);
  if (threadIdx.x == 0 && gtimer() > tc.deadline && ld_volatile_u32(&ctx.control->error) != 0u) mirror_error(ctx);   // a wait ran out
  if (inst >= 0 && ctx.trace_capacity) {
    asm volatile("bar.sync 1, %0;" ::"r"(WORKER_THREADS) : "memory");
    if (threadIdx.x == 0) write_trace(ctx, (uint32_t)inst, (uint32_t)node_idx, blockIdx.x, 0, n.cls, frame, t0, gtimer());
  }
  if (tmem_cols) {
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x < 32) tmem_dealloc(tmem_base_s, tmem_cols);
  }
}

// ------------------------------------------------------------------ pick probe (tests)
__global__ void vla_pick_probe_kernel(int n_cls, const int* tau, unsigned pending, unsigned feasible, PickState* st,
                                      int rr_start, int policy, int u_max, const int* grid, const int* res, int* out) {
  int phase;
  unsigned group_mask[PICK_MAX_CLASSES];
  for (int i = 0; i < PICK_MAX_CLASSES; ++i) group_mask[i] = 1u << i;   // one class per group: the paper's listing
  int k = pick_choose(n_cls, tau, group_mask, pending, feasible, *st, rr_start, policy, u_max, &phase, grid, res);
  if (k >= 0) pick_commit(*st, k, tau);
  out[0] = k;
  out[1] = phase;
}

}  // namespace vla
