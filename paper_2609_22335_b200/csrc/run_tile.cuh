// Which body runs a tile of a node.  Included behind the bodies (tiles.cuh); the CPU tests include it behind stand-ins.
#pragma once

namespace vla {

// LOAD_TIME: also the operations of the load-time constant program (sincosf's slow path is not code to keep in a kernel
// whose tile bodies compete for the instruction cache).  An operation that the kernel does not have is an error.
template <bool LOAD_TIME>
__device__ __forceinline__ void run_tile(const DeviceCtx& ctx, const TileCtx& c, const NodeDesc& n, int tile, int inst,
                                         uint64_t frame) {
  switch (n.op) {
    case OP_GEMM: tile_gemm(c, n.u.gemm, tile); break;
    case OP_RMSNORM: tile_rmsnorm(c, n.u.norm, tile); break;
    case OP_ATTN: tile_attention(c, n.u.attn, tile); break;
    case OP_PATCHIFY: tile_patchify(c, n.u.patch, tile); break;
    case OP_EMBED: tile_embed(c, n.u.embed, tile); break;
    case OP_ADDROWS: tile_addrows(c, n.u.addrows, tile); break;
    case OP_EMIT:
    case OP_EMIT_PART:
      tile_emit(c, n.u.emit, ctx.chunk_host + (size_t)inst * ctx.chunk_elems, ctx.done_host + inst, frame, n.op == OP_EMIT);
      break;
    case OP_TIMEEMB:
      if constexpr (LOAD_TIME) { tile_timeemb(c, n.u.timeemb, tile); break; }
      [[fallthrough]];
    default:
      if (worker_tid() == 0) set_error(ctx, DEV_ERR_BAD_OP, (unsigned)n.op);
  }
}

}  // namespace vla
