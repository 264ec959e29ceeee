// Host build of the switch over a tile's operation (csrc/run_tile.cuh) with stand-ins for the bodies, for the CPU tests.
#include <cstddef>
#include <cstdint>

#define __device__
#define __forceinline__ inline
#include "../paper_2609_22335_b200/csrc/vla_types.h"

namespace vla {

struct TileCtx {};
static int ran;              // operation whose body ran, -1 none
static unsigned error_code;

inline int worker_tid() { return 0; }
inline void set_error(const DeviceCtx&, unsigned code, unsigned) { error_code = code; }
#define BODY(name, Args, op) inline void name(const TileCtx&, const Args&, int) { ran = op; }
BODY(tile_gemm, GemmArgs, OP_GEMM)
BODY(tile_rmsnorm, NormArgs, OP_RMSNORM)
BODY(tile_attention, AttnArgs, OP_ATTN)
BODY(tile_patchify, PatchArgs, OP_PATCHIFY)
BODY(tile_embed, EmbedArgs, OP_EMBED)
BODY(tile_addrows, AddRowsArgs, OP_ADDROWS)
BODY(tile_timeemb, TimeEmbArgs, OP_TIMEEMB)
inline void tile_emit(const TileCtx&, const EmitArgs&, float*, DoneRec*, uint64_t, bool last) { ran = last ? OP_EMIT : OP_EMIT_PART; }

}  // namespace vla

#include "../paper_2609_22335_b200/csrc/run_tile.cuh"

extern "C" int run_tile_host(int load_time, int op, unsigned* error) {
  vla::DeviceCtx ctx = {};
  vla::TileCtx c;
  vla::NodeDesc n = {};
  n.op = op;
  vla::ran = -1;
  vla::error_code = 0;
  if (load_time) vla::run_tile<true>(ctx, c, n, 0, 0, 0);
  else vla::run_tile<false>(ctx, c, n, 0, 0, 0);
  *error = vla::error_code;
  return vla::ran;
}
