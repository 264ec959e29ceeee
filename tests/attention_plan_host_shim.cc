// Host build of the stand-alone attention's launch plan for the CPU tests.
#include "../paper_2609_22335_b200/csrc/attention_plan.h"

extern "C" void attention_plan_host(int tiles, int tkv, int hs, int causal, int sms, const int* alone, const int* two,
                                    int* out /*[7]: split, stages, smem, tmem_cols, s_bufs, terms, min parts*/) {
  vla::OpRoom room;
  for (int s = 0; s <= vla::OPA_MAX_SPLIT; ++s) { room.alone[s] = alone[s]; room.two[s] = two[s]; }
  const vla::OpAttnLaunch p = vla::opa_plan(tiles, tkv, hs, causal != 0, sms, room);
  out[0] = p.split; out[1] = p.stages; out[2] = p.smem; out[3] = p.tmem_cols; out[4] = p.s_bufs; out[5] = p.terms;
  out[6] = vla::opa_min_parts(tiles, hs, (tkv + 63) / 64, p.smem, sms);
}
