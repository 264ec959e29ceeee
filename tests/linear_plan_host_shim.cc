// Host build of the linear layer's tile plan for the CPU tests.
#include "../paper_2609_22335_b200/csrc/linear_plan.h"

// clusters of four CTAs as a B200 answers, and not known
static vla::LinearRoom room(int sms) { return sms == 148 ? vla::LinearRoom{33, 71} : vla::LinearRoom{0, 0}; }

extern "C" void linear_plan_host(int m, int n, int k, int f32, int sms, int* out /*[6]: bm, bn, ks, tiles_m, tiles, stages*/) {
  const vla::LinearPlan p = vla::linear_plan(m, n, k, f32 != 0, sms, room(sms));
  out[0] = p.bm; out[1] = p.bn; out[2] = p.ks; out[3] = p.tiles_m; out[4] = p.tiles; out[5] = p.stages;
}
extern "C" void linear_pair_plan_host(int m, int n, int k, int f32, int sms, int* out /*[5]: bm, bn, tiles_m, tiles, stages*/) {
  const vla::LinearPlan p = vla::linear_plan(m, n, k, f32 != 0, sms, room(sms));
  const vla::LinearPairPlan q = vla::linear_pair_plan(m, n, k, p, sms);
  out[0] = q.bm; out[1] = q.bn; out[2] = q.tiles_m; out[3] = q.tiles; out[4] = q.stages;
}
