// Launch shape of a stand-alone attention call (op_attention.cuh): plain arithmetic, compiled for the host in the CPU tests too.
#pragma once
#include "vla_types.h"

namespace vla {

constexpr int ATTN_BQ = 128;   // queries per tile (MMA M)
constexpr int ATTN_BN = 64;    // keys per block (MMA N of S, MMA K of P V; one 128-byte swizzle row of P)
constexpr int OPA_MAX_S = 3;             // score buffers
constexpr int OPA_MAX_SPLIT = 8;         // CTAs of a cluster
constexpr int OPA_MAX_SMEM = 208 * 1024;
constexpr int OPA_MAX_STAGES = 4;

struct OpAttnLaunch { int split, stages, smem, tmem_cols, s_bufs, terms; };   // (terms: bf16 numbers that a probability is given in)

inline int opa_smem(int hs, int stages) {
  const int nbox = (hs + 63) / 64;
  return nbox * (128 * 128 + stages * 2 * 64 * 128);
}
inline bool opa_split_fits(int s, int hs, int blocks, int smem) {
  return s <= blocks && (hs / 16 + s - 1) / s * s * 8192 <= smem;                 // (the partial rows meet in the stages)
}
// Parts of the keys that a call needs if a probability is one bf16 number.  Each part has a maximum of its own, whose probability of 1 is
// exact, so fewer parts round more (87 x 956, 36 heads of 128: rel-L2 2.0e-3 in eight parts, 2.2e-3 in three; the result's own rounding
// alone 1.65e-3).  Powers of two up to two CTAs per SM (one above a head width of 128) are what the operator's precision is stated for.
inline int opa_min_parts(int tiles, int hs, int blocks, int smem, int sms) {
  const int per_sm = hs <= 128 ? 2 : 1;
  int s = 1;
  while (s < OPA_MAX_SPLIT && (long long)tiles * s * 2 <= (long long)per_sm * sms && opa_split_fits(2 * s, hs, blocks, smem)) s *= 2;
  return s;
}
// The split of the keys is the one with the least estimated time, in units of a key block of a CTA that has its SM to itself (0.7 us
// up to a head width of 128, 1.05 at 256): its CTAs' blocks, 1.55 times that where two share an SM (up to a width of 128), 7 for a call
// and 4 for every further wave, 1.8 (3 above 128) for meeting in the cluster.  `clusters[s]`: clusters of s CTAs the chip holds, one CTA per SM -- from
// three CTAs on a cluster is not given an SM that has one already (288 CTAs in clusters of three take two waves, in pairs one).
// Fitted to 60 shapes of 16..2048 queries and keys with every split timed: the split chosen is at most 6 % behind the best.  (Powers of
// two up to the chip's two CTAs per SM: 725 x 687, 12 heads of 128, 19.6 us split four ways and 12.2 two ways; 87 x 956, 36 heads over 12
// of 128, 20.6 eight and 10.7 three ways.)
// A split into fewer parts than opa_min_parts takes its probabilities in two terms, which costs a block 0.16 more (0.12 above 128, 0.35
// where two CTAs share an SM): 87 x 956 in three parts 9.9 -> 10.8 us, 725 x 687 in two 11.4 -> 12.5, 1024 x 1024 of 12 heads of 64 in two 13.6 -> 15.7.
inline OpAttnLaunch opa_plan(int tiles, int tkv, int hs, int sms, const int* clusters) {
  OpAttnLaunch p;
  const int per_sm = hs <= 128 ? 2 : 1, budget = per_sm == 2 ? OPA_MAX_SMEM / 2 : OPA_MAX_SMEM, blocks = (tkv + 63) / 64;
  p.stages = OPA_MAX_STAGES;
  while (p.stages > 2 && opa_smem(hs, p.stages) > budget) --p.stages;
  p.smem = opa_smem(hs, p.stages);
  p.split = 1; p.terms = 1;
  const int min_parts = opa_min_parts(tiles, hs, blocks, p.smem, sms);
  double best = 1e300;
  for (int s = 1; s <= OPA_MAX_SPLIT; ++s) {
    if (!opa_split_fits(s, hs, blocks, p.smem)) continue;
    const long long ctas = (long long)tiles * s, room = s > 2 ? (long long)clusters[s] * s : (long long)per_sm * sms;
    const long long waves = room > 0 ? (ctas - 1) / room + 1 : ctas;
    const bool shared = per_sm == 2 && s <= 2 && ctas > sms;
    const double block = (shared ? 1.55 : 1.0) + (s >= min_parts ? 0.0 : (shared ? 0.35 : (hs <= 128 ? 0.16 : 0.12)));
    const double t = (double)waves * ((blocks + s - 1) / s * block + 4.0) + 3.0 + (s == 1 ? 0.0 : (hs <= 128 ? 1.8 : 3.0));
    if (t < best) { best = t; p.split = s; p.terms = s >= min_parts ? 1 : 2; }
  }
  p.tmem_cols = hs <= 128 ? 256 : 512;
  p.s_bufs = (p.tmem_cols - hs) / ATTN_BN < OPA_MAX_S ? (p.tmem_cols - hs) / ATTN_BN : OPA_MAX_S;
  return p;
}

}  // namespace vla
