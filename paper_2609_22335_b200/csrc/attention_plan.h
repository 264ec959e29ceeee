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
// Clusters of s CTAs that the chip holds, s = 1 .. 8: one CTA per SM, and two (0: not known).
struct OpRoom { int alone[OPA_MAX_SPLIT + 1], two[OPA_MAX_SPLIT + 1]; };
// The split of the keys is the one with the least estimated time, in units of a key block of a CTA that has its SM to itself (0.7 us
// up to a head width of 128, 1.05 at 256): its CTAs' blocks, 1.05 + 0.28 width / 128 times that where there are more CTAs than one per SM, 5
// (6) for a wave's set-up, 1.2 (2.4; 2.4 above 128 too) for meeting in the cluster.  A wave is what runs at once; causal waves but the last
// cost 0.57 of their longest CTA, since the next ones start as the short ones end.  Clusters of any size get two CTAs an SM, but whole
// clusters have to fit the chip's parts (148 SMs: 284 CTAs in clusters of four, 264 of eight).
// Fitted to 162 shapes of 1..2048 queries and 65..2048 keys with every split timed: 0.6 % behind the best of them on average, and none more than
// 5 % behind the largest power of two that the chip has room for.  (With one CTA per SM counted for clusters of three and more, and all causal
// waves at their longest: 687 x 687 causal, 64 heads over 32 of 80, in two parts 30 us, whole 22; 582 x 1908, 12 heads of 64, in two 18.3, in four 14.1.)
// A split into fewer parts than opa_min_parts takes its probabilities in two terms, which costs a block 0.16 more (0.11 above 128, 0.35
// where two CTAs share an SM): 87 x 956 in three parts 9.9 -> 10.8 us, 725 x 687 in two 11.4 -> 12.5, 1024 x 1024 of 12 heads of 64 in two 13.6 -> 15.7.
inline OpAttnLaunch opa_plan(int tiles, int tkv, int hs, bool causal, int sms, const OpRoom& room) {
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
    const long long ctas = (long long)tiles * s, alone = s > 2 ? (long long)room.alone[s] * s : sms;
    const long long at_once = s > 2 ? (long long)(per_sm == 2 ? room.two[s] : room.alone[s]) * s : (long long)per_sm * sms;
    const long long waves = at_once > 0 ? (ctas - 1) / at_once + 1 : ctas;
    const bool shared = per_sm == 2 && ctas > alone;
    const double block = (shared ? 1.05 + 0.28 / 128 * hs : 1.0) + (s >= min_parts ? 0.0 : (shared ? 0.35 : (per_sm == 2 ? 0.16 : 0.11)));
    const double over = (shared ? 6.0 : 5.0) + (s == 1 ? 0.0 : (shared || per_sm == 1 ? 2.4 : 1.2)), chain = (blocks + s - 1) / s * block;
    const double t = (double)(waves - 1) * ((causal ? 0.57 : 1.0) * chain + over) + chain + over;
    if (t < best) { best = t; p.split = s; p.terms = s >= min_parts ? 1 : 2; }
  }
  p.tmem_cols = hs <= 128 ? 256 : 512;
  p.s_bufs = (p.tmem_cols - hs) / ATTN_BN < OPA_MAX_S ? (p.tmem_cols - hs) / ATTN_BN : OPA_MAX_S;
  return p;
}

}  // namespace vla
