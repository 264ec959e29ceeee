// Tile shape of a stand-alone linear layer (op_linear.cuh): plain arithmetic, compiled for the host in the CPU tests too.
#pragma once
#include "vla_types.h"

namespace vla {

constexpr int LIN_MAX_STAGES = 12;
constexpr int LIN_SMEM = 110 * 1024;          // half an SM

struct LinearPlan {
  int bm, bn, ks, tiles_m, tiles, stages;   // tokens and features of a tile, CTAs that share its K, tiles, pipeline depth
  double cost;                              // estimated cycles
};

// (Every call of the operator pays for this arithmetic, and divisions are most of it: bm and bn are multiples of 16, so what is
// divided by them comes from tables.)
struct LinearTables {
  int stages[25] = {};            // by (bm + bn) / 16
  uint64_t recip[17] = {};        // by j: x * recip >> 36 = x / j for x below 2^32
  constexpr LinearTables() {
    for (int i = 2; i <= 24; ++i) {
      const int stage = i * 16 * GEMM_BK * 2, tail = stage < 16384 ? 16384 - stage : 0;       // the MMA always reads 128 rows
      const int s = (LIN_SMEM - tail) / stage;
      stages[i] = s > LIN_MAX_STAGES ? LIN_MAX_STAGES : s;
    }
    for (int j = 1; j <= 16; ++j) recip[j] = ((1ull << 36) + j - 1) / j;
  }
};
constexpr LinearTables kLinearTables;
inline int linear_stages(int bm, int bn) { return kLinearTables.stages[(bm + bn) >> 4]; }
inline long long linear_tiles_n(int n, int bn) {                              // features / bn, rounded up
  return (long long)(((uint64_t)((unsigned)(n - 1) >> 4) * kLinearTables.recip[bn >> 4]) >> 36) + 1;
}
// Whether a cluster of `ks` CTAs can share the K range of a tile of `bn` features: each finishes a whole number of 32-column
// groups, and the others' partial sums of those have to fit its stages.
inline bool linear_split_fits(int bm, int bn, int ks, int nkb) {
  return ks == 1 || ((bn & (bn - 1)) == 0 && bn >= 32 * ks && nkb >= 2 * ks &&
                     128 * (bn / ks) * (ks - 1) * 4 <= linear_stages(bm, bn) * (bm + bn) * GEMM_BK * 2);
}
// Clusters of four CTAs that run at once with an SM to each CTA, and with two CTAs to an SM, as the driver answers (0: not known; 33 and 71 on
// 148 SMs, since whole clusters have to fit the chip's parts).
struct LinearRoom { int alone, two; };
// Split of a call with fp32 results, and the width that goes with it.  A split shortens the tensor core's sums (K = 4096: rel-L2
// 2.4e-6 for 5.1e-6), which shows in fp32 and vanishes in bf16; so here it is not traded for the time that a width without one
// gains.  An estimate over powers of two: per k-block max(operand bytes over 47 B/clk, MMA issue) cycles for a CTA alone on its
// SM, max(2 x bytes over 90 B/clk, 2 x MMA) beside another one, a round trip and an epilogue per tile, an exchange per split.
inline void linear_split_f32(LinearPlan& g, int n, int k, int nkb, int sms, int fours) {
  double best = 1e300;
  for (int bn = 256; bn >= 16; bn >>= 1)
    for (int ks = 1; ks <= 8; ks <<= 1) {
      const long long ctas = g.tiles_m * linear_tiles_n(n, bn) * ks, rounds = ctas <= 2 * sms ? 1 : (ctas - 1) / (2 * sms) + 1;
      if (!linear_split_fits(g.bm, bn, ks, nkb) || (ks > 1 && ctas > 2 * sms)) continue;         // (a split tile is a cluster of its own)
      const double bytes = (double)(g.bm + bn) * GEMM_BK * 2, mma = bn <= 64 ? 200 : 2.0 * bn;
      const double kb = ctas > sms ? (2 * bytes / 90 > 2 * mma ? 2 * bytes / 90 : 2 * mma) : (bytes / 47 > mma ? bytes / 47 : mma);
      const double t = (double)(rounds * ((nkb + ks - 1) / ks)) * kb + (bn <= 128 ? 1 : rounds) * (1500 + 16.0 * bn / ks) + (ks > 1 ? 2500 + 8.0 * bn : 0);
      if (t < best) { best = t; g.bn = bn; g.ks = ks; }
    }
  if (g.ks > 1) {     // what it really takes, for the choice between the kernels: two CTAs of an SM get 52 B/clk, 45 where rows start in
                      // the middle of a 32-byte sector and with clusters of four, a CTA alone as many as it asks for
    const long long ctas = g.tiles_m * linear_tiles_n(n, g.bn) * g.ks, room = g.ks == 4 ? fours : 2 * sms;
    const double bytes = (double)(g.bm + g.bn) * GEMM_BK * (k % 16 == 0 ? 2.0 : 2.3), mma = g.bn <= 64 ? 200 : 2.0 * g.bn;
    const double beside = (2 * bytes / 52 > 2 * mma ? 2 * bytes / 52 : 2 * mma) * (g.ks == 4 ? 1.15 : 1.0), alone = bytes / 120 > mma ? bytes / 120 : mma;
    const int steps = (nkb + g.ks - 1) / g.ks;
    const double over = 7000 + 16.0 * g.bn / g.ks + 8.0 * g.bn;
    g.cost = (g.ks == 4 ? 6300 : 1000) + 1.05 * (over + steps * (ctas > sms ? beside : alone) + (ctas > room ? over + steps * alone : 0));     // (the few clusters that start late have the chip to themselves)
  }
}
// Tile width and K split of a call: the pair with the least estimated time.  A k-block of a tile costs a CTA that has its SM to
// itself max(400, 4 x width, 2600 / stages) cycles -- issue, MMA with its operands, a load's round trip -- and two on an SM
// twice the first two, or the time of their operands at 58 B/clk (42 where K is no multiple of 64: rows then straddle 128-byte
// lines; 39 where it is none of 16, and every other row starts in the middle of a 32-byte sector, 34 where two stages have to
// hide that).  A tile adds its epilogue (behind the next tile's main loop where there are two accumulators), a split its exchange.
// Where more clusters of four are asked for than the chip has room for, the call takes the last ones' time alone on their SMs as well; 256-wide
// tiles share SMs from 104 CTAs on, not from 132.
// Fitted to 280 shapes of 1..8192 x 7..16384 x 64..12288 with every width and split timed: the pair chosen is 1.8 % behind the
// best one on average, more than 10 % behind on 20, 24 % at most.  (By the estimate above, with powers of two alone up to the
// chip's two CTAs per SM: 8 %, 87 shapes, 83 %; 3455 x 1392 x 8448 100 us at width 256 and 71 at 144, 653 x 7782 x 2248 with GELU
// 96 and 60, 91 x 9152 x 1344 with its K split four ways 1.8 times the 64-wide tiles that need no split.)
inline LinearPlan linear_plan(int m, int n, int k, bool f32, int sms, const LinearRoom& room) {
  LinearPlan g;
  g.tiles_m = (m - 1) / 128 + 1;
  g.bm = ((m - 1) / g.tiles_m / 16 + 1) * 16;
  g.bn = 16; g.ks = 1; g.cost = 0;
  const int nkb = (k - 1) / GEMM_BK + 1, fours = room.two > 0 ? 4 * room.two : 2 * sms, lone_fours = room.alone > 0 ? 4 * room.alone : sms;
  if (f32) linear_split_f32(g, n, k, nkb, sms, fours);
  if (g.ks == 1) {
    const double operand_rate = k % GEMM_BK == 0 ? 2.0 / 58 : (k % 16 == 0 ? 2.0 / 42 : 2.0 / 39);      // cycles a byte of two CTAs' operands takes
    double best = 1e300;
    for (int ks = 1, shift = 0; ks <= (f32 ? 1 : 8) && nkb >= ks; ks <<= 1, ++shift)
      for (int bn = ks == 1 ? 16 : 32 * ks; bn <= 256 && (ks > 1 || bn < n + 16); bn += ks == 1 ? 16 : bn) {       // (of equals the narrowest)
        const long long ctas = g.tiles_m * linear_tiles_n(n, bn) * ks;
        if (!linear_split_fits(g.bm, bn, ks, nkb) || (ks > 1 && ctas > 2 * sms)) continue;
        const long long rounds = ctas <= 2 * sms ? 1 : (ctas - 1) / (2 * sms) + 1;
        const double own = bn > 100 ? 4.0 * bn : 400.0, slow = k % 16 != 0 && linear_stages(g.bm, bn) == 2 ? 1.15 : 1.0;
        const double operands = (g.bm + bn) * GEMM_BK * 2 * operand_rate * slow;
        double kb = 2 * own > operands ? 2 * own : operands;
        const bool beside = ctas > (ks < 4 ? sms : (bn < 256 ? lone_fours : sms - sms * 3 / 10));
        if (!beside) {
          const double trip = 2600.0 / linear_stages(g.bm, bn);
          kb = own > trip ? own : (trip < kb ? trip : kb);
        }
        double t = (double)(rounds * ((nkb + ks - 1) >> shift)) * kb + (bn <= 128 ? 1 : rounds) * 2400.0 + (ks == 1 ? 0 : 50.0 * bn + (ks == 4 && beside ? 600.0 : 0));
        if (ks > 2 && ctas > fours) t += ((nkb + ks - 1) >> shift) * own + 2400.0;
        if (t < best) { best = t; g.bn = bn; g.ks = ks; }
      }
    g.cost = best;
  }
  g.tiles = (int)(g.tiles_m * linear_tiles_n(n, g.bn));
  g.stages = linear_stages(g.bm, g.bn);
  return g;
}


// The same call as tiles of two SMs (op_linear_pair.cuh): bm tokens and half of bn features a CTA; bn = 0 where the plan above is
// the faster one.  Under 129 tokens one of the CTAs would idle.  A split of K becomes as many accumulators in tensor memory, so that
// sums stay as short as they were.  A k-block of a pair's tile costs max(560, its CTA's operands at 43 B/clk), a tile 600 cycles more and its
// whole epilogue where tensor memory has no room for a second set of accumulators, and a call 6800 more than the other kernel's (9500 where
// that one splits K): two CTAs have to meet, and the last epilogue stands alone.
// Fitted to 2104 shapes of 1..8192 x 7..16384 x 64..12288, most of them near the line between two choices, with every width and split of both
// kernels timed: the choice is 1.6 % behind the best one on average for bf16 results and 0.5 % for fp32 (0.62 to 0.99 of the other kernel's time
// where it goes this way: 2077 x 4944 x 7144 227 -> 145 us, 4096 x 4096 x 4096 114 -> 96, 8192 x 3072 x 768 40 -> 35; fp32 with a split 2997 x 731 x 1200
// 31 -> 15, 452 x 6648 x 6024 84 -> 51).  With k-blocks from 350 cycles on, clusters of four counted for one CTA per SM and their waves for whole ones,
// 214 of the 2104 were more than 5 % slower than the other kernel or a wider split, by up to half: 4390 x 149 x 6736 fp32 38 for 26 us, 2330 x 1891 x 8768 fp32 95 for 75,
// 948 x 786 x 6656 28 for 21.
constexpr int LINP_SMEM = 224 * 1024;         // a CTA of a pair has its SM to itself
struct LinearPairPlan { int bm, bn, tiles_m, tiles, stages; };
inline LinearPairPlan linear_pair_plan(int m, int n, int k, const LinearPlan& single, int sms) {
  LinearPairPlan g = {0, 0, 0, 0, 0};
  const int parts = single.ks, widest = parts <= 2 ? 256 : 512 / parts;
  const double more = parts == 1 ? 6800.0 : 9500.0;
  if (m <= 128 || n <= 112 || sms < 2 || widest < 128 || single.cost <= more) return g;
  g.tiles_m = (m - 1) / 256 + 1;
  g.bm = ((m - 1) / (2 * g.tiles_m) / 16 + 1) * 16;
  const int nkb = (k - 1) / GEMM_BK + 1, pairs = sms / 2;
  double best = 0.95 * (single.cost - more);       // (a margin: the two estimates err by as much)
  for (int bn = 128; bn <= widest && bn < n + 16; bn += 16) {
    const long long tiles = g.tiles_m * linear_tiles_n(n, bn), rounds = tiles <= pairs ? 1 : (tiles - 1) / pairs + 1;
    const double operands = (g.bm + bn / 2) * GEMM_BK * 2 / 43.0;
    const double loop = nkb * (operands > 560.0 ? operands : 560.0) + 600.0, least = 350.0 * nkb + 2000.0;
    const double t = (double)rounds * ((loop > least ? loop : least) + (2 * parts * bn <= 512 ? 0.0 : 2200.0 + 10.0 * bn));
    if (t < best) { best = t; g.bn = bn; g.tiles = (int)tiles; }
  }
  if (g.bn > 0) {     // (behind the start of the last stage there are the 16 KB that the MMA reads of any token tile)
    const int stage = (g.bm + g.bn / 2) * GEMM_BK * 2, s = (LINP_SMEM - 16384) / stage;
    g.stages = s > LIN_MAX_STAGES ? LIN_MAX_STAGES : s;
  }
  return g;
}

}  // namespace vla
