// Launch geometry of kernel 1 (quantize_kernel.cuh): what a CTA covers, its shared memory, and the plan that divides a call's
// rows and groups among CTAs.  Plain C++, no CUDA types.
#pragma once

#include <stddef.h>
#include <stdint.h>

namespace w4a4 {

constexpr int kQuantWarps = 8;                               // element-wise warps at most
constexpr int quantize_rows(int steps, int warps = kQuantWarps) { return 4 * warps * steps; }
constexpr int quantize_threads(int R, int warps = kQuantWarps) { return 32 * (warps + (R > 0 ? 1 : 0)); }
constexpr int kL1Stages = 3, kXhBuffers = 2;
constexpr uint32_t xh_tile_bytes(int steps, int warps) { return quantize_rows(steps, warps) * 128u; }   // rows x 64 channels in BF16

// One stage of the activation ring: what the element-wise warps read for one group, 16 bytes per lane and step and the
// group's 64 reciprocals once per warp.
constexpr uint32_t x_stage_bytes(int steps, int warps) { return warps * (steps * 512u + 256u); }
constexpr int kXStages(int R, int steps) { return steps == 2 ? (R >= 96 ? 3 : 4) : (R == 0 ? 5 : (R <= 64 ? 3 : 2)); }

// Dynamic shared memory: alignment slack, L1 ring, x_hat tiles, activation ring (and what the 128-row operand reads behind
// the last x_hat tile), and in a K-split launch this CTA's share of all partial sums of T.
constexpr uint32_t x_ring_bytes(int R, int steps, int warps) {
  const uint32_t ring = kXStages(R, steps) * x_stage_bytes(steps, warps), behind = 128 * 128 - xh_tile_bytes(steps, warps);
  return R == 0 || ring > behind ? ring : behind;
}
constexpr size_t quantize_smem_bytes(int R, int steps, int warps, int splits) {
  return (R == 0 ? 0 : 1024 + kL1Stages * R * 128 + kXhBuffers * xh_tile_bytes(steps, warps)) + x_ring_bytes(R, steps, warps) +
         (splits > 1 ? (quantize_rows(steps, warps) + splits) * R * 4 : 0);
}

// How a launch divides M rows x G groups.  fitting_clusters[k], k <= 8, and wide_clusters: clusters of k and of kMaxKSplits CTAs
// that run at a time, one CTA to an SM, as the device answers (0: such a cluster cannot be launched there).
// `image`: bytes of an INT4 layer's weight image, which its forwards expand in this launch and whose codes take longer (0: MXFP4).
// With a low-rank branch every launch for a layer has the same K split, also one without the expansion (a stage called alone, a
// search's later candidates, later chunks of a host forward): the split is the summation order of T, and the same rows have to
// give the same bits.  (Without an expansion 1560 x 5120, r = 32, takes 14.2 us with it and 12.9 with one of its own, a search of
// 12 forwards 1194 and 1173.)
struct QuantizePlan {
  int steps, warps, splits;   // a CTA owns 4 steps warps rows and a 1 / splits share of the groups
  int spare = 0;              // warps without rows for a launch whose other CTAs expand weights
};
constexpr int kMaxKSplits = 16;

// Clocks that a launch of 16-row warps takes, as a model: a group takes an SM as long as its element-wise warps need to issue it, or
// one warp's own chain; every CTA adds its start and the end with T.  `int4`: INT4 codes, else MXFP4.
inline int quantize_clocks(int M, int G, int r, int fitting, int w, int k, bool int4) {
  const int slots = quantize_smem_bytes(r, 4, w, k) <= 114688 ? 2 : 1;   // CTAs that share an SM
  const int ctas = ((M + 16 * w - 1) / (16 * w) + fitting - 1) / fitting;     // CTAs that an SM takes in all
  const int groups = (G + k - 1) / k;
  auto wave = [&](int n) {   // n CTAs at a time
    const int issue = (int4 ? 142 : 160) * w * n + 23 * n, chain = int4 ? 1300 : 1250;
    return groups * (issue > chain ? issue : chain) + 4300 + 820 * n + (k > 1 ? 13 : 1) * r * w * n / 2;
  };
  const int last = ctas % slots;
  return ctas / slots * wave(slots) + (last > 0 ? wave(last) : 0) + (k > 1 ? 2000 + 190 * k : 0);
}

inline QuantizePlan quantize_plan(int M, int G, int r, int sms, const int* fitting_clusters, int wide_clusters, size_t image) {
  const bool int4 = image > 0;
  const int few = 448;   // rows up to which 2 steps per warp beat 4
  if (r == 0) {
    // The splits are independent CTAs.  About five to an SM at any size, so that no SM is left with a CTA more than others:
    // 32760 x 5120 in 256 CTAs of 128 rows 105.7 us, in 768 95.1 us.  Beside an expansion too: with 1.25 per SM there, forwards of
    // 20000 x 13824 -> 1024 took 664 us instead of 612, of 6000 x 13824 -> 1024 211 instead of 182.
    const int steps = M <= few ? 2 : 4, per_warp = 4 * steps;
    const int warps = M < kQuantWarps * per_warp ? (M + per_warp - 1) / per_warp : kQuantWarps;
    const int splits = 5 * sms / ((M + per_warp * warps - 1) / (per_warp * warps));
    return {steps, warps, splits < 1 || G < 4 ? 1 : (splits > G / 2 ? G / 2 : splits)};
  }
  // Beside an expansion, which takes longer than the activations and wants its share of the machine from the start: smaller
  // CTAs, two to an SM, about one per SM in all.  Eight forwards of 5120 -> 5120 replayed from one graph, each: 700 rows,
  // r = 64 60.0 -> 51.2 us; 1560, r = 64 96.8 -> 90.3; 4097, r = 96 204 -> 194.   Above 34 x 128 rows
  // it no longer pays: 4480 rows, r = 32 201.4 us with this plan and 200.0 with the general one, 4736 209.2 | 199.7; r = 96 209.7 |
  // 210.6 and 215.2 | 213.0.
  if (int4 && M > few && M <= 34 * 128) {
    const int k = M <= 1024 ? 8 : 4, clusters = k == 8 ? 16 : 33, warps = (M + 8 * clusters - 1) / (8 * clusters);
    if (k <= G / 2 && fitting_clusters[k] > 0) return {2, warps < kQuantWarps ? warps : kQuantWarps, k};
  }
  // The splits of a row block form a cluster, which stays within a GPC.  With few rows: the most splits that still run all row
  // blocks at once, one CTA to an SM, and the fewest warps that cover the rows.  Above a byte image of 2^24 (5120 x 5120 is 1.6 of
  // that) its expansion is what the launch takes long for, on CTAs of the same form, so these get six warps: 1 x 5120 -> 13824, r = 16
  // 107 us with one, 53 with six; 1 x 5120 -> 5120 33.8 and 22.5.  Where many row blocks would make many clusters of 16, which
  // leave more SMs out, clusters of 8 do: 448 x 5120 -> 13824 94 and 85.  Smaller layers lose by either: 64 x 13824 -> 1024 22.5 us in
  // clusters of 16, 28.6 of 8.
  const bool large = image > (1u << 24);
  if (M <= few) for (int k = large && M > 256 ? 8 : kMaxKSplits; k > 1; k = k > 8 ? 8 : k - 1) {
    const int clusters = k > 8 ? wide_clusters : fitting_clusters[k];
    const int steps = k > 8 || large ? 2 : 4, per_warp = 4 * steps;
    if (clusters > 0 && k <= G / 2 && M <= clusters * kQuantWarps * per_warp) {
      const int warps = (M + clusters * per_warp - 1) / (clusters * per_warp);
      return {steps, warps, k, large && warps < 6 ? 6 - warps : 0};
    }
  }
  // Otherwise what takes the fewest clocks.  The model's constants are fitted to 444 measured surfaces (449 to 32760 rows, K 256 to
  // 13824, r 16 to 96, all warps and splits): its choice is 1.6 % (MXFP4) and 2.5 % (INT4) slower than the best one on average and
  // 3 | 5 % faster than the rule before it (the most splits with one CTA to an SM, else none), nowhere by more than 3 % slower.
  // That rule left the middle of the range half empty: 6000 x 13824, r = 16, MXFP4 73 -> 53 us, 9600 rows 135 -> 82.  32760 rows
  // keep 293 CTAs of 7 warps.
  QuantizePlan best = {4, kQuantWarps, 1};
  int least = quantize_clocks(M, G, r, sms, kQuantWarps, 1, int4);
  for (int k = 1; k <= kMaxKSplits; k = k == 8 ? kMaxKSplits : k + 1) {
    const int clusters = k == 1 ? sms : (k > 8 ? wide_clusters : fitting_clusters[k]);
    if (clusters == 0 || (k > 1 && k > G / 2)) continue;
    for (int w = kQuantWarps; w >= (M <= 2048 ? 2 : 4); --w) {
      const int clocks = quantize_clocks(M, G, r, clusters, w, k, int4);
      if (clocks < least) least = clocks, best = {4, w, k};
    }
  }
  return best;
}

}  // namespace w4a4
