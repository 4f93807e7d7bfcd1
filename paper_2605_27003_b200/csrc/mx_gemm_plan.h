// Which form of the MXFP4 GEMM a launch takes (mx_gemm_kernel.cuh), where K is not split.  Plain C++, no CUDA types.
#pragma once

namespace w4a4 {

// CTA pairs (cta_group::2) on 256 x 256 tiles, or single CTAs on 128 x 256 ones?  tiles_m x tiles_n tiles of 128 x 256; `fused`: the
// epilogue quantizes for the next layer, which exists in the pair kernel only.
// Pairs need at least two row tiles and an even number of CTAs.  A wave of pairs takes less time than one of
// single CTAs, but single CTAs win where a tile each is about all there is (900 x 5120 -> 5120 25.1 -> 20.7 us, 700 17.6 -> 15.9)
// and where they need two waves and pairs three (600 x 5120 -> 13824 31.1 -> 25.1); at 1.22 waves and K = 13824 they lose (43.6 | 45.1),
// and with two row tiles the pairs' shared weight reads count (200 x 13824 -> 13824 30.7 | 35.0).
inline bool mx_gemm_pairs(int tiles_m, int tiles_n, int sms, bool fused) {
  const int tiles = tiles_m * tiles_n, pair_tiles = (tiles_m + 1) / 2 * tiles_n;
  const bool singles = !fused && tiles_m > 2 && (tiles <= sms + sms / 8 || (tiles <= 2 * sms && pair_tiles > 2 * (sms / 2)));
  return tiles_m >= 2 && sms >= 2 && !singles;
}

}  // namespace w4a4
