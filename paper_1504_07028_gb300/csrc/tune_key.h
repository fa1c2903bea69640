// What the autotuner tells images and tilings apart by (host only; the CPU tests compile it).
//
// An image's z-update takes the pixel-domain form where its plan leaves that choice to the library
// (Plan::zl) and the squares of its shift weights sum to no more than that form's limit. Only
// then have the fields of the transform passes no effect: tilings that differ in them are one
// tiling to time, while an image with larger weights runs the passes and has all of them to try.
// For the same reason a tiling found for one form is not handed to an image that runs the other.
#pragma once

#include <tuple>
#include <vector>

namespace sgs {

struct TuneKey {
  int precision, M, K, size_class, pixel;
  bool operator<(const TuneKey& o) const {
    return std::tie(precision, M, K, size_class, pixel) <
           std::tie(o.precision, o.M, o.K, o.size_class, o.pixel);
  }
};

// The largest l with 4^l <= H W: images of one class differ by less than a factor of four.
inline int size_class_of(int H, int W) {
  const long long n = (long long)H * W;
  int l = 0;
  while ((2LL << l) <= n) ++l;  // l = floor(log2 n)
  return l / 2;
}

// pixel: the weights allow the pixel-domain z-update (FP32 and their sum of squares small enough).
inline TuneKey make_tune_key(int precision, int M, int K, int H, int W, bool pixel) {
  return TuneKey{precision, M, K, size_class_of(H, W), pixel ? 1 : 0};
}

// Append what a resolved tiling makes an image run.
template <typename Plan>
inline void append_tiling_key(std::vector<int>& key, const Plan& pl, bool pixel) {
  const bool zl = pl.zl && pixel;
  key.push_back(pl.THmax); key.push_back(zl);
  if (zl) return;                  // no row or column pass to tile
  key.push_back(pl.QB); key.push_back(pl.CB);
  key.push_back(pl.row.threads); key.push_back(pl.NSEG); key.push_back(pl.zf_cs);
  key.push_back(pl.rp);
  key.push_back(pl.p2);
}

}  // namespace sgs
