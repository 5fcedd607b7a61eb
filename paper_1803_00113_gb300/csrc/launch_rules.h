// Which form a launch takes, from its numbers of items and pixels (host code
// without CUDA types).  Private to the library.
#pragma once

#include <cstdint>

namespace celeste {

// Into how many shares an item's background goes: up to one item for each
// resident warp of the rendering background (20 per SM), a warp does 64 pixels
// (a pass of its lanes) or more, four at most sharing an item.  The chain of an
// item's neighbours, staging and passes, is what such a launch waits for.  600
// field sources, three classes: 85 -> 75 us; at 60 items per SM 82, and with
// 12,000 items split 125 against 92.  Shares of 32 pixels and less cost more
// than they save: 60 sources in 1,600 items of 64 pixels 40 us against 29.
constexpr int kSplitItems = 20;
inline int background_shares(int64_t n_pixels, int n_items, int sm_count) {
  if (n_items <= 0 || n_items > kSplitItems * sm_count) return 1;
  const int64_t mean = n_pixels / n_items;
  return mean >= 256 ? 4 : (mean >= 128 ? 2 : 1);
}

}  // namespace celeste
