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

// A block of eight warps per item instead of a warp: where its blocks are
// resident together (two per SM in the derivative pass, five in the value
// pass), and, in the derivative pass, an item has more than one pass; longer
// items also in two rounds (from three passes in derivatives, six in values),
// since part of a class's sources have often stopped: fits of 56 sources lose
// up to 1 % without.  Beyond, the persistent kernels fill the GPU and are
// faster.  One 41 x 41 source, a Newton
// iteration: derivatives 26.5 -> 14.2 us, values 14.0 -> 8.7.  Calls on n
// sources of one item, a warp against a block an item: derivatives of 304
// items of 100 pixels 1.10, of 608 items of 25 pixels 0.83; values of 760
// items of 64 pixels 1.00, of 912 0.93, of 810 items of 1,024 pixels 1.30;
// 600 field sources, a class of 1,100 items: 249 us of derivatives in a pass
// with eight items per SM, 236 with four.
inline bool block_per_item_derivs(int64_t n_pixels, int n_items, int sm_count) {
  if (n_items <= 0) return false;
  const int64_t mean = n_pixels / n_items;
  return mean > 32 && n_items <= (mean >= 96 ? 4 : 2) * sm_count;
}
inline bool block_per_item_values(int64_t n_pixels, int n_items, int sm_count) {
  if (n_items <= 0) return false;
  const int64_t mean = n_pixels / n_items;
  return n_items <= (mean >= 192 ? 8 : 5) * sm_count;
}

}  // namespace celeste
