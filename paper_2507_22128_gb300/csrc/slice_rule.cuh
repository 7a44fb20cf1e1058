// How finely the gridders cut their work items (k_grid.cu).  Plain C++, so that
// the rule can be checked on the host.
#pragma once

#include <cstdint>

namespace rix {

// most entries of a gridder work item (a run of sorted entries of one uv tile
// and w-plane block): the partition cuts by it, the gridders size by it
constexpr int kItemEntries = 2048;

// Entries of a slice, a power of two of at least 64, for a partition of
// `entries` entries on `slots` resident CTAs.  A work item is up to 2048 entries
// of one uv tile, so a small or centrally crowded observation has a few long
// items and most SMs idle (19,841 samples at 128^2 in whole items: 207 us per
// gridding launch and 31 us per degridding, the time of one full item; 17 and 5 us
// in slices).  A slice is at most a quarter of a slot's share of the entries:
// each stages and flushes its tile, about the work of ten entries.
//
// Sums in FP32 bound the cut from below; `crowded` is then the entries of the
// fullest tile, otherwise 0.  Of m entries added in pieces of s, the additions
// within the pieces leave s^2 / (3 m) and those of the pieces to the grid
// m / (3 s) squared roundings of the total (entries of one sign, where each
// addition rounds by the size of the running sum).  That is no more than in whole
// items of I = 2048 while m^2 <= s I (s + I): tiles of up to 16,600 entries may be
// cut to 64, tiles from 92,700 on not at all.  Relative error of such images of
// 300,000 samples at 64^2, three observations: in whole items 1.38 - 1.44e-7, by
// the rule 1.44 - 1.47e-7, in slices of 64 1.7 - 2.8e-7; of 20,000 samples at 128^2
// 2.1e-7 in whole items and 1.5 - 1.9e-7 by the rule.
inline int slice_entries(int64_t entries, int64_t slots, int64_t crowded) {
  const int64_t share = entries / (4 * (slots > 1 ? slots : 1));
  const double m = (double)crowded, I = kItemEntries;
  int s = 64;
  while (s < kItemEntries && (s < share || m * m > s * I * (s + I))) s *= 2;
  return s;
}

// log2 of the slices that every item is numbered with: as many as the fullest
// tile needs
inline int slices_log2(int64_t fullest, int slice) {
  const int64_t longest = fullest < 1 ? 1 : fullest < kItemEntries ? fullest : kItemEntries;
  int l = 0;
  while (((int64_t)slice << l) < longest) ++l;
  return l;
}

// CTAs for `total` slices (those of an item side by side): all that fit, an odd
// number, so that a CTA, which takes every gridDim-th slice, does not get the same
// place of every item: in most items of a sparse observation only the first slice
// holds entries, and of 1,216 CTAs 76 did all the work of items of 16 slices.
inline int64_t slice_blocks(int64_t total, int64_t slots) {
  return total <= slots ? total : slots - (slots + 1) % 2;
}

}  // namespace rix
