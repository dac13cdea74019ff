// adjoint_levels.h -- which levels of the adjoint's V-cycle run as one CTA (host only).
#pragma once
#include <stddef.h>

namespace mg {

constexpr int kAdjTailCells = 4096, kAdjTailLevels = 5;

// The first level of the one-block tail among the levels' sides n[0 .. nlev-1], or -1:
// the first with at most kAdjTailCells cells and at most kAdjTailLevels levels from
// there on; the finest only in the natural layout.  (The product in 64 bits: from a
// side of 1291 it passes 2^31.)
static inline int adj_tail_level(const int* n, int nlev, bool split) {
  for (int l = split ? 1 : 0; l < nlev; ++l)
    if (nlev - l <= kAdjTailLevels && (long long)n[l] * n[l] * n[l] <= kAdjTailCells) return l;
  return -1;
}

// Shared memory of a tail of T levels of sides n: four arrays a level, at most 4 x 4096
// (1 + 1/8 + ...) cells.
static inline size_t adj_tail_smem(const int* n, int T) {
  size_t cells = 0;
  for (int l = 0; l < T; ++l) cells += (size_t)n[l] * n[l] * n[l];
  return cells * 4 * sizeof(float);
}

constexpr int kAdjTailSmem = 80 * 1024;

}  // namespace mg
