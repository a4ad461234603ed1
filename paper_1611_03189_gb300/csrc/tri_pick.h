// Which on-chip form of the tridiagonalisation (kernels_cluster.cu) takes a block
// of m unknowns: class 0 is one CTA, class q a cluster of 2^q.
#pragma once

#include <algorithm>

namespace hs {

constexpr int kTriClasses = 5;

// max_m[q]: the largest block class q holds on the device, 0 when its clusters
// cannot be resident there (fewer SMs per GPC, a partition of the GPU).
// mode: 0, or 1 (one CTA only) or 2 (the smallest class that fits).
// Preferred class first -- FP32: one CTA while it fits, then 4 CTAs (a step is
// bound by its barriers and distributed reads, which cost 2 CTAs as much), then 8,
// then 16.  FP64: the arithmetic itself (3 n^2 FMAs a step at 1/64 of the FP32
// rate) outgrows the barriers from about n = 112 on, so 8 CTAs share it from there
// (88: the same) and 16 from n = 161 on (a 331 x 198 factorization 171.6 ms with 8
// only, 166.3 with 16 from 161, 166.1 from 129, 167.0 from 113).
// Without the preferred class or a larger one that holds m, the next smaller one
// does: -1 means m > tri_pick_max(max_m, mode), and nothing else.
inline int tri_pick(const int (&max_m)[kTriClasses], int m, bool fp64, int mode) {
  const int n = mode == 1 ? 1 : kTriClasses;
  int first = 0;
  if (mode == 0) {
    if (fp64 && m > 112)
      first = m > 160 ? 4 : 3;
    else if (m > max_m[0])
      first = 2;
  }
  for (int q = first; q < n; ++q)
    if (m <= max_m[q]) return q;
  for (int q = first - 1; q >= 0; --q)
    if (m <= max_m[q]) return q;
  return -1;
}

// the largest block any class of the mode holds
inline int tri_pick_max(const int (&max_m)[kTriClasses], int mode) {
  return mode == 1 ? max_m[0] : *std::max_element(max_m, max_m + kTriClasses);
}

}  // namespace hs
