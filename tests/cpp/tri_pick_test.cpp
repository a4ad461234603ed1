// The class of the on-chip tridiagonalisation on devices where some clusters
// cannot be resident: a block that any class holds gets one that holds it.
#include <cstdio>
#include <cstdlib>

#include "../../paper_1611_03189_gb300/csrc/tri_pick.h"

using namespace hs;

int main() {
  const int full[2][kTriClasses] = {{237, 331, 465, 653, 914}, {167, 232, 327, 464, 656}};   // FP32, FP64
  for (int fp64 = 0; fp64 < 2; ++fp64)
    for (int mask = 0; mask < 32; ++mask)        // classes that are resident
      for (int mode = 0; mode < 3; ++mode) {
        int max_m[kTriClasses];
        for (int q = 0; q < kTriClasses; ++q) max_m[q] = (mask >> q & 1) ? full[fp64][q] : 0;
        const int top = tri_pick_max(max_m, mode);
        for (int m = 9; m <= 1000; ++m) {
          const int q = tri_pick(max_m, m, fp64, mode);
          const bool ok = m > top ? q == -1 : q >= 0 && q < (mode == 1 ? 1 : kTriClasses) && m <= max_m[q];
          if (!ok) {
            std::printf("fp64 %d classes %d mode %d m %d: class %d, largest %d\n", fp64, mask, mode, m, q, top);
            return 1;
          }
        }
        // the leading steps of a larger block leave a tail that has a class
        if (top > 0 && tri_pick(max_m, top, fp64, mode) < 0) return 2;
      }
  // all classes there: the preferred ones
  const int want[2][4] = {{0, 2, 3, 4}, {0, 3, 4, 4}};
  const int at[2][4] = {{237, 238, 466, 700}, {112, 113, 161, 600}};
  for (int fp64 = 0; fp64 < 2; ++fp64)
    for (int i = 0; i < 4; ++i)
      if (tri_pick(full[fp64], at[fp64][i], fp64, 0) != want[fp64][i]) return 3;
  std::printf("ok\n");
  return 0;
}
