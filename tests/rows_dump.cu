// Host-only dump of the streamed kernel's rows (stream_row from csrc/common.cuh):
// one line "L RS y0 k off yp ym act" for every layout that is walked row by row
// without a branch.
#include <cstdio>

#include "common.cuh"

int main() {
  for (int L = 4; L <= 64; L += 2)
    for (int RS = 1; RS <= L; ++RS)
      for (int y0 = 0; y0 < RS && mpk::stream_four_rows(L, RS); ++y0)
        for (int k = 0; k < 4; ++k) {
          const mpk::StreamRow r = mpk::stream_row(mpk::stream_rows(L, RS, y0), L / 2, RS, k);
          std::printf("%d %d %d %d %d %d %d %d\n", L, RS, y0, k, r.off, r.yp, r.ym, r.act ? 1 : 0);
        }
  return 0;
}
