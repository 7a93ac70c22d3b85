// Schedules of the plane kernel whose rows are widened to whole memory sectors: every row of every window keeps its results'
// distance to the sectors, i.e. position minus output index is a multiple of a sector's results.  Random layers.
#include <algorithm>
#include <cstdio>

#include "b2c_internal.h"

using namespace b2c;

int main() {
  unsigned long long x = 88172645463325252ull;  // xorshift64
  auto pick = [&](int lo, int hi) {
    x ^= x << 13, x ^= x >> 7, x ^= x << 17;
    return lo + (int)(x % (unsigned long long)(hi - lo + 1));
  };
  int widened = 0, wrong = 0;
  for (int t = 0; t < 3000; ++t) {
    b2c_conv_desc d = {};
    d.N = pick(1, 40), d.C = pick(8, 64), d.H = pick(0, 1) ? pick(3, 16) : pick(8, 130), d.K = 16 * pick(1, 4);
    d.out_mode = pick(1, 3);
    d.W = d.out_mode == B2C_OUT_I8 ? 8 * pick(26, 60) : pick(40, 250);
    d.R = d.S = 3, d.stride_h = d.stride_w = 1, d.pad_h = d.pad_w = 1, d.dil_h = d.dil_w = 1, d.shift = 8;
    Geom g;
    if (resolve_geom(&d, &g) != B2C_OK) continue;
    const int outputs = d.out_mode & B2C_OUT_I32 ? kSectorOutputs : 4 * kSectorOutputs;
    PlaneArgs pl;
    int narrow = 1 << 30;
    for (int i = 0; plane_plan(g, 1, i, &pl); ++i) narrow = std::min(narrow, pl.pitch);
    for (int i = 0; plane_plan(g, 1, i, &pl); ++i) {
      if (pl.pitch == narrow || pl.runw > 0) continue;
      ++widened;
      bool kept = true;
      const int total = pl.spi > 0 ? g.P : pl.total_rows;
      for (int s0 = 0; s0 < total; s0 += pl.seg_rows)
        for (int w0 = s0; w0 < std::min(total, s0 + pl.seg_rows); w0 += pl.th)
          for (int r = w0; r < std::min(std::min(total, s0 + pl.seg_rows), w0 + pl.th); ++r) {
            const int row = pl.spi > 0 ? r : r % pl.rpi;  // of its image
            if (row < g.P && ((long long)(r - w0) * pl.pitch - (long long)row * g.Q) % outputs != 0) kept = false;
          }
      if (!kept && ++wrong <= 5)
        std::printf("N %d C %d %dx%d outputs %d: rows of %d widened to %d, %d rows a window, %d a segment, %s\n", d.N, d.C, d.H, d.W, d.out_mode, narrow, pl.pitch,
                    pl.th, pl.seg_rows, pl.spi > 0 ? "image by image" : "over the batch");
    }
  }
  std::printf("%d widened schedules, %d off the sectors\n", widened, wrong);
  return wrong || widened < 100 ? 1 : 0;
}
