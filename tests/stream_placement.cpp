// Replays where the stream kernel's builder threads put the pixels of a layer, tile by tile, with the functions that the
// kernel itself uses, and reports layers in which two threads store to one unit of a window or a tap reads anything
// but its pixel (or, outside the image, zero).  Arguments: the number of random layers, then nothing; or one layer.
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "stream_tile.h"

using namespace b2c;

namespace {

constexpr int kPairs = 3;         // pairs of blocks: each walks several tiles
constexpr long long kZero = 0, kStale = -1;

// 0: not a layer of this kernel, 1: right, 2: wrong.
int replay(const b2c_conv_desc& d, int tile_n) {
  Geom g;
  if (resolve_geom(&d, &g) != B2C_OK) return 0;
  StreamArgs sa;
  std::vector<uint64_t> table;
  std::vector<int32_t> wsrc;
  if (!stream_plan(g, tile_n, &sa, &table, &wsrc)) return 0;
  ConvArgs args = {};
  args.H = d.H;
  args.W = d.W;
  args.pad_h = d.pad_h;
  args.pad_w = d.pad_w;
  args.out_P = g.P;
  const int stride = d.stride_h, tiles_m = sa.num_tiles / sa.cols, units = sa.win_bytes / 16;
  const int per_row = sa.ndh * sa.ndw, plane_units = sa.plane_bytes / 16;
  const bool same_rows = stream_same_rows(sa);
  long long doubled = 0, outside = 0, wrong = 0, checked = 0;
  auto pixel = [&](int n, int h, int w) { return 1 + ((long long)n * d.H + h) * d.W + w; };
  for (int pair = 0; pair < kPairs; ++pair)
    for (int rank = 0; rank < 2; ++rank) {
      std::vector<long long> window(units, kZero);
      std::vector<int> writers(units);
      TileRows first = {};
      for (int t = pair; t < tiles_m; t += kPairs) {
        const TileRows tr = stream_tile_rows(args, sa, (t * 2 + rank) * sa.th);
        if (t == pair) first = tr;
        // rows outside the images
        if (!same_rows)
          for (int j = 0; j < tr.end - tr.r0; ++j)
            for (int a = 0; a < sa.ndh; ++a) {
              const int gr = tr.r0 + j, n = gr / sa.rpi, h = (gr - n * sa.rpi) * stride + sa.row_phase[a] - d.pad_h;
              if (n < d.N && h >= 0 && h < d.H) continue;
              for (int u = 0; u < 2; ++u)
                for (int b = 0; b < sa.ndw; ++b)
                  for (int q = 0; q < sa.pitch; ++q) window[(u * per_row + a * sa.ndw + b) * plane_units + j * sa.pitch + q] = kZero;
            }
        // Pixels.  (Where tiles repeat, a thread's first places are those of its first tile.)
        writers.assign(units, 0);
        for (int e = 0; e < stream_items(sa); ++e) {
          StreamItem it;
          const int y = stride == 1 ? (e >> 1) & 3 : ((e >> 2) & 1) * 2;
          const TileRows& at = same_rows ? first : tr;
          if (!stream_item(args, sa, at, e, y, stride, &it)) continue;
          const int p = (int)it.src / sa.img_slot, c_step = (int)stream_channel_step(args, sa);
          const int n_at = at.n_a + p, n = tr.n_a + p;
          const RawRows rr = stream_raw_rows(args, sa, at, n_at, stride);
          const int f = (int)it.src % sa.img_slot % (16 * c_step) + (sa.box_bytes > 0 ? (rr.lo * d.W) & ~15 : 0);
          if ((int)it.src + 15 * c_step + 4 > sa.raw_bytes || (it.src & 3) != 0) ++outside;
          const bool loaded = tr.end > tr.r0 && n < d.N && n * sa.rpi < tr.end && stream_raw_rows(args, sa, tr, n, stride).hi > rr.lo;
          for (int k = 0; k < 4; ++k) {
            const uint32_t unit = (it.dst[k >> 1] >> (16 * (k & 1))) & 0xFFFFu;
            if (unit == kStreamNoUnit) continue;
            if ((int)unit >= units) {
              ++outside;
              continue;
            }
            if (++writers[unit] == 2) ++doubled;
            const int fp = f + (k ^ y);
            window[unit] = loaded ? pixel(n, fp / d.W, fp % d.W) : kStale;
          }
        }
        // what the taps of the valid outputs read
        for (int row = 0; row < kTileM; ++row) {
          const int j = row / sa.pitch, q = row % sa.pitch, gr = tr.r0 + j, n = gr / sa.rpi, i = gr - n * sa.rpi;
          if (j >= sa.th || q >= g.Q || i >= g.P || n >= d.N) continue;
          ++checked;
          for (int r = 0; r < d.R; ++r)
            for (int s = 0; s < d.S; ++s) {
              const uint64_t a = table[r * d.S + s];
              const int h = i * stride - d.pad_h + r * d.dil_h, w = q * stride - d.pad_w + s * d.dil_w;
              const long long expect = h >= 0 && h < d.H && w >= 0 && w < d.W ? pixel(n, h, w) : kZero;
              for (int u = 0; u < 2; ++u) {
                const int at = (int)(a & 0x3FFF) + row + u * (int)(a >> 16);
                if (at >= units || window[at] != expect) ++wrong;
              }
            }
        }
      }
    }
  const bool right = !doubled && !outside && !wrong && checked == (long long)d.N * g.PQ;
  if (!right)
    std::printf("N %d C %d %dx%d K %d filter %dx%d stride %d pad %d,%d dil %d,%d: %lld units with two writers, %lld places outside, "
                "%lld wrong reads, %lld of %lld outputs\n",
                d.N, d.C, d.H, d.W, d.K, d.R, d.S, stride, d.pad_h, d.pad_w, d.dil_h, d.dil_w, doubled, outside, wrong, checked,
                (long long)d.N * g.PQ);
  return right ? 1 : 2;
}

}  // namespace

int main(int argc, char** argv) {
  int seen[3] = {0, 0, 0};
  b2c_conv_desc d = {};
  d.out_mode = B2C_OUT_I32;
  auto layer = [&](int N, int C, int H, int W, int K, int R, int S, int stride, int ph, int pw, int dh, int dw) {
    d.N = N, d.C = C, d.H = H, d.W = W, d.K = K, d.R = R, d.S = S;
    d.stride_h = d.stride_w = stride;
    d.pad_h = ph, d.pad_w = pw, d.dil_h = dh, d.dil_w = dw;
    int tile_n = 64;
    while (tile_n < K && tile_n < 256) tile_n <<= 1;
    ++seen[replay(d, tile_n)];
  };
  if (argc == 13) {
    int v[12];
    for (int i = 0; i < 12; ++i) v[i] = std::atoi(argv[i + 1]);
    layer(v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7], v[8], v[9], v[10], v[11]);
  } else {
    unsigned long long x = 88172645463325252ull;  // xorshift64
    auto pick = [&](int lo, int hi) {
      x ^= x << 13, x ^= x >> 7, x ^= x << 17;
      return lo + (int)(x % (unsigned long long)(hi - lo + 1));
    };
    for (int i = argc > 1 ? std::atoi(argv[1]) : 1000; i > 0; --i)
      layer(pick(1, 40), 16 * pick(3, 8), pick(2, 60), pick(4, 60), pick(16, 64), pick(1, 6), pick(1, 5), pick(1, 2), pick(0, 3), pick(0, 3), pick(1, 3),
            pick(1, 3));
  }
  std::printf("layers: %d right, %d wrong, %d of other kernels\n", seen[1], seen[2], seen[0]);
  return seen[2] ? 1 : 0;
}
