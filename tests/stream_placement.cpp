// Replays where the stream kernel's builder threads put the pixels of a layer, tile by tile, with the functions that the
// kernel itself uses, and reports layers in which two threads store to one unit of a window or a tap reads anything
// but its pixel (or, outside the image, zero).  Arguments: the number of random layers, or one layer.  "rings" instead runs
// the waits of the window and raw rings in random orders.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
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

unsigned long long g_random = 88172645463325252ull;  // xorshift64
int pick(int lo, int hi) {
  g_random ^= g_random << 13, g_random ^= g_random >> 7, g_random ^= g_random << 17;
  return lo + (int)(g_random % (unsigned long long)(hi - lo + 1));
}
b2c_conv_desc random_layer() {
  b2c_conv_desc d = {};
  d.out_mode = B2C_OUT_I32;
  d.N = pick(1, 40), d.C = 16 * pick(3, 8), d.H = pick(2, 60), d.W = pick(4, 60), d.K = pick(16, 64), d.R = pick(1, 6), d.S = pick(1, 5);
  d.stride_h = d.stride_w = pick(1, 2);
  d.pad_h = pick(0, 3), d.pad_w = pick(0, 3), d.dil_h = pick(1, 3), d.dil_w = pick(1, 3);
  return d;
}

// A barrier as the waits see it: a wait for a parity passes when the phase in progress has the other one.
struct Phases {
  long long done = 0;
  bool passes(long long use) const { return (done & 1) != (use & 1); }
};

// Windows of a block in the order of its roles, which advance in random order: the raw producer, the loads in flight, the
// builder groups and the MMA warp.  False if a role gets past a wait before the phase that it waits for is complete.
bool ring_waits_hold(const StreamArgs& sa) {
  const int windows = 40, S = sa.win_stages, R = sa.raw_stages, groups = stream_groups(sa);
  Phases win_full[4], win_empty[4], raw_full[4], raw_empty[4];
  std::vector<int> loads;                       // windows whose raw rows are in flight
  std::vector<int> next(groups), state(groups);  // window of each group; 0: waits for its buffer, 1: for its rows, 2: builds
  for (int g = 0; g < groups; ++g) next[g] = g;
  int produced = 0, consumed = 0;
  std::vector<int> commits;  // windows whose MMAs are in flight
  for (int step = 0; step < 4000 && consumed < windows; ++step) {
    const int role = pick(0, groups + 3);
    if (role < groups) {
      const int g = role, w = next[g];
      if (w >= windows) continue;
      if (state[g] == 0) {
        if (!win_empty[w % S].passes(w / S - 1)) continue;
        if (win_empty[w % S].done < w / S) return false;
        state[g] = 1;
      } else if (state[g] == 1) {
        if (!raw_full[w % R].passes(w / R)) continue;
        if (raw_full[w % R].done < w / R + 1) return false;
        state[g] = 2;
      } else {
        ++raw_empty[w % R].done;
        ++win_full[w % S].done;
        next[g] = w + groups;
        state[g] = 0;
      }
    } else if (role == groups) {
      const int w = produced;
      if (w >= windows || !raw_empty[w % R].passes(w / R - 1)) continue;
      if (raw_empty[w % R].done < w / R) return false;
      loads.push_back(w);
      ++produced;
    } else if (role == groups + 1) {
      if (loads.empty()) continue;
      const int i = pick(0, (int)loads.size() - 1);  // copies complete in any order
      ++raw_full[loads[i] % R].done;
      loads.erase(loads.begin() + i);
    } else if (role == groups + 2) {
      const int w = consumed;
      if (!win_full[w % S].passes(w / S)) continue;
      if (win_full[w % S].done < w / S + 1) return false;
      commits.push_back(w);
      ++consumed;
    } else if (!commits.empty()) {
      ++win_empty[commits.front() % S].done;
      commits.erase(commits.begin());
    }
  }
  return consumed == windows;
}

// Every pair of ring lengths that the planner gives to random layers.
int rings() {
  std::map<std::pair<int, int>, StreamArgs> seen;
  for (int i = 0; i < 50000; ++i) {
    const b2c_conv_desc d = random_layer();
    Geom g;
    StreamArgs sa;
    if (resolve_geom(&d, &g) == B2C_OK && stream_plan(g, 64 << pick(0, 2), &sa)) seen[{sa.win_stages, sa.raw_stages}] = sa;
  }
  int wrong = 0;
  for (const auto& s : seen) {
    bool holds = true;
    for (int i = 0; i < 20000 && holds; ++i) holds = ring_waits_hold(s.second);
    std::printf("%d windows, %d raw buffers, %d groups: %s\n", s.first.first, s.first.second, stream_groups(s.second),
                holds ? "every wait holds" : "a wait passes early");
    wrong += !holds;
  }
  return wrong || seen.size() < 3 ? 1 : 0;
}

}  // namespace

int main(int argc, char** argv) {
  if (argc == 2 && !std::strcmp(argv[1], "rings")) return rings();
  int seen[3] = {0, 0, 0};
  auto layer = [&](const b2c_conv_desc& d) {
    int tile_n = 64;
    while (tile_n < d.K && tile_n < 256) tile_n <<= 1;
    ++seen[replay(d, tile_n)];
  };
  if (argc == 13) {
    int v[12];
    for (int i = 0; i < 12; ++i) v[i] = std::atoi(argv[i + 1]);
    b2c_conv_desc d = {};
    d.out_mode = B2C_OUT_I32;
    d.N = v[0], d.C = v[1], d.H = v[2], d.W = v[3], d.K = v[4], d.R = v[5], d.S = v[6];
    d.stride_h = d.stride_w = v[7];
    d.pad_h = v[8], d.pad_w = v[9], d.dil_h = v[10], d.dil_w = v[11];
    layer(d);
  } else {
    for (int i = argc > 1 ? std::atoi(argv[1]) : 1000; i > 0; --i) layer(random_layer());
  }
  std::printf("layers: %d right, %d wrong, %d of other kernels\n", seen[1], seen[2], seen[0]);
  return seen[2] ? 1 : 0;
}
