// Where the stream kernel (conv_mma_stream.cu) finds the pixels of a tile in the raw rows and where it puts them in the
// window.  One definition for the kernel, its planner and the test that replays it on the host.
#pragma once

#include "b2c_internal.h"

#ifdef __CUDACC__
#define B2C_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define B2C_HOST_DEVICE inline
#endif

namespace b2c {

B2C_HOST_DEVICE int stream_min(int a, int b) { return a < b ? a : b; }
B2C_HOST_DEVICE int stream_max(int a, int b) { return a > b ? a : b; }

// Grid rows [r0, end) that a block's tile needs units of: its th output rows and what their taps reach below, up to the
// last row that a valid output reads (the overhang rows of an image are no outputs).
struct TileRows {
  int r0, end, n_a;  // n_a: image of row r0
};
B2C_HOST_DEVICE TileRows stream_tile_rows(const ConvArgs& args, const StreamArgs& sa, int r0) {
  TileRows t;
  t.r0 = r0;
  t.end = r0;
  t.n_a = sa.images;
  if (r0 >= sa.total_rows) return t;
  t.n_a = (int)sa.div_rpi.div((uint32_t)r0);
  const int last = stream_min(r0 + sa.th, sa.total_rows) - 1;
  const int n_l = (int)sa.div_rpi.div((uint32_t)last);
  const int i_l = stream_min(last - n_l * sa.rpi, args.out_P - 1);
  t.end = stream_max(r0, n_l * sa.rpi + i_l + sa.max_ri + 1);
  return t;
}

// Raw rows [lo, hi) of image n that those grid rows need (none: hi <= lo).  No row past the image's own rpi grid rows: with
// stride 2 its last row may be one that no output reads (2 x 2 filters on an odd height), and the grid row it would fill
// is the first of the next image.
struct RawRows {
  int lo, hi;
};
B2C_HOST_DEVICE RawRows stream_raw_rows(const ConvArgs& args, const StreamArgs& sa, const TileRows& t, int n, int stride) {
  RawRows r;
  r.lo = stream_max(0, (t.r0 - n * sa.rpi) * stride - args.pad_h);
  r.hi = stream_min(args.H, (stream_min(t.end - n * sa.rpi, sa.rpi) - 1) * stride + sa.max_dh - args.pad_h + 1);
  return r;
}

// Builder groups that take the windows in turn: no more than the ring has windows.  A wait tells the phases of a barrier apart
// by parity only, so a group must not come to a buffer two uses ahead of the MMAs.  Window w, in a ring of S, waits for the
// MMAs of w - S; that those of w - 2 S are through is known from the group's own last window, w - groups, which waited for
// those of w - groups - S.  (With three groups and two buffers, a group overwrote windows that were still to be read.)
constexpr int kStreamGroups = 3;
B2C_HOST_DEVICE int stream_groups(const StreamArgs& sa) { return stream_min(kStreamGroups, sa.win_stages); }

// The work of one builder thread on a window: four consecutive pixels of 16 channels.
struct StreamItem {
  uint32_t src;     // byte offset of channel 0 of the group in the raw rows
  uint32_t dst[2];  // units of the four pixels in the window, 16 bits each, kStreamNoUnit: not stored
};
constexpr uint32_t kStreamNoUnit = 0xFFFFu;

B2C_HOST_DEVICE int stream_items(const StreamArgs& sa) { return sa.max_images * 2 * sa.img_groups; }
// Bytes between two channels of the raw rows.
B2C_HOST_DEVICE uint32_t stream_channel_step(const ConvArgs& args, const StreamArgs& sa) {
  return (uint32_t)(sa.box_bytes > 0 ? sa.box_bytes : args.H * args.W);
}

// Item e = (image of the tile, block of 16 channels, four consecutive pixels); false: nothing to store.  Entry k of dst is
// pixel k ^ y (the order in which the thread stores them).
B2C_HOST_DEVICE bool stream_item(const ConvArgs& args, const StreamArgs& sa, const TileRows& tr, int e, int y, int stride, StreamItem* it) {
  const int iu = (int)sa.div_groups.div((uint32_t)e);
  const int p = iu >> 1, u = iu & 1;
  const int n = tr.n_a + p;
  if (e >= stream_items(sa) || n >= sa.images || n * sa.rpi >= tr.end) return false;
  const RawRows rr = stream_raw_rows(args, sa, tr, n, stride);
  const int f0 = rr.lo * args.W, f1 = rr.hi * args.W;
  const int f = ((f0 >> 2) + e - iu * sa.img_groups) * 4;
  if (f >= f1) return false;
  it->src = (uint32_t)(p * sa.img_slot) + (uint32_t)(u * 16) * stream_channel_step(args, sa) + (uint32_t)(f - (sa.box_bytes > 0 ? (f0 & ~15) : 0));
  const int h0 = (int)sa.div_w.div((uint32_t)f);
  const int w0 = f - h0 * args.W;
  const int row0 = n * sa.rpi - tr.r0;  // window row of the image's grid row 0
  const int plane_units = sa.plane_bytes >> 4;
  const int per_row = sa.ndh * sa.ndw;  // planes of 16 channels
  uint32_t d[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int q = k ^ y;
    // (W >= 4: a group crosses one row end at most)
    const bool wrap = w0 + q >= args.W;
    const int hp = h0 + (wrap ? 1 : 0) + args.pad_h, wp = w0 + q - (wrap ? args.W : 0) + args.pad_w;
    const int ra = stride == 1 ? 0 : (int)sa.row_index[hp & 1], cbi = stride == 1 ? 0 : (int)sa.col_index[wp & 1];
    const int j = row0 + (stride == 1 ? hp : hp >> 1), jc = stride == 1 ? wp : wp >> 1;
    const bool stored = f + q >= f0 && f + q < f1 && jc < sa.pitch && (stride == 1 || (ra >= 0 && cbi >= 0)) && j < tr.end - tr.r0;
    d[k] = stored ? (uint32_t)((u * per_row + ra * sa.ndw + cbi) * plane_units + j * sa.pitch + jc) : kStreamNoUnit;
  }
  it->dst[0] = d[0] | (d[1] << 16);
  it->dst[1] = d[2] | (d[3] << 16);
  return true;
}

// Tiles that all start an image have their rows outside the images at the same places: zero from the start, never written.
B2C_HOST_DEVICE bool stream_same_rows(const StreamArgs& sa) { return sa.th % sa.rpi == 0; }

}  // namespace b2c
