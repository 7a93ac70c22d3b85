// Host-side embedding planner: which convolution axes feed the MMA's M / N / K dimensions, with
// which layout rewrite, tile width and reduction split.
//
// The paper finds embeddings by constraint solving over the scalar data-flow graph (Section 4)
// and derives the layout rewrites of Table 2 from the solution.  For a 2-D convolution on a
// matrix-multiply intrinsic the legal, axis-aligned, dense solutions form a small closed family
// (the hyper-rectangle and linear-access constraints of Section 4.2 leave only: feed K from the
// padded channel axis, or from the unrolled stencil), so this planner writes that family out
// directly, ranks it with the overhead terms of Section 4.4 and leaves the final choice to
// measured device time, as Section 6.1 does with its five best candidates.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <utility>

#include "b2c_internal.h"
#include "stream_tile.h"

namespace b2c {

int round_up(int v, int m) { return (v + m - 1) / m * m; }

static int out_extent(int in, int k, int stride, int pad, int dil) {
  long long span = (long long)in + 2LL * pad - (long long)dil * (k - 1) - 1;
  if (span < 0) return 0;
  return (int)(span / stride) + 1;
}

int resolve_geom(const b2c_conv_desc* d, Geom* g) {
  if (!d || !g) return B2C_E_INVALID_ARG;
  if (d->N < 1 || d->C < 1 || d->H < 1 || d->W < 1 || d->K < 1 || d->R < 1 || d->S < 1) return B2C_E_INVALID_ARG;
  if (d->stride_h < 1 || d->stride_w < 1 || d->pad_h < 0 || d->pad_w < 0 || d->dil_h < 1 || d->dil_w < 1)
    return B2C_E_INVALID_ARG;
  if (d->shift < 0 || d->shift > 31) return B2C_E_INVALID_ARG;
  if (d->in_layout != B2C_LAYOUT_NCHW && d->in_layout != B2C_LAYOUT_NHWC) return B2C_E_INVALID_ARG;
  if (d->out_layout != B2C_LAYOUT_NCHW && d->out_layout != B2C_LAYOUT_NHWC) return B2C_E_INVALID_ARG;
  if ((d->out_mode & ~3) != 0 || (d->out_mode & 3) == 0) return B2C_E_INVALID_ARG;
  g->d = *d;
  g->P = out_extent(d->H, d->R, d->stride_h, d->pad_h, d->dil_h);
  g->Q = out_extent(d->W, d->S, d->stride_w, d->pad_w, d->dil_w);
  long long kg = (long long)d->C * d->R * d->S;
  if (g->P == 0 || g->Q == 0) return B2C_E_UNSUPPORTED;
  if (kg > kMaxKg) return B2C_E_UNSUPPORTED;
  // A padding of a million pixels per side serves no convolution and would let the products below
  // leave 64 bits for extreme images; P*Q must fit 31 bits before anything is derived from it.
  if (d->pad_h > (1 << 20) || d->pad_w > (1 << 20)) return B2C_E_UNSUPPORTED;
  const long long pq = (long long)g->P * g->Q;
  if (pq > 0x7FFFFF00LL) return B2C_E_UNSUPPORTED;
  g->PQ = (int)pq;
  g->Mg = (long long)d->N * pq;
  g->Kg = (int)kg;
  g->x_elems = (long long)d->N * d->C * d->H * d->W;
  g->w_elems = (long long)d->K * kg;
  g->y_elems = g->Mg * d->K;
  // Index arithmetic in the kernels is 32-bit for rows/columns and 64-bit for byte offsets.
  if (g->Mg > 0x7FFFFF00LL || g->x_elems > (1LL << 40) || g->y_elems > (1LL << 40)) return B2C_E_UNSUPPORTED;
  if ((long long)d->H * d->W * d->C > 0x7FFFFFFFLL) return B2C_E_UNSUPPORTED;
  return B2C_OK;
}

// Pad rule (Table 2, rule 2) for the channel axis: the intrinsic consumes 32 channels per
// instruction, so C is padded to a multiple of 32.
int cp_channel_pad(int C) { return round_up(C, kMmaK); }

// Split rule (Table 2, rule 3): the padded channel axis is cut into blocks of the largest of
// 128 / 64 / 32 bytes that divides it (one shared-memory swizzle row per block).
int cp_block_bytes(int C_pad) {
  if (C_pad % 128 == 0) return 128;
  if (C_pad % 64 == 0) return 64;
  return 32;
}

int im2col_k_pad(int Kg) { return round_up(Kg, kMmaK); }

bool staged_word_mode(const Geom& g) { return g.d.dil_w == 1; }
int staged_run_len(const Geom& g) { return staged_word_mode(g) ? round_up(g.d.S, 4) : g.d.S; }
int variant_k_pad(const Geom& g, int variant) {
  if (variant == B2C_VARIANT_IM2COL_WINDOW) return round_up(g.d.C * g.d.R * round_up(g.d.S, 4), kMmaK);
  if (variant == B2C_VARIANT_IM2COL_STAGED) return round_up(g.d.C * g.d.R * staged_run_len(g), kMmaK);
  return im2col_k_pad(g.Kg);
}

size_t workspace_bytes_for(const Geom& g, int variant, int tile_n, int split_k, bool swap) {
  size_t ws = 0;
  const b2c_conv_desc& d = g.d;
  TmaView v;
  if (is_tma_view_variant(variant) && tma_view_for(g, variant, &v)) {
    bool direct = shift_base_variant(variant) == B2C_VARIANT_CP_TMA && d.in_layout == B2C_LAYOUT_NHWC && v.C == d.C;
    if (!direct) ws += (size_t)v.bytes();
  } else if (variant == B2C_VARIANT_IM2COL_EXPLICIT) {
    ws += (size_t)g.Mg * im2col_k_pad(g.Kg);
  }
  ws = (ws + 255) / 256 * 256;
  // A split reduction accumulates int32 partial sums in scratch unless the int32 output itself
  // can serve (int32-only output in any layout).
  if (split_k > 1 && !cluster_split_ok(variant, tile_n, split_k, swap) && (d.out_mode & B2C_OUT_I8))
    ws += (size_t)g.y_elems * 4;
  return ws;
}

// Limits of the 4-D im2col-mode tensor map: corners in [-128, 127], tap offsets in [0, 255],
// traversal strides in [1, 8].
static bool view_fits_tensor_map(const TmaView& v) {
  int up_w = v.pad_w - (v.S - 1) * v.dil_w, up_h = v.pad_h - (v.R - 1) * v.dil_h;
  if (v.pad_w > 128 || v.pad_h > 128 || up_w < -128 || up_h < -128 || up_w > 127 || up_h > 127) return false;
  if ((v.S - 1) * v.dil_w > 255 || (v.R - 1) * v.dil_h > 255) return false;
  if (v.stride_w > 8 || v.stride_h > 8) return false;
  if (v.bytes() > (1LL << 40) || (long long)v.H * v.W * v.C > 0x7FFFFFFFLL) return false;
  return true;
}

int s2d_pack_factor(const Geom& g) {
  const int cphase = g.d.C * g.d.stride_h * g.d.stride_w;
  const int Sp = (g.d.S + g.d.stride_w - 1) / g.d.stride_w;
  if (cphase > kMmaK / 2) return 1;
  return std::max(1, std::min(kMmaK / cphase, Sp));
}

bool shift_geom(const Geom& g, const TmaView& v, ShiftGeom* sg, bool tiles_2d) {
  if (v.stride_h != 1 || v.stride_w != 1 || g.d.K > 256) return false;
  sg->cb = cp_block_bytes(v.C);
  sg->ncb = v.C / sg->cb;
  sg->tiles_h = sg->tiles_w = 0;
  long long rows;
  sg->two_d = 0;
  sg->valid_w = 0;
  // Two-dimensional tiles for the multi-tap views: a tile is 128/pitch rows of `pitch` window origins
  // (pitch a power of two), its window one TMA box of the rows those origins and their taps touch.
  // Narrow rows (padded width up to 128, at most a quarter lost to rounding the pitch up): the pitch
  // covers the whole padded row and a tile is several image rows.  Wide rows (padded width >= 192):
  // one-row tiles of 128 origins of which the last (S - 1)*dil_w only serve as the taps' overhang
  // (tiles advance by the valid width).  In between, and for anything else, the window is whole
  // padded rows (below).
  const int wp_real = v.W + 2 * v.pad_w;
  const long long wp_full = round_up(wp_real, 8);
  const int overhang = (v.S - 1) * v.dil_w;
  int pitch = 16;
  while (pitch < wp_real) pitch <<= 1;
  const bool narrow_2d = !tiles_2d && pitch <= kTileM && (long long)pitch * 100 <= wp_full * 125;
  const bool wide_2d = !tiles_2d && v.S > 1 && wp_full >= 192 && overhang <= kTileM / 4;
  if (narrow_2d || wide_2d) {
    sg->two_d = 1;
    sg->wps = narrow_2d ? pitch : kTileM;
    sg->valid_w = narrow_2d ? wp_real - overhang : kTileM - overhang;
    sg->hp = v.H + 2 * v.pad_h;
    const int tile_h = kTileM / sg->wps;
    rows = tile_h + (long long)(v.R - 1) * v.dil_h + (overhang > 0 ? 1 : 0);
    if (rows > 256) return false;
    sg->tiles_h = (g.P + tile_h - 1) / tile_h;
    sg->tiles_w = (g.Q + sg->valid_w - 1) / sg->valid_w;
  } else if (tiles_2d) {
    // tiles of 128/tw x tw pixels over an unpadded view with one tap per filter row: the window is one
    // box of (128/tw + R - 1) rows of tw pixels, and a tap moves the tile by one row of tw pixels
    if (v.S != 1 || v.pad_h != 0 || v.pad_w != 0 || v.dil_h != 1) return false;
    sg->two_d = 1;
    // tile width: the widest power of two up to 128 that wastes at most 15 % of its columns on the
    // ragged right edge (wide tiles give long contiguous output runs), else 16
    int tile_w = kShiftTileW;
    for (int tw = kTileM; tw > kShiftTileW; tw >>= 1)
      if ((long long)((g.Q + tw - 1) / tw) * tw * 100 <= (long long)g.Q * 115) {
        tile_w = tw;
        break;
      }
    const int tile_h = kTileM / tile_w;
    sg->wps = tile_w;
    sg->valid_w = tile_w;
    sg->hp = v.H;
    rows = tile_h + v.R - 1;
    if (rows > 256) return false;
    sg->tiles_h = (g.P + tile_h - 1) / tile_h;
    sg->tiles_w = (g.Q + tile_w - 1) / tile_w;
  } else {
    const int wp = v.W + 2 * v.pad_w;
    sg->wps = round_up(wp, 8);
    sg->hp = v.H + 2 * v.pad_h;
    if (sg->wps > 256) return false;  // one copy per staged image row
    const long long shift_max = (long long)(v.R - 1) * v.dil_h * sg->wps + (long long)(v.S - 1) * v.dil_w;
    // a tile starts anywhere inside its first staged row and reads 128 positions plus the largest shift
    rows = (sg->wps - 1 + kTileM - 1 + shift_max) / sg->wps + 1;
    if (rows > 4096) return false;
  }
  sg->rows = (int)rows;
  sg->row_bytes = sg->wps * sg->cb;
  const long long cblk = rows * sg->row_bytes;
  const long long win = (cblk * sg->ncb + 1023) / 1024 * 1024;
  int tile_n = 16;
  while (tile_n < g.d.K) tile_n <<= 1;
  const long long wbytes = (long long)v.R * v.S * sg->ncb * tile_n * sg->cb;
  if (2 * win + wbytes + 2048 > 200 * 1024) return false;
  sg->cblk_bytes = (int)cblk;
  sg->win_bytes = (int)win;
  sg->w_bytes = (int)wbytes;
  sg->tile_n = tile_n;
  // Window buffers per block and blocks per SM: as many windows in flight per SM as fit (each block
  // at least two, at most six), preferring more resident blocks on a tie.
  sg->stages = 2;
  sg->blocks_per_sm = 1;
  for (int bps = 3; bps >= 1; --bps) {
    const long long room = (220 * 1024) / bps - wbytes - 2048;
    const int st = (int)std::min<long long>(6, std::min<long long>(room, 198 * 1024 - wbytes) / win);
    if (st >= 2 && st * bps > sg->stages * sg->blocks_per_sm) {
      sg->stages = st;
      sg->blocks_per_sm = bps;
    }
  }
  sg->mtot = sg->two_d ? (long long)v.N * sg->tiles_h * sg->tiles_w * kTileM : (long long)v.N * sg->hp * sg->wps;
  return sg->mtot <= 0x7FFFFF00LL;
}

bool tma_view_for(const Geom& g, int variant, TmaView* v) {
  const b2c_conv_desc& d = g.d;
  if (variant == B2C_VARIANT_ROWPHASE_SHIFT) {
    // Stencil Unroll along s and Image Pack of the vertical stride in one rewrite:
    // U[n][h'][q][(dh, s, c)] = x[n][c][h'*stride_h + dh - pad_h][q*stride_w - pad_w + s*dil_w], and an
    // R' x 1, stride-1, unpadded convolution over U remains (r = r'*stride_h + dh).
    if (d.dil_h != 1) return false;
    const int Rp = (d.R + d.stride_h - 1) / d.stride_h;
    const long long cq = (long long)d.stride_h * d.S * d.C;
    if (cq > 4096) return false;
    if ((long long)d.C * d.stride_h * row_phase_seg(d.stride_w, d.S, d.dil_w) > kRowPhaseSmemMax) return false;
    *v = TmaView{d.N, round_up((int)cq, kMmaK), g.P + Rp - 1, g.Q, Rp, 1, 1, 1, 0, 0, 1, 1};
    ShiftGeom sg;
    return view_fits_tensor_map(*v) && shift_geom(g, *v, &sg, true);
  }
  if (is_shift_variant(variant)) {
    ShiftGeom sg;
    return tma_view_for(g, shift_base_variant(variant), v) && shift_geom(g, *v, &sg);
  }
  if (variant == B2C_VARIANT_CP_TMA) {
    // Pad + Split + Reorder of the channel axis (Table 2).  An NHWC source with a multiple of 32
    // channels is read in place; any other NHWC source is re-padded into the scratch tensor.
    *v = TmaView{d.N, cp_channel_pad(d.C), d.H, d.W, d.R, d.S, d.stride_h, d.stride_w, d.pad_h, d.pad_w, d.dil_h, d.dil_w};
  } else if (variant == B2C_VARIANT_ROW_UNROLL) {
    // Stencil Unroll along s only: U[n][h][q][(s, c)] = x[n][c][h][q*stride_w - pad_w + s*dil_w].
    // What is left is an R x 1 convolution over U with the vertical geometry unchanged.
    if (d.S == 1) return false;  // nothing to unroll: same as the channel-pack map
    *v = TmaView{d.N, round_up(d.S * d.C, kMmaK), d.H, g.Q, d.R, 1, d.stride_h, 1, d.pad_h, 0, d.dil_h, 1};
  } else if (variant == B2C_VARIANT_SPACE_TO_DEPTH) {
    // Image Pack of a strided convolution: with hp = h + pad_h = (p + r')*stride_h + dh the stride
    // phases (dh, dw) become channels of X'[n][hp / stride_h][wp / stride_w][(c, dh, dw)], and a
    // stride-1, unpadded R' x S' convolution over X' remains (R' = ceil(R / stride_h)).
    if (d.dil_h != 1 || d.dil_w != 1 || (d.stride_h == 1 && d.stride_w == 1)) return false;
    const int Rp = (d.R + d.stride_h - 1) / d.stride_h, Sp = (d.S + d.stride_w - 1) / d.stride_w;
    // horizontal tap packing: X''[..][w'][(ui, c, dh, dw)] = X'[..][w' + ui][(c, dh, dw)], taps at w' + pack*s''
    const int pack = s2d_pack_factor(g);
    const int Sv = (Sp + pack - 1) / pack;
    *v = TmaView{d.N, round_up(pack * d.C * d.stride_h * d.stride_w, kMmaK), g.P + Rp - 1, g.Q + pack * (Sv - 1), Rp, Sv,
                 1, 1, 0, 0, 1, pack};
  } else if (variant == B2C_VARIANT_DILATION_PACK) {
    // Image Pack of a dilated convolution (Section 6.1): with h - pad_h = i*dil_h + a every tap of an
    // output pixel reads phase a of the image, X_a[j] = x[j*dil_h + a], at j = i + r.  The dil_h*dil_w
    // phase sub-images (extent ceil(H / dil_h), zeros past the image) are fused into the batch and a
    // dense, stride-1 R x S convolution with padding ceil(pad / dil) remains.
    if ((d.dil_h == 1 && d.dil_w == 1) || d.stride_h != 1 || d.stride_w != 1) return false;
    const long long n_sub = (long long)d.N * d.dil_h * d.dil_w;
    if (n_sub > 0x7FFFFFFF) return false;
    *v = TmaView{(int)n_sub, cp_channel_pad(d.C), (d.H + d.dil_h - 1) / d.dil_h, (d.W + d.dil_w - 1) / d.dil_w, d.R, d.S,
                 1, 1, (d.pad_h + d.dil_h - 1) / d.dil_h, (d.pad_w + d.dil_w - 1) / d.dil_w, 1, 1};
    const long long rows = (long long)v->N * (v->H + 2 * v->pad_h - v->R + 1) * (v->W + 2 * v->pad_w - v->S + 1);
    if (rows > 0x7FFFFF00LL) return false;
  } else {
    return false;
  }
  return view_fits_tensor_map(*v);
}

long long view_rows(const Geom& g, int variant, const TmaView& v) {
  if (is_shift_variant(variant)) {
    // window origins on the padded grid (width rounded up to 8), not only the valid output pixels
    ShiftGeom sg;
    return shift_geom(g, v, &sg, shift_tiles_2d(variant)) ? sg.mtot : g.Mg;
  }
  if (variant != B2C_VARIANT_DILATION_PACK) return g.Mg;
  return (long long)v.N * (v.H + 2 * v.pad_h - v.R + 1) * (v.W + 2 * v.pad_w - v.S + 1);
}

// The staged stencil unroll keeps, per image a tile can touch, the zero-padded input rows that
// feed the tile's 128 output pixels: C x rows x pitch bytes, with the left margin rounded up to 16
// so that aligned 16-byte copies land on aligned shared-memory addresses.
bool staged_window(const Geom& g, WindowGeom* w) {
  const b2c_conv_desc& d = g.d;
  if (d.in_layout != B2C_LAYOUT_NCHW) return false;  // the window is staged from whole NCHW rows
  const int rows_out = std::min(g.P, (kTileM - 2) / g.Q + 2);  // output rows 128 consecutive pixels can span
  const int parts = (int)std::min<long long>(d.N, (kTileM - 2) / g.PQ + 2);
  const long long rows = (long long)(rows_out - 1) * d.stride_h + (long long)(d.R - 1) * d.dil_h + 1;
  const long long left = round_up(d.pad_w, 16);
  // columns read: up to (Q-1)*stride_w - pad_w + (S-1)*dil_w
  const long long right_edge = (long long)(g.Q - 1) * d.stride_w - d.pad_w + (long long)(d.S - 1) * d.dil_w + 1;
  const long long width = std::max<long long>(d.W, right_edge);
  const long long pitch = (left + width + 15) / 16 * 16;
  const long long bytes = (long long)parts * d.C * rows * pitch;
  if (bytes > 64 * 1024 || variant_k_pad(g, B2C_VARIANT_IM2COL_STAGED) > 4096) return false;
  w->rows = (int)rows;
  w->pitch = (int)pitch;
  w->left = (int)left;
  w->parts = parts;
  w->bytes = (int)bytes;
  return true;
}

// Small images: whole images as the window, linear tiles.
static bool window_linear_geom(const Geom& g, WindowTile* wt) {
  const b2c_conv_desc& d = g.d;
  const long long chw = (long long)d.C * d.H * d.W;
  // an image is one bulk copy (16-byte multiple, a few KB); a tile of 128 consecutive pixels touches
  // at most four images; runs of at most two words; the margin in front of the window covers the
  // negative offsets of the padding (those taps are masked, but their addresses must be valid)
  if ((chw % 16) != 0 || chw > 16 * 1024 || d.S > 8 || d.R > 32 || g.PQ < 43) return false;
  if ((long long)d.pad_h * d.W + d.pad_w + 8 > 128) return false;
  const int parts = (kTileM - 2) / g.PQ + 2;
  wt->linear = 1;
  wt->tile_w = kTileM;
  wt->tile_h = 1;
  wt->win_w = d.W;
  wt->win_h = d.H;
  wt->left = 128;
  wt->off0 = 0;
  wt->tiles_h = wt->tiles_w = 1;
  wt->box_bytes = (int)chw;
  // rows below the image that masked taps may address: up to (R-1)*dil_h rows past the last output row's first tap
  const long long slack = round_up((int)((long long)(d.R - 1) * d.dil_h * d.W + d.S + 16), 128) + 128;
  const long long win = 128 + (long long)parts * chw + slack;
  if (win > 60 * 1024 || chw >= (1 << 16) || win >= (1 << 16)) return false;
  wt->win_bytes = round_up((int)win, 128);
  wt->mtot = g.Mg;
  return true;
}

bool window_tile_geom(const Geom& g, WindowTile* wt) {
  const b2c_conv_desc& d = g.d;
  // words of an A row are unaligned words of a window row: unit horizontal dilation
  if (d.in_layout != B2C_LAYOUT_NCHW || d.dil_w != 1 || d.C > 64 || d.K > 256) return false;
  wt->linear = 0;
  wt->S_run = round_up(d.S, 4);
  wt->K_pad = round_up(d.C * d.R * wt->S_run, kMmaK);
  if (wt->K_pad > 1024) return false;
  wt->num_kb = (wt->K_pad + 127) / 128;
  wt->tile_n = 16;
  while (wt->tile_n < d.K) wt->tile_n <<= 1;
  // small images: linear tiles over whole images (no padded positions at all)
  if (((d.W % 16) != 0 || g.PQ <= 1024) && window_linear_geom(g, wt)) {
    wt->smem = 1024 + 2 * (size_t)wt->num_kb * kTileM * 128 + (size_t)wt->num_kb * wt->tile_n * 128 + kWindowStages * (size_t)wt->win_bytes +
               (size_t)round_up(wt->K_pad, 128) + 256;
    return wt->mtot <= 0x7FFFFF00LL && wt->smem <= 200 * 1024;
  }
  wt->linear = 0;
  // the window is one tiled TMA box of the NCHW tensor: rows must be multiples of 16 bytes, every box
  // extent at most 256
  if ((d.W % 16) != 0) return false;
  wt->left = round_up(d.pad_w, 16);
  wt->off0 = wt->left - d.pad_w;
  long long best_tiles = -1;
  for (int tw = kTileM; tw >= 16; tw >>= 1) {
    const int th = kTileM / tw;
    // last byte a row can touch: the last pixel's last (padded) tap, plus the second word of an unaligned read
    const long long ww = round_up((int)std::min<long long>((long long)(tw - 1) * d.stride_w + wt->off0 + wt->S_run + 8, 1 << 20), 16);
    const long long wh = (long long)(th - 1) * d.stride_h + (long long)(d.R - 1) * d.dil_h + 1;
    if (ww > 256 || wh > 256 || (long long)d.C * wh * ww > 24 * 1024) continue;
    const long long tiles = (long long)((g.P + th - 1) / th) * ((g.Q + tw - 1) / tw);
    if (best_tiles < 0 || tiles < best_tiles) {
      best_tiles = tiles;
      wt->tile_w = tw;
      wt->tile_h = th;
      wt->win_w = (int)ww;
      wt->win_h = (int)wh;
    }
  }
  if (best_tiles < 0) return false;
  wt->tiles_h = (g.P + wt->tile_h - 1) / wt->tile_h;
  wt->tiles_w = (g.Q + wt->tile_w - 1) / wt->tile_w;
  wt->box_bytes = d.C * wt->win_h * wt->win_w;
  wt->win_bytes = round_up(wt->box_bytes + 32, 128);
  wt->mtot = (long long)d.N * wt->tiles_h * wt->tiles_w * kTileM;
  wt->smem = 1024 + 2 * (size_t)wt->num_kb * kTileM * 128 + (size_t)wt->num_kb * wt->tile_n * 128 + kWindowStages * (size_t)wt->win_bytes +
             (size_t)round_up(wt->K_pad, 128) + 256;
  return wt->mtot <= 0x7FFFFF00LL && wt->smem <= 200 * 1024 && (long long)d.N * wt->tiles_h * wt->tiles_w < 0x7FFFFFFFLL;
}

// ---- window unroll over planes of units (B2C_VARIANT_IM2COL_WINDOW) ------------------------------------------------------------------
namespace {

// One form of the units (see conv_mma_plane.cu): which units a position has, and where the MMAs find them.
struct PlaneForm {
  int runw, ndh, ndw, planes, run_groups;
  int qb;  // row form: columns of a builder item
  int max_dh, max_ri, max_si;  // largest row phase, vertical and horizontal shift in grid positions
  int8_t row_phase[kMaxStridePhases], col_phase[kMaxStridePhases];
  int pitch, rpi;
  struct Unit {
    int plane, ri, si;
    int src[16];  // filter element of every byte, -1 = zero
  };
  std::vector<Unit> units;
};

bool plane_form(const Geom& g, bool row_form, bool whole_sectors, PlaneForm* f) {
  const b2c_conv_desc& d = g.d;
  const int sh = d.stride_h, sw = d.stride_w;
  if (sh > kMaxStridePhases || sw > kMaxStridePhases) return false;
  // (row form: from 8 channels on the 16-channel units are at least half full, and their builder moves more per load:
  // 16 x 14 x 14, 15501 images, 97 us against 117)
  if (row_form && (d.dil_w != 1 || d.S > 24 || d.C >= 8)) return false;
  int rowidx[kMaxStridePhases];
  std::fill(rowidx, rowidx + kMaxStridePhases, -1);
  std::fill(f->row_phase, f->row_phase + kMaxStridePhases, (int8_t)0);
  std::fill(f->col_phase, f->col_phase + kMaxStridePhases, (int8_t)-1);
  f->max_dh = f->max_ri = f->max_si = 0;
  for (int r = 0; r < d.R; ++r) {
    rowidx[(long long)r * d.dil_h % sh] = 0;
    f->max_ri = std::max<long long>(f->max_ri, (long long)r * d.dil_h / sh);
  }
  f->ndh = 0;
  for (int p = 0; p < sh; ++p)
    if (rowidx[p] == 0) {
      f->row_phase[f->ndh] = (int8_t)p;
      rowidx[p] = f->ndh++;
      f->max_dh = p;
    }
  f->units.clear();
  if (row_form) {
    // Runs of RUNW words of one (channel, row phase); G of them make U units.
    f->ndw = 1;
    f->runw = d.S <= 4 ? 1 : (d.S <= 8 ? 2 : (d.S <= 16 ? 4 : 6));
    const int G = f->runw == 1 ? 4 : (f->runw == 4 ? 1 : 2), U = G * f->runw / 4;
    f->run_groups = (d.C * f->ndh + G - 1) / G;
    f->qb = sw <= 2 ? 4 : 1;
    f->planes = f->run_groups * U;
    if (f->planes > 64) return false;
    for (int plane = 0; plane < f->planes; ++plane)
      for (int ri = 0; ri <= f->max_ri; ++ri) {
        PlaneForm::Unit u;
        u.plane = plane;
        u.ri = ri;
        u.si = 0;
        bool any = false;
        for (int b = 0; b < 16; ++b) {
          const int word = (plane % U) * 4 + b / 4;
          const int run = plane / U * G + word / f->runw;
          const int s = word % f->runw * 4 + b % 4, c = run / f->ndh, dh = f->row_phase[run % f->ndh];
          const long long off = (long long)ri * sh + dh;
          const int r = (int)(off / d.dil_h);
          u.src[b] = (c < d.C && s < d.S && off % d.dil_h == 0 && r < d.R) ? (c * d.R + r) * d.S + s : -1;
          any |= u.src[b] >= 0;
        }
        if (any) f->units.push_back(u);
      }
  } else {
    f->runw = 0;
    f->run_groups = 0;
    f->qb = 4;
    int colidx[kMaxStridePhases];
    std::fill(colidx, colidx + kMaxStridePhases, -1);
    for (int s = 0; s < d.S; ++s) {
      colidx[(long long)s * d.dil_w % sw] = 0;
      f->max_si = std::max<long long>(f->max_si, (long long)s * d.dil_w / sw);
    }
    f->ndw = 0;
    for (int p = 0; p < sw; ++p)
      if (colidx[p] == 0) f->col_phase[p] = (int8_t)(colidx[p] = f->ndw++);
    const int ncb = (d.C + 15) / 16;
    if ((long long)ncb * f->ndh * f->ndw > 64 || (long long)ncb * d.R * d.S > 1024) return false;
    f->planes = ncb * f->ndh * f->ndw;
    for (int cb = 0; cb < ncb; ++cb)
      for (int r = 0; r < d.R; ++r)
        for (int s = 0; s < d.S; ++s) {
          PlaneForm::Unit u;
          u.plane = (cb * f->ndh + rowidx[r * d.dil_h % sh]) * f->ndw + colidx[s * d.dil_w % sw];
          u.ri = r * d.dil_h / sh;
          u.si = s * d.dil_w / sw;
          for (int b = 0; b < 16; ++b) u.src[b] = cb * 16 + b < d.C ? ((cb * 16 + b) * d.R + r) * d.S + s : -1;
          f->units.push_back(u);
        }
  }
  // Grid of an image: P + max_ri rows of Q + max_si positions; with stride 1 the zero rows (columns) below
  // (right of) an image are the ones above (left of) the next image (row).
  const int cols = g.Q + f->max_si, rows = g.P + f->max_ri;
  const int share_w = (row_form || sw != 1) ? 0 : std::max(0, std::min(std::min(d.pad_w, f->max_si), cols - (d.W + d.pad_w)));
  const int share_h = sh != 1 ? 0 : std::max(0, std::min(std::min(d.pad_h, f->max_ri), rows - (d.H + d.pad_h)));
  f->pitch = cols - share_w;
  // (the added columns stay zero)
  if (whole_sectors) f->pitch = g.Q + round_up(f->pitch - g.Q, (d.out_mode & B2C_OUT_I32) ? kSectorOutputs : 4 * kSectorOutputs);
  f->rpi = rows - share_h;
  return true;
}

// Grid rows after which NKPQ results start on a memory sector again (1: every row does; 0: no schedule can keep to sectors).
// The channel form takes windows of so many rows; the row form's tiles start before a window that does not start on a boundary.
// A grid row's outputs are one run of memory, and the next row's follow without a gap; so where the row's overhang is a
// multiple of a sector's outputs, a warp's 32 positions lie the same way to the sectors all through a window, and windows
// that start on a boundary keep every store on it.  Stores of 32 int32 results from any start took 67 us for 253 MB, from sector
// boundaries 47: the memory side pays for the two partly written sectors, not the SM.  H * W of the results decides how many
// channels start on a boundary: all (a multiple of 8; 32 for int8), or every other one (4, 16); fewer are not worth it.
int plane_sector_rows(const Geom& g, int pitch) {
  const b2c_conv_desc& d = g.d;
  if (d.out_layout != B2C_LAYOUT_NCHW) return 0;
  const int outputs = (d.out_mode & B2C_OUT_I32) ? kSectorOutputs : 4 * kSectorOutputs;
  if ((pitch - g.Q) % outputs != 0 || g.PQ % (outputs / 2) != 0) return 0;
  int rows = 1;
  while ((long long)rows * g.Q % outputs != 0) rows <<= 1;
  return rows;
}

// Schedule of one form with per_sm blocks per SM, windows of min_tiles to max_tiles accumulator tiles, dealt one by one
// (`dealt`) or in segments, at most `stages` (see plane_choices): window height,
// column tile and stages with the lowest estimated time (returned; negative if nothing fits).  The estimate adds up,
// in SM cycles, what a window costs each role (constants measured on the kernel: builder items, 39 cycles and up per
// MMA, the store path) and takes the slowest role per window, the way of the first window to its MMAs and the stores
// of the last one.
double plane_schedule(const Geom& g, int groups, const PlaneForm& f, int per_sm, bool dealt, int min_tiles, int max_tiles, int stages,
                      bool whole_sectors, PlaneArgs* pl) {
  const b2c_conv_desc& d = g.d;
  const int HW = d.H * d.W;
  const long long total_rows = (long long)d.N * f.rpi;
  if (total_rows > 0x3FFFFFFF || (total_rows + 64) * f.pitch > 0x3FFFFFFFLL) return -1;
  const int num_mma = ((int)f.units.size() + 1) / 2;
  const int n16 = round_up(d.K, 16);
  const int nruns = d.C * f.ndh, ncb = (d.C + 15) / 16;
  const double out_bytes = (d.out_mode & B2C_OUT_I32 ? 4.0 : 0.0) + (d.out_mode & B2C_OUT_I8 ? 1.0 : 0.0);
  const int step = whole_sectors ? plane_sector_rows(g, f.pitch) : 1;  // rows of windows and segments come in multiples of it
  const int outputs = (d.out_mode & B2C_OUT_I32) ? kSectorOutputs : 4 * kSectorOutputs;
  const int max_lead = f.runw > 0 && plane_sector_rows(g, f.pitch) > 1 ? outputs - 1 : 0;
  const double out_cost = (d.out_mode & B2C_OUT_I32 ? (whole_sectors ? 4.0 : 5.0) : 0.0) + (d.out_mode & B2C_OUT_I8 ? 3.0 : 0.0);
  const int kb = per_sm == 2 ? 4 : 8, sets = per_sm == 2 ? 1 : 2;  // builder warps; sets of four epilogue warps
  const int smem_max = per_sm == 2 ? 110 * 1024 : kPlaneSmemMax;
  double best = -1;
  int tile_list[6], ntl = 0;
  // column tiles: all channels if they fit; narrower ones repeat the building of the units, and are tried only while
  // there are too few tiles for every SM
  const bool few = total_rows * f.pitch * groups < 2LL * kNumSMs * kTileM;
  for (int t = few ? 16 : 64; t < n16 && t <= 256; t <<= 1)
    if (few || n16 > 128) tile_list[ntl++] = t;
  if (n16 <= 256) tile_list[ntl++] = n16;
  for (int ti = 0; ti < ntl; ++ti) {
    const int tile_n = tile_list[ti];
    const long long w_bytes = (long long)num_mma * 32 * tile_n;
    if (w_bytes > 150 * 1024) continue;
    const int cols = (d.K + tile_n - 1) / tile_n;
    if ((long long)cols * groups > 65535) continue;
    // (two accumulators at least: with one, a set of epilogue warps that takes every other tile would find its wait
    // already satisfied by the phase of two tiles before)
    const int nbuf = std::min(kMaxAcc, 512 / per_sm / tile_n);
    if (nbuf < 2) continue;
    int tmem_cols = 32;
    while (tmem_cols < nbuf * tile_n) tmem_cols <<= 1;
    const int places = (int)std::max<long long>(1, (long long)kNumSMs * per_sm / ((long long)cols * groups));
    for (int th = 1; th <= 128; th += 1 + th / 16) {
      const int tiles = (th * f.pitch + kTileM - 1) / kTileM;  // (the estimate leaves out what a lead can add)
      if (th % step != 0) continue;
      if (th > 1 && (tiles > max_tiles || th > total_rows)) break;
      if (tiles < min_tiles) continue;
      const int wr = th + f.max_ri;
      const long long plane_units = (long long)wr * f.pitch;
      const long long last_read = (long long)(th * f.pitch + max_lead + kTileM - 1) / kTileM * kTileM + (long long)f.max_ri * f.pitch + f.max_si + 1;
      const long long win_bytes = (((f.planes - 1) * plane_units + std::max(plane_units, last_read)) * 16 + 127) / 128 * 128;
      if (win_bytes > 200 * 1024) break;
      // Segments: single windows; or a block's share of all rows, cut further when the outputs that are being written
      // at the same time spread over more than about 100 MB; each segment builds its first max_ri rows anew.
      int blocks = (int)std::min<long long>(places, (total_rows + th - 1) / th);
      long long share = (total_rows + blocks - 1) / blocks;
      if (dealt) share = std::min<long long>(share, th);
      // Images of several windows: windows and segments end with the image (its overhang rows are no output rows, and
      // no window needs rows of two images); equal parts of it.
      int spi = 0;
      if (f.rpi >= 2 * th) {
        const long long want = std::max<long long>(th, std::min<long long>(share, g.P));  // rows of a segment
        spi = (int)((g.P + want - 1) / want);
        share = (g.P + spi - 1) / spi;
        if (share > th && !dealt) share = (share + th - 1) / th * th;
        spi = (int)((g.P + share - 1) / share);
        blocks = (int)std::min<long long>(places, (long long)d.N * spi);
      }
      if (whole_sectors && (spi == 0 ? g.Q % outputs != 0 : spi > 1 && share % step != 0)) continue;
      // (a window in the middle of an image that does not start on a boundary)
      const int lead_mask = spi > 0 && max_lead > 0 && ((long long)th * g.Q % outputs != 0 || share * g.Q % outputs != 0) ? max_lead : 0;
      const double active = (double)blocks * share * f.pitch * d.K * groups * out_bytes;
      if (spi == 0 && active > 100e6 && share > th) {
        const int parts = (int)std::min<double>((double)((share + th - 1) / th), std::ceil(active / 100e6));
        share = (total_rows + (long long)blocks * parts - 1) / ((long long)blocks * parts);
      }
      const long long segs = spi ? (long long)d.N * spi : (total_rows + share - 1) / share, segs_per_block = (segs + blocks - 1) / blocks;
      const long long per_block = (share + th - 1) / th * segs_per_block;
      const double conc = (double)std::min<long long>(per_sm, std::max<long long>(1, ((long long)blocks * cols * groups + kNumSMs - 1) / kNumSMs));
      const double mma = tiles * (num_mma * std::max(40.0, tile_n / 2.0) + 150.0);
      const double valid = (double)g.P / f.rpi * g.Q / f.pitch;
      const double tile_out = 4.0 * tile_n * out_cost * (0.4 + 0.6 * valid);  // store path of the SM
      const double tile_lat = 600.0 + tile_n * 2.5 * out_cost;                // one set of warps, start to end
      const double epi = std::max(conc * th * f.pitch / kTileM * tile_out, (double)((tiles + sets - 1) / sets) * tile_lat);
      // raw chunks of the window's new rows; also of the whole first window when a block has only that one
      for (int cr = th; cr <= wr; cr += std::max(1, f.max_ri)) {
        const bool whole_first = cr == wr && (dealt || per_block == 1);
        if (dealt ? !whole_first : (cr != th && !whole_first)) continue;
        if (share > th && cr != th) continue;  // segments of several windows: the kernel's overlap move relies on it
        // raw staging: rows of at most two images per channel, or whole images when a chunk spans more (or they
        // are small enough not to matter: one copy per image instead of one per channel)
        const int images = (int)std::min<long long>(d.N, cr <= 1 ? 1 : (cr - 2) / f.rpi + 2);
        const int raw_rows = std::min(cr * d.stride_h, images * d.H);
        const long long rows_bytes = (long long)d.C * (round_up(raw_rows * d.W, 16) + 64);
        const int img_slot = round_up(d.C * HW + 15, 16) + 16;
        const long long whole_bytes = (long long)images * img_slot;
        const bool whole = images > 2 || whole_bytes <= rows_bytes + rows_bytes / 4 || whole_bytes <= 8192;
        // one tiled copy for all channels: they start on 16 bytes, the segment fits a box, and no chunk has two images
        const int box = round_up(raw_rows * d.W + 15, 16);
        const bool tiled = !whole && spi > 0 && HW % 16 == 0 && d.C >= 4 && d.C <= 256 && box <= 1024;
        const long long raw_data = whole ? whole_bytes : (tiled ? (long long)d.C * box : rows_bytes);
        const double copies = whole ? images : (tiled ? 1.0 : (double)d.C * (spi ? 1.0 : 1.0 + (double)cr / f.rpi));
        const long long raw_bytes = (raw_data + 2 * kPlaneMargin + 127) / 128 * 128;
        const int first_chunks = (int)((std::min<long long>(share, th) + f.max_ri + cr - 1) / cr);
        const long long row_items = f.runw ? (f.pitch + f.qb - 1) / f.qb : (long long)ncb * f.ndh * ((d.W + 3) / 4);
        auto build_cycles = [&](long long rows, double* lat) {
          // SM issue and shared-memory cycles of the items, and the way of one warp through its share of them
          const double item = f.runw ? 15.0 + nruns * (4.0 + f.qb * 2.0 + 1.5 * f.runw) + f.planes * (6.0 + 6.0 * f.qb) : 150.0;
          const double one = f.runw ? 250.0 + f.run_groups * (130.0 + 12.0 * f.qb * f.runw) : 900.0;
          const long long items = rows * row_items;
          *lat = (double)((items + kb * 32 - 1) / (kb * 32)) * one;
          return (double)items / 32 * item;
        };
        double build_lat, first_lat;
        const long long new_rows = dealt ? wr : th;
        const double move = dealt || f.max_ri == 0 ? 0.0 : (double)f.planes * f.max_ri * f.pitch / 32 * 12.0 + 300.0;
        const double build = build_cycles(new_rows, &build_lat) + move;
        (void)build_cycles(std::min<long long>(share, th) + f.max_ri, &first_lat);
        build_lat += move / kb + 300.0;
        const double copy = 900.0 + (double)raw_data / 24.0 + copies * 60.0;
        for (int st = 2 - stages; st < 3; ++st) {
          const bool single = per_block == 1;
          const int ws = st < 2 ? 2 : 1, rs = (single && whole_first) ? 1 : (st < 1 ? 2 : 1);
          if (single && st < 2) continue;
          if (ws == 1 && !dealt && !single && th < f.max_ri) continue;  // the overlap rows are moved inside the buffer
          const long long smem = 128 + (lead_mask ? (lead_mask + 1) * 16 : 0) + ws * win_bytes + rs * raw_bytes + w_bytes + 8LL * round_up(num_mma, 4);
          if (smem > smem_max) continue;
          // one buffer between two roles makes them take turns
          double chain = rs == 1 ? copy + build_lat : std::max(copy, build_lat);
          if (ws == 1) chain = build_lat + std::max(rs == 1 ? copy : 0.0, mma);
          const double steady = std::max(std::max(conc * build, conc * mma), std::max(epi, chain));
          // (a last, partly filled round of segments: the stores of the others' get its share of the memory)
          const double windows = std::max(1.0, (dealt || spi) ? (double)((share + th - 1) / th) * 0.5 * (std::ceil((double)segs / blocks) + (double)segs / blocks) : (double)total_rows / blocks / th);
          const double t = 3000 + copy * (rs == 1 ? first_chunks : 1) + first_lat + first_chunks * 150.0 + mma / tiles + epi + w_bytes / 40.0 * conc +
                           (windows - 1) * steady + (dealt ? 0.0 : (double)(segs_per_block - 1) * f.max_ri / th * conc * build);
          if (best >= 0 && t >= best * 0.999) continue;
          best = t;
          pl->pitch = f.pitch;
          pl->total_rows = (int)total_rows;
          pl->tile_n = tile_n;
          pl->cols = cols;
          pl->tmem_cols = tmem_cols;
          pl->nbuf = nbuf;
          pl->per_sm = per_sm;
          pl->th = th;
          pl->cr = cr;
          pl->tiles = tiles;
          pl->seg_rows = (int)share;
          pl->segs = (int)segs;
          pl->blocks = std::min<int>(blocks, pl->segs);
          pl->plane_bytes = (int)plane_units * 16;
          pl->win_bytes = (int)win_bytes;
          pl->whole_images = whole ? 1 : 0;
          pl->img_slot = img_slot;
          pl->c_pitch = tiled ? box : round_up(raw_rows * d.W, 16) + 64;
          pl->box_bytes = tiled ? box : 0;
          pl->spi = spi;
          pl->lead_mask = lead_mask;
          pl->raw_bytes = (int)raw_bytes;
          pl->win_stages = ws;
          pl->raw_stages = rs;
          pl->w_bytes = (int)w_bytes;
          pl->smem = (int)smem;
        }
      }
    }
  }
  return best;
}

// Form and schedules of the plane kernel, the lowest estimate first: the best one for each number of blocks per SM,
// way of dealing windows, range of window heights and number of buffers, rows as narrow as can be or widened to whole sectors
// (their order depends on how the store path, the builders and DRAM share the time, which the estimate knows to 10 to
// 25 %; the timed selection tries them all).
struct PlaneChoice {
  double t;
  PlaneArgs pl;
};
bool plane_choices(const Geom& g, int groups, PlaneForm* form, std::vector<PlaneChoice>* out) {
  const b2c_conv_desc& d = g.d;
  // (enumerating a problem and creating a plan for one of its embeddings search the same descriptor one after the
  // other: the last search of this thread is kept, by the descriptor's values)
  struct Last {
    b2c_conv_desc d;
    int groups = 0;
    PlaneForm form;
    std::vector<PlaneChoice> list;
  };
  static thread_local Last last;
  if (last.groups == groups && std::memcmp(&last.d, &d, sizeof(d)) == 0) {
    *form = last.form;
    *out = last.list;
    return !out->empty();
  }
  out->clear();
  if (d.in_layout != B2C_LAYOUT_NCHW || d.pad_h > 32 || d.pad_w > 32 || d.K > 1024) return false;
  // (above 96 channels the weights of a column tile and the units of a window no longer fit beside each other: 30
  // images of 128 x 28 x 28 -> 128, 3x3, 19.7 us against 11.3 by the channel pack)
  if (d.C > 96) return false;
  // Images of a few pixels would fill a window with the overhang of many images; the channel-pack maps do those.
  if ((d.W % 16) != 0 && g.PQ < 43) return false;
  if ((long long)d.C * d.H * d.W > (1 << 26) || d.W > 8192) return false;
  double best = -1;
  for (int f = 0; f < 2; ++f) {
    PlaneForm cand;
    std::vector<PlaneChoice> list;
    // blocks per SM, dealt, fewest and most tiles of a window, buffers (2: two windows and two raw chunks, 1: two and
    // one, 0: one of each; fewer are often better although no role waits less: they leave the L1 more room)
    static const int kStyles[10][5] = {{1, 1, 4, 5, 0}, {1, 1, 5, 8, 1}, {1, 1, 4, 8, 2},  {1, 1, 9, 16, 2}, {2, 1, 1, 4, 2},
                                       {2, 1, 5, 16, 0}, {2, 1, 5, 8, 1}, {2, 1, 9, 16, 1}, {2, 0, 5, 16, 2}, {1, 0, 1, 16, 2}};
    int narrow = 0;
    for (int whole_sectors = 0; whole_sectors < 2; ++whole_sectors) {
      if (!plane_form(g, f == 1, whole_sectors != 0, &cand)) break;
      // Rows widened to whole sectors are listed beside the others where they cost little: every tile of 128 positions then holds
      // fewer outputs.  Best schedule of either kind, 3x3, us: 57 -> 64 positions, 64 x 56 x 56 -> 64, 315 images 79 and 74, 100
      // 28.9 and 24.5, 16 9.2 and 8.9, 8 and fewer the same; 101 -> 108, 20 images of 32 x 100 x 100 -> 64 17.2 and 15.5, but 4 images
      // 7.1 and 7.8; 61 -> 68 and 113 -> 120 2 % less; 51 -> 58 and 53 -> 60 10 % more; 29 -> 36, depth-wise on 28 x 28, no gain.
      if (whole_sectors && (cand.pitch == narrow || cand.pitch * 20 > narrow * 23 || plane_sector_rows(g, cand.pitch) == 0)) break;
      narrow = cand.pitch;
      for (const int* style : kStyles) {
        PlaneChoice c;
        std::memset(&c.pl, 0, sizeof(c.pl));
        c.t = plane_schedule(g, groups, cand, style[0], style[1] != 0, style[2], style[3], style[4], whole_sectors != 0, &c.pl);
        if (c.t < 0) continue;
        bool same = false;
        for (const PlaneChoice& o : list)
          same |= o.pl.pitch == c.pl.pitch && o.pl.per_sm == c.pl.per_sm && o.pl.th == c.pl.th && o.pl.seg_rows == c.pl.seg_rows &&
                  o.pl.tile_n == c.pl.tile_n && o.pl.win_stages == c.pl.win_stages && o.pl.raw_stages == c.pl.raw_stages;
        if (!same) list.push_back(c);
      }
    }
    if (list.empty()) continue;
    std::stable_sort(list.begin(), list.end(), [](const PlaneChoice& a, const PlaneChoice& b) { return a.t < b.t; });
    if (best >= 0 && list[0].t >= best) continue;
    best = list[0].t;
    *form = cand;
    *out = list;
  }
  last.d = d;
  last.groups = groups;
  last.form = *form;
  last.list = *out;
  return !out->empty();
}

}  // namespace

bool plane_plan(const Geom& g, int groups, int nth, PlaneArgs* pl, std::vector<uint64_t>* table, std::vector<int32_t>* wsrc) {
  const b2c_conv_desc& d = g.d;
  std::memset(pl, 0, sizeof(*pl));
  PlaneForm f;
  std::vector<PlaneChoice> list;
  if (!plane_choices(g, groups, &f, &list)) return false;
  if (nth < 0 || nth >= (int)list.size()) return false;
  *pl = list[nth].pl;
  f.pitch = pl->pitch;  // (the form was searched with rows of two widths)
  const int HW = d.H * d.W;
  pl->runw = f.runw;
  pl->sh = d.stride_h;
  pl->sw = d.stride_w;
  pl->ndh = f.ndh;
  pl->ndw = f.ndw;
  pl->max_dh = f.max_dh;
  std::memcpy(pl->row_phase, f.row_phase, sizeof(pl->row_phase));
  std::memcpy(pl->col_phase, f.col_phase, sizeof(pl->col_phase));
  pl->planes = f.planes;
  pl->rpi = f.rpi;
  pl->max_ri = f.max_ri;
  pl->num_mma = ((int)f.units.size() + 1) / 2;
  pl->gpr = f.runw ? (f.pitch + f.qb - 1) / f.qb : (d.W + 3) / 4;
  pl->run_groups = f.run_groups;
  pl->zero_fill = f.runw == 0 ? 1 : 0;
  // words: rows start on one when W does and every channel starts on one (segments: 16 bytes, the alignment of
  // all channels is then the same)
  pl->aligned = (d.W % 4 == 0 && (pl->whole_images || HW % 16 == 0)) ? 1 : 0;
  // flat groups: channels start on words (of memory, hence of the staged copy), and a group crosses one row end at most
  if (f.runw == 0 && d.stride_h == 1 && d.stride_w == 1 && HW % 4 == 0 && d.W >= 4) pl->aligned = 2;
  pl->div_rpi = make_fastdiv((uint32_t)f.rpi);
  pl->div_pitch = make_fastdiv((uint32_t)f.pitch);
  pl->div_gpr = make_fastdiv((uint32_t)pl->gpr);
  pl->div_nu = make_fastdiv((uint32_t)std::max(1, f.planes / f.ndw));
  pl->div_w = make_fastdiv((uint32_t)d.W);
  pl->div_spi = make_fastdiv((uint32_t)std::max(1, pl->spi));
  pl->img_channels = d.C * groups;
  pl->div_hw4 = make_fastdiv((uint32_t)std::max(1, HW / 4));
  pl->div_overlap = make_fastdiv((uint32_t)std::max(1, f.max_ri * f.pitch));
  pl->div_sw = make_fastdiv((uint32_t)d.stride_w);
  if (table && wsrc) {
    // units in address order, two per MMA; a last odd one is paired with its neighbour under zero weights
    std::vector<std::pair<int, int>> order;
    for (size_t i = 0; i < f.units.size(); ++i)
      order.push_back({f.units[i].plane * (pl->plane_bytes / 16) + f.units[i].ri * f.pitch + f.units[i].si, (int)i});
    std::sort(order.begin(), order.end());
    table->clear();
    wsrc->assign((size_t)pl->num_mma * 32, -1);
    for (int m = 0; m < pl->num_mma; ++m) {
      const bool two = 2 * m + 1 < (int)order.size();
      const int a0 = order[2 * m].first, a1 = two ? order[2 * m + 1].first : a0 + 1;
      table->push_back((uint64_t)a0 | ((uint64_t)(a1 - a0) << 16));
      for (int u = 0; u < (two ? 2 : 1); ++u)
        for (int b = 0; b < 16; ++b) (*wsrc)[(size_t)(2 * m + u) * 16 + b] = f.units[order[2 * m + u].second].src[b];
    }
    // (the issuing warp reads the table four entries at a time)
    while (table->size() % 4 != 0) table->push_back(table->back());
  }
  return true;
}

bool stream_plan(const Geom& g, int tile_n, StreamArgs* sa, std::vector<uint64_t>* table, std::vector<int32_t>* wsrc) {
  const b2c_conv_desc& d = g.d;
  std::memset(sa, 0, sizeof(*sa));
  const int HW = d.H * d.W;
  if (d.in_layout != B2C_LAYOUT_NCHW || d.stride_h != d.stride_w || d.stride_h > 2 || d.W < 4 || d.pad_h > 32 || d.pad_w > 32) return false;
  // (bulk copies of a channel block start and end on 16 bytes)
  if ((long long)d.C * HW % 16 != 0 || (long long)d.C * HW > (1 << 26) || d.K > 4096) return false;
  // the grid and the units of a block of 32 channels
  Geom block = g;
  block.d.C = 32;
  PlaneForm f;
  if (!plane_form(block, false, false, &f) || f.pitch > kTileM) return false;
  const long long total_rows = (long long)d.N * f.rpi;
  if (total_rows > 0x3FFFFFF0 / f.pitch) return false;
  const int sh = d.stride_h;
  sa->stride = sh;
  sa->words = HW % 4 == 0 ? 1 : 0;
  sa->ndh = f.ndh;
  sa->ndw = f.ndw;
  sa->max_dh = f.max_dh;
  for (int p = 0; p < 2; ++p) {
    sa->row_phase[p] = f.row_phase[p];
    sa->row_index[p] = -1;
    sa->col_index[p] = f.col_phase[p];
  }
  for (int i = 0; i < f.ndh; ++i) sa->row_index[f.row_phase[i]] = (int8_t)i;
  sa->pitch = f.pitch;
  sa->rpi = f.rpi;
  sa->total_rows = (int)total_rows;
  sa->max_ri = f.max_ri;
  sa->images = d.N;
  sa->th = kTileM / f.pitch;
  sa->ncb = (d.C + 31) / 32;
  sa->taps = d.R * d.S;
  const int wr = sa->th + f.max_ri;
  const int plane_units = wr * f.pitch;
  const int last_read = kTileM + f.max_ri * f.pitch + f.max_si;
  sa->plane_bytes = plane_units * 16;
  sa->win_bytes = (((f.planes - 1) * plane_units + std::max(plane_units, last_read)) * 16 + 127) / 128 * 128;
  if ((long long)f.ndh * f.ndw * plane_units > 16000) return false;  // (14 bits of the descriptor)
  // images of a tile whose rows it needs, and the most raw rows of one (the tiles repeat after rpi of them)
  sa->div_rpi = make_fastdiv((uint32_t)f.rpi);
  ConvArgs rows = {};  // (what the row functions read of it)
  rows.H = d.H;
  rows.pad_h = d.pad_h;
  rows.out_P = g.P;
  int raw_rows = 0;
  const long long tiles_m = (total_rows + sa->th - 1) / sa->th;
  for (long long t = 0; t < std::min<long long>(tiles_m, f.rpi); ++t) {
    const TileRows tr = stream_tile_rows(rows, *sa, (int)(t * sa->th));
    for (int n = tr.n_a; n * f.rpi < tr.end; ++n) {
      const RawRows r = stream_raw_rows(rows, *sa, tr, n, sh);
      if (r.hi <= r.lo) continue;
      sa->max_images = std::max(sa->max_images, n - tr.n_a + 1);
      raw_rows = std::max(raw_rows, r.hi - r.lo);
    }
  }
  if (sa->max_images < 1 || sa->max_images > 32) return false;
  // raw rows: whole images of a channel block, one bulk copy each, or one tiled copy per image of the rows needed
  const int box = round_up(raw_rows * d.W + 15, 16);
  const bool tiled = HW % 16 == 0 && box <= 1024 && (long long)box < HW;
  if (!tiled && 32LL * HW * sa->max_images > 40 * 1024) return false;
  sa->box_bytes = tiled ? box : 0;
  sa->img_slot = round_up(32 * (tiled ? box : HW), 128);
  sa->img_groups = tiled ? (raw_rows * d.W + 6) / 4 : (std::min(HW, raw_rows * d.W) + 6) / 4;
  sa->raw_bytes = sa->img_slot * sa->max_images;
  sa->tile_n = tile_n;
  sa->cols = (d.K + tile_n - 1) / tile_n;
  sa->tmem_cols = 2 * tile_n;
  sa->num_tiles = (int)((tiles_m + 1) / 2) * sa->cols;
  // weights: 16 KB a stage and block; the run of a half column tile is read in 1 KB rows
  sa->b_group = 1024 / tile_n;
  sa->b_stage_bytes = sa->b_group * tile_n * 16;
  const int total_mma = sa->ncb * sa->taps;
  sa->w_steps = (total_mma + sa->b_group - 1) / sa->b_group;
  sa->w_run_rows = total_mma * tile_n / 64;
  const int table_bytes = 8 * (round_up(sa->taps, 4) + 4);
  // rings: four windows and raw blocks where they leave room for six weight stages, else fewer
  static const int kRings[6][3] = {{4, 4, 6}, {4, 3, 5}, {3, 3, 5}, {3, 3, 4}, {2, 2, 4}, {2, 2, 3}};
  int ring = 0;
  for (; ring < 6; ++ring) {
    sa->win_stages = kRings[ring][0];
    sa->raw_stages = kRings[ring][1];
    const int rest = kStreamSmemMax - 128 - table_bytes - sa->win_stages * sa->win_bytes - sa->raw_stages * sa->raw_bytes;
    sa->b_stages = rest < 0 ? 0 : std::min(std::min(kStreamMaxStages, sa->w_steps + 1), rest / sa->b_stage_bytes);
    if (sa->b_stages >= std::min(kRings[ring][2], sa->w_steps + 1)) break;
  }
  if (ring == 6) return false;
  sa->smem = 128 + table_bytes + sa->win_stages * sa->win_bytes + sa->raw_stages * sa->raw_bytes + sa->b_stages * sa->b_stage_bytes;
  sa->pairs = kNumSMs / 2;
  sa->div_pitch = make_fastdiv((uint32_t)f.pitch);
  sa->div_w = make_fastdiv((uint32_t)d.W);
  sa->div_groups = make_fastdiv((uint32_t)sa->img_groups);
  sa->div_cols = make_fastdiv((uint32_t)sa->cols);
  if (table && wsrc) {
    // one MMA per tap: the two 16-channel blocks at one position
    table->clear();
    wsrc->assign((size_t)total_mma * 32, -1);
    const int half = f.ndh * f.ndw * plane_units;
    for (int r = 0; r < d.R; ++r)
      for (int s = 0; s < d.S; ++s) {
        const PlaneForm::Unit& u = f.units[r * d.S + s];  // (of the first 16 channels)
        table->push_back((uint64_t)(u.plane * plane_units + u.ri * f.pitch + u.si) | ((uint64_t)half << 16));
        for (int cb = 0; cb < sa->ncb; ++cb)
          for (int c = 0; c < 32 && cb * 32 + c < d.C; ++c)
            (*wsrc)[((size_t)cb * sa->taps + r * d.S + s) * 32 + c] = ((cb * 32 + c) * d.R + r) * d.S + s;
      }
    while (table->size() % 4 != 0) table->push_back(table->back());
  }
  return true;
}

// The plane kernel builds every input row once per window and needs windows of several tiles to pay for the rows the
// taps reach below; the window kernel's tiles are independent of each other and spread a small problem over more
// blocks.  Up to kPlaneMinTiles accumulator tiles a problem that the window kernel takes is listed for it alone; above,
// both are listed and the timed selection decides: which is faster depends on more than the number of tiles (7x7
// stride 2 of 3 x 224 x 224, 98 tiles an image: 16 images 14.3 us by the window kernel, 15.3 by this one, 100 images 72
// and 65; but 3x3 stride 2 of 12 x 36 x 256, 159 images, 64 channels, 2862 tiles, 31.5 and 42.2, and 3x3 of
// 8 x 154 x 48, 158 images, 24 channels, 9480 tiles, 96 and 119).
static bool plane_wanted(const WindowTile* wt) { return wt == nullptr || wt->mtot > (long long)kPlaneMinTiles * kTileM; }

// Accumulator rows that a schedule of the plane kernel issues: whole tiles of every window, the taps' overhang among
// them (see seg_rows and window_span in conv_mma_plane.cu).
long long plane_rows_issued(const Geom& g, const PlaneArgs& pl) {
  if (pl.lead_mask) {
    long long sum = 0;  // of one image, window by window: a window's tiles start up to lead_mask positions before it
    for (int r0 = 0; r0 < g.P; r0 += pl.seg_rows)
      for (int r = r0; r < std::min(r0 + pl.seg_rows, g.P); r += pl.th)
        sum += ((long long)std::min(pl.th, std::min(r0 + pl.seg_rows, g.P) - r) * pl.pitch + ((long long)r * g.Q & pl.lead_mask) + kTileM - 1) / kTileM;
    return sum * g.d.N * kTileM;
  }
  auto tiles = [&](long long rows) {  // of a segment
    const long long full = ((long long)pl.th * pl.pitch + kTileM - 1) / kTileM;
    return rows / pl.th * full + (rows % pl.th * pl.pitch + kTileM - 1) / kTileM;
  };
  const long long all = pl.spi > 0 ? g.P : pl.total_rows;  // rows that are cut into segments: an image's, or the batch's
  return ((all / pl.seg_rows) * tiles(pl.seg_rows) + tiles(all % pl.seg_rows)) * (pl.spi > 0 ? g.d.N : 1) * kTileM;
}

static void add(std::vector<Candidate>* out, const Geom& g, int variant, int tile_n, int split_k,
                bool swap = false, int tile_m = kTileM, int schedule = -1, long long plane_rows = 0, int plane_k = 0) {
  const b2c_conv_desc& d = g.d;
  Candidate e = {};
  e.schedule = schedule;
  e.map_m = swap ? B2C_AXIS_K : B2C_AXIS_NPQ;
  e.map_n = swap ? B2C_AXIS_NPQ : B2C_AXIS_K;
  e.variant = variant;
  e.tile_m = tile_m;
  e.tile_n = tile_n;
  e.split_k = split_k;
  e.device_us = -1.0f;
  long long M_pad = (g.Mg + tile_m - 1) / tile_m * tile_m;
  long long N_pad = (long long)round_up(d.K, tile_n);
  if (swap) {
    M_pad = (long long)round_up(d.K, kTileM);
    N_pad = (g.Mg + tile_n - 1) / tile_n * tile_n;
  }
  long long k_issued, moved;
  long long mac_min = g.Mg * d.K * g.Kg;
  long long data_min = g.x_elems + g.w_elems + g.y_elems;
  TmaView v;
  if (is_tma_view_variant(variant) && tma_view_for(g, variant, &v)) {
    e.map_k = (variant == B2C_VARIANT_CP_TMA || variant == B2C_VARIANT_DILATION_PACK || variant == B2C_VARIANT_CP_SHIFT)
                  ? B2C_AXIS_C
                  : ((variant == B2C_VARIANT_ROW_UNROLL || variant == B2C_VARIANT_ROWPHASE_SHIFT) ? B2C_AXIS_SC
                                                                                                  : B2C_AXIS_C_PHASES);
    if (!swap) M_pad = (view_rows(g, variant, v) + tile_m - 1) / tile_m * tile_m;
    k_issued = (long long)v.R * v.S * v.C;
    long long packed = v.bytes();
    bool direct = shift_base_variant(variant) == B2C_VARIANT_CP_TMA && d.in_layout == B2C_LAYOUT_NHWC && v.C == d.C;
    moved = (direct ? 0 : g.x_elems + packed) + packed + (long long)d.K * k_issued + g.y_elems;
  } else {
    e.map_k = B2C_AXIS_CRS;
    int K_pad = variant_k_pad(g, variant);
    k_issued = K_pad;
    WindowTile wt;
    if (schedule >= 0) {
      M_pad = plane_rows;
      K_pad = plane_k;
      k_issued = K_pad;
    } else if (variant == B2C_VARIANT_IM2COL_WINDOW && window_tile_geom(g, &wt)) {
      M_pad = wt.mtot;  // whole two-dimensional tiles
    }
    if (variant == B2C_VARIANT_IM2COL_EXPLICIT)
      moved = g.x_elems + 2 * g.Mg * K_pad + (long long)d.K * K_pad + g.y_elems;
    else if (variant == B2C_VARIANT_IM2COL_STAGED)
      moved = g.x_elems + (long long)d.K * K_pad + g.y_elems;
    else
      moved = g.x_elems + (long long)d.K * K_pad + g.y_elems;
  }
  if (split_k > 1 && !cluster_split_ok(variant, tile_n, split_k, swap)) moved += 2 * g.y_elems;  // partial sums through memory
  e.o_mac = M_pad * N_pad * k_issued - mac_min;
  e.o_data = moved - data_min;
  e.workspace_bytes = (int64_t)workspace_bytes_for(g, variant, tile_n, split_k, swap);
  // two-SM channel-pack schedule on NCHW input: room for the work counters of the pack that runs
  // inside the MMA kernel (1 + N integers after the rewritten operand)
  if (tile_m == 2 * kTileM && variant == B2C_VARIANT_CP_TMA && d.in_layout == B2C_LAYOUT_NCHW)
    e.workspace_bytes = (e.workspace_bytes + 255) / 256 * 256 + ((int64_t)(d.N + 1) * 4 + 255) / 256 * 256;
  out->push_back(e);
}

void enumerate_embeddings(const Geom& g, std::vector<Candidate>* out) {
  out->clear();
  const b2c_conv_desc& d = g.d;
  // Tile widths: every MMA N extent up to the first one that covers K.
  std::vector<int> tiles;
  for (int t = 16; t <= 256; t <<= 1) {
    tiles.push_back(t);
    if (t >= d.K) break;
  }
  for (int variant = 0; variant < kNumVariants; ++variant) {
    TmaView view;
    if (is_tma_view_variant(variant) && !tma_view_for(g, variant, &view)) continue;
    const long long tiles_m =
        ((is_tma_view_variant(variant) ? view_rows(g, variant, view) : g.Mg) + kTileM - 1) / kTileM;
    WindowGeom wg;
    if (variant == B2C_VARIANT_IM2COL_STAGED && !staged_window(g, &wg)) continue;
    if (variant == B2C_VARIANT_IM2COL_WINDOW) {
      // window kernel: one schedule, all output channels in one column tile (the weights are resident), no split
      WindowTile wt;
      const bool window = window_tile_geom(g, &wt);
      if (window) add(out, g, variant, wt.tile_n, 1);
      // plane kernel: one entry per schedule
      PlaneForm form;
      std::vector<PlaneChoice> plane;
      if (plane_wanted(window ? &wt : nullptr) && plane_choices(g, 1, &form, &plane))
        for (int i = 0; i < (int)plane.size(); ++i)
          add(out, g, variant, plane[i].pl.tile_n, 1, false, kTileM, i, plane_rows_issued(g, plane[i].pl),
              ((int)form.units.size() + 1) / 2 * kMmaK);
      // Stream kernel: more channels than the plane kernel takes, taps enough to pay for the building of the units, and tiles for
      // more than a few pairs of SMs.  The widest column tile builds the units least often; half of it where it leaves half
      // of the pairs without a tile (16 images of 192 x 28 x 28 -> 192, 3x3, 58 tiles: 11.9 us; half the tile a fifth more).
      if (d.C >= 48 && d.R * d.S >= 4) {
        int wide = 64;
        while (wide < d.K && wide < 256) wide <<= 1;
        StreamArgs sa;
        for (int t = wide; t >= std::max(64, wide / 2); t >>= 1) {
          if (!stream_plan(g, t, &sa) || sa.num_tiles < 8 || (t < wide && sa.num_tiles >= kNumSMs / 2)) break;
          add(out, g, variant, t, 1, false, kTileM, kStreamSchedule, (long long)sa.num_tiles / sa.cols * 2 * kTileM, sa.ncb * sa.taps * kMmaK);
        }
      }
      continue;
    }
    int num_kb;
    if (is_tma_view_variant(variant)) {
      num_kb = view.R * view.S * (view.C / cp_block_bytes(view.C));
    } else {
      num_kb = (variant_k_pad(g, variant) + 127) / 128;
    }
    // The in-kernel gather keeps its lookup table in shared memory.
    if (variant == B2C_VARIANT_IM2COL_GATHER && im2col_k_pad(g.Kg) > 4096) continue;
    if (is_shift_variant(variant)) {
      // one schedule: all output channels in one column tile (the weights are resident), no split
      ShiftGeom sg;
      if (shift_geom(g, view, &sg, shift_tiles_2d(variant))) add(out, g, variant, sg.tile_n, 1);
      continue;
    }
    for (int t : tiles) {
      // Skip widths that only add padding: keep t if it is the covering width or K % t == 0
      // or it wastes less than a quarter of the columns.
      int n_pad = round_up(d.K, t);
      if (t < tiles.back() && (n_pad - d.K) * 4 > n_pad) continue;
      long long ctas = tiles_m * (n_pad / t);
      for (int split = 1; split <= 32; split <<= 1) {
        if (split > num_kb) break;
        // A split reduction only helps while the grid is smaller than the machine.
        if (split > 1 && ctas * (split / 2) >= kNumSMs) break;
        add(out, g, variant, t, split);
      }
      // two-SM schedule of the same map: 256-row tiles, each block of the pair loads half of the column tile
      if (pair_schedule_ok(variant, t, 1, false, tiles_m * kTileM)) add(out, g, variant, t, 1, false, 2 * kTileM);
    }
    // Swapped axis map (M <- k, N <- fused pixels) for the TMA-fed variants: the 128 accumulator rows
    // are output channels, so it is only listed when K fills at least half of them; the pixel tile
    // widths are those that waste less than a quarter of their columns (or the covering one).
    if ((is_tma_view_variant(variant) || variant == B2C_VARIANT_IM2COL_EXPLICIT) && d.K >= kTileM / 2 &&
        variant != B2C_VARIANT_DILATION_PACK && !is_shift_variant(variant)) {
      const long long tiles_k = (d.K + kTileM - 1) / kTileM;
      for (int t = 32; t <= 256; t <<= 1) {
        const long long n_pad = (g.Mg + t - 1) / t * t;
        const bool covering = t >= g.Mg || t == 256;
        if (!covering && (n_pad - g.Mg) * 4 > n_pad) continue;
        const long long ctas = tiles_k * (n_pad / t);
        for (int split = 1; split <= 32; split <<= 1) {
          if (split > num_kb) break;
          if (split > 1 && ctas * (split / 2) >= kNumSMs) break;
          add(out, g, variant, t, split, true);
        }
        if (t >= g.Mg) break;
      }
    }
  }
  std::stable_sort(out->begin(), out->end(), [](const Candidate& a, const Candidate& b) {
    return a.o_mac + a.o_data < b.o_mac + b.o_data;
  });
  for (size_t i = 0; i < out->size(); ++i) (*out)[i].id = (int)i;
}

int pick_by_policy(const std::vector<Candidate>& all, int policy) {
  if (all.empty()) return -1;
  if (policy >= 0) return policy < (int)all.size() ? policy : -1;
  if (policy == B2C_POLICY_MIN_WORKSPACE) {
    int best = 0;
    for (size_t i = 1; i < all.size(); ++i)
      if (all[i].workspace_bytes < all[best].workspace_bytes) best = (int)i;
    return best;
  }
  return 0;  // MIN_OVERHEAD (AUTO_TIMED is resolved by the caller)
}

}  // namespace b2c
