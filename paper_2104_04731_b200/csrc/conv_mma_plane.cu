// Stencil unroll (Table 2, rule 1) formed from an input window in shared memory, for layers whose packed
// weights fit in shared memory (the low-channel shapes of Section 6.1, and any layer of moderate size).
//
// What makes the unroll cheap is that it is never written out.  The MMA's A operand is described to the tensor
// core without a swizzle: 16-byte units, 8 rows of a core matrix 16 bytes apart, row groups 128 bytes apart, and
// the two 16-byte halves of the 32-byte reduction slice a free distance apart.  An A operand of 128 rows is then
// ANY 128 consecutive units of shared memory plus the 128 units at a constant distance from them, starting at
// any unit.  So the window is kept as planes of 16-byte units, one unit per grid position and plane, and every
// MMA reads two taps (or two channel planes) of all 128 positions by start address and distance alone: no byte
// of the window is copied per tap.  Two forms of the units:
//   channel form   unit = 16 channels of one input pixel.  Planes: blocks of 16 channels x the stride phases the
//                  taps use.  Tap (r, s) is the same plane read further on.
//   row form       unit = the taps of one filter row, i.e. runs of RUNW 32-bit words of consecutive input bytes
//                  (one run per channel and vertical stride phase); only the vertical taps are shifts.  For one
//                  to a few channels, where 16 channels per unit would be mostly padding.
// Grid: every image is rpi rows of `pitch` positions; row i, column j holds output (i, j) where i < P and j < Q,
// the rest is the taps' overhang (zero rows and columns of the padding are shared by neighbours where possible).
// A window is `th` grid rows (of the whole batch, so it may end in one image and go on in the next) plus the
// max_ri rows the taps reach below, and feeds up to `tiles` accumulator tiles of 128 positions each.  A block
// walks consecutive windows, so the last max_ri rows of one are the first of the next: they are moved as units,
// and every input row is fetched and turned into units once per block.
//
// Roles: warp 0 fetches the raw NCHW rows of a window in chunks of at most `cr` grid rows: whole images or one row
// segment per channel by bulk copies (any width, the 16-byte boundaries around a segment are fetched with it), or all
// channels by one tiled copy where every channel starts on 16 bytes (bulk copies cost about 60 cycles each to issue,
// 7600 a window of 64 channels; 315 images of 64 x 56 x 56, 3x3, 84 us with them, 70 without); warp 1 issues the MMAs,
// the builder warps turn raw rows into units (byte transposes or unaligned words, zeros outside the image), the
// epilogue warps drain the accumulators (activation step, shift / clip, NKPQ or NPQK stores).  The weights stay
// resident.
// What bounds it now: the stores of the results (4 to 5 cycles of the SM's store path per 128 bytes; runs of 32 lanes that start
// inside a sector cost the memory side more, see plane_sector_rows) beside the builders' shared-memory traffic.  Before (operand
// rows written out by builder warps, or a rewrite through memory) and after: 64 images of 3 x 227 x 227, 7x7 stride 2, 64 channels 97 -> 49 us; 32 of 1 x 700 x 161,
// 20x5 stride 2, 76 -> 30; 15501 of 16 x 14 x 14, 3x3, 125 -> 95; 315 of 64 x 56 x 56, 3x3, 99 -> 74 (of the first and the last,
// tiles on sector boundaries gave 51.6 -> 49.2 and 79.2 -> 73.6).
// Copies of window w + 2, units of w + 1, MMAs of w and stores of w - 1 overlap.  Every wait is
// bounded as in the other kernels.
#include <algorithm>

#include "conv_mma_common.cuh"

namespace b2c {

namespace {

constexpr unsigned kSleepWindow = 200;  // ns between polls of a wait for a whole window

struct __align__(8) PlaneCtl {
  unsigned long long raw_full[2], raw_empty[2];
  unsigned long long win_full[2], win_empty[2];
  unsigned long long acc_full[kMaxAcc], acc_empty[kMaxAcc];
  unsigned long long w_full;
  unsigned long long build_sync;  // the builders' rendezvous (an mbarrier, so that a builder that gives up ends the others' wait)
  SharedCtl base;  // abort flag and tensor-memory base (the bounded waits take this)
};

// Up to four MMAs from a list of A descriptors; the B descriptor advances by a constant step.
__device__ __forceinline__ void mma_i8_list4(uint32_t d_tmem, uint64_t a0, uint64_t a1, uint64_t a2, uint64_t a3,
                                             uint64_t bdesc, uint64_t b_step, uint32_t idesc, uint32_t accumulate,
                                             uint32_t on, int count) {
  asm volatile(
      "{\n"
      ".reg .pred pacc, ptrue, q0, q1, q2, q3;\n"
      ".reg .b64 b1, b2, b3;\n"
      "setp.ne.b32 pacc, %8, 0;\n"
      "setp.eq.b32 ptrue, 0, 0;\n"
      "setp.ne.b32 q0, %9, 0;\n"
      "setp.gt.and.s32 q1, %10, 1, q0;\n"
      "setp.gt.and.s32 q2, %10, 2, q0;\n"
      "setp.gt.and.s32 q3, %10, 3, q0;\n"
      "add.u64 b1, %5, %6;\n"
      "add.u64 b2, b1, %6;\n"
      "add.u64 b3, b2, %6;\n"
      "@q0 tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %5, %7, pacc;\n"
      "@q1 tcgen05.mma.cta_group::1.kind::i8 [%0], %2, b1, %7, ptrue;\n"
      "@q2 tcgen05.mma.cta_group::1.kind::i8 [%0], %3, b2, %7, ptrue;\n"
      "@q3 tcgen05.mma.cta_group::1.kind::i8 [%0], %4, b3, %7, ptrue;\n"
      "}" ::"r"(d_tmem),
      "l"(a0), "l"(a1), "l"(a2), "l"(a3), "l"(bdesc), "l"(b_step), "r"(idesc), "r"(accumulate), "r"(on), "r"(count)
      : "memory");
}

// Bounded wait with back-off: polling a barrier takes the same shared-memory pipe as the builders' and the
// epilogue's loads and stores, and most warps of this kernel wait for whole windows (microseconds), so a warp that
// finds its barrier not ready sleeps between polls.  (Waits for a tile poll: sleeping there costs 2 to 5 us a call.)
__device__ __forceinline__ bool mbar_wait_sleep(uint32_t bar, uint32_t parity, SharedCtl* ctl, int* status, unsigned ns) {
  if (mbar_try_wait(bar, parity)) return true;
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_ns();
  while (true) {
    __nanosleep(ns);
    if (mbar_try_wait(bar, parity)) return true;
    if (ctl->abort_flag) return false;
    if (global_ns() - t0 > kWaitLimitNs) {
      ctl->abort_flag = 1;
      atomicCAS(status, 0, B2C_E_TIMEOUT);
      return false;
    }
  }
}

// Debug build: is the unit at this offset in shared memory inside the window of `bytes` bytes at `lo`?
#ifdef B2C_DEBUG_BOUNDS
#define B2C_WINDOW_OK(d, site, lo, bytes, at) b2c_dbg_in_range((d).status, site, smem + (lo), bytes, smem + (at), 16)
#else
#define B2C_WINDOW_OK(d, site, lo, bytes, at) true
#endif

// Which raw rows a chunk of grid rows [gr0, gr0 + cnt) needs: those of images n_a .. n_b (none if the chunk lies
// past the batch: images == 0).
struct ChunkRows {
  int n_a, images;
  int lo_a, rows_a;  // first raw row and row count of image n_a
  int rows_b;        // row count of image n_a + 1, from its first row on (row mode: a chunk touches two at most)
};
__device__ __forceinline__ ChunkRows chunk_rows(const ConvArgs& args, const PlaneArgs& pl, int gr0, int cnt) {
  ChunkRows r = {0, 0, 0, 0, 0};
  if (gr0 >= pl.total_rows) return r;
  const int last = min(gr0 + cnt, pl.total_rows) - 1;
  r.n_a = (int)pl.div_rpi.div((uint32_t)gr0);
  const int n_b = (int)pl.div_rpi.div((uint32_t)last);
  r.images = n_b - r.n_a + 1;
  const int i_a = gr0 - r.n_a * pl.rpi, i_b = last - n_b * pl.rpi;
  const int end_a = r.images == 1 ? i_b : pl.rpi - 1;
  r.lo_a = max(0, i_a * pl.sh - args.pad_h);
  r.rows_a = max(0, min(args.H - 1, end_a * pl.sh + pl.max_dh - args.pad_h) - r.lo_a + 1);
  r.rows_b = max(0, min(args.H - 1, i_b * pl.sh + pl.max_dh - args.pad_h) + 1);
  return r;
}
// The grid rows are cut into segments, dealt to the blocks in turn; a segment is walked in windows of th output
// rows.  Segment seg, and its window w: output rows [gr0, gr0 + rows), new unit rows [new0, new1).  With spi > 0 the
// segments are those of one image each (spi per image, its P output rows only), else seg_rows rows of the batch.
struct SegRows {
  int begin, end, windows;
  int out0;  // (segments of one image) output row of the image at which it begins
};
__device__ __forceinline__ SegRows seg_rows(const ConvArgs& args, const PlaneArgs& pl, int seg) {
  SegRows b;
  if (pl.spi > 0) {
    const int n = (int)pl.div_spi.div((uint32_t)seg);
    const int r0 = (seg - n * pl.spi) * pl.seg_rows;
    b.begin = n * pl.rpi + r0;
    b.out0 = r0;
    b.end = n * pl.rpi + min(r0 + pl.seg_rows, args.out_P);
  } else {
    b.begin = seg * pl.seg_rows;
    b.out0 = 0;
    b.end = min(b.begin + pl.seg_rows, pl.total_rows);
  }
  b.windows = (b.end - b.begin + pl.th - 1) / pl.th;
  return b;
}
struct WindowSpan {
  int gr0, rows, new0, new1;
  int lead;  // positions between the start of the first tile and the window's first output
};
template <bool LEAD>
__device__ __forceinline__ WindowSpan window_span(const ConvArgs& args, const PlaneArgs& pl, const SegRows& b, int w) {
  WindowSpan s;
  s.gr0 = b.begin + w * pl.th;
  s.rows = min(pl.th, b.end - s.gr0);
  s.new0 = w == 0 ? s.gr0 : s.gr0 + pl.max_ri;
  s.new1 = s.gr0 + s.rows + pl.max_ri;
  s.lead = LEAD ? ((b.out0 + w * pl.th) * args.out_Q) & pl.lead_mask : 0;
  return s;
}
// Bytes of one channel's slot for a segment of `rows` raw rows: any start inside 16 bytes, rounded up.
__device__ __forceinline__ int segment_bytes(int rows, int W) { return (rows * W + 30) & ~15; }

// RUNW: 0 = channel form, else row form with runs of RUNW words.  VAR: channel form 2 = unit strides and H * W a
// multiple of 4 (pixels are taken four at a time across row ends, so that any width reads whole words), 1 = every
// row of every channel starts on a word, 0 = any; row form 1, 2 = the horizontal stride (four neighbouring columns per builder item), 0 = any
// stride (one column).  KB builder warps, KE epilogue warps, MINB blocks per SM.  LEAD (row form): tiles may start before
// their window, so that stores start on sectors.  An instantiation of its own: the few instructions cost layers that have no
// use for it 5 % (15501 images of 16 x 14 x 14, 95 -> 100 us).
template <int RUNW, int VAR, int KB, int KE, int MINB, bool LEAD>
__global__ void __launch_bounds__(64 + 32 * (KB + KE), MINB)
    conv_mma_plane_kernel(const __grid_constant__ CUtensorMap tmap_x, const ConvArgs args, const PlaneArgs pl) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ PlaneCtl pc;
  SharedCtl* ctl = &pc.base;
  constexpr int kThreadsAll = 64 + 32 * (KB + KE);

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
  const int lane = threadIdx.x & 31;
  const int grp = args.groups > 1 ? (int)blockIdx.z : 0;
  const int n0 = (int)blockIdx.y * args.tile_n;
  const int HW = args.H * args.W;
  const int nbuf = pl.nbuf;

  // shared memory: [windows][raw rows, margins around each stage][weights][A descriptor offsets]
  const uint32_t smem_base = (smem_u32(smem_raw) + 127u) & ~127u;
  uint8_t* smem = smem_raw + (smem_base - smem_u32(smem_raw));
  const uint32_t win_off = LEAD ? (uint32_t)(pl.lead_mask + 1) * 16u : 0u;  // a first tile may start before the window
  const uint32_t raw_off = win_off + (uint32_t)(pl.win_stages * pl.win_bytes);
  const uint32_t w_off = raw_off + (uint32_t)(pl.raw_stages * pl.raw_bytes);
  const uint32_t tab_off = w_off + (uint32_t)pl.w_bytes;

  if (warp == 0) {
    if (lane < 2) {
      mbar_init(smem_u32(&pc.raw_full[lane]), 1);
      mbar_init(smem_u32(&pc.raw_empty[lane]), KB);
      mbar_init(smem_u32(&pc.win_full[lane]), KB);
      mbar_init(smem_u32(&pc.win_empty[lane]), 1);
    }
    if (lane >= 8 && lane < 8 + kMaxAcc) {
      mbar_init(smem_u32(&pc.acc_full[lane - 8]), 1);
      mbar_init(smem_u32(&pc.acc_empty[lane - 8]), 4);
    }
    if (lane == 16) {
      mbar_init(smem_u32(&pc.w_full), 1);
      mbar_init(smem_u32(&pc.build_sync), KB);
      ctl->abort_flag = 0;
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)),
                 "r"(args.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  {
    // A descriptor offsets (a plan constant, written by no kernel)
    uint64_t* t = reinterpret_cast<uint64_t*>(smem + tab_off);
    for (int i = threadIdx.x; i < pl.num_mma; i += kThreadsAll) t[i] = pl.mma_table[i];
  }
  if (pl.zero_fill) {
    // columns that are padding in every window: no builder ever writes them
    for (int i = threadIdx.x * 16; i < pl.win_stages * pl.win_bytes; i += kThreadsAll * 16)
      *reinterpret_cast<uint4*>(smem + win_off + i) = make_uint4(0, 0, 0, 0);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_acc = __shfl_sync(0xffffffffu, ctl->tmem_base, 0);
  pdl_wait();
  pdl_launch_dependents();

  const int seg_first = (int)blockIdx.x, seg_step = (int)gridDim.x, seg_end = pl.segs;
  const int8_t* xg = args.x + (size_t)grp * args.group_x_stride;

  if (warp == 0) {
    // ---------------------------------------------------------------- raw rows and weights
    const uint32_t leader = elect_one() ? 1u : 0u;
    {
      const uint8_t* wsrc = pl.w + (size_t)((size_t)grp * gridDim.y + blockIdx.y) * pl.w_bytes;
      mbar_arrive_expect_tx(smem_u32(&pc.w_full), (uint32_t)pl.w_bytes, leader);
      asm volatile(
          "{\n.reg .pred q;\nsetp.ne.b32 q, %4, 0;\n"
          "@q cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n}" ::"r"(smem_base + w_off),
          "l"(wsrc), "r"((uint32_t)pl.w_bytes), "r"(smem_u32(&pc.w_full)), "r"(leader)
          : "memory");
    }
    const uintptr_t x_end = reinterpret_cast<uintptr_t>(args.x) + (size_t)pl.x_bytes;
    int s = 0;
    uint32_t ph = 0;
    bool alive = true;
    for (int seg = seg_first; seg < seg_end && alive; seg += seg_step) {
    const SegRows blk = seg_rows(args, pl, seg);
    for (int win = 0; win < blk.windows && alive; ++win) {
      const WindowSpan sp = window_span<LEAD>(args, pl, blk, win);
      for (int c0 = sp.new0; c0 < sp.new1; c0 += pl.cr) {
      const ChunkRows r = chunk_rows(args, pl, c0, min(pl.cr, sp.new1 - c0));
      alive = __all_sync(0xffffffffu, mbar_wait_sleep(smem_u32(&pc.raw_empty[s]), ph ^ 1u, ctl, args.status, kSleepWindow));
      if (!alive) break;
      const uint32_t full = smem_u32(&pc.raw_full[s]);
      const uint32_t raw = raw_off + (uint32_t)(s * pl.raw_bytes) + kPlaneMargin;
      if (pl.box_bytes > 0) {
        // one tiled copy: box_bytes of every channel of the image from the 16-byte boundary before row lo_a on
        if (r.rows_a > 0 && B2C_X_OK(args.dbg, 53, xg + (size_t)r.n_a * args.x_stride_n + r.lo_a * args.W,
                                     (long long)(args.C - 1) * HW + r.rows_a * args.W)) {
          mbar_arrive_expect_tx(full, (uint32_t)(args.C * pl.box_bytes), leader);
          tma_load_2d(smem_base + raw, &tmap_x, ((r.lo_a * args.W) & ~15) >> 2, r.n_a * pl.img_channels + grp * args.C, full, leader);
        } else {
          mbar_arrive_expect_tx(full, 0u, leader);
        }
        if (++s == pl.raw_stages) {
          s = 0;
          ph ^= 1u;
        }
        continue;
      }
      // Copies of this chunk, dealt to the lanes twice: first the byte count, then the copies.  Each fetches
      // the 16-byte units its bytes lie in; bytes in the tensor's last, incomplete unit are copied by hand.
      const int copies = pl.whole_images ? r.images : args.C * r.images;
      uint32_t my_bytes = 0;
      for (int pass = 0; pass < 2; ++pass) {
        for (int c = lane; c < copies; c += 32) {
          const int8_t* src;
          int bytes;
          uint32_t dst;
          if (pl.whole_images) {
            src = xg + (size_t)(r.n_a + c) * args.x_stride_n;
            bytes = args.C * HW;
            dst = raw + (uint32_t)(c * pl.img_slot);
          } else {
            const int ch = c >= args.C ? c - args.C : c;
            const bool second = c >= args.C;
            src = xg + (size_t)(r.n_a + (second ? 1 : 0)) * args.x_stride_n + (size_t)ch * HW + (second ? 0 : r.lo_a) * args.W;
            bytes = (second ? r.rows_b : r.rows_a) * args.W;
            dst = raw + (uint32_t)(ch * pl.c_pitch) + (second ? (uint32_t)segment_bytes(r.rows_a, args.W) : 0u);
          }
          const uintptr_t a0 = reinterpret_cast<uintptr_t>(src) & ~(uintptr_t)15;
          const uintptr_t e1 = reinterpret_cast<uintptr_t>(src) + bytes;
          uintptr_t e0 = (e1 + 15) & ~(uintptr_t)15;
          if (e0 > x_end) e0 -= 16;
          if (bytes == 0 || !B2C_X_OK(args.dbg, 50, src, bytes)) continue;
          if (pass == 0) {
            if (e0 > a0) my_bytes += (uint32_t)(e0 - a0);
            const uintptr_t from = max(e0, reinterpret_cast<uintptr_t>(src));
            for (uintptr_t b = from; b < e1; ++b)  // fewer than 16 bytes, in the last window only
              smem[dst + (uint32_t)(b - a0)] = *reinterpret_cast<const uint8_t*>(b);
          } else if (e0 > a0) {
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                             smem_base + dst),
                         "l"(a0), "r"((uint32_t)(e0 - a0)), "r"(full)
                         : "memory");
          }
        }
        if (pass == 0) {
          const uint32_t total = __reduce_add_sync(0xffffffffu, my_bytes);
          __syncwarp();
          mbar_arrive_expect_tx(full, total, leader);
          __syncwarp();
        }
      }
      if (++s == pl.raw_stages) {
        s = 0;
        ph ^= 1u;
      }
      }
    }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    const uint32_t idesc = make_idesc_i8(args.tile_n);
    const uint32_t leader = elect_one() ? 1u : 0u;
    const uint64_t b0 = make_plain_desc(smem_base + w_off, (uint32_t)args.tile_n * 16u);
    const uint64_t b_step = (uint64_t)(args.tile_n * 2);
    const uint32_t tab = smem_base + tab_off;
    bool alive = __all_sync(0xffffffffu, mbar_wait(smem_u32(&pc.w_full), 0u, ctl, args.status));
    int s = 0, buf = 0;
    uint32_t ph = 0, aph = 0;
    for (int seg = seg_first; seg < seg_end && alive; seg += seg_step) {
    const SegRows blk = seg_rows(args, pl, seg);
    for (int win = 0; win < blk.windows && alive; ++win) {
      alive = __all_sync(0xffffffffu, mbar_wait(smem_u32(&pc.win_full[s]), ph, ctl, args.status));
      if (!alive) break;
      const WindowSpan sp = window_span<LEAD>(args, pl, blk, win);
      const int tiles = (sp.rows * pl.pitch + sp.lead + kTileM - 1) / kTileM;
      uint64_t abase = make_plain_desc(smem_base + win_off + (uint32_t)(s * pl.win_bytes) - (uint32_t)(sp.lead * 16), 0u);
      for (int t = 0; t < tiles; ++t) {
        alive = __all_sync(0xffffffffu, mbar_wait(smem_u32(&pc.acc_empty[buf]), aph ^ 1u, ctl, args.status));
        if (!alive) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t d_tmem = tmem_acc + (uint32_t)(buf * args.tile_n);
        uint64_t bdesc = b0;
        for (int m = 0; m < pl.num_mma; m += 4) {
          uint64_t o0, o1, o2, o3;
          asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(o0), "=l"(o1) : "r"(tab + (uint32_t)m * 8u));
          asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(o2), "=l"(o3) : "r"(tab + (uint32_t)m * 8u + 16u));
          mma_i8_list4(d_tmem, abase + o0, abase + o1, abase + o2, abase + o3, bdesc, b_step, idesc, m ? 1u : 0u, leader,
                       pl.num_mma - m);
          bdesc += 4 * b_step;
        }
        mma_commit(smem_u32(&pc.acc_full[buf]), leader);
        abase += kTileM;  // 128 units further on
        if (++buf == nbuf) {
          buf = 0;
          aph ^= 1u;
        }
      }
      mma_commit(smem_u32(&pc.win_empty[s]), leader);
      if (++s == pl.win_stages) {
        s = 0;
        ph ^= 1u;
      }
    }
    }
    __syncwarp();
  } else if (warp < 2 + KB) {
    // ---------------------------------------------------------------- builders
    const int tid = (int)threadIdx.x - 64;
    const uint32_t x_low = (uint32_t)reinterpret_cast<uintptr_t>(xg);
    const uint32_t hw_low = pl.whole_images ? 0u : (uint32_t)HW;  // (a whole image keeps one alignment)
    const uint32_t c_step = (uint32_t)(pl.whole_images ? HW : pl.c_pitch);
    int rs = 0, ws = 0;
    uint32_t rph = 0, wph = 0, sph = 0;
    bool ok = true;
    auto rendezvous = [&]() -> bool {
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&pc.build_sync));
      const bool met = __all_sync(0xffffffffu, mbar_wait(smem_u32(&pc.build_sync), sph, ctl, args.status));
      sph ^= 1u;
      return met;
    };
    // After a wait that gave up, a warp leaves a window by vote and the role where a segment begins, so that its lanes stay
    // together; what it still builds and arrives on is of no use to anyone, and harmless.  (ok is a lane's own.)
    for (int seg = seg_first; seg < seg_end; seg += seg_step) {
    if (__any_sync(0xffffffffu, ctl->abort_flag != 0)) break;
    const SegRows blk = seg_rows(args, pl, seg);
    for (int win = 0; win < blk.windows; ++win) {
      const WindowSpan sp = window_span<LEAD>(args, pl, blk, win);
      ok = mbar_wait_sleep(smem_u32(&pc.win_empty[ws]), wph ^ 1u, ctl, args.status, kSleepWindow);
      if (!__all_sync(0xffffffffu, ok)) break;
      const uint32_t win_s = win_off + (uint32_t)(ws * pl.win_bytes);
      if (win > 0 && pl.max_ri > 0) {
        // The overlap rows: the last max_ri rows of the previous window become the first of this one.
        // With two buffers a builder that is done with the last window of a segment goes on to the next segment, whose
        // first window has no rendezvous and is built where a slower builder may still be reading rows to move.  These
        // are rows th and up, and they arrive there in a second raw chunk, because segments of several windows have
        // cr == th (the planner lists no others): it lands in the raw stage of the slower builder's window, which
        // that builder releases after its move.
        const uint32_t prev = win_off + (uint32_t)((pl.win_stages == 1 ? 0 : ws ^ 1) * pl.win_bytes) + (uint32_t)(pl.th * pl.pitch) * 16u;
        ok = rendezvous();  // every builder has finished the previous window
        if (!ok) break;
        const int per_plane = pl.max_ri * pl.pitch;
        for (int i = tid; i < pl.planes * per_plane; i += KB * 32) {
          const int plane = (int)pl.div_overlap.div((uint32_t)i);
          const uint32_t at = (uint32_t)(plane * pl.plane_bytes) + (uint32_t)(i - plane * per_plane) * 16u;
          *reinterpret_cast<uint4*>(smem + win_s + at) = *reinterpret_cast<const uint4*>(smem + prev + at);
        }
        // (a single buffer: the rows just moved are about to be overwritten; th >= max_ri, so the move itself is disjoint)
        if (pl.win_stages == 1) ok = rendezvous();
        if (!ok) break;
      }
      for (int c0 = sp.new0; c0 < sp.new1; c0 += pl.cr) {
      const int cnt = min(pl.cr, sp.new1 - c0);
      const int j0 = c0 - sp.gr0;  // window row of the chunk's first grid row
      const ChunkRows r = chunk_rows(args, pl, c0, cnt);
      ok = mbar_wait(smem_u32(&pc.raw_full[rs]), rph, ctl, args.status);
      if (!__all_sync(0xffffffffu, ok)) break;
      const uint32_t raw_s = raw_off + (uint32_t)(rs * pl.raw_bytes) + kPlaneMargin;
      const uint32_t seg_b = (uint32_t)segment_bytes(r.rows_a, args.W);
      // offset of byte (channel 0, row h, column 0) of image n in shared memory, without the channel's own
      // alignment term ((low + c * HW) & 15), whose base `low` it returns as well
      auto row_offset = [&](int n, int h, uint32_t* low) -> uint32_t {
        const uint32_t image = x_low + (uint32_t)n * (uint32_t)args.x_stride_n;
        if (pl.whole_images) {
          *low = image & 15u;
          return raw_s + (uint32_t)((n - r.n_a) * pl.img_slot) + (uint32_t)(h * args.W);
        }
        const bool second = n != r.n_a;
        const int lo = second ? 0 : r.lo_a;
        *low = (image + (uint32_t)(lo * args.W)) & 15u;
        return raw_s + (second ? seg_b : 0u) + (uint32_t)((h - lo) * args.W);
      };
      // alignment term of channel c (whole images: the image's own, the channels follow without gaps)
      auto channel_low = [&](uint32_t low, int c) -> uint32_t { return pl.whole_images ? low : ((low + (uint32_t)c * hw_low) & 15u); };
      auto word = [&](uint32_t off) -> uint32_t { return *reinterpret_cast<const uint32_t*>(smem + off); };
      // Four neighbouring 16-byte units of a lane: store t takes unit t ^ y with y from the lane, so that the eight
      // lanes of a store phase (their groups are 64 bytes apart) hit eight different 16-byte bank groups.
      const int y = (lane >> 1) & 3;
      auto rotate = [&](uint32_t (&px)[4][4]) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint32_t b0 = (y & 1) ? px[1][k] : px[0][k], b1 = (y & 1) ? px[0][k] : px[1][k];
          const uint32_t b2 = (y & 1) ? px[3][k] : px[2][k], b3 = (y & 1) ? px[2][k] : px[3][k];
          px[0][k] = (y & 2) ? b2 : b0;
          px[1][k] = (y & 2) ? b3 : b1;
          px[2][k] = (y & 2) ? b0 : b2;
          px[3][k] = (y & 2) ? b1 : b3;
        }
      };
      if constexpr (RUNW == 0) {
        if constexpr (VAR == 2) {
          // flat groups: item = (image of the chunk, block of 16 channels, four consecutive pixels); rows of the chunk
          // that lie outside the image become zeros first
          for (int jc = warp - 2; jc < cnt; jc += KB) {
            const int gr = c0 + jc;
            const int n = (int)pl.div_rpi.div((uint32_t)gr);
            if (gr < pl.total_rows && (unsigned)(gr - n * pl.rpi - args.pad_h) < (unsigned)args.H) continue;
            for (int u = 0; u < pl.planes; ++u)
              for (int q = lane; q < pl.pitch; q += 32)
                *reinterpret_cast<uint4*>(smem + win_s + (uint32_t)(u * pl.plane_bytes) + (uint32_t)((j0 + jc) * pl.pitch + q) * 16u) =
                    make_uint4(0, 0, 0, 0);
          }
          // (whole images: all of them in one loop, HW / 4 groups each; row segments: image by image)
          const int passes = pl.whole_images ? min(r.images, 1) : r.images;
          for (int pass = 0; pass < passes; ++pass) {
            int n = r.n_a + pass;
            int first = c0 - n * pl.rpi - args.pad_h;  // raw row of the chunk's first grid row
            const int rows_end = pl.total_rows - c0;   // grid rows from the chunk's first one to the end of the batch
            // rows [h_lo, h_hi) of the image belong to this chunk
            int f0 = max(0, first) * args.W, f1 = min(args.H, first + min(cnt, rows_end)) * args.W;
            if (!pl.whole_images && f0 >= f1) continue;
            const int g0 = pl.whole_images ? 0 : f0 >> 2;
            const int groups = pl.whole_images ? HW >> 2 : ((f1 + 3) >> 2) - g0;
            uint32_t low;
            uint32_t a_row = pl.whole_images ? row_offset(n, 0, &low) : row_offset(n, max(0, first), &low) - (uint32_t)(f0 & 3);
            if (!pl.whole_images) a_row += low;
            const int items = groups * pl.planes * (pl.whole_images ? r.images : 1);
            for (int e = tid; e < items; e += KB * 32) {
              int u, g;
              if (pl.whole_images) {
                const int t = (int)pl.div_hw4.div((uint32_t)e);
                g = e - t * groups;
                const int im = (int)pl.div_nu.div((uint32_t)t);
                u = t - im * pl.planes;
                n = r.n_a + im;
                first = c0 - n * pl.rpi - args.pad_h;
                f0 = max(0, first) * args.W;
                f1 = min(args.H, first + min(cnt, rows_end)) * args.W;
                a_row = row_offset(n, 0, &low) + low;
              } else {
                u = pl.planes == 1 ? 0 : (int)((unsigned)e / (unsigned)groups);
                g = e - u * groups;
              }
              const int f = (g0 + g) * 4;
              if (f + 4 <= f0 || f >= f1) continue;
              const int pos0 = (j0 - first) * pl.pitch + args.pad_w;  // position of raw row 0, column 0: negative if it lies above the window
              const uint32_t a = a_row + (uint32_t)(g * 4) + (uint32_t)(u * 16) * c_step;
              const int left = args.C - u * 16;
              uint32_t px[4][4];
#pragma unroll
              for (int k4 = 0; k4 < 4; ++k4) {
                uint32_t v[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                  const int c = k4 * 4 + k;
                  v[k] = c < left ? word(a + (uint32_t)c * c_step + (channel_low(low, u * 16 + c) - low)) : 0u;
                }
                const uint32_t t0 = __byte_perm(v[0], v[1], 0x5140), t1 = __byte_perm(v[2], v[3], 0x5140);
                const uint32_t t2 = __byte_perm(v[0], v[1], 0x7362), t3 = __byte_perm(v[2], v[3], 0x7362);
                px[0][k4] = __byte_perm(t0, t1, 0x5410);
                px[1][k4] = __byte_perm(t0, t1, 0x7632);
                px[2][k4] = __byte_perm(t2, t3, 0x5410);
                px[3][k4] = __byte_perm(t2, t3, 0x7632);
              }
              rotate(px);
              const int h = (int)pl.div_w.div((uint32_t)f);
              const int wcol = f - h * args.W;
              // Offset of the group's first pixel in shared memory, in 32 bits that may wrap: where a window starts inside an
              // image, the group of its first pixel can begin in the row above (30 x 30, segments of 6 rows: pixel 150 is in
              // the group of 148), before the window.  Only the whole sum, of a pixel that is stored, becomes a pointer.
              const uint32_t dst = win_s + (uint32_t)(u * pl.plane_bytes) + (uint32_t)(pos0 + h * pl.pitch + wcol) * 16u;
              const uint32_t wrap = (uint32_t)(pl.pitch - args.W) * 16u;  // W >= 4: at most one row end inside a group
#pragma unroll
              for (int p = 0; p < 4; ++p) {
                const int q = p ^ y;
                const uint32_t at = dst + (uint32_t)q * 16u + (wcol + q >= args.W ? wrap : 0u);
                if (f + q >= f0 && f + q < f1 && B2C_WINDOW_OK(args.dbg, 52, win_s, pl.win_bytes, at))
                  *reinterpret_cast<uint4*>(smem + at) = make_uint4(px[p][0], px[p][1], px[p][2], px[p][3]);
              }
            }
          }
        } else {
        // channel form: item = (window row, block of 16 channels and row phase, group of 4 pixels)
        const int nu = (pl.planes / pl.ndw);
        const int items = cnt * nu * pl.gpr;
        for (int e = tid; e < items; e += KB * 32) {
          const int t = (int)pl.div_gpr.div((uint32_t)e);
          const int w = (e - t * pl.gpr) * 4;
          const int jc0 = (int)pl.div_nu.div((uint32_t)t);
          const int u = t - jc0 * nu;  // channel block * ndh + row phase
          const int j = j0 + jc0;
          const int cb = pl.ndh == 1 ? u : u / pl.ndh;
          const int hi = u - cb * pl.ndh;
          const int gr = c0 + jc0;
          const int n = (int)pl.div_rpi.div((uint32_t)gr);
          const int h = (gr - n * pl.rpi) * pl.sh + (int)pl.row_phase[hi] - args.pad_h;
          uint32_t px[4][4];  // [pixel][word of the unit]
          if (gr < pl.total_rows && (unsigned)h < (unsigned)args.H) {
            uint32_t low;
            uint32_t a = row_offset(n, h, &low) + (uint32_t)w + (uint32_t)(cb * 16) * c_step;
            const int left = args.C - cb * 16;  // channels of this block that exist
            if (VAR == 1) a += low;
#pragma unroll
            for (int k4 = 0; k4 < 4; ++k4) {
              uint32_t v[4];
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                const int c = k4 * 4 + k;
                v[k] = 0;
                if (c < left) {
                  if (VAR == 1) {
                    v[k] = word(a + (uint32_t)c * c_step);
                  } else {
                    const uint32_t ac = a + (uint32_t)c * c_step + ((low + (uint32_t)(cb * 16 + c) * hw_low) & 15u);
                    v[k] = __byte_perm(word(ac & ~3u), word((ac & ~3u) + 4u), 0x3210u + 0x1111u * (ac & 3u));
                  }
                }
              }
              const uint32_t t0 = __byte_perm(v[0], v[1], 0x5140), t1 = __byte_perm(v[2], v[3], 0x5140);
              const uint32_t t2 = __byte_perm(v[0], v[1], 0x7362), t3 = __byte_perm(v[2], v[3], 0x7362);
              px[0][k4] = __byte_perm(t0, t1, 0x5410);
              px[1][k4] = __byte_perm(t0, t1, 0x7632);
              px[2][k4] = __byte_perm(t2, t3, 0x5410);
              px[3][k4] = __byte_perm(t2, t3, 0x7632);
            }
          } else {
#pragma unroll
            for (int p = 0; p < 4; ++p) px[p][0] = px[p][1] = px[p][2] = px[p][3] = 0;
          }
          rotate(px);
          if (pl.sw == 1) {
            uint8_t* dst = smem + win_s + (uint32_t)(u * pl.plane_bytes) + (uint32_t)(j * pl.pitch + w + args.pad_w) * 16u;
#pragma unroll
            for (int p = 0; p < 4; ++p) {
              const int q = p ^ y;
              if (w + q < args.W) *reinterpret_cast<uint4*>(dst + q * 16) = make_uint4(px[p][0], px[p][1], px[p][2], px[p][3]);
            }
          } else {
#pragma unroll
            for (int p = 0; p < 4; ++p) {
              const int wq = w + (p ^ y) + args.pad_w;
              const int jc = (int)pl.div_sw.div((uint32_t)wq);
              const int ci = (int)pl.col_phase[wq - jc * pl.sw];
              if (w + (p ^ y) < args.W && ci >= 0 && jc < pl.pitch)
                *reinterpret_cast<uint4*>(smem + win_s + (uint32_t)((u * pl.ndw + ci) * pl.plane_bytes) + (uint32_t)(j * pl.pitch + jc) * 16u) =
                    make_uint4(px[p][0], px[p][1], px[p][2], px[p][3]);
            }
          }
        }
        }
      } else {
        // Row form: item = (window row, QB neighbouring output columns); G runs make U units per column.  A run of
        // all QB columns is one stream of NS words, aligned once; the columns' words are words of the stream or
        // byte permutes of two.  No branches: rows outside the image read a valid address and are cleared, so that
        // the loads of a group of runs are in flight together.
        constexpr int QB = VAR == 0 ? 1 : 4;
        constexpr int G = RUNW == 1 ? 4 : (RUNW == 4 ? 1 : 2);
        constexpr int U = G * RUNW / 4;
        constexpr int NS = ((QB - 1) * VAR + 4 * RUNW + 3) / 4;
        const int items = cnt * pl.gpr;
        for (int e = tid; e < items; e += KB * 32) {
          const int jc0 = (int)pl.div_gpr.div((uint32_t)e);
          const int q0 = (e - jc0 * pl.gpr) * QB;
          const int gr = c0 + jc0;
          const int n = (int)pl.div_rpi.div((uint32_t)gr);
          const int h0 = (gr - n * pl.rpi) * pl.sh - args.pad_h;
          const bool live = gr < pl.total_rows;
          const int col0 = q0 * pl.sw - args.pad_w;
          uint32_t mask[NS];
#pragma unroll
          for (int k = 0; k < NS; ++k) mask[k] = 0xFFFFFFFFu;
          if (col0 < 0 || col0 + 4 * NS > args.W) {
#pragma unroll
            for (int k = 0; k < NS; ++k) {
              // bytes [first, last) of this word are image columns
              const int first = min(4, max(0, -(col0 + 4 * k))), last = min(4, max(0, args.W - (col0 + 4 * k)));
              const uint32_t below = last == 4 ? 0xFFFFFFFFu : ((1u << (8 * last)) - 1u);
              mask[k] = first == 4 ? 0u : (below & (0xFFFFFFFFu << (8 * first)));
            }
          }
          uint32_t low;
          const uint32_t a0 = row_offset(n, h0, &low) + (uint32_t)col0;  // (rows outside the image are never read)
          uint8_t* dst = smem + win_s + (uint32_t)((j0 + jc0) * pl.pitch + q0) * 16u;
          int c = 0, hi = 0;
          uint32_t c_off = 0, c_low = low;
#pragma unroll 2
          for (int g = 0; g < pl.run_groups; ++g) {
            uint32_t v[G][NS];
#pragma unroll
            for (int x = 0; x < G; ++x) {
              const int dh = (int)pl.row_phase[hi];
              const bool valid = live && c < args.C && (unsigned)(h0 + dh) < (unsigned)args.H;
              const uint32_t a = valid ? a0 + c_off + (uint32_t)(dh * args.W) + (c_low & 15u) : raw_s;
              const uint32_t sel = 0x3210u + 0x1111u * (a & 3u);
              uint32_t prev = word(a & ~3u);
#pragma unroll
              for (int k = 0; k < NS; ++k) {
                const uint32_t next = word((a & ~3u) + 4u * (uint32_t)(k + 1));
                v[x][k] = valid ? (__byte_perm(prev, next, sel) & mask[k]) : 0u;
                prev = next;
              }
              if (++hi == pl.ndh) {
                hi = 0;
                ++c;
                c_off += c_step;
                c_low += hw_low;
              }
            }
#pragma unroll
            for (int k = 0; k < U; ++k) {
              uint32_t px[4][4];
#pragma unroll
              for (int p = 0; p < QB; ++p)
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                  const int x = (k * 4 + b) / RUNW, off = p * VAR + (k * 4 + b) % RUNW * 4;
                  const int i = off >> 2, sft = off & 3;
                  px[p][b] = sft == 0 ? v[x][i] : __byte_perm(v[x][i], v[x][i + 1 < NS ? i + 1 : i], 0x3210 + 0x1111 * sft);
                }
              if (QB == 1) {
                *reinterpret_cast<uint4*>(dst) = make_uint4(px[0][0], px[0][1], px[0][2], px[0][3]);
              } else {
                rotate(px);
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                  const int q = p ^ y;
                  if (q0 + q < pl.pitch) *reinterpret_cast<uint4*>(dst + q * 16) = make_uint4(px[p][0], px[p][1], px[p][2], px[p][3]);
                }
              }
              dst += pl.plane_bytes;
            }
          }
        }
      }
      // the raw rows have been read
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&pc.raw_empty[rs]));
      if (++rs == pl.raw_stages) {
        rs = 0;
        rph ^= 1u;
      }
      }
      // the units are visible to the tensor core's async proxy
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&pc.win_full[ws]));
      if (++ws == pl.win_stages) {
        ws = 0;
        wph ^= 1u;
      }
    }
    }
  } else {
    // ---------------------------------------------------------------- epilogue warps
    // Four warps drain a tile (one per tensor-memory lane quadrant); with eight, two sets take turns.
    const int quad = warp & 3;
    const int set = (warp - 2 - KB) >> 2;
    constexpr int kSets = KE / 4;
    const int row = quad * 32 + lane;
    const int pitch = pl.pitch;
    const int step_j = kTileM / pitch, step_q = kTileM - step_j * pitch;  // a tile further: rows and columns
    const int row_j = (int)pl.div_pitch.div((uint32_t)row), row_q = row - row_j * pitch;
    int buf = 0, ti = 0;
    uint32_t aph = 0;
    // (As the builders; tiles after a wait that gave up are drained as they are, and the status says so.)
    for (int seg = seg_first; seg < seg_end; seg += seg_step) {
    if (__any_sync(0xffffffffu, ctl->abort_flag != 0)) break;
    const SegRows blk = seg_rows(args, pl, seg);
    for (int win = 0; win < blk.windows; ++win) {
      const WindowSpan sp = window_span<LEAD>(args, pl, blk, win);
      const int positions = sp.rows * pitch;
      const int tiles = (positions + sp.lead + kTileM - 1) / kTileM;
      int j = row_j, q = row_q - sp.lead;  // this lane's grid row and column in the window
      if constexpr (LEAD)
        for (; q < 0; q += pitch) --j;
      for (int t = 0; t < tiles; ++t, ++ti) {
        if (kSets == 1 || (ti & (kSets - 1)) == set) {
          const int n = (int)pl.div_rpi.div((uint32_t)(sp.gr0 + j));
          const int i = sp.gr0 + j - n * pl.rpi;
          bool row_valid = t * kTileM + row < positions && q < args.out_Q && i < args.out_P;
          if constexpr (LEAD)  // (one comparison: positions before the window wrap to large values)
            row_valid = (unsigned)(t * kTileM + row - sp.lead) < (unsigned)positions && q < args.out_Q && i < args.out_P;
          const int out_pq = i * args.out_Q + q;
          (void)mbar_wait(smem_u32(&pc.acc_full[buf]), aph, ctl, args.status);
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const long long base_nkpq = (long long)n * args.y_stride_n + out_pq + (long long)grp * args.K * args.out_PQ;
          const long long base_npqk = ((long long)n * args.out_PQ + out_pq) * args.K;
          const uint32_t taddr = tmem_acc + ((uint32_t)(quad * 32) << 16) + (uint32_t)(buf * args.tile_n);
          int c = 0;
          for (; c + 32 <= args.tile_n; c += 32)
            epilogue_columns<32>(args, taddr + (uint32_t)c, n0 + c, row_valid, base_nkpq, base_npqk, 0u, grp * args.K);
          if (c < args.tile_n)
            epilogue_columns<16>(args, taddr + (uint32_t)c, n0 + c, row_valid, base_nkpq, base_npqk, 0u, grp * args.K);
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_u32(&pc.acc_empty[buf]));
        }
        q += step_q;
        j += step_j;
        if (q >= pitch) {
          q -= pitch;
          ++j;
        }
        if (++buf == nbuf) {
          buf = 0;
          aph ^= 1u;
        }
      }
    }
    }
  }

  // ---------------------------------------------------------------- teardown
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (ctl->abort_flag) {
    if (threadIdx.x == 0) {
      const unsigned long long t0 = global_ns();
      while (global_ns() - t0 < 50000ull) __nanosleep(1000);
    }
    __syncthreads();
  }
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_acc), "r"(args.tmem_cols) : "memory");
  }
}

template <int RUNW, int VAR, int KB, int KE, int MINB, bool LEAD>
cudaError_t launch_one(const CUtensorMap& tmap, const ConvArgs& args, const PlaneArgs& pl, dim3 grid, cudaStream_t st) {
  static std::atomic<unsigned long long> configured{0};
  cudaError_t e =
      set_max_dynamic_smem_once(configured, (const void*)conv_mma_plane_kernel<RUNW, VAR, KB, KE, MINB, LEAD>, kPlaneSmemMax);
  if (e != cudaSuccess) return e;
  return launch_pdl(conv_mma_plane_kernel<RUNW, VAR, KB, KE, MINB, LEAD>, grid, dim3(64 + 32 * (KB + KE)), (size_t)pl.smem, st, tmap, args, pl);
}

template <int RUNW, int VAR, bool LEAD>
cudaError_t launch_blocks(const CUtensorMap& tmap, const ConvArgs& args, const PlaneArgs& pl, dim3 grid, cudaStream_t st) {
  // One block per SM: eight builder and eight epilogue warps; two blocks: four of each.
  if (pl.per_sm == 1) return launch_one<RUNW, VAR, 8, 8, 1, LEAD>(tmap, args, pl, grid, st);
  return launch_one<RUNW, VAR, 4, 4, 2, LEAD>(tmap, args, pl, grid, st);
}
template <int RUNW, int VAR>
cudaError_t launch_form(const CUtensorMap& tmap, const ConvArgs& args, const PlaneArgs& pl, dim3 grid, cudaStream_t st) {
  if constexpr (RUNW > 0)
    if (pl.lead_mask) return launch_blocks<RUNW, VAR, true>(tmap, args, pl, grid, st);
  return launch_blocks<RUNW, VAR, false>(tmap, args, pl, grid, st);
}
template <int RUNW>
cudaError_t launch_row_form(const CUtensorMap& tmap, const ConvArgs& args, const PlaneArgs& pl, dim3 grid, cudaStream_t st) {
  if (pl.sw == 1) return launch_form<RUNW, 1>(tmap, args, pl, grid, st);
  if (pl.sw == 2) return launch_form<RUNW, 2>(tmap, args, pl, grid, st);
  return launch_form<RUNW, 0>(tmap, args, pl, grid, st);
}

}  // namespace

cudaError_t launch_conv_mma_plane(const CUtensorMap& tmap, const ConvArgs& args, const PlaneArgs& pl, cudaStream_t st) {
  const dim3 grid((unsigned)pl.blocks, (unsigned)pl.cols, (unsigned)std::max(1, args.groups));
  cudaError_t e;
  switch (pl.runw) {
    case 0:
      e = pl.aligned == 2 ? launch_form<0, 2>(tmap, args, pl, grid, st)
                          : (pl.aligned == 1 ? launch_form<0, 1>(tmap, args, pl, grid, st) : launch_form<0, 0>(tmap, args, pl, grid, st));
      break;
    case 1: e = launch_row_form<1>(tmap, args, pl, grid, st); break;
    case 2: e = launch_row_form<2>(tmap, args, pl, grid, st); break;
    case 4: e = launch_row_form<4>(tmap, args, pl, grid, st); break;
    default: e = launch_row_form<6>(tmap, args, pl, grid, st); break;
  }
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace b2c
