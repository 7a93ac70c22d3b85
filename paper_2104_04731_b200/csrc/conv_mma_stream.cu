// Stencil unroll (Table 2, rule 1) from planes of 16-byte units in shared memory, as in conv_mma_plane.cu, for layers
// whose weights do not fit beside the window: the channels are taken in blocks of 32, and the weights of a block stream
// through a ring while its units are built.  A pair of blocks on neighbouring SMs (cluster of two) owns a tile of
// 256 positions x tile_n channels (tcgen05.mma.cta_group::2): each block builds the units of its own 128 positions and
// loads half of the weights, and the tensor cores of both SMs read both halves.
//
// Why: the channel pack writes the rewritten input and reads it back R x S times through L2 (an SM takes about 50 bytes
// a clock from there, the pair schedule needs 64 per MMA clock), and the rewrite's stores disturb those loads.  Here the
// input is read once per column tile, as it lies in memory, and only the weights stream: 32 bytes per MMA clock, 11 more
// for the raw rows.  What it pays is the overhang of the position grid (7 x 7 outputs with stride 2: 49 of 64 positions).
// Measured in a loop over three sets of buffers, the fastest other embedding and this kernel: 128 images of 256 x 7 x 7 -> 512, 3x3,
// 19.5 and 13.8 us; 40 of 160 x 20 x 44 -> 130, 5x5, 62.8 and 35.8; 64 of 96 x 28 x 28 -> 192, 5x5, 43.0 and 29.4; 16 of
// 192 x 28 x 28 -> 192, 3x3, 13.1 and 11.9; 84 of 128 x 14 x 28 -> 256, 3x3 stride 2, 17.9 and 10.8.  1440 of 256 x 14 x 14 -> 512, 3x3
// stride 2: 92.7 and 94 (the overhang takes more than the missing rewrite saves).  Large windows leave rings of two, and other
// embeddings are faster: 80 of 128 x 56 x 56 -> 64, 5x5 stride 2, 34.7 and 40.4; 17 of 176 x 48 x 45 -> 428, 22.3 and 34.2.
// What bounds it: no unit is full (1536 images of the last shape under ncu: tensor pipe 58 % of the time, issue slots 45, L1 41);
// a window's way through the builders, whose waits and fences take the most issue opportunities, and at the boards' power limit the
// clock.  By count, of 1152 MMA clocks that a block of 32 channels takes with 9 taps and 256 columns, shared memory is busy for all:
// operand reads 576, arriving weights and raw rows 386, builders about 200.
//
// A tile is th grid rows of the whole batch per block (th x pitch <= 128 positions), so that both blocks' operands start
// at the same address, which the pair's one descriptor needs.  Grid, phases and units are those of the plane kernel's channel
// form; strides 1 and 2.
//
// Roles of a block: warp 0 weights (tiled copies of weight chunks that complete on the leader's barrier), warp 1 MMA issue (in
// the leader), warp 2 raw NCHW rows of a channel block (whole images by bulk copies, or one tiled copy per image part), three
// groups of builder warps turn them into units, eight warps drain the accumulators.  The builders of both blocks arrive on the leader's
// win_full.  Every wait is bounded as in the other kernels.
#include <algorithm>

#include "conv_mma_cluster.cuh"
#include "stream_tile.h"

namespace b2c {

namespace {

constexpr int kGroupWarps = 4;  // of a builder group; stream_groups of the groups take windows in turn
constexpr int kBuilders = kStreamGroups * kGroupWarps, kEpilogue = 8;
constexpr int kFirstBuilder = 3, kFirstEpilogue = kFirstBuilder + kBuilders;
constexpr int kStreamThreads = 32 * (kFirstEpilogue + kEpilogue);

struct __align__(8) StreamCtl {
  unsigned long long b_full[kStreamMaxStages], b_empty[kStreamMaxStages];
  unsigned long long win_full[4], win_empty[4];
  unsigned long long raw_full[4], raw_empty[4];
  unsigned long long acc_full[2], acc_empty[2];
  SharedCtl base;  // abort flag and tensor-memory base (the bounded waits take this)
};

// Up to four two-SM MMAs from a list of A descriptors; the B descriptor advances by a constant step.
__device__ __forceinline__ void mma_i8_pair_list4(uint32_t d_tmem, uint64_t a0, uint64_t a1, uint64_t a2, uint64_t a3,
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
      "@q0 tcgen05.mma.cta_group::2.kind::i8 [%0], %1, %5, %7, pacc;\n"
      "@q1 tcgen05.mma.cta_group::2.kind::i8 [%0], %2, b1, %7, ptrue;\n"
      "@q2 tcgen05.mma.cta_group::2.kind::i8 [%0], %3, b2, %7, ptrue;\n"
      "@q3 tcgen05.mma.cta_group::2.kind::i8 [%0], %4, b3, %7, ptrue;\n"
      "}" ::"r"(d_tmem),
      "l"(a0), "l"(a1), "l"(a2), "l"(a3), "l"(bdesc), "l"(b_step), "r"(idesc), "r"(accumulate), "r"(on), "r"(count)
      : "memory");
}

// Debug build: do the n bytes at this offset in shared memory lie inside the `bytes` bytes at `lo`?
#ifdef B2C_DEBUG_BOUNDS
#define B2C_SMEM_OK(d, site, lo, bytes, at, n) b2c_dbg_in_range((d).status, site, smem + (lo), bytes, smem + (at), n)
#else
#define B2C_SMEM_OK(d, site, lo, bytes, at, n) true
#endif

// STRIDE 1 or 2 on both axes.  WORDS: H * W is a multiple of 4, so four consecutive pixels of a channel are one word.
template <int STRIDE, bool WORDS>
__global__ void __launch_bounds__(kStreamThreads, 1)
    conv_mma_stream_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_w, const ConvArgs args,
                           const StreamArgs sa) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ StreamCtl sc;
  SharedCtl* ctl = &sc.base;

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();  // 0: leader (issues the MMAs), 1: peer
  const int tile_first = (int)(blockIdx.x >> 1), tile_step = (int)(gridDim.x >> 1), tile_end = sa.num_tiles;

  // shared memory: [windows][weight stages][raw rows][A descriptor offsets]
  const uint32_t smem_base = (smem_u32(smem_raw) + 127u) & ~127u;
  uint8_t* smem = smem_raw + (smem_base - smem_u32(smem_raw));
  const uint32_t b_off = (uint32_t)(sa.win_stages * sa.win_bytes);
  const uint32_t raw_off = b_off + (uint32_t)(sa.b_stages * sa.b_stage_bytes);
  const uint32_t tab_off = raw_off + (uint32_t)(sa.raw_stages * sa.raw_bytes);

  if (warp == 0) {
    if (lane < sa.b_stages) {
      mbar_init(smem_u32(&sc.b_full[lane]), 1);  // used in the leader: its producer's arrival and the bytes of both blocks
      mbar_init(smem_u32(&sc.b_empty[lane]), 1);
    }
    if (lane >= 16 && lane < 20) {
      mbar_init(smem_u32(&sc.win_full[lane - 16]), 2 * kGroupWarps);  // used in the leader: the builder warps of a group in both blocks
      mbar_init(smem_u32(&sc.win_empty[lane - 16]), 1);
      mbar_init(smem_u32(&sc.raw_full[lane - 16]), 1);
      mbar_init(smem_u32(&sc.raw_empty[lane - 16]), kGroupWarps);
    }
    if (lane >= 24 && lane < 26) {
      mbar_init(smem_u32(&sc.acc_full[lane - 24]), 1);
      mbar_init(smem_u32(&sc.acc_empty[lane - 24]), 2 * kEpilogue);
    }
    if (lane == 28) ctl->abort_flag = 0;
    if (lane == 29) asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_w) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)),
                 "r"(sa.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  {
    // A descriptor offsets (a plan constant, written by no kernel)
    uint64_t* t = reinterpret_cast<uint64_t*>(smem + tab_off);
    for (int i = threadIdx.x; i < sa.taps; i += kStreamThreads) t[i] = sa.mma_table[i];
  }
  // columns that are padding: no builder ever writes them
  for (int i = threadIdx.x * 16; i < sa.win_stages * sa.win_bytes; i += kStreamThreads * 16)
    *reinterpret_cast<uint4*>(smem + i) = make_uint4(0, 0, 0, 0);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  // the other block's barriers must be initialised before anything arrives on them
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_acc = __shfl_sync(0xffffffffu, ctl->tmem_base, 0);
  pdl_wait();
  if (rank != 0) pdl_launch_dependents();

  const int HW = args.H * args.W;

// tile t: grid rows of this block, column tile
#define B2C_STREAM_TILE(t)                                              \
  const int mt_ = (int)sa.div_cols.div((uint32_t)(t));                 \
  const int ct = (t) - mt_ * sa.cols;                                  \
  const int r0 = (mt_ * 2 + (int)rank) * sa.th;

  if (warp == 0) {
    // ---------------------------------------------------------------- weights (both blocks)
    const uint32_t leader_lane = elect_one() ? 1u : 0u;
    int s = 0;
    uint32_t ph = 0;
    bool alive = true;
    for (int t = tile_first; t < tile_end && alive; t += tile_step) {
      const int ct = t - (int)sa.div_cols.div((uint32_t)t) * sa.cols;
      int row = (ct * 2 + (int)rank) * sa.w_run_rows;
      for (int st = 0; st < sa.w_steps; ++st) {
        alive = __all_sync(0xffffffffu, mbar_wait(smem_u32(&sc.b_empty[s]), ph ^ 1u, ctl, args.status));
        if (!alive) break;
        const uint32_t full = map_to_rank(smem_u32(&sc.b_full[s]), 0u);
        if (rank == 0) mbar_arrive_expect_tx(smem_u32(&sc.b_full[s]), 2u * (uint32_t)sa.b_stage_bytes, leader_lane);
        tma_pair_load_2d(smem_base + b_off + (uint32_t)(s * sa.b_stage_bytes), &tmap_w, 0, row, full, leader_lane);
        row += sa.b_stage_bytes >> 10;
        if (++s == sa.b_stages) {
          s = 0;
          ph ^= 1u;
        }
      }
    }
    __syncwarp();
  } else if (warp == 1 && rank != 0) {
    // (the peer's warp 1 only allocates and frees tensor memory)
  } else if (warp == 1) {
    // ---------------------------------------------------------------- leader: MMA issue for the pair
    const uint32_t idesc = make_idesc_i8_pair(args.tile_n);
    const uint32_t leader_lane = elect_one() ? 1u : 0u;
    const uint64_t b_step = (uint64_t)args.tile_n;  // tile_n / 2 channels x 32 bytes, in units of 16
    const uint32_t tab = smem_base + tab_off;
    int ws = 0, bs = 0, in_b = 0, ti = 0;
    uint32_t wph = 0, bph = 0;
    uint64_t bdesc = 0;
    bool alive = true;
    for (int t = tile_first; t < tile_end && alive; t += tile_step, ++ti) {
      const int buf = ti & 1;
      // the epilogue warps of both blocks must have drained this accumulator
      alive = __all_sync(0xffffffffu, mbar_wait_cluster(smem_u32(&sc.acc_empty[buf]), (uint32_t)((ti >> 1) & 1) ^ 1u, ctl, args.status));
      if (!alive) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t d_tmem = tmem_acc + (uint32_t)(buf * args.tile_n);
      for (int cb = 0; cb < sa.ncb; ++cb) {
        alive = __all_sync(0xffffffffu, mbar_wait_cluster(smem_u32(&sc.win_full[ws]), wph, ctl, args.status));
        if (!alive) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint64_t abase = make_plain_desc(smem_base + (uint32_t)(ws * sa.win_bytes), 0u);
        for (int tap = 0; tap < sa.taps;) {
          if (in_b == 0) {
            alive = __all_sync(0xffffffffu, mbar_wait(smem_u32(&sc.b_full[bs]), bph, ctl, args.status));
            if (!alive) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            bdesc = make_plain_desc(smem_base + b_off + (uint32_t)(bs * sa.b_stage_bytes), (uint32_t)args.tile_n * 8u);
          }
          const int cnt = min(4, min(sa.taps - tap, sa.b_group - in_b));
          uint64_t o[4];
#pragma unroll
          for (int k = 0; k < 4; ++k)  // (the table is padded: entries past the last are read, not used)
            asm volatile("ld.shared.b64 %0, [%1];" : "=l"(o[k]) : "r"(tab + (uint32_t)(tap + k) * 8u));
          mma_i8_pair_list4(d_tmem, abase + o[0], abase + o[1], abase + o[2], abase + o[3], bdesc, b_step, idesc, (cb | tap) ? 1u : 0u,
                            leader_lane, cnt);
          tap += cnt;
          in_b += cnt;
          bdesc += (uint64_t)cnt * b_step;
          if (in_b == sa.b_group || (cb == sa.ncb - 1 && tap == sa.taps)) {
            mma_commit_pair(smem_u32(&sc.b_empty[bs]), leader_lane);
            in_b = 0;
            if (++bs == sa.b_stages) {
              bs = 0;
              bph ^= 1u;
            }
          }
        }
        if (!alive) break;
        mma_commit_pair(smem_u32(&sc.win_empty[ws]), leader_lane);
        if (++ws == sa.win_stages) {
          ws = 0;
          wph ^= 1u;
        }
      }
      if (alive) mma_commit_pair(smem_u32(&sc.acc_full[buf]), leader_lane);
    }
    pdl_launch_dependents();
    __syncwarp();
  } else if (warp == 2) {
    // ---------------------------------------------------------------- raw rows of a channel block (both blocks)
    const uint32_t leader_lane = elect_one() ? 1u : 0u;
    int s = 0;
    uint32_t ph = 0;
    bool alive = true;
    for (int t = tile_first; t < tile_end && alive; t += tile_step) {
      B2C_STREAM_TILE(t)
      (void)ct;
      const TileRows tr = stream_tile_rows(args, sa, r0);
      // lane p copies image n_a + p
      const int n = tr.n_a + lane;
      RawRows rr = {0, 0};
      if (tr.end > tr.r0 && lane < sa.max_images && n < sa.images && n * sa.rpi < tr.end) rr = stream_raw_rows(args, sa, tr, n, STRIDE);
      const bool mine = rr.hi > rr.lo;
      for (int cb = 0; cb < sa.ncb; ++cb) {
        alive = __all_sync(0xffffffffu, mbar_wait(smem_u32(&sc.raw_empty[s]), ph ^ 1u, ctl, args.status));
        if (!alive) break;
        const uint32_t full = smem_u32(&sc.raw_full[s]);
        const uint32_t dst = smem_base + raw_off + (uint32_t)(s * sa.raw_bytes + lane * sa.img_slot);
        const int channels = min(32, args.C - cb * 32);
        const int8_t* src = args.x + (size_t)n * args.x_stride_n + (size_t)(cb * 32) * HW;
        bool copy = mine;
        // (what the copy reads: whole channels, or the rows and what their tensor map clips)
        if (mine && !(sa.box_bytes > 0 ? B2C_X_OK(args.dbg, 57, src + rr.lo * args.W, (long long)(channels - 1) * HW + (rr.hi - rr.lo) * args.W)
                                       : B2C_X_OK(args.dbg, 57, src, (long long)channels * HW)))
          copy = false;
        const uint32_t bytes = !copy ? 0u : (uint32_t)(sa.box_bytes > 0 ? 32 * sa.box_bytes : channels * HW);
        const uint32_t total = __reduce_add_sync(0xffffffffu, bytes);
        mbar_arrive_expect_tx(full, total, leader_lane);
        __syncwarp();
        if (sa.box_bytes > 0) {
          tma_load_2d(dst, &tmap_x, ((rr.lo * args.W) & ~15) >> 2, n * args.C + cb * 32, full, copy ? 1u : 0u);
        } else if (copy) {
          asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src),
                       "r"(bytes), "r"(full)
                       : "memory");
        }
        if (++s == sa.raw_stages) {
          s = 0;
          ph ^= 1u;
        }
      }
    }
    __syncwarp();
  } else if (warp < kFirstEpilogue) {
    // ---------------------------------------------------------------- builders (both blocks)
    // The way of one window through a group (waits, loads, transposes, stores, arrival) is longer than its MMAs take, so
    // groups of four warps work on consecutive windows side by side (1440 images of 256 x 14 x 14 -> 512, 3x3 stride 2, cool GPU:
    // one group of eight 222 us, three of four 115, and 80 with the items kept; two of six 92, three of five 82).
    const int group = (warp - kFirstBuilder) / kGroupWarps, bw = (warp - kFirstBuilder) % kGroupWarps, tid = bw * 32 + lane;
    const int groups = stream_groups(sa);  // (a group past them takes no window)
    int turn = 0;  // the group whose window is next
    int rs = 0, ws = 0;
    uint32_t rph = 0, wph = 0;
    bool ok = true;
    auto next_window = [&]() {
      if (++turn == groups) turn = 0;
      if (++rs == sa.raw_stages) {
        rs = 0;
        rph ^= 1u;
      }
      if (++ws == sa.win_stages) {
        ws = 0;
        wph ^= 1u;
      }
    };
    const int per_row = sa.ndh * sa.ndw;      // planes of 16 channels
    const uint32_t c_step = stream_channel_step(args, sa);
    // An item's places in the raw rows and in the window are worked out once for a tile (once in all where every tile
    // starts an image) and used for its ncb channel blocks: with the divisions of every pixel in every block the builders
    // took most of the SM's issue slots (115 us, so 80).
    constexpr int kKept = 3;  // items a thread keeps; further ones are worked out anew
    const int items = stream_items(sa);
    // Store t of a lane takes pixel t ^ y, with y from the lane, so that the eight lanes of a store phase (their groups are 64
    // bytes apart, 32 with stride 2) hit eight different 16-byte bank groups; the transposes' selectors do the exchange.
    const int y = STRIDE == 1 ? (lane >> 1) & 3 : ((lane >> 2) & 1) * 2;
    const uint32_t sel_a = (y & 2) ? 0x7362u : 0x5140u, sel_b = (y & 2) ? 0x5140u : 0x7362u;
    const uint32_t sel_c = (y & 1) ? 0x7632u : 0x5410u, sel_d = (y & 1) ? 0x5410u : 0x7632u;
    auto build_item = [&](const StreamItem& it, uint32_t raw_s, uint32_t win_s) {
      const uint32_t a = raw_s + it.src;
      // (the second word of an unaligned pixel group may lie behind the stage: it is read, not used)
      if (!B2C_SMEM_OK(args.dbg, 60, raw_s, sa.raw_bytes + 8, a & ~3u, 15 * c_step + (WORDS ? 4u : 8u))) return;
      uint32_t px[4][4];
#pragma unroll
      for (int k4 = 0; k4 < 4; ++k4) {
        uint32_t v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint32_t ac = a + (uint32_t)(k4 * 4 + k) * c_step;
          if (WORDS) {
            v[k] = *reinterpret_cast<const uint32_t*>(smem + ac);
          } else {
            v[k] = __byte_perm(*reinterpret_cast<const uint32_t*>(smem + (ac & ~3u)), *reinterpret_cast<const uint32_t*>(smem + (ac & ~3u) + 4),
                               0x3210u + 0x1111u * (ac & 3u));
          }
        }
        const uint32_t t0 = __byte_perm(v[0], v[1], sel_a), t1 = __byte_perm(v[2], v[3], sel_a);
        const uint32_t t2 = __byte_perm(v[0], v[1], sel_b), t3 = __byte_perm(v[2], v[3], sel_b);
        px[0][k4] = __byte_perm(t0, t1, sel_c);
        px[1][k4] = __byte_perm(t0, t1, sel_d);
        px[2][k4] = __byte_perm(t2, t3, sel_c);
        px[3][k4] = __byte_perm(t2, t3, sel_d);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t unit = (it.dst[q >> 1] >> (16 * (q & 1))) & 0xFFFFu;
        const uint32_t at = win_s + unit * 16u;
        if (unit != kStreamNoUnit && B2C_SMEM_OK(args.dbg, 59, win_s, sa.win_bytes, at, 16))
          *reinterpret_cast<uint4*>(smem + at) = make_uint4(px[q][0], px[q][1], px[q][2], px[q][3]);
      }
    };
    const bool same_rows = stream_same_rows(sa);
    StreamItem kept[kKept];
    uint32_t live = 0;  // bit i: kept[i] stores something
    for (int t = tile_first; t < tile_end && ok; t += tile_step) {
      B2C_STREAM_TILE(t)
      (void)ct;
      const TileRows tr = stream_tile_rows(args, sa, r0);
      const int rows = tr.end - tr.r0;
      // (then the places are those of the first tile; a tile that ends behind the batch builds units of outputs that do not exist)
      if (t == tile_first || !same_rows) live = 0;
#pragma unroll
      for (int i = 0; i < kKept; ++i)
        if ((t == tile_first || !same_rows) && stream_item(args, sa, tr, tid + i * kGroupWarps * 32, y, STRIDE, &kept[i])) live |= 1u << i;
      for (int cb = 0; cb < sa.ncb; ++cb, next_window()) {
        if (turn != group) continue;
        ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&sc.win_empty[ws]), wph ^ 1u, ctl, args.status));
        if (!ok) break;
        const uint32_t win_s = (uint32_t)(ws * sa.win_bytes);
        // rows outside the image (a buffer's later windows of the tile find them cleared)
        if (!same_rows && cb < sa.win_stages) {
          for (int e = bw; e < rows * sa.ndh; e += kGroupWarps) {
            const int j = STRIDE == 1 || sa.ndh == 1 ? e : e >> 1, a = e - j * sa.ndh;
            const int gr = tr.r0 + j;
            const int n = (int)sa.div_rpi.div((uint32_t)gr);
            const int h = (gr - n * sa.rpi) * STRIDE + (int)sa.row_phase[a] - args.pad_h;
            if (n < sa.images && (unsigned)h < (unsigned)args.H) continue;
            for (int u = 0; u < 2; ++u)
              for (int b = 0; b < sa.ndw; ++b)
                for (int q = lane; q < sa.pitch; q += 32) {
                  const uint32_t at = win_s + (uint32_t)((u * per_row + a * sa.ndw + b) * sa.plane_bytes) + (uint32_t)(j * sa.pitch + q) * 16u;
                  if (B2C_SMEM_OK(args.dbg, 58, win_s, sa.win_bytes, at, 16)) *reinterpret_cast<uint4*>(smem + at) = make_uint4(0, 0, 0, 0);
                }
          }
        }
        ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&sc.raw_full[rs]), rph, ctl, args.status));
        if (!ok) break;
        const uint32_t raw_s = raw_off + (uint32_t)(rs * sa.raw_bytes);
#pragma unroll
        for (int i = 0; i < kKept; ++i)
          if ((live >> i) & 1u) build_item(kept[i], raw_s, win_s);
        for (int e = tid + kKept * kGroupWarps * 32; e < items; e += kGroupWarps * 32) {
          StreamItem it;
          if (stream_item(args, sa, tr, e, y, STRIDE, &it)) build_item(it, raw_s, win_s);
        }
        // the raw rows have been read; the units are visible to the tensor cores' async proxy
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(smem_u32(&sc.raw_empty[rs]));
          mbar_arrive_cluster(map_to_rank(smem_u32(&sc.win_full[ws]), 0u));
        }
      }
    }
  } else {
    // ---------------------------------------------------------------- epilogue warps (both blocks)
    const int quad = warp & 3;                     // tensor-memory lane quadrant this warp may read
    const int half = (warp - kFirstEpilogue) >> 2;  // the two warps of a quadrant split the columns
    const int row = quad * 32 + lane;
    const int j = (int)sa.div_pitch.div((uint32_t)row), q = row - j * sa.pitch;
    bool ok = true;
    int ti = 0;
    for (int t = tile_first; t < tile_end && ok; t += tile_step, ++ti) {
      B2C_STREAM_TILE(t)
      const int gr = r0 + j;
      const int n = (int)sa.div_rpi.div((uint32_t)gr);
      const int i = gr - n * sa.rpi;
      const bool row_valid = j < sa.th && q < args.out_Q && i < args.out_P && n < sa.images;
      const int out_pq = i * args.out_Q + q;
      const int buf = ti & 1;
      ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&sc.acc_full[buf]), (uint32_t)((ti >> 1) & 1), ctl, args.status));
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (!ok) break;
      const long long base_nkpq = (long long)n * args.y_stride_n + out_pq;
      const long long base_npqk = ((long long)n * args.out_PQ + out_pq) * args.K;
      const int cols = args.tile_n >> 1, c_begin = half * cols;  // (tile_n >= 64)
      const uint32_t taddr = tmem_acc + ((uint32_t)(quad * 32) << 16) + (uint32_t)(buf * args.tile_n + c_begin);
      for (int c = 0; c < cols; c += 32)
        epilogue_columns<32>(args, taddr + (uint32_t)c, ct * args.tile_n + c_begin + c, row_valid, base_nkpq, base_npqk, 0u);
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(map_to_rank(smem_u32(&sc.acc_empty[buf]), 0u));
    }
  }
#undef B2C_STREAM_TILE

  // ---------------------------------------------------------------- teardown
  // No block of the pair leaves, or frees tensor memory, while the other may still read its shared memory, arrive on its
  // barriers or write its accumulator.
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (ctl->abort_flag) {
    if (threadIdx.x == 0) {
      const unsigned long long t0 = global_ns();
      while (global_ns() - t0 < 50000ull) __nanosleep(1000);
    }
    __syncthreads();
  }
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_acc), "r"(sa.tmem_cols) : "memory");
  }
}

template <int STRIDE, bool WORDS>
cudaError_t launch_one(const CUtensorMap& tmap_x, const CUtensorMap& tmap_w, const ConvArgs& args, const StreamArgs& sa, int* resident,
                       cudaStream_t st) {
  static std::atomic<unsigned long long> configured{0};
  cudaError_t e = set_max_dynamic_smem_once(configured, (const void*)conv_mma_stream_kernel<STRIDE, WORDS>, kStreamSmemMax);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(2 * std::min(sa.num_tiles, sa.pairs)));
  cfg.blockDim = dim3(kStreamThreads);
  cfg.dynamicSmemBytes = (size_t)sa.smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 2;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  if (resident) return cudaOccupancyMaxActiveClusters(resident, conv_mma_stream_kernel<STRIDE, WORDS>, &cfg);
  e = cudaLaunchKernelEx(&cfg, conv_mma_stream_kernel<STRIDE, WORDS>, tmap_x, tmap_w, args, sa);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_form(const CUtensorMap& tmap_x, const CUtensorMap& tmap_w, const ConvArgs& args, const StreamArgs& sa, int* resident,
                        cudaStream_t st) {
  if (sa.stride == 1)
    return sa.words ? launch_one<1, true>(tmap_x, tmap_w, args, sa, resident, st) : launch_one<1, false>(tmap_x, tmap_w, args, sa, resident, st);
  return sa.words ? launch_one<2, true>(tmap_x, tmap_w, args, sa, resident, st) : launch_one<2, false>(tmap_x, tmap_w, args, sa, resident, st);
}

}  // namespace

// Pairs of blocks that the device keeps resident at once: the persistent grid is one wave of them.
int stream_resident_pairs(const StreamArgs& sa) {
  StreamArgs s = sa;
  s.pairs = kNumSMs / 2;
  int resident = 0;
  if (launch_form(CUtensorMap{}, CUtensorMap{}, ConvArgs{}, s, &resident, nullptr) != cudaSuccess) (void)cudaGetLastError();
  return resident > 0 ? std::min(resident, kNumSMs / 2) : kNumSMs / 2;
}

cudaError_t launch_conv_mma_stream(const CUtensorMap& tmap_x, const CUtensorMap& tmap_w, const ConvArgs& args, const StreamArgs& sa,
                                   cudaStream_t st) {
  return launch_form(tmap_x, tmap_w, args, sa, nullptr, st);
}

}  // namespace b2c
