"""Parity of the window unroll's forms and of the epilogue's branches against the CPU oracle, at the sizes where
they can go wrong.  All sums are exact integers, so every comparison is element by element."""
import numpy as np
import pytest
import torch

import oracle
import paper_2104_04731_b200 as b2c
from paper_2104_04731_b200.synth import int8_uniform

from gpu_util import check_against_oracle, to_dev

pytestmark = pytest.mark.gpu


# ---- per-channel bias: whole runs of channels with one load per four values, ragged runs one by one ----------
@pytest.mark.parametrize("K,groups", [(64, 1), (48, 1), (33, 1), (20, 1), (24, 4), (128, 2)])   # 24 / 4 = 6: bias not on 16 bytes
def test_bias_vector_and_scalar_loads(lib, K, groups):
    N, C, H, W = 2, 32, 9, 8
    x = int8_uniform((N, C, H, W), 1011)
    w = int8_uniform((K, C // groups, 3, 3), 1012)
    bias = int8_uniform((K,), 1013).astype(np.int32) * 701
    want = oracle.conv2d_int8(x, w, 1, 1, 1, 6, bias=bias, relu=True, groups=groups)
    d = lib.make_desc(N, C, H, W, K, 3, 3, 1, 1, 1, 6, out_mode=3)
    for e in [None] if groups > 1 else lib.enumerate_embeddings(d):
        plan = lib.Plan(d, groups=groups) if groups > 1 else lib.Plan(d, e.id)
        plan.set_weights(to_dev(w))
        plan.set_activation(to_dev(bias), True)
        y32 = torch.full((N, K, H, W), -7777777, dtype=torch.int32, device="cuda")
        y8 = torch.full((N, K, H, W), 77, dtype=torch.int8, device="cuda")
        ws = torch.zeros(max(16, plan.workspace_bytes()), dtype=torch.uint8, device="cuda")
        plan.run(to_dev(x), y32, y8, ws)
        torch.cuda.synchronize()
        assert plan.device_status() == b2c.OK
        assert np.array_equal(y32.cpu().numpy(), want[0]) and np.array_equal(y8.cpu().numpy(), want[1])
        plan.destroy()


# ---- window unroll over planes of units: forms, staging and window dealing at the edges of their ranges -----------
# (batches above the size from which this kernel runs, or shapes the window kernel does not take; every listed schedule)
@pytest.mark.parametrize("case", [
    # N, C, H, W, K, R, S, stride, pad, dil, shift
    (3, 1, 40, 61, 32, 20, 5, 2, 0, 1, 9),             # one channel, odd width: runs of two words, 20 filter rows
    (5, 3, 27, 35, 64, 7, 7, 2, 3, 1, 8),              # 7x7 stem on an odd image: six runs, columns outside on both sides
    (2, 1, 12, 75, 17, 3, 21, 2, 4, 1, 7),             # runs of six words; 17 channels
    (2, 2, 15, 33, 40, 2, 12, 1, 3, 1, 6),             # runs of four words, stride 1
    (3, 5, 14, 22, 24, 3, 3, (1, 3), 1, (2, 1), 6),    # stride 3: one column per builder item; vertical dilation
    (4, 17, 13, 15, 20, 3, 3, 1, 1, 1, 8),             # channel form, H * W odd: unaligned words
    (2, 40, 18, 10, 96, 3, 3, 1, 1, 1, 9),             # channel form, flat groups across row ends, ragged channel block
    (3, 24, 17, 12, 33, 3, 3, 2, 1, 1, 8),             # channel form, stride 2: four phase planes
    (2, 12, 16, 20, 300, 1, 1, 1, 0, 1, 6),            # 1x1; three column tiles
    (2, 9, 20, 18, 16, 3, 3, 1, (4, 0), 4, 7),         # dilation 4, padding on one axis
    (1, 8, 9, 50, 16, 2, 2, 1, 32, 1, 5),              # padding as wide as the kernel takes
    (60, 8, 7, 7, 8, 3, 3, 1, 1, 1, 7),                # small images: a window spans many (7 rows each)
    (300, 18, 14, 14, 16, 3, 3, 1, 1, 1, 8),           # whole images staged (3528 bytes: two alignments in turn)
    (30, 3, 225, 223, 16, 5, 5, 2, 2, 1, 7),           # segments of one window dealt to the blocks in turn; blocks that walk one segment
    (100, 48, 30, 30, 64, 3, 3, 1, 1, 1, 9),           # the same in channel form: flat groups, moved overlap rows
    (20, 64, 56, 24, 40, 3, 3, 1, 1, 1, 9),            # one tiled copy for all channels: segments of single images
    (12, 20, 96, 44, 32, 3, 5, 2, (1, 2), 1, 8),       # the same with stride 2; ragged last segment of an image
])
@pytest.mark.parametrize("out_layout,out_mode", [(0, 3), (1, 2)])
def test_plane_kernel(lib, case, out_layout, out_mode):
    N, C, H, W, K, R, S, stride, pad, dil, shift = case
    x = int8_uniform((N, C, H, W), 1021)
    w = int8_uniform((K, C, R, S), 1022)
    ref = oracle.conv2d_int8(x, w, stride, pad, dil, shift)
    d = lib.make_desc(N, C, H, W, K, R, S, stride, pad, dil, shift, 0, out_layout, out_mode)
    ids = [e.id for e in lib.enumerate_embeddings(d) if e.variant == b2c.VARIANT_IM2COL_WINDOW]
    assert ids
    for i in ids:
        check_against_oracle(x, w, stride, pad, dil, shift, out_mode, i, ref=ref, out_layout=out_layout)


# ---- blocks that walk several segments of several windows (moved overlap rows, then a fresh segment in the same rings), and
# accumulator rings of odd length between two sets of epilogue warps: combinations that only larger batches list ----------
@pytest.mark.parametrize("case", [
    # N, C, H, W, K, R, stride, out_layout, out_mode
    (90, 17, 40, 36, 16, 3, 1, 0, 2),      # one tiled copy, flat groups: 180 segments of 20 rows, windows of 10
    (160, 48, 16, 34, 16, 3, 2, 1, 1),     # one tiled copy, unaligned words, stride 2: 160 segments of 8 rows, windows of 4
    (150, 48, 42, 44, 16, 3, 2, 0, 2),     # row segments by bulk copies: 150 segments of 22 rows, windows of 11
    (160, 64, 38, 37, 16, 3, 1, 1, 2),     # two blocks per SM, one window buffer and one raw chunk: 320 segments
    (160, 16, 40, 35, 96, 3, 1, 0, 3),     # segments across images, ring of five accumulators
    (300, 5, 29, 30, 96, 3, 1, 0, 1),      # the same in row form
    (310, 1, 23, 37, 144, 3, 1, 0, 1),     # whole images, row form, ring of three accumulators
])
def test_plane_kernel_walks_segments(lib, case):
    N, C, H, W, K, R, stride, out_layout, out_mode = case
    x = int8_uniform((N, C, H, W), 1081)
    w = int8_uniform((K, C, R, R), 1082)
    ref = oracle.conv2d_int8(x, w, stride, R // 2, 1, 8)
    d = lib.make_desc(N, C, H, W, K, R, R, stride, R // 2, 1, 8, 0, out_layout, out_mode)
    ids = [e.id for e in lib.enumerate_embeddings(d) if e.variant == b2c.VARIANT_IM2COL_WINDOW]
    assert len(ids) > 1
    for i in ids:
        check_against_oracle(x, w, stride, R // 2, 1, 8, out_mode, i, ref=ref, out_layout=out_layout)


# ---- NKPQ stores from sector boundaries: tiles that start before their window (row form), rows widened to whole sectors ----------
@pytest.mark.parametrize("case", [
    # N, C, H, W, K, R, stride, pad, out_mode
    (20, 3, 60, 92, 16, 7, 2, 3, 1),       # row form, rows of 46: windows start at every even distance from a boundary
    (7, 2, 96, 100, 24, 3, 1, 1, 2),       # int8 alone: sectors of 32 results, up to 28 positions of lead
    (9, 17, 64, 54, 33, 3, 1, 1, 3),       # channel form, rows widened from 55 to 62 positions
    (40, 64, 56, 56, 48, 3, 1, 1, 1),      # 57 to 64: every row starts on a boundary
    (11, 20, 52, 50, 16, 3, 1, 1, 1),      # rows of 50 widened to 58, segments of several windows
    (3, 1, 82, 30, 16, 5, 1, 2, 1),        # a short last window with a lead
])
def test_plane_kernel_aligned_stores(lib, case):
    N, C, H, W, K, R, stride, pad, out_mode = case
    x = int8_uniform((N, C, H, W), 1091)
    w = int8_uniform((K, C, R, R), 1092)
    ref = oracle.conv2d_int8(x, w, stride, pad, 1, 8)
    d = lib.make_desc(N, C, H, W, K, R, R, stride, pad, 1, 8, out_mode=out_mode)
    ids = [e.id for e in lib.enumerate_embeddings(d) if e.variant == b2c.VARIANT_IM2COL_WINDOW]
    assert len(ids) > 1
    # (the row form, fewer than 8 channels, begins tiles before their windows)
    assert (C < 8) == any(lib.test_kernel_of(d, i) == b2c.KERNEL_PLANE_LEAD for i in ids)
    for i in ids:
        check_against_oracle(x, w, stride, pad, 1, 8, out_mode, i, ref=ref)


def test_plane_kernel_reads_the_last_incomplete_16_bytes(lib):
    """The tensor ends inside a 16-byte unit: its last bytes are copied one by one, nothing behind them is read."""
    N, C, H, W, K = 3, 3, 29, 31, 16                     # 8091 bytes, 11 past the last whole unit
    x = int8_uniform((N, C, H, W), 1031)
    w = int8_uniform((K, C, 3, 3), 1032)
    ref = oracle.conv2d_int8(x, w, 1, 1, 1, 5)
    d = lib.make_desc(N, C, H, W, K, 3, 3, 1, 1, 1, 5, out_mode=3)
    assert x.size % 16 == 11
    for e in lib.enumerate_embeddings(d):
        if e.variant == b2c.VARIANT_IM2COL_WINDOW:
            check_against_oracle(x, w, 1, 1, 1, 5, 3, e.id, ref=ref)


# ---- units built while the weights stream (two SMs): staging forms, ragged blocks, walks of several tiles -------------------------
@pytest.mark.parametrize("case", [
    # N, C, H, W, K, R, S, stride, pad, dil, shift
    (37, 256, 14, 14, 130, 3, 3, 2, 1, 1, 11),      # whole images, four phase planes, ragged column tile, a pair with an empty half
    (130, 64, 7, 7, 64, 3, 3, 1, 1, 1, 9),          # H * W odd: unaligned words
    (21, 80, 28, 28, 96, 3, 3, 1, 1, 1, 10),        # one tiled copy per image part; ragged last block of 16 channels
    (9, 96, 44, 40, 70, 5, 5, 2, 2, 1, 11),         # 25 MMAs a block: weight stages that end inside one
    (11, 64, 28, 52, 300, 2, 3, 1, (0, 1), 3, 9),   # dilation 3, six taps, padding on one axis (30 rows are no form of this kernel)
    (60, 48, 12, 20, 256, 4, 1, 1, 2, 1, 9),        # half a block of channels, padding wider than the taps need
    (400, 64, 14, 14, 512, 3, 3, 2, 1, 1, 10),      # several tiles a pair: both accumulators, rings that run on
    (2, 48, 112, 126, 64, 3, 3, 1, 1, 1, 9),        # one grid row of 127 positions a tile
    (34, 112, 44, 40, 32, 5, 5, 2, 2, 1, 11),       # rings of two windows, several tiles of four windows each
])
@pytest.mark.parametrize("out_layout,out_mode", [(0, 3), (1, 2)])
def test_stream_kernel(lib, case, out_layout, out_mode):
    N, C, H, W, K, R, S, stride, pad, dil, shift = case
    x = int8_uniform((N, C, H, W), 1095)
    w = int8_uniform((K, C, R, S), 1096)
    ref = oracle.conv2d_int8(x, w, stride, pad, dil, shift)
    d = lib.make_desc(N, C, H, W, K, R, S, stride, pad, dil, shift, 0, out_layout, out_mode)
    ids = [e.id for e in lib.enumerate_embeddings(d) if e.variant == b2c.VARIANT_IM2COL_WINDOW and e.tile_n >= 64]
    assert any(lib.test_kernel_of(d, i) == b2c.KERNEL_STREAM for i in ids)
    for i in ids:
        check_against_oracle(x, w, stride, pad, dil, shift, out_mode, i, ref=ref, out_layout=out_layout)


@pytest.mark.parametrize("case", [
    # N, C, H, W, K, R, S, pad, dil: stride 2, the last row of every image is read by no output
    (64, 64, 15, 15, 128, 2, 2, 0, 1),
    (64, 128, 13, 12, 128, 2, 2, 0, 1),
    (60, 64, 17, 22, 96, 4, 3, (0, 1), 1),
    (40, 96, 27, 20, 70, 6, 3, (0, 1), 1),
    (50, 64, 21, 26, 64, 2, 2, 0, (3, 1)),
])
def test_stream_kernel_unread_last_row(lib, case):
    """It belongs to no grid row of its image; stored, it would lie on the next image's first row."""
    N, C, H, W, K, R, S, pad, dil = case
    x = int8_uniform((N, C, H, W), 1097)
    w = int8_uniform((K, C, R, S), 1098)
    ref = oracle.conv2d_int8(x, w, 2, pad, dil, 9)
    d = lib.make_desc(N, C, H, W, K, R, S, 2, pad, dil, 9, 0, 0, 3)
    ids = [e.id for e in lib.enumerate_embeddings(d) if lib.test_kernel_of(d, e.id) == b2c.KERNEL_STREAM]
    assert ids
    for i in ids:
        for _ in range(3):
            check_against_oracle(x, w, 2, pad, dil, 9, 3, i, ref=ref)


@pytest.mark.parametrize("case", [
    # N, C, H, W, K, R, stride, pad: space to depth is a fifth or more faster than the plane kernel, and has a higher overhead
    (8, 93, 93, 9, 364, 3, 2, 1),
    (3, 96, 28, 14, 192, 3, 2, 1),
])
def test_timed_selection_runs_the_other_families_beside_the_plane_kernel(lib, case):
    N, C, H, W, K, R, stride, pad = case
    d = lib.make_desc(N, C, H, W, K, R, R, stride, pad)
    assert any(e.variant == b2c.VARIANT_IM2COL_WINDOW for e in lib.enumerate_embeddings(d))
    plan = lib.Plan(d, b2c.POLICY_AUTO_TIMED)
    assert plan.info().variant == b2c.VARIANT_SPACE_TO_DEPTH
    plan.destroy()


@pytest.mark.parametrize("case", [
    # N, C, H, W, K, groups, R, shift, out_mode
    (40, 64, 28, 28, 64, 64, 3, 5, 3),       # depth-wise: groups merged 16 at a time and more
    (30, 96, 17, 23, 96, 96, 3, 5, 1),       # odd image: every group's channel slice at another alignment
    (16, 128, 20, 20, 256, 8, 3, 7, 2),      # 16 -> 32 channels a group, nothing to merge
])
def test_grouped_plane_kernel(lib, case):
    N, C, H, W, K, groups, R, shift, out_mode = case
    x = int8_uniform((N, C, H, W), 1041)
    w = int8_uniform((K, C // groups, R, R), 1042)
    bias = int8_uniform((K,), 1043).astype(np.int32) * 97
    want = oracle.conv2d_int8(x, w, 1, 1, 1, shift, bias=bias, relu=True, groups=groups)
    d = lib.make_desc(N, C, H, W, K, R, R, 1, 1, 1, shift, out_mode=out_mode)
    plan = lib.Plan(d, b2c.POLICY_AUTO_TIMED, groups=groups)
    assert plan.info().device_us > 0
    assert plan.info().variant == b2c.VARIANT_IM2COL_WINDOW   # well ahead of the staged window and of the dense form here
    plan.set_weights(to_dev(w))
    plan.set_activation(to_dev(bias), True)
    y32 = torch.full((N, K, H, W), -7777777, dtype=torch.int32, device="cuda") if out_mode & 1 else None
    y8 = torch.full((N, K, H, W), 77, dtype=torch.int8, device="cuda") if out_mode & 2 else None
    ws = torch.zeros(max(16, plan.workspace_bytes()), dtype=torch.uint8, device="cuda")
    plan.run(to_dev(x), y32, y8, ws)
    torch.cuda.synchronize()
    assert plan.device_status() == b2c.OK
    assert y32 is None or np.array_equal(y32.cpu().numpy(), want[0])
    assert y8 is None or np.array_equal(y8.cpu().numpy(), want[1])
    plan.destroy()


# ---- one-shot call: weights packed by the launch that packs the activations -----------------------------------------
@pytest.mark.parametrize("case", [
    # N, C, H, W, K, R, stride, pad, dil
    (1, 64, 56, 56, 64, 3, 1, 1, 1),     # rows by bulk copies
    (2, 48, 14, 14, 72, 3, 1, 1, 1),     # whole images by bulk copies; 48 channels padded to 64
    (3, 33, 9, 11, 40, 3, 2, 1, 1),      # odd image: the loads of the plain pack kernel; 33 channels
    (2, 70, 12, 10, 129, 1, 1, 0, 1),    # 1x1
    (160, 130, 4, 4, 600, 3, 1, 1, 1),   # as many blocks of activations as SMs: fewer of weights, several words a thread
    (2, 256, 14, 14, 512, 3, 2, 1, 1),   # eight rows of channel tiles, weight blocks dealt to them
])
def test_one_shot_packs_weights_with_the_activations(lib, case):
    N, C, H, W, K, R, stride, pad, dil = case
    xs = [int8_uniform((N, C, H, W), 1051 + i) for i in range(2)]
    ws = [int8_uniform((K, C, R, R), 1061 + i) for i in range(2)]
    lib.oneshot_cache_clear()
    for x, w in zip(xs + xs[::-1], ws + ws):   # weights and activations change from call to call
        want = oracle.conv2d_int8(x, w, stride, pad, dil, 9)
        y32 = torch.full(want[0].shape, -7777777, dtype=torch.int32, device="cuda")
        y8 = torch.full(want[1].shape, 77, dtype=torch.int8, device="cuda")
        lib.conv2d_int8(to_dev(x), to_dev(w), stride, pad, dil, 9, y32, y8)
        torch.cuda.synchronize()
        assert np.array_equal(y32.cpu().numpy(), want[0]) and np.array_equal(y8.cpu().numpy(), want[1])
    assert lib.oneshot_status() == b2c.OK
    lib.oneshot_cache_clear()


# ---- channel-pack weights of more than 2^32 words: the filter index needs 64 bits -----------------------------------------
def test_channel_pack_of_weights_beyond_32_bit_indices(lib):
    """One channel is packed as 32, so 32769 filters of 128 x 128 taps are 2^32 + 131072 words (17 GB) from 0.5 GB."""
    K, R = 32769, 128
    assert K * R * R * 8 == 2**32 + 131072
    if torch.cuda.mem_get_info()[0] < 30 << 30:
        pytest.skip("needs 30 GB of free device memory")
    gen = torch.Generator(device="cuda").manual_seed(1071)
    w = torch.randint(-128, 128, (K, 1, R, R), dtype=torch.int8, device="cuda", generator=gen)
    x = torch.randint(-128, 128, (1, 1, R, R), dtype=torch.int8, device="cuda", generator=gen)
    want = torch.mv(w.view(K, R * R).double(), x.view(R * R).double()).to(torch.int32)   # (exact: sums below 2^28)
    d = lib.make_desc(1, 1, R, R, K, R, R)
    e = max((e for e in lib.enumerate_embeddings(d) if e.variant == b2c.VARIANT_CP_TMA and e.split_k == 1
             and e.map_m == b2c.AXIS_NPQ), key=lambda e: e.tile_n)
    plan = lib.Plan(d, e.id)
    try:
        plan.set_weights(w)
        y32 = torch.full((1, K, 1, 1), -7777777, dtype=torch.int32, device="cuda")
        ws = torch.zeros(max(16, plan.workspace_bytes()), dtype=torch.uint8, device="cuda")
        plan.run(x, y32, None, ws)
        torch.cuda.synchronize()
        assert plan.device_status() == b2c.OK
        assert torch.equal(y32.view(K), want)
    finally:
        plan.destroy()


# ---- NPQK results in 16-byte pieces: exchanged between four lanes (int32 sums), a last run of channels shorter than a tile ----
@pytest.mark.parametrize("K", [4, 12, 16, 36, 48, 80, 272])
@pytest.mark.parametrize("in_layout,case", [
    # N, C, H, W, R, S, stride, pad, dil, shift: pixel counts that are no multiple of 4, 32 or 128
    (1, (3, 32, 7, 9, 3, 3, 1, 1, 1, 8)),
    (0, (1, 3, 21, 17, 3, 3, 2, 1, 1, 6)),
    (1, (2, 16, 13, 11, 2, 2, 1, 0, 3, 7)),     # dilation: rows that fall outside the output
])
def test_npqk_results_in_pieces(lib, K, in_layout, case):
    N, C, H, W, R, S, st, pad, dil, shift = case
    x = int8_uniform((N, C, H, W), 1021)
    w = int8_uniform((K, C, R, S), 1022)
    bias = int8_uniform((K,), 1023).astype(np.int32) * 311
    want = [np.ascontiguousarray(v.transpose(0, 2, 3, 1))
            for v in oracle.conv2d_int8(x, w, st, pad, dil, shift, bias=bias, relu=True)[:2]]
    xd = to_dev(np.ascontiguousarray(x.transpose(0, 2, 3, 1)) if in_layout else x)
    for mode in (1, 2, 3):
        d = lib.make_desc(N, C, H, W, K, R, S, st, pad, dil, shift, in_layout, 1, mode)
        for e in lib.enumerate_embeddings(d):
            plan = lib.Plan(d, e.id)
            plan.set_weights(to_dev(w))
            plan.set_activation(to_dev(bias), True)
            y32 = torch.full(want[0].shape, -7777777, dtype=torch.int32, device="cuda") if mode & 1 else None
            y8 = torch.full(want[0].shape, 77, dtype=torch.int8, device="cuda") if mode & 2 else None
            ws = torch.zeros(max(16, plan.workspace_bytes()), dtype=torch.uint8, device="cuda")
            plan.run(xd, y32, y8, ws)
            torch.cuda.synchronize()
            assert plan.device_status() == b2c.OK
            assert y32 is None or np.array_equal(y32.cpu().numpy(), want[0]), (mode, e.id)
            assert y8 is None or np.array_equal(y8.cpu().numpy(), want[1]), (mode, e.id)
            plan.destroy()
