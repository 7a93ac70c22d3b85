"""The stream kernel's placement of pixels (csrc/stream_tile.h), replayed on the host for random layers: no unit of a window
has two writers, and every tap of every output reads its pixel, or zero outside the image.  And the waits of its rings,
whose barriers tell phases apart by parity only, with the roles in random order."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2104_04731_b200", "csrc")


@pytest.fixture(scope="module")
def replay(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("placement") / "stream_placement")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", os.path.join(cuda, "include"), "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                           os.path.join(HERE, "stream_placement.cpp"), os.path.join(CSRC, "planner.cpp"), "-o", exe])
    return lambda *args: subprocess.run([exe, *map(str, args)], capture_output=True, text=True, timeout=300)


def test_random_layers(replay):
    r = replay(20000)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
    right = int(r.stdout.rsplit("layers: ", 1)[1].split()[0])
    assert right > 5000, r.stdout


@pytest.mark.parametrize("layer", [
    # N, C, H, W, K, R, S, stride, pad (rows, columns), dilation: the last row of an image is read by no output
    (64, 64, 15, 15, 128, 2, 2, 2, 0, 0, 1, 1),
    (64, 128, 13, 12, 128, 2, 2, 2, 0, 0, 1, 1),
    (60, 64, 17, 22, 96, 4, 3, 2, 0, 1, 1, 1),
    (40, 96, 27, 20, 70, 6, 3, 2, 0, 1, 1, 1),
    (50, 64, 21, 26, 64, 2, 2, 2, 0, 0, 3, 1),
])
def test_even_filters_with_stride_two(replay, layer):
    r = replay(*layer)
    assert r.returncode == 0 and "1 right" in r.stdout, r.stdout + r.stderr


def test_ring_waits(replay):
    r = replay("rings")
    assert r.returncode == 0 and "2 windows" in r.stdout, r.stdout + r.stderr
