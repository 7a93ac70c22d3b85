"""Every bounded wait of the convolution kernels is voted on by its warp before the warp acts on it.

A wait gives up after its time limit or when another warp has.  If the lanes of a warp disagreed (the barrier completes while
one of them gives up), some would leave the role and the others wait for them at the next warp-wide instruction for good.
The time limit cannot be made to run out between two lanes on purpose, so this reads the sources.
"""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2104_04731_b200", "csrc")


def test_results_of_waits_are_voted():
    waits = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "conv_mma*.cu")) + [os.path.join(CSRC, "mma_rate.cu")]):
        lines = open(path).read().split("\n")
        own = False  # a lane's own result is kept in `ok`
        for n, line in enumerate(lines):
            call = re.search(r"\bmbar_wait(_\w+)?\(", line)
            if not call or "__device__" in line or line.lstrip().startswith("//"):
                continue
            waits += 1
            before = line[:call.start()].strip()
            if before in ("", "(void)") or before.endswith("__all_sync(0xffffffffu,"):  # not used, or voted at once
                continue
            assert before == "ok =" and lines[n + 1].strip() == "if (!__all_sync(0xffffffffu, ok)) break;", (os.path.basename(path), n + 1, line)
            own = True
        if own:  # then nothing but the vote looks at it
            assert not re.search(r"&& ok\b", "\n".join(lines)), os.path.basename(path)
    assert waits > 20


def test_staged_window_warps_leave_together():
    """They meet at a barrier in every tile after the first; a warp whose wait gave up still comes there, with its word for it."""
    source = open(os.path.join(CSRC, "conv_mma.cu")).read()
    role = source[source.index("gather + epilogue warps"):]
    assert "(ok || AMODE == A_STAGED)" in role.split("B2C_TILE_ORIGIN", 1)[0]
    first = re.search(r'if \(ti > 0[^\n]*', role).group(0)
    assert "!barrier_and(1, kGatherWarps * 32, ok)) break;" in first
