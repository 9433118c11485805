"""Barriers of the kernels whose warps take different roles, read from the source (no GPU needed)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2104_08309_gb300", "csrc")


def _block(text, at):
    """The brace block that opens at or after `at`, and the index after it."""
    i = text.index("{", at)
    depth = 0
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i:j + 1], j + 1
    raise AssertionError("unbalanced braces")


def test_k_small3_roles_meet_at_named_barriers():
    """The FP64 and the FP32 warps of k_small3 run in the two arms of one branch.  __syncthreads() may only be
    reached on a condition that is the same for the whole block, so the arms meet at a named barrier of all
    its threads, apart from those of each half."""
    text = open(os.path.join(CSRC, "pft_small.cu")).read()
    kernel, _ = _block(text, text.index(") k_small3("))
    arm64, end = _block(kernel, kernel.index("if (warp < kGW)"))
    assert kernel[end:].lstrip().startswith("else")
    arm32, _ = _block(kernel, end)
    for arm in (arm64, arm32):
        assert "__syncthreads" not in arm
        assert arm.count("both_sync()") == 1      # one a round of the loop over the batches
    whole = re.search(r"void both_sync\(\).*?bar\.sync (\d+), %0;\" ::\"n\"\((\w+)\)", text)
    assert whole.group(2) == "kNT"
    ids = {1, 2}                                  # half_sync of the two halves
    assert re.search(r"half_sync\(1\)", arm64) and "lane, warp, 1)" in arm64 and "warp - kGW, 2)" in arm32
    assert int(whole.group(1)) not in ids | {0}
