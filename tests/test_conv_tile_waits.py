"""Bounded waits of the tiled convolutions, in the source: what a role does after a wait
are warp-wide instructions, so the lanes of a warp have to agree on its outcome also
when it ran out (one lane may have seen the phase complete, the next the abort flag)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_03617_gb300", "csrc")


def test_a_warp_agrees_on_the_outcome_of_a_wait():
    with open(os.path.join(CSRC, "conv_tile.cu")) as fh:
        src = re.sub(r"//[^\n]*", "", fh.read())
    kernels = [k.split("\ntemplate")[0] for k in src.split("__global__")[1:] if "bar_wait(" in k]
    assert len(kernels) == 2
    for k in kernels:
        # the role of one lane: from "warp == 4" and "lane == 0" to the warp's reunion
        role = re.search(r"else if \(warp == 4\) \{\s*if \(lane == 0\) \{(.*?)\n        \}\s*__syncwarp\(\);\s*\} else", k, re.S)
        assert role, "the MMA issuer is one lane"
        assert "__syncwarp" not in role.group(1) and "_sync(" not in role.group(1)
        rest = k[:role.start()] + k[role.end():]
        uses = [ln.strip() for ln in rest.splitlines() if "bar_wait(" in ln]
        assert uses
        for u in uses:
            voted = "all_of_128(bar_wait(" in u or "__all_sync(0xffffffffu, bar_wait(" in u
            assert voted or u.startswith("bar_wait("), u            # or nothing depends on it
