"""Programmatic dependent launch in the kernels' sources.  A kernel that lets the next
one start before it has waited for the one before it lets a whole queue of waiting
grids become resident; so the release follows the wait (the complex128 sweep releases
earlier on grids of at most one warp an SM, or larger than the SMs hold, by template)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_03617_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as fh:
        return re.sub(r"//[^\n]*", "", fh.read())


@pytest.mark.parametrize("name", ["tma3d2.cu", "conv_tile.cu"])
def test_release_follows_the_wait(name):
    # one place in the source where a kernel waits, and the release right behind it
    assert re.findall(r"griddepcontrol\.(\w+)", _source(name)) == ["wait", "launch_dependents"]


def _chained_sources():
    return [f for f in sorted(os.listdir(CSRC)) if f.endswith(".cu") and "griddepcontrol.wait" in _source(f)]


def test_no_read_only_loads_of_a_predecessors_output():
    """A chained kernel runs while its predecessor writes its inputs: they must not be
    read by loads for memory that is constant over the kernel's life (ld.global.nc,
    __ldg).  Tables that no chained kernel writes are const __restrict__ arguments."""
    assert len(_chained_sources()) == 3
    for name in _chained_sources():
        assert not re.findall(r"\.nc\b|__ldg\w*\s*\(", _source(name)), name
