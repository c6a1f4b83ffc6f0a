"""Counts behind bench.py's roofline lines (no GPU)."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402
from paper_2506_03617_gb300 import inputs as I  # noqa: E402


@pytest.mark.parametrize("ni,npml", [((5, 7), 0), ((5, 7), 2), ((9, 4), 3), ((4, 5, 6), 0), ((4, 5, 3), 2)])
def test_fp64_instructions_count_every_cell(ni, npml):
    g = I.Grid(len(ni), ni, npml)
    total = 0
    for flat in range(g.n_total):
        k, q = 0, flat
        for d in range(g.dim):
            q, i = divmod(q, g.n[d])
            k += i < npml or i >= npml + ni[d]
        total += bench.FP64_INSTR[g.dim][k]
    assert bench.fp64_instr_per_update(g) == pytest.approx(total / g.n_total, rel=1e-14)


def test_a_launch_of_two_steps_counts_its_bytes_once():
    assert bench.sweep_bytes("c64", 1000, 7) == 28 * 1000 * 7
    with open(os.path.join(ROOT, "bench.py")) as fh:
        src = fh.read()
    row = src[src.index("# HBM-resident case"):src.index('extra["hbm_resident_3d"]')]
    assert "BYTES_PER_PT" not in row and row.count("sweep_bytes(") == 2      # by launches, not by steps
