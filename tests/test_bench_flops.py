"""The roofline's numerator and traffic are those of the kept counters of the cell kernel: bench.py's executed
flops and DRAM bytes per cell against the table of profiles/newton_kernels_lognormal_hhe_128.md."""
import os
import re

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_executed_flops_are_the_counted_ones():
    with open(os.path.join(ROOT, "profiles", "newton_kernels_lognormal_hhe_128.md")) as fh:
        row = next(line for line in fh if line.startswith("| `k_cell<3,ITER>`"))
    cells = [c.strip() for c in row.split("|")]
    dfma, dmul, dadd = (float(v) for v in cells[5].split("/"))
    assert bench.EXECUTED_FLOPS["cell_residual_schur"] == 2 * dfma + dmul + dadd
    read, written = (float(v) for v in re.findall(r"[\d.]+", cells[6]))
    assert abs(bench.TRAFFIC_PER_CELL["cell_residual_schur"] - (read + written) * 1e6 / 128 ** 3) < 0.1
    assert bench.EXECUTED_FLOPS.keys() == bench.ALU_FLOPS.keys()
