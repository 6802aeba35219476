"""CPU tests of the bench's bookkeeping for plans whose inner solve runs by grid
groups, and of the list of sources that ties a profile to the kernel code."""
import os
import re
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2309_14584_gb300", "csrc")
sys.path.insert(0, ROOT)

import bench  # noqa: E402

INFO = {"N": 5, "K": 3, "R": 4, "M": 7}
REP = {"iterations": 4, "refinements": 1}


def test_bytes_of_an_inner_solve_by_grid_groups():
    """N = 5, K = 3, two groups: 12 K N + 16 G N + 24 N = 180 + 160 + 120 = 460 an
    iteration; DCT 8 M + 8 R = 88; the FP64 sweep 8 K N + 8 (8 N + 5 R) = 600."""
    layout = {"groups": 2, "grids_per_group": 2, "slices": 1, "slice_coefs": 32}
    assert bench.algorithmic_bytes(INFO, REP, "mixed", layout) == 88 + 4 * 460 + 600
    none = dict.fromkeys(layout, 0)
    assert bench.algorithmic_bytes(INFO, REP, "mixed", none) == bench.algorithmic_bytes(INFO, REP, "mixed")
    hbm, gather = bench.sparse_rooflines(INFO, REP, 1e-3, {"hbm_gbs": 1.0}, "measured", 0.3, layout)
    assert gather is None and hbm["algorithmic_bytes_per_launch"] == 88 + 4 * 460 + 600
    assert bench.sparse_rooflines(INFO, REP, 1e-3, {"hbm_gbs": 1.0}, "measured", 0.3, none)[1]["loads_per_launch"] == 150


def test_profiles_are_tied_to_every_source_of_the_solver_kernels():
    seen, todo = set(), ["fct_solver.cuh"]
    while todo:
        name = todo.pop()
        if name in seen or not os.path.exists(os.path.join(CSRC, name)):
            continue
        seen.add(name)
        todo += re.findall(r'#include "([^"]+)"', open(os.path.join(CSRC, name)).read())
    assert "fct_cells.cuh" in seen
    assert seen == set(bench.SOLVER_SOURCES)
