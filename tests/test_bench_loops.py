"""What bench.py says about the loops that keep vectors in shared memory (no GPU):
their kernel's name, their bytes, and the bound at sizes in and beyond L2."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402

LOOP = {"l2_window": "none", "persistent": True, "persistent_single_reduction": True,
        "cluster": False, "stream_single_reduction": False}


@pytest.mark.parametrize("vectors,rows,per_cell", [(5, True, 16), (5, False, 52), (4, False, 60),
                                                   (3, False, 76)])
def test_resident_loop_on_all_cells(vectors, rows, per_cell):
    tf = dict(LOOP, resident_vectors=vectors, resident_rows=rows)
    assert bench.loop_name(tf).startswith("k_resident_cg")
    assert ("rows" in bench.loop_name(tf)) == rows
    assert bench.loop_bytes(tf) == per_cell
    r = bench.roofline(tf, 400_000, 1000, 0.011, 6800.0, "measured", 0)
    assert r["bound"].startswith("fp64 issue") and r["bytes_per_cell_iter"] == 108


def test_streamed_loop_on_all_cells():
    tf = dict(LOOP, resident_vectors=0, resident_rows=False)
    assert bench.loop_name(tf).startswith("k_persistent_gear")
    assert bench.loop_bytes(tf) == bench.BYTES_PER_CELL_ITER_FP64_1RED
    assert bench.roofline(tf, 2_000_000, 1000, 0.05, 6800.0, "measured", 0)["bound"] == "hbm"


@pytest.mark.parametrize("cells,where", [(2_093_058, "84 MB, stay in L2"),
                                         (33_538_050, "1342 MB, come from HBM")])
def test_two_cyclic_loop_names_what_bounds_it(cells, where):
    tf = dict(LOOP, two_cyclic=True)
    r = bench.roofline(tf, cells, 1000, 0.1, 6800.0, "measured", 0)
    assert r["bound"].startswith("fp64 issue") and where in r["bound"] and r["bytes_per_cell_iter"] == 36
