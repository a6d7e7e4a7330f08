"""bench.roofline reports DRAM traffic for every layout that the autotuner keeps by itself."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("snap,ckpt", [(0, 64), (1, 4000)])
@pytest.mark.parametrize("layout", [4, 5])
def test_lean_steps_have_their_traffic(layout, snap, ckpt):
    sys.path.insert(0, ROOT)
    import bench
    info = {"padded_cells": 1_000_000, "ckpt_interval": ckpt, "stored_steps": 2784, "stencil": 3, "adj_stencil": 2,
            "tile_x": 32, "tile_z": 16, "adj_tile_x": 32, "adj_tile_z": 16, "layout": layout, "staged_stores": 0,
            "adj_persistent": 0, "adj_layout": layout, "adj_form": 2, "snap_store": snap}
    for r in bench.roofline("batched", info, {"step": (10.0, 100), "adj": (20.0, 100)}, nt=4000, ns=32):
        # less than the algorithmic bytes (CPML cells and the L2's hits between neighbours aside)
        assert 0.8 * r["bytes_per_cell"] * 1e6 < r["traffic"] < r["bytes_per_cell"] * 1e6
        assert r["frac_traffic"] > 0
