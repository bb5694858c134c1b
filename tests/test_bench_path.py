"""The benchmark's record names the kernels of the path that served the call."""
import pytest

import bench
import zef_synth as zs


@pytest.mark.parametrize("grids,launches,kernel,bound", [
    (1, 2, "k_grid_label", "hbm"),                       # one kernel, and the one that clears the statistics
    (1, 4, "k_grid_stream + k_grid_pending", "hbm"),     # a listed call
    (0, 3, "k_label32<256, 2, 2>", "alu"),               # the general kernels, however few
    (0, 17, "k_label32<256, 2, 2>", "alu")])
def test_record_names_the_path(grids, launches, kernel, bound):
    w = zs.config0()
    st = {"cell_grids": grids, "kernel_launches": launches, "pairs_evaluated": 10 ** 9, "pairs_rescued": 0,
          "block_threads": 256, "points_per_thread": 2}
    r = bench.label_roofline(st, w, w.points.shape[0], 1.0, 80.0, 152)
    assert r["kernel"] == kernel and r["bound"] == bound and r["frac"] > 0
