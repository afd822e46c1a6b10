"""The kernel that a bench line names is the one that the statistics say ran."""
import pytest

import bench


@pytest.mark.parametrize("precision,n_tiles,kernel", [("fp32", 0, "k_scatter_sf "), ("fp64", 0, "k_scatter_sf64 "),
                                                      ("fp64", 12, "k_scatter_fp64 "), ("fp16x3", 12, "k_scatter_tc ")])
def test_roofline_names_the_kernel(precision, n_tiles, kernel):
    st = {"scatter_flops": 1e12, "ms_scatter": 10.0, "n_chunks": 1, "n_tiles": n_tiles}
    assert bench.roofline_for(precision, st)["kernel"].startswith(kernel)
