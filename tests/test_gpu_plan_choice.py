"""The autotuner times what it chooses between: slice strides on the
lane-per-row kernel, which they order, and staged blocks against it."""

import pytest

import workloads as W
from gpu_helpers import torch_mod  # noqa: F401  (skips without a GPU)

pytestmark = pytest.mark.gpu


def test_slice_strides_are_timed_on_the_lane_kernel():
    import paper_2105_00578_gb300 as spx
    g = W.grid3d(128, 128, 96, 27)
    h = spx.sphynx_create(g.row_ptr, g.col)
    try:
        for retune in (False, True):
            if retune:
                spx.sphynx_set_spmm_sell_stride(h, -1)
            info, plan = spx.sphynx_get_info(h), spx.sphynx_get_plan_info(h)
            assert info["spmm_variant"] == 2 and plan["staged_used"] == 1 and plan["staged_threads"] == 128
            assert plan["lane_variant"] in (1, 2)
            # the float product here: about 55 us staged, 90 us a lane per row
            assert min(plan["tuned_us_stride"]) > 1.2 * plan["tuned_us_staged"] > 0, plan
            assert plan["tuned_us_stride"].index(min(plan["tuned_us_stride"])) == [1, 2, 4, 8, 16].index(
                info["sell_stride"])
            assert info["tuned_us_pattern"] == plan["tuned_us_staged"]
    finally:
        spx.sphynx_destroy(h)


def test_graphs_without_blocks_have_one_choice():
    import paper_2105_00578_gb300 as spx
    g = W.rgg(3000, seed=1)
    h = spx.sphynx_create(g.row_ptr, g.col)
    try:
        info, plan = spx.sphynx_get_info(h), spx.sphynx_get_plan_info(h)
        assert plan["staged_threads"] == 0 and plan["staged_used"] == 0 and plan["tuned_us_staged"] == 0
        assert plan["lane_variant"] == info["spmm_variant"]
    finally:
        spx.sphynx_destroy(h)
