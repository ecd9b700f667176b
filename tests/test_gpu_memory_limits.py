"""Calls whose faster plan needs more memory than the one before it still run
where only the smaller one fits."""

import contextlib

import numpy as np
import pytest

import workloads as W
from gpu_helpers import torch_mod

pytestmark = pytest.mark.gpu


@contextlib.contextmanager
def only(torch, free):
    """Leaves `free` bytes of device memory to the library."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    have, _ = torch.cuda.mem_get_info()
    hold = torch.empty(have - free, dtype=torch.uint8, device="cuda") if have > free else None
    try:
        yield
    finally:
        del hold
        torch.cuda.synchronize()
        torch.cuda.empty_cache()


def test_multijagged_without_room_for_its_keys():
    import paper_2105_00578_gb300 as spx
    torch = torch_mod()
    n, K = 24_000_000, 5                        # permutations 192 MB, keys 384 MB more
    gen = torch.Generator(device="cuda").manual_seed(1)
    c = torch.randn((n, 2), generator=gen, device="cuda", dtype=torch.float64)
    ref = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    got = torch.full((n,), -2, dtype=torch.int32, device="cuda")
    spx.sphynx_mj(spx.DT_F64, c, 2, 2, n, None, K, ref)
    with only(torch, 420 << 20):
        spx.sphynx_mj(spx.DT_F64, c, 2, 2, n, None, K, got)
        torch.cuda.synchronize()
    assert torch.equal(ref, got)


def _least_create(torch, g, before):
    """The least free memory (in steps of 8 MB) in which sphynx_create succeeds, and the plan it then has."""
    import paper_2105_00578_gb300 as spx
    for mb in range(64, 4096, 8):
        before()
        with only(torch, mb << 20):
            try:
                h = spx.sphynx_create(g.row_ptr, g.col)
            except spx.SphynxError as e:
                assert e.code == spx.ERR_OOM
                continue
            plan = spx.sphynx_get_plan_info(h)
            spx.sphynx_destroy(h)
            return mb, plan
    raise AssertionError("never fits")


def test_create_goes_without_the_layouts_that_only_add_speed():
    import paper_2105_00578_gb300 as spx
    torch = torch_mod()
    for g, field in ((W.rgg(1_200_000, seed=2), "degree_slices"), (W.grid3d(128, 128, 90, 27), "staged_threads")):
        h = spx.sphynx_create(g.row_ptr, g.col)     # modules loaded
        assert spx.sphynx_get_plan_info(h)[field] > 0
        spx.sphynx_destroy(h)
        mb, plan = _least_create(torch, g, lambda: None)
        assert plan[field] == 0, (mb, plan)
