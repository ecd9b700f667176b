"""The staged-block product (shared-pattern schedule of unweighted graphs with
wide rows) against the explicit SELL-32 schedule: both add a row's entries in
ascending column order, so every result is the same bit for bit."""

import numpy as np
import pytest

import workloads as W
from gpu_helpers import torch_mod

pytestmark = pytest.mark.gpu


def _pair(run):
    """run(variant) under the explicit and the shared-pattern schedule."""
    return run(1), run(2)


# n around multiples of a block's 192 or 384 rows, an odd n (a last 8-byte row
# of bfloat16), lines shorter and longer than a block
@pytest.mark.parametrize("dims", [(8, 8, 6), (8, 8, 3), (7, 11, 5), (5, 7, 11), (97, 3, 3), (17, 13, 11),
                                  (400, 4, 3), (61, 53, 41)])
@pytest.mark.parametrize("cols", [2, 7, 10, 14])
def test_staged_block_products_equal_explicit_slices(dims, cols):
    import paper_2105_00578_gb300 as spx
    torch = torch_mod()
    g = W.grid3d(*dims, 27)
    ld = (cols + 3) & ~3
    gen = torch.Generator(device="cuda").manual_seed(cols)
    h = spx.sphynx_create(g.row_ptr, g.col)
    try:
        assert spx.sphynx_get_info(h)["sell_pattern_slices"] > 0
        x32 = torch.randn((g.n, ld), generator=gen, device="cuda")
        for code, x in ((spx.DT_F32, x32), (spx.DT_BF16, x32.bfloat16())):
            def product(variant):
                spx.sphynx_set_spmm_variant(h, variant)
                y = torch.full((g.n, ld), np.nan, device="cuda")
                spx.sphynx_laplacian_apply(h, "combinatorial", code, x, ld, y, ld, cols)
                return y
            a, b = _pair(product)
            assert torch.equal(a, b)
        for code_in, code_out in ((spx.DT_F32, spx.DT_F32), (spx.DT_F32, spx.DT_BF16), (spx.DT_BF16, spx.DT_BF16)):
            t = x32.bfloat16() if code_in == spx.DT_BF16 else x32
            for yterms, first in ((2, 1), (2, 0), (1, 0), (0, 0)):
                def step(variant):
                    spx.sphynx_set_spmm_variant(h, variant)
                    out = torch.zeros((g.n, ld), device="cuda",
                                      dtype=torch.bfloat16 if code_out == spx.DT_BF16 else torch.float32)
                    y = x32.clone()
                    spx.sphynx_poly_step(h, "combinatorial", code_in, t, code_out, out, y, ld, cols, 30.0, 7.0,
                                         yterms, first)
                    return torch.cat([out.float(), y])
                a, b = _pair(step)
                assert torch.equal(a, b), (code_in, code_out, yterms, first)
    finally:
        spx.sphynx_destroy(h)


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 3e38])
def test_staged_blocks_keep_non_finite_values_to_their_neighbours(value):
    import paper_2105_00578_gb300 as spx
    torch = torch_mod()
    g = W.grid3d(12, 11, 10, 27)
    h = spx.sphynx_create(g.row_ptr, g.col)
    try:
        for code, dt in ((spx.DT_F32, torch.float32), (spx.DT_BF16, torch.bfloat16)):
            x = torch.randn((g.n, 8), device="cuda").to(dt)
            for row in (0, 11, 12, g.n // 2, g.n - 1):   # line ends: the next row in memory is not a neighbour
                x[row, row % 8] = value

            def product(variant):
                spx.sphynx_set_spmm_variant(h, variant)
                y = torch.zeros((g.n, 8), device="cuda")
                spx.sphynx_laplacian_apply(h, "combinatorial", code, x, 8, y, 8, 8)
                return y.cpu().numpy()
            a, b = _pair(product)
            np.testing.assert_array_equal(a, b)   # NaNs compare equal in place
    finally:
        spx.sphynx_destroy(h)
