"""Double products in degree-ordered slices (graphs of short rows of uneven
length) against the CSR schedule, which adds each row's entries in the same
order: the results are the same bit for bit."""

import numpy as np
import pytest

import workloads as W
from gpu_helpers import torch_mod

pytestmark = pytest.mark.gpu


# below and above one 1024-row window, ragged last slices and windows
@pytest.mark.parametrize("n", [60, 1000, 1024, 1031, 5000, 20011])
@pytest.mark.parametrize("weighted", [False, True])
def test_double_products_equal_csr(n, weighted):
    import paper_2105_00578_gb300 as spx
    torch = torch_mod()
    g = W.rgg(n, seed=n)
    if weighted:
        g = W.random_edge_weights(g)
    h = spx.sphynx_create(g.row_ptr, g.col, g.w)
    gen = torch.Generator(device="cuda").manual_seed(n)
    try:
        for cols in (1, 4, 7, 12):
            ld = 1 if cols == 1 else (cols + 3) & ~3
            x = torch.randn((g.n, ld), generator=gen, device="cuda", dtype=torch.float64)
            for lap in ("combinatorial", "normalized"):
                out = []
                for variant in (0, 1):
                    spx.sphynx_set_spmm_variant(h, variant)
                    y = torch.full_like(x, np.nan)
                    spx.sphynx_laplacian_apply(h, lap, spx.DT_F64, x, ld, y, ld, cols)
                    out.append(y)
                    if cols > 1:
                        t, acc = torch.zeros_like(x), x.clone()
                        spx.sphynx_poly_step(h, lap, spx.DT_F64, x, spx.DT_F64, t, acc, ld, cols, 3.0, 5.0, 2, 0)
                        out += [t, acc]
                half = len(out) // 2
                for a, b in zip(out[:half], out[half:]):
                    assert torch.equal(a, b), (cols, lap)
    finally:
        spx.sphynx_destroy(h)
