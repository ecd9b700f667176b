"""FP64 products use degree-ordered slices where they pay: from nine slices an SM
on, and not for what gains nothing by them.  Every product equals the CSR
schedule's bit for bit."""

import pytest

import workloads as W
from gpu_helpers import torch_mod
from test_gpu_degree_slices_choice import _first_rows

pytestmark = pytest.mark.gpu

LEAST = 9 * 32 * 152


def _create(n, weighted):
    import paper_2105_00578_gb300 as spx
    row_ptr, col = _first_rows(n)
    g = W.CSRGraph(n=n, row_ptr=row_ptr, col=col, name="first rows")
    if weighted:
        g = W.random_edge_weights(g)
    return g, spx.sphynx_create(g.row_ptr, g.col, g.w)


@pytest.mark.parametrize("n", [2000, LEAST - 1, LEAST])
def test_size_of_the_graphs_that_have_them(n):
    import paper_2105_00578_gb300 as spx
    g, h = _create(n, False)
    try:
        assert spx.sphynx_get_plan_info(h)["degree_slices"] == int(n >= LEAST)
    finally:
        spx.sphynx_destroy(h)


# whole and ragged slices and 1024-row windows; 63232 rows are 13 slices an SM
@pytest.mark.parametrize("n", [LEAST, 44 * 1024, 44 * 1024 + 1, 50_017, 63_231, 63_232, 70_001])
@pytest.mark.parametrize("weighted", [False, True])
def test_products_equal_csr_and_take_them_where_they_pay(n, weighted):
    import paper_2105_00578_gb300 as spx
    torch = torch_mod()
    g, h = _create(n, weighted)
    try:
        for cols in (1, 4, 7, 12):
            ld = 1 if cols == 1 else (cols + 3) & ~3
            x = torch.randn((n, ld), device="cuda", dtype=torch.float64)
            for lap in ("combinatorial", "normalized"):
                pays = lap == "combinatorial" or weighted or (cols > 1 and n >= 63_232)
                out = []
                for variant in (0, 1, -1):
                    spx.sphynx_set_spmm_variant(h, variant)
                    y, t, acc = torch.zeros_like(x), torch.zeros_like(x), x.clone()
                    spx.sphynx_laplacian_apply(h, lap, spx.DT_F64, x, ld, y, ld, cols)
                    assert spx.sphynx_get_plan_info(h)["degree_last"] == {0: 0, 1: 1, -1: int(pays)}[variant]
                    if cols > 1:
                        spx.sphynx_poly_step(h, lap, spx.DT_F64, x, spx.DT_F64, t, acc, ld, cols, 3.0, 5.0, 2, 0)
                    out.append((y, t, acc))
                for other in out[1:]:
                    for a, b in zip(out[0], other):
                        assert torch.equal(a, b), (cols, lap)
    finally:
        spx.sphynx_destroy(h)
