"""Which graphs have degree-ordered slices for FP64 products: a last slice of a
few rows, whose offsets always share a pattern, does not decide it."""

import numpy as np
import pytest

import workloads as W
from gpu_helpers import torch_mod

pytestmark = pytest.mark.gpu


def _first_rows(n, path=0, seed=4):
    """The first n vertices of a geometric graph, whose numbers are not sorted by
    place; one left without an edge is joined to the next.  The last `path`
    vertices lose their edges and end a path instead (offsets -1 and 1)."""
    from scipy import sparse
    g = W.rgg(2 * n, seed=seed)
    assert g.n >= n
    a = sparse.csr_matrix((np.ones(g.nnz), g.col, g.row_ptr), shape=(g.n, g.n))[:n, :n].tocsr()
    if path:
        keep = sparse.diags((np.arange(n) < n - path).astype(float))
        ends = np.arange(n - path, n)
        b = sparse.csr_matrix((np.ones(path), (ends, ends - 1)), shape=(n, n))
        a = (keep @ a @ keep + b + b.T).tocsr()
        a.eliminate_zeros()
    alone = np.nonzero(np.diff(a.indptr) == 0)[0]
    b = sparse.csr_matrix((np.ones(len(alone)), (alone, (alone + 1) % n)), shape=(n, n))
    a = (a + b + b.T).tocsr()
    a.sort_indices()
    return a.indptr.astype(np.int64), a.indices.astype(np.int32)


def _products(h, n, torch):
    """FP64 products under the CSR schedule and the tuner's."""
    import paper_2105_00578_gb300 as spx
    for cols in (1, 4, 7, 12):
        ld = 1 if cols == 1 else (cols + 3) & ~3
        x = torch.randn((n, ld), device="cuda", dtype=torch.float64)
        out = []
        for variant in (0, -1):
            spx.sphynx_set_spmm_variant(h, variant)
            y = torch.full_like(x, np.nan)
            spx.sphynx_laplacian_apply(h, "combinatorial", spx.DT_F64, x, ld, y, ld, cols)
            out.append(y[:, :cols])
        assert torch.equal(*out), cols


@pytest.mark.parametrize("last", [1, 2, 3, 32])
def test_a_ragged_last_slice_does_not_turn_them_off(last):
    import paper_2105_00578_gb300 as spx
    torch = torch_mod()
    n = 32 * 1600 + last
    row_ptr, col = _first_rows(n, path=last if last < 32 else 0)
    h = spx.sphynx_create(row_ptr, col)
    try:
        assert spx.sphynx_get_info(h)["sell_pattern_slices"] >= (last < 32)
        assert spx.sphynx_get_plan_info(h)["degree_slices"] == 1
        _products(h, n, torch)
    finally:
        spx.sphynx_destroy(h)


def test_meshes_have_none():
    import paper_2105_00578_gb300 as spx
    g = W.grid2d(400, 300)
    h = spx.sphynx_create(g.row_ptr, g.col)
    try:
        assert spx.sphynx_get_plan_info(h)["degree_slices"] == 0
    finally:
        spx.sphynx_destroy(h)
