"""Multi-jagged at the sizes where its passes change form: 11-bit digits up to
2048 parts and 8-bit digits above, and tiles of 4096 points in the scatter.
Integers: bit for bit the oracle's."""

import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_helpers import torch_mod

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,K", [(20011, 2047), (20011, 2048), (20011, 2049), (4097, 4099), (4095, 3), (4096, 3),
                                 (4097, 3), (8193, 2048)])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("weighted", [False, True])
def test_mj_digit_widths_and_tiles(n, K, dtype, weighted):
    import paper_2105_00578_gb300 as spx
    torch = torch_mod()
    dims = max(1, K.bit_length() - 1)
    c = W.random_coords(n, dims, seed=n + K, dtype=np.float64 if dtype == "f64" else np.float32, ties=weighted)
    vw = W.random_vertex_weights(n, 1, 9, seed=K) if weighted else None
    part = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    spx.sphynx_mj(spx.DT_F64 if dtype == "f64" else spx.DT_F32, torch.from_numpy(c).cuda(), dims, dims, n,
                  None if vw is None else torch.from_numpy(vw).cuda(), K, part)
    torch.cuda.synchronize()
    assert np.array_equal(part.cpu().numpy(), O.multijagged(c, vw, K))
