"""What the library's scratch pool holds after a call: at most 64 MB."""

import pytest

from gpu_helpers import torch_mod

pytestmark = pytest.mark.gpu

KEEP = 64 << 20


def test_a_large_gram_gives_its_scratch_back():
    import paper_2105_00578_gb300 as spx
    torch = torch_mod()
    n, ld = 48_000_000, 4                       # its float copy of diag(B) alone is 192 MB
    s = torch.ones((n, ld), device="cuda")
    b = torch.ones(n, device="cuda", dtype=torch.float64)

    def call(rows):
        return spx.sphynx_gram(spx.DT_F32, [s], [s], ld, rows, b)

    call(1000)                                  # modules loaded, pool made
    torch.cuda.synchronize()
    free0, _ = torch.cuda.mem_get_info()
    ga, gb = call(n)
    free1, _ = torch.cuda.mem_get_info()        # no synchronisation after the call
    assert ga[0, 0] == n and gb[0, 0] == n
    assert free0 - free1 <= KEEP, (free0 - free1) >> 20
