"""Rayleigh-Ritz vectors of close and of equal values are B-orthonormal to FP64
rounding, whatever the distance of the values."""

import numpy as np
import pytest

from gpu_helpers import torch_mod  # noqa: F401  (skips without a GPU)
from test_gpu_ritz_selection import _blocks, _check

pytestmark = pytest.mark.gpu

GAPS = [0.0, 1e-14, 1e-12, 1e-10, 1e-9, 1e-8, 1e-7, 1e-6, 1e-5, 1e-4, 1e-3]


@pytest.mark.parametrize("gap", GAPS)
@pytest.mark.parametrize("m,nev", [(8, 4), (12, 4), (21, 7)])
def test_close_wanted_values(m, nev, gap):
    rng = np.random.default_rng(m)
    for _ in range(10):
        lam = np.concatenate([np.linspace(0.1, 0.5, nev - 1), [0.5 + gap], np.linspace(0.9, 2.5, m - nev)])
        _check(*_blocks([(lam[rng.permutation(m)], 2.0)], rng), nev, lam, 2.0)


@pytest.mark.parametrize("gap", GAPS)
@pytest.mark.parametrize("m,nev", [(8, 3), (12, 4), (21, 7)])
def test_close_values_across_the_boundary(m, nev, gap):
    rng = np.random.default_rng(m)
    for _ in range(10):
        lam = np.concatenate([np.linspace(0.1, 0.5, nev), [0.5 + gap], np.linspace(0.9, 2.5, m - nev - 1)])
        _check(*_blocks([(lam[rng.permutation(m)], 2.0)], rng), nev, lam, 2.0)
