"""The refined Rayleigh-Ritz path (float eigendecomposition, FP64 refinement of
the wanted columns) against numpy's FP64 generalized eigensolve."""

import numpy as np
import pytest

from gpu_helpers import torch_mod  # noqa: F401  (skips without a GPU)

pytestmark = pytest.mark.gpu


def _pencil(m, lam, seed, cond=10.0, scale=1.0):
    """G_A, G_B with generalized eigenvalues lam and G_B of condition about cond^2, columns of unequal length."""
    rng = np.random.default_rng(seed)
    q, _ = np.linalg.qr(rng.standard_normal((m, m)))
    x = q * np.geomspace(1.0, cond, m) @ np.linalg.qr(rng.standard_normal((m, m)))[0]
    d = 10.0 ** rng.uniform(-2, 2, m)
    ga = d[:, None] * (x.T @ (lam[:, None] * x)) * d * scale
    gb = d[:, None] * (x.T @ x) * d
    return 0.5 * (ga + ga.T), 0.5 * (gb + gb.T)


def _check(ga, gb, nev, lam, scale=1.0, cond=10.0):
    import paper_2105_00578_gb300 as spx
    m = ga.shape[0]
    th, y, svqb = spx.sphynx_rayleigh_ritz(ga, gb, np.ones(m), nev, 2.0 ** -53)
    assert not svqb
    # FP64 backward error of the scaled pencil, times the basis' condition: 50 m u cond^2
    top = np.max(np.abs(lam)) * scale
    tol = 50 * m * 2.0 ** -53 * cond ** 2
    assert np.all(np.abs(th - np.sort(lam)[:nev] * scale) <= tol * top)
    assert np.all(np.diff(th) >= -tol * top)
    d = np.sqrt(np.diag(gb))
    ys = d[:, None] * y                                   # scaled coordinates
    bs, as_ = gb / np.outer(d, d), ga / np.outer(d, d)
    assert np.max(np.abs(ys.T @ bs @ ys - np.eye(nev))) <= tol
    res = as_ @ ys - bs @ ys * th
    assert np.max(np.abs(res)) <= tol * np.linalg.norm(as_, 2)


@pytest.mark.parametrize("m,nev", [(2, 1), (2, 2), (5, 2), (12, 4), (13, 4), (21, 7), (24, 8), (31, 10), (32, 11),
                                   (32, 16), (33, 11)])
def test_separated_values(m, nev):
    lam = np.linspace(0.0, 2.0, m) ** 2 + 1e-3 * np.arange(m)
    _check(*_pencil(m, lam, m), nev, lam)


@pytest.mark.parametrize("gap", [0.0, 1e-12, 1e-8, 1e-5])
def test_multiple_wanted_values(gap):
    lam = np.concatenate([[0.0, 1e-3], 0.5 + gap * np.arange(3), np.linspace(1, 3, 16)])
    _check(*_pencil(21, lam, 5), 7, lam)


@pytest.mark.parametrize("gap", [0.0, 1e-10, 1e-7])
def test_wanted_value_meeting_an_unwanted_one(gap):
    lam = np.concatenate([np.linspace(0.0, 0.5, 6), 0.7 + gap * np.arange(3), np.linspace(1, 3, 12)])
    _check(*_pencil(21, lam, 6), 7, lam)


@pytest.mark.parametrize("scale", [1e-200, 1e-30, 1e30, 1e200])
def test_scales_beyond_float(scale):
    lam = np.linspace(0.1, 2.0, 12)
    _check(*_pencil(12, lam, 7, scale=scale), 4, lam, scale=scale)


def test_indefinite_and_ill_conditioned():
    lam = np.linspace(-1.0, 2.0, 15)
    _check(*_pencil(15, lam, 8), 5, lam)
    lam = np.linspace(0.0, 2.0, 15)
    _check(*_pencil(15, lam, 9, cond=1e4), 5, lam, cond=1e4)   # no float start: the general path
