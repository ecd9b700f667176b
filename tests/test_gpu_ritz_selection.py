"""Rayleigh-Ritz returns the nev smallest values when the nev-th and the next one
are closer than float arithmetic can tell and their vectors do not couple
(diagonal pencils, decoupled blocks): checked against the values that the
pencils are built from."""

import numpy as np
import pytest

from gpu_helpers import torch_mod  # noqa: F401  (skips without a GPU)

pytestmark = pytest.mark.gpu


def _gram_pair(lam, cond, rng):
    """G_A, G_B of a basis of condition `cond` whose pencil has the values lam."""
    m = len(lam)
    if cond == 1.0:
        return np.diag(lam), np.eye(m)
    q, _ = np.linalg.qr(rng.standard_normal((m, m)))
    x = q * np.geomspace(1.0, cond, m) @ np.linalg.qr(rng.standard_normal((m, m)))[0]
    ga, gb = x.T @ (lam[:, None] * x), x.T @ x
    return 0.5 * (ga + ga.T), 0.5 * (gb + gb.T)


def _blocks(parts, rng):
    """Block-diagonal pencil of the given (values, condition) parts, its columns shuffled."""
    m = sum(len(lam) for lam, _ in parts)
    ga, gb, at = np.zeros((m, m)), np.zeros((m, m)), 0
    for lam, cond in parts:
        k = len(lam)
        ga[at:at + k, at:at + k], gb[at:at + k, at:at + k] = _gram_pair(lam, cond, rng)
        at += k
    p = rng.permutation(m)
    return np.ascontiguousarray(ga[np.ix_(p, p)]), np.ascontiguousarray(gb[np.ix_(p, p)])


def _check(ga, gb, nev, lam, cond):
    import paper_2105_00578_gb300 as spx
    m = len(lam)
    th, y, svqb = spx.sphynx_rayleigh_ritz(ga, gb, np.ones(m), nev, 2.0 ** -53)
    assert not svqb
    # FP64 backward error of the scaled pencil times the basis' condition
    tol = 50 * m * 2.0 ** -53 * cond ** 2
    top = np.max(np.abs(lam))
    assert np.max(np.abs(th - np.sort(lam)[:nev])) <= tol * top
    assert np.max(np.abs(y.T @ gb @ y - np.eye(nev))) <= tol
    assert np.max(np.abs(ga @ y - gb @ y * th)) <= tol * top * np.linalg.norm(gb, 2) * np.max(np.abs(y))


GAPS = [1e-6, 1e-7, 1e-8, 1e-10, 1e-12, 0.0]


@pytest.mark.parametrize("gap", GAPS)
@pytest.mark.parametrize("wanted", [1.0, 1e-2, 1e-4])
def test_diagonal_pencils(gap, wanted):
    rng = np.random.default_rng(11)
    for _ in range(20):
        low = np.sort(rng.uniform(0.1, 1.0, 3)) * wanted
        lam = np.concatenate([low, [low[2] + gap * wanted], wanted * rng.uniform(1.5, 2.0, 2), [2.0, 3.0]])
        lam = lam[rng.permutation(len(lam))]
        _check(*_blocks([(lam, 1.0)], rng), 3, lam, 1.0)


@pytest.mark.parametrize("gap", GAPS)
@pytest.mark.parametrize("wanted", [1.0, 1e-2, 1e-4])
@pytest.mark.parametrize("m1,m2,nev", [(5, 5, 3), (9, 12, 7), (16, 16, 8)])
def test_decoupled_blocks(gap, wanted, m1, m2, nev):
    rng = np.random.default_rng(m1 + m2)
    for _ in range(10):
        low = wanted * (0.2 + 0.8 * np.sort(rng.permutation(nev) + rng.uniform(0.2, 0.8, nev)) / nev)
        rest = np.concatenate([[low[-1] + gap * wanted], np.linspace(1.5, 3.0, m1 + m2 - nev - 1)])
        # the nev-th value and the next one in different blocks, the others spread over both
        one, two = [low[-1]], [rest[0]]
        for v in rng.permutation(np.concatenate([low[:-1], rest[1:]])):
            (one if len(one) < m1 and (len(two) == m2 or rng.random() < 0.5) else two).append(v)
        lam = np.concatenate([one, two])
        _check(*_blocks([(np.array(one), 2.0), (np.array(two), 2.0)], rng), nev, lam, 2.0)
