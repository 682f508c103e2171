"""The Gaussian fit's paired-FP32 sums against FP64 at the edges of its chunks,
feature tiles and value ranges.

A chunk holds 64 to 2,048 rows (512 at least above 65,536 rows), a tile 32
features, the finish kernel's tile 256.  Tolerances: a pair keeps 48 bits; its
low part, at most n 2^-24 of the sum, rounds by 2^-24 of itself at each of n
additions, so a class mean is within n^2 2^-48 of its largest value in the
worst case and within n 2^-47 by far in any case here (n <= 2,048 / 8 rows per
run and up to 64 runs joined); 1e-11 covers that, and the squares likewise.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

nb = pytest.importorskip("paper_1905_13746_gb300")

TOL = 1e-11


def _check(X, y, C, vs=1e-9):
    m = nb.fit(torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda(), C, kind=nb.NB_GAUSSIAN,
               var_smoothing=vs)
    mu, var, log_pi = m.params()
    X64 = X.astype(np.float64)
    eps = vs * X64.var(axis=0).max()
    for c in range(C):
        r = X64[y == c]
        big = np.abs(r).max(axis=0)
        mean = r.mean(axis=0)
        assert (np.abs(mu[c] - mean) <= TOL * big).all(), c
        v = np.square(r - mean).mean(axis=0) + eps
        # the mean's own error enters squared; differences are exact
        assert (np.abs(var[c] - v) <= TOL * v + (TOL * big) ** 2).all(), c
        assert log_pi[c] == pytest.approx(np.log(len(r)) - np.log(len(y)), abs=1e-14)
    return m


def _labels(rng, n, C, skew):
    p = np.ones(C) if not skew else 1.0 / (1.0 + np.arange(C)) ** 2
    y = rng.choice(C, size=n, p=p / p.sum()).astype(np.int32)
    y[:2 * C] = np.arange(2 * C) % C
    return y


@pytest.mark.parametrize("n,F,C,skew", [
    (4, 1, 2, False), (63, 31, 2, True), (64, 32, 3, False), (65, 33, 2, False),
    (512, 257, 64, False), (513, 16, 64, True), (2049, 64, 33, True), (4097, 5, 32, False),
    (65_537, 7, 5, True), (70_000, 129, 2, True)])
def test_moments_at_tile_edges(n, F, C, skew):
    rng = np.random.default_rng(n + 7 * F + C)
    y = _labels(rng, n, C, skew)
    X = (rng.normal(size=(n, F)) * rng.uniform(0.5, 3, F) +
         rng.uniform(0, 10, (C, F))[y]).astype(np.float32)
    _check(X, y, C)


@pytest.mark.parametrize("scale", [1e-36, 1e-20, 1e15, 1e30])
def test_moments_over_the_float_range(scale):
    rng = np.random.default_rng(5)
    y = _labels(rng, 700, 3, False)
    X = (rng.normal(size=(700, 40)) * scale).astype(np.float32)
    X[:, 1] += np.float32(1e4 * scale)    # far from zero: exact differences
    _check(X, y, 3)


def test_sums_beyond_float_range():
    """FP32 sums above 3.4e38 take the FP64 row loop."""
    rng = np.random.default_rng(6)
    y = _labels(rng, 200, 2, False)
    X = rng.uniform(1e38, 3e38, size=(200, 3)).astype(np.float32)
    _check(X, y, 2)


def test_constant_features_have_zero_variance_and_order_does_not_matter_to_a_repeat():
    rng = np.random.default_rng(8)
    n, F = 3000, 35
    y = _labels(rng, n, 4, True)
    X = rng.normal(size=(n, F)).astype(np.float32)
    X[:, 3] = np.float32(0.1)
    X[:, 4] = 0.0
    m = _check(X, y, 4, vs=0.01)
    again = nb.fit(torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda(), 4,
                   kind=nb.NB_GAUSSIAN, var_smoothing=0.01)
    eps = 0.01 * X.astype(np.float64).var(axis=0).max()
    mu, var, _ = m.params()
    assert np.abs(var[:, 3:5] - eps).max() <= 1e-12 * eps
    assert np.array_equal(mu, again.params()[0]) and np.array_equal(var, again.params()[1])


def test_refit_keeps_results_while_its_workspace_grows():
    rng = np.random.default_rng(9)
    y = _labels(rng, 500, 2, False)
    X = rng.normal(size=(500, 20)).astype(np.float32)
    m = nb.fit(torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda(), 2, kind=nb.NB_GAUSSIAN)
    for n in (5000, 300, 40_000):
        y2 = _labels(rng, n, 2, False)
        X2 = torch.from_numpy(rng.normal(size=(n, 20)).astype(np.float32)).cuda()
        y2 = torch.from_numpy(y2).cuda()
        nb.refit(m, X2, y2)
        fresh = nb.fit(X2, y2, 2, kind=nb.NB_GAUSSIAN)
        for a, b in zip(m.params(), fresh.params()):
            assert np.array_equal(a, b)
