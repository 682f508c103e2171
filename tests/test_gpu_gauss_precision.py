"""The Gaussian fit's class moments are as exact as FP64 sums.

A run's sum is rounded to FP64 once; sums of runs are added in FP64: at most three pieces
of a class per chunk, ceil(chunks / 8) chunks per warp, eight warps.  Every addition and
the final divisions and subtraction round by at most 2^-53 of the sum of magnitudes, so
a moment is within (additions + 4) 2^-53 of it (mean: of mean |x|; variance: of itself and
of the square by which K, the FP32 mean, may miss the mean, at most 2^-48 of the mean's).
The reference is summed in NumPy's long double (64 bits of mantissa or more).
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

nb = pytest.importorskip("paper_1905_13746_gb300")


@pytest.mark.parametrize("n,F,C,offset", [(700, 40, 2, 0.0), (4096, 400, 2, 10.0), (9000, 33, 5, 3.0),
                                          (70_000, 40, 3, 100.0), (20_000, 64, 64, 5.0)])
def test_moments_round_like_fp64_sums(n, F, C, offset):
    rng = np.random.default_rng(n + F)
    y = (np.arange(n) % C).astype(np.int32)
    rng.shuffle(y)
    X = (rng.normal(size=(n, F)) * rng.uniform(0.5, 3, F) + offset * rng.uniform(0, 1, F)).astype(np.float32)
    mu, var, _ = nb.fit(torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda(), C,
                        kind=nb.NB_GAUSSIAN, var_smoothing=0.0).params()
    rows = 64 if n <= 65536 else 512          # the fewest rows of a chunk: the most chunks
    adds = 3 + -(-n // rows) // 8 + 1 + 8
    u = (adds + 4) * 2.0 ** -53
    for c in range(C):
        r = X[y == c].astype(np.longdouble)
        m = r.mean(axis=0)
        v = np.square(r - m).mean(axis=0)
        assert (np.abs(mu[c] - m) <= u * np.abs(r).mean(axis=0)).all(), c
        assert (np.abs(var[c] - v) <= u * (v + 2.0 ** -48 * m * m)).all(), \
            (c, float(np.max(np.abs(var[c] - v) / v)), u)


def _huge(n, F, C, seed):
    """Finite values whose FP32 class sums overflow in every run of rows, and their labels."""
    rng = np.random.default_rng(seed)
    y = (np.arange(n) % C).astype(np.int32)
    X = (rng.uniform(1.0, 1.9, size=(n, F)) * 2.0 ** 127).astype(np.float32)
    X[:, 1::2] *= -1
    X[::3, 0] *= np.float32(2.0 ** -20)
    return X, y


@pytest.mark.parametrize("n,F,C", [(65, 3, 2), (5000, 33, 3), (70_000, 5, 2)])
def test_overflowing_sums_of_several_chunks(n, F, C):
    """The same moments as those of the values scaled by 2^-64, where nothing overflows."""
    X, y = _huge(n, F, C, n)
    yd = torch.from_numpy(y).cuda()
    mu, var, _ = nb.fit(torch.from_numpy(X).cuda(), yd, C, kind=nb.NB_GAUSSIAN, var_smoothing=0.0).params()
    small = torch.from_numpy(np.ldexp(X, -64)).cuda()
    m2, v2, _ = nb.fit(small, yd, C, kind=nb.NB_GAUSSIAN, var_smoothing=0.0).params()
    # FP64 sums of runs in place of exact ones: 2^-53 for each of a run's rows at most
    u = 2048 * 2.0 ** -53
    assert (np.abs(np.ldexp(mu, -64) - m2) <= u * np.abs(m2).max()).all()
    assert (np.abs(np.ldexp(var, -128) - v2) <= 8 * u * (v2 + np.square(m2))).all()


def test_overflowing_sums_cost_a_run_not_the_matrix():
    """Each run of rows is summed again by itself: no lane walks all rows (which took over a
    thousand times as long)."""
    X, y = _huge(400_000, 32, 2, 1)
    yd = torch.from_numpy(y).cuda()
    times = []
    for x in (np.ldexp(X, -64), X):
        xd = torch.from_numpy(x).cuda()
        m = nb.fit(xd, yd, 2, kind=nb.NB_GAUSSIAN, no_sync=True)
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        best = 1e30
        for _ in range(3):
            a.record()
            nb.refit(m, xd, yd, no_sync=True)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        times.append(best)
    assert times[1] <= 20 * times[0], times


def test_more_features_than_a_grid_dimension_holds_tiles():
    """2.1M features are 65,626 tiles of 32."""
    F, n = 2_100_003, 6
    rng = np.random.default_rng(3)
    X = rng.normal(size=(n, F)).astype(np.float32)
    y = np.array([0, 1, 0, 1, 1, 0], np.int32)
    mu, var, _ = nb.fit(torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda(), 2,
                        kind=nb.NB_GAUSSIAN, var_smoothing=0.0).params()
    for c in range(2):
        r = X[y == c].astype(np.longdouble)
        m = r.mean(axis=0)
        v = np.square(r - m).mean(axis=0)
        u = 16 * 2.0 ** -53              # at most three pieces of one chunk
        assert (np.abs(mu[c] - m) <= u * np.abs(r).mean(axis=0)).all()
        assert (np.abs(var[c] - v) <= u * (v + 2.0 ** -48 * m * m)).all()
