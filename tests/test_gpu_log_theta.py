"""log theta of a many-class fit: the device logarithm is correctly rounded but for a share.

With alpha = 1 a feature that a class never has gives log 1 - log(N_c + F), which is the
class's logarithm of the total itself, so every other entry is known: the rounded logarithm
of its count less that number, rounded.  The logarithm is within 0.5 + 2^-8 units in the
last place for counts of four and more (its own error stays below 2^-60, a unit there is
2^-52 at least), so at most 2^-7 of them round the other way.
"""
import numpy as np
import pytest
import torch

from _common import stored

pytestmark = pytest.mark.gpu

nb = pytest.importorskip("paper_1905_13746_gb300")


@pytest.mark.parametrize("C,F,top", [(3, 4001, 60), (5, 3000, 60_000), (64, 1024, 255)])
def test_log_theta_is_the_rounded_logarithm(C, F, top):
    rng = np.random.default_rng(C)
    n = 40 * C
    X = np.maximum(4, np.exp(rng.uniform(1.4, np.log(top), (n, F)))).astype(np.uint16)
    X[:, 0] = 0
    y = (np.arange(n) % C).astype(np.int32)
    f, vals = stored(X, "u16")
    lt, _, _ = nb.fit(f, torch.from_numpy(y).cuda(), C).params()
    counts = np.stack([vals[y == c].sum(0) for c in range(C)])
    assert (counts[:, 0] == 0).all()
    # (long double: 64 bits of mantissa or more)
    exact = np.log(counts.astype(np.longdouble) + 1).astype(np.float64) + lt[:, :1]
    off = lt != exact
    assert off.mean() <= 2.0 ** -7, off.mean()
    # and what rounds the other way is one unit of the logarithm away
    assert (np.abs(lt - exact) <= np.spacing(np.maximum(np.abs(exact), np.log(counts + 1)))).all()
