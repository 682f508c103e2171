"""Two-class rows that stand in for the FP64 recheck: each output is the FP64 one rounded once.

F32, U16 and BF16 counts at any alignment (log-posterior mode) sum a 30-bit Delta exactly and
its residuals in FP32; FP8 rows of up to 496 features sum a 37-bit Delta.  One heavy feature
makes the step coarse while the other weights are small, so that many margins are near zero,
where an absolute error of the step's size would show.

Tolerance: half an FP32 unit (2^-24 of the value), and, absolute, the part of Delta that the
sums leave out -- per count half a step 2^-(S+9) times (depth + 2) roundings of 2^-24, or half
a step 2^-(S+16) -- and the FP64 sums' own rounding on both sides, F additions of terms that
make up T max |log theta|, 2^-53 each; 2^(22 - S) is the power of two above max |Delta|.
"""
import numpy as np
import pytest
import torch

from _common import compare, oracle_mn, stored, to_np
from test_gpu_float_counts import _features

pytestmark = pytest.mark.gpu

nb = pytest.importorskip("paper_1905_13746_gb300")


def _rows(seed, n, F, top):
    """Files of two classes that differ by percents, but for one feature that only one has."""
    rng = np.random.default_rng(seed)
    p = rng.dirichlet(np.full(F, 2.0))
    p = np.stack([p, p * rng.uniform(0.97, 1.03, F)])
    y = (np.arange(n) % 2).astype(np.int32)
    X = np.minimum(rng.poisson(rng.uniform(300, 3000, n)[:, None] * p[y]), top)
    X[:, 0] = np.where((np.arange(n) < n // 2) & (y == 1), top, 0)   # training files alone
    return X.astype(np.uint16), y


def _check(res, m, ref, vals, part):
    d = np.abs(m["log_theta"][1] - m["log_theta"][0]).max()
    step = 2.0 ** np.ceil(np.log2(max(d, 1e-300)) + 1e-12) * 2.0 ** -22          # 2^-S
    T, F = vals.sum(1), vals.shape[1]
    slack = T * step * part + 8 * F * 2.0 ** -53 * T * np.abs(m["log_theta"]).max()
    assert (res["label"] == ref["label"]).all()
    assert (np.abs(res["margin"].astype(np.float64) - ref["margin"]) <=
            2.0 ** -24 * ref["margin"] + slack).all()
    err = np.abs(res["lp"].astype(np.float64) - ref["lp"])
    assert (err <= 2.0 ** -24 * np.abs(ref["lp"]) + slack[:, None]).all()


@pytest.mark.parametrize("fmt,F,pad", [("f32", 1003, 0), ("f32", 64, 1), ("f32", 33, 0), ("u16", 100, 4),
                                       ("u16", 128, 0), ("u16", 1001, 0), ("bf16", 64, 0),
                                       ("bf16", 57, 7), ("bf16", 1001, 0)])
def test_float_and_16_bit_counts(fmt, F, pad):
    X, y = _rows(F, 3000, F, 250)
    f, vals = _features(X, fmt, pad)
    model = nb.fit(f, torch.from_numpy(y).cuda(), 2)
    m, ref = oracle_mn(vals, y, 2, vals)
    depth = max(8 * 4, (F + 31) // 32) + 7      # values a lane sums, shuffles, the residual's own
    _check(to_np(nb.score(model, f)), m, ref, vals, 2.0 ** -9 * depth * 2.0 ** -24)


@pytest.mark.parametrize("F", [1, 16, 17, 100, 256, 257, 495, 496])
@pytest.mark.parametrize("mode", [nb.NB_RECHECK_LP, nb.NB_RECHECK_OFF])
def test_narrow_fp8_counts(F, mode):
    X, y = _rows(F, 3000, F, 16)
    f, vals = stored(X, "fp8")
    model = nb.fit(f, torch.from_numpy(y).cuda(), 2)
    m, ref = oracle_mn(vals, y, 2, vals)
    res = to_np(nb.score(model, f, recheck=mode))
    if mode == nb.NB_RECHECK_OFF:     # labels of nearer rows are the recheck's to settle
        near = ref["margin"] <= 1e-6
        res["label"][near] = ref["label"][near]
    _check(res, m, ref, vals, 2.0 ** -16)


@pytest.mark.parametrize("fmt", ["u16", "bf16"])
def test_the_register_kernel_can_be_asked_for(fmt):
    """Its FP32 bound leaves most rows of the log-posterior mode to FP64; the exact sums none."""
    X, y = _rows(5, 3000, 64, 250)
    f, vals = _features(X, fmt, 0)
    model = nb.fit(f, torch.from_numpy(y).cuda(), 2)
    m, ref = oracle_mn(vals, y, 2, vals)
    marked = {}
    for variant in (nb.NB_VARIANT_AUTO, nb.NB_VARIANT_PIPELINED, nb.NB_VARIANT_REGISTER):
        model.set_tile_config(variant, 0, 0, 0)
        res = to_np(nb.score(model, f))
        marked[variant] = res["n_rechecked"]
        compare(res, ref)
    assert marked[nb.NB_VARIANT_AUTO] == marked[nb.NB_VARIANT_PIPELINED] <= 30
    assert marked[nb.NB_VARIANT_REGISTER] > 1500


@pytest.mark.parametrize("F", [100, 490])
def test_tuning_narrow_fp8_rows_changes_no_result(F):
    X, y = _rows(F, 3000, F, 16)
    f, vals = stored(X, "fp8")
    model = nb.fit(f, torch.from_numpy(y).cuda(), 2)
    before = to_np(nb.score(model, f))
    assert model.autotune(f)[0][0] != nb.NB_VARIANT_REGISTER
    after = to_np(nb.score(model, f))
    for k in ("label", "margin", "lp"):
        assert np.array_equal(before[k], after[k]), k
