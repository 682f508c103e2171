"""Class counts of the windowed fit kernel (any class count) and its finish
tables, at the edges of its steps (32 rows), slabs (128 bytes), overflow moves
(256 rows of u8, 255 of float counts per class) and class limits.

Counts are integers and must be equal.  log theta is a difference of two
logarithms of up to 40, each within one unit in the last place: 4e-14 absolute.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

nb = pytest.importorskip("paper_1905_13746_gb300")

DT = {"u8": torch.uint8, "u16": torch.uint16, "bf16": torch.bfloat16, "f32": torch.float32}
MAX = {"u8": 255, "u16": 65535, "bf16": 256, "f32": 16777215, "fp8": 448}


def _check(fmt, n, F, C, pad=0, skew=False, shift=0, seed=0, big=False):
    rng = np.random.default_rng(seed + n + 3 * F + C)
    y = np.zeros(n, np.int32) if skew else rng.integers(0, C, n).astype(np.int32)
    y[:C] = np.arange(C)[:n]
    X = rng.poisson(2.0, (n, F)).astype(np.int64)
    X[rng.random((n, F)) < 0.02] = MAX[fmt] if big else 9
    ld = F + pad
    flat = np.zeros(n * ld + shift, np.float64)
    flat[shift:].reshape(n, ld)[:, :F] = X
    flat[shift:].reshape(n, ld)[:, F:] = 3        # padding must not be counted
    t = torch.from_numpy(flat)
    if fmt == "fp8":
        d = t.float().cuda().to(torch.float8_e4m3fn)
        f = nb.Features(d.view(torch.uint8)[shift:].view(n, ld)[:, :F], nb.NB_FP8E4M3,
                        row_exp=torch.zeros(n, dtype=torch.int8, device="cuda"))
    else:
        d = (t.to(torch.int32) if fmt == "u16" else t.float()).to(DT[fmt]).cuda()
        f = nb.Features(d[shift:].view(n, ld)[:, :F])
    m = nb.fit(f, torch.from_numpy(y).cuda(), C)
    counts, nc = m.counts()
    ref = np.zeros((C, F), np.int64)
    np.add.at(ref, y, X)
    assert np.array_equal(counts.astype(np.int64), ref)
    assert np.array_equal(nc.astype(np.int64), np.bincount(y, minlength=C))
    lt, _, log_pi = m.params()
    want = np.log(ref + 1.0) - np.log(ref.sum(1, keepdims=True) + float(F))
    assert np.abs(lt - want).max() <= 4e-14
    assert np.abs(log_pi - (np.log(np.bincount(y, minlength=C)) - np.log(n))).max() <= 1e-14


@pytest.mark.parametrize("n,F,C", [
    (3, 1, 3), (31, 3, 3), (33, 128, 5), (64, 129, 64), (65, 127, 64), (700, 516, 33),
    (3000, 64, 64), (40_000, 260, 16), (500, 4100, 64), (900, 40, 150), (300, 70, 255)])
@pytest.mark.parametrize("fmt", ["u8", "u16", "bf16", "f32", "fp8"])
def test_counts_of_every_type(fmt, n, F, C):
    es = {"u8": 1, "fp8": 1, "u16": 2, "bf16": 2, "f32": 4}[fmt]
    _check(fmt, n, F, C, pad=-F % (16 // es))


@pytest.mark.parametrize("fmt", ["u8", "u16", "bf16", "f32", "fp8"])
def test_one_class_moves_before_its_words_overflow(fmt):
    """Every row of one class, a share of the values at the type's largest."""
    es = {"u8": 1, "fp8": 1, "u16": 2, "bf16": 2, "f32": 4}[fmt]
    _check(fmt, 70_000, 36, 4, pad=-36 % (16 // es), skew=True, big=True)


@pytest.mark.parametrize("fmt,F,pad,shift,C", [
    ("f32", 1003, 0, 0, 2), ("f32", 1003, 0, 1, 7), ("f32", 33, 0, 0, 200), ("u16", 66, 0, 2, 3),
    ("u8", 37, 3, 4, 3), ("u8", 37, 0, 0, 3), ("bf16", 33, 0, 1, 5), ("fp8", 50, 2, 0, 4)])
def test_rows_of_any_alignment(fmt, F, pad, shift, C):
    _check(fmt, 2100, F, C, pad=pad, shift=shift)
