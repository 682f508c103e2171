"""Many-class rows of 2^17 and more counts: the exact sums on the CUDA cores (up to
768 such rows a call, 1,024 of FP8 and BF16) and, above that for u8, the chunked tensor-core pass.

A row's sums are exact integers, so labels equal the FP64 oracle's and the log
posteriors lie within the library's 1e-5; none of these rows needs FP64 unless the
margin is within the weight quantisation, which the separated profiles exclude.
"""
import numpy as np
import pytest
import torch

from _common import compare, count_matrix, oracle_mn, stored, to_np

pytestmark = pytest.mark.gpu

nb = pytest.importorskip("paper_1905_13746_gb300")


def _heavy(fmt, n, F, C, every, seed=0):
    """Counts of C separated classes; every `every`-th row holds 2^17 counts and more."""
    top = {"u8": 255, "u8ovf": 2000, "bf16": 256, "fp8": 240}[fmt]
    X, y, _ = count_matrix(seed + F + C, n, F, C=C, clip=16 if fmt == "fp8" else 255, conc=0.3)
    X = X.astype(np.int64)
    rng = np.random.default_rng(seed)
    need = -(-(1 << 17) // top)
    for i in range(0, n, every):
        at = rng.permutation(F)[:need]
        X[i, at] = top
    assert (X[::every].sum(1) >= 1 << 17).all()
    return X.astype(np.uint16), y


@pytest.mark.parametrize("fmt,F,C", [
    ("u8", 1030, 3), ("u8", 1024, 64), ("u8", 1029, 9), ("u8ovf", 600, 17), ("u8ovf", 601, 64),
    ("bf16", 704, 16), ("bf16", 705, 33), ("fp8", 800, 8), ("fp8", 1001, 40)])
@pytest.mark.parametrize("every", [1, 7, 300])
def test_few_heavy_rows_are_exact(fmt, F, C, every):
    X, y = _heavy(fmt, 301, F, C, every)
    f, vals = stored(X, fmt)
    yd = torch.from_numpy(y).cuda()
    y2 = y.copy()
    y2[:C] = np.arange(C)
    model = nb.fit(f, torch.from_numpy(y2).cuda(), C)
    assert nb.score_path(model, f) == nb.NB_PATH_TENSOR
    _, ref = oracle_mn(vals, y2, C, vals)
    compare(to_np(nb.score(model, f)), ref)
    off = to_np(nb.score(model, f, recheck=nb.NB_RECHECK_OFF))
    assert off["n_rechecked"] == 0          # the fast path computes every row
    del yd


@pytest.mark.parametrize("n", [768, 774])
def test_the_limit_between_the_two_passes(n):
    X, y = _heavy("u8", n, 520, 5, 1, seed=3)
    f, vals = stored(X, "u8")
    model = nb.fit(f, torch.from_numpy(y).cuda(), 5)
    _, ref = oracle_mn(vals, y, 5, vals)
    res = to_np(nb.score(model, f))
    compare(res, ref)


def test_calls_on_two_streams_do_not_share_scratch():
    """A model's own scratch serves one call at a time; a second stream gets other memory."""
    X, y = _heavy("u8", 3000, 520, 5, 3, seed=8)
    f, vals = stored(X, "u8")
    model = nb.fit(f, torch.from_numpy(y).cuda(), 5)
    _, ref = oracle_mn(vals, y, 5, vals)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(3)]
    outs = []
    for k in range(9):
        with torch.cuda.stream(streams[k % 3]):
            outs.append(nb.score(model, f, stream=streams[k % 3]))
    torch.cuda.synchronize()
    for o in outs:
        compare(to_np(o), ref)
