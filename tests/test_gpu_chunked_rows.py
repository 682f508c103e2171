"""Heavy u8 rows beyond what the CUDA cores take: the chunked tensor-core pass in each of its
class parts, over more than two chunks, with overflow entries, and on several streams.

The sums are exact integers, so labels equal the FP64 oracle's and the log posteriors lie
within the library's 1e-5.
"""
import numpy as np
import pytest
import torch

from _common import compare, count_matrix, oracle_mn, stored, to_np

pytestmark = pytest.mark.gpu

nb = pytest.importorskip("paper_1905_13746_gb300")

FEW = 768     # heavy rows of a call that go to the CUDA cores


def _rows(seed, n, F, C, heavy, overflow):
    """n files of C separated classes; row i is heavy (2^17 and more stored counts) where heavy[i]."""
    X, y, _ = count_matrix(seed, n, F, C=C, clip=255, conc=0.3, mu=7.0)
    X = X.astype(np.uint16)
    rng = np.random.default_rng(seed)
    for i in np.nonzero(heavy)[0]:
        at = rng.permutation(F)[:515]              # 515 x 255 > 2^17
        X[i, at] = 255
        if overflow:
            X[i, at[:7]] += rng.integers(1, 3000, 7).astype(np.uint16)
    return X, y


def _model(fmt, X, y, C):
    y = y.copy()
    y[:C] = np.arange(C)
    f, vals = stored(X, fmt)
    return nb.fit(f, torch.from_numpy(y).cuda(), C), f, oracle_mn(vals, y, C, vals)[1]


@pytest.mark.parametrize("fmt", ["u8", "u8ovf"])
@pytest.mark.parametrize("C,F", [(5, 520), (17, 1100), (33, 1536), (64, 1100), (64, 2061)])
@pytest.mark.parametrize("heavy", [FEW + 1, 900])
def test_more_heavy_rows_than_the_cuda_cores_take(fmt, C, F, heavy):
    n = 1000
    h = np.zeros(n, bool)
    h[np.random.default_rng(C + F).permutation(n)[:heavy]] = True
    X, y = _rows(C + F, n, F, C, h, fmt == "u8ovf")
    assert (np.minimum(X, 255).astype(np.int64).sum(1) >= 1 << 17).sum() == heavy
    model, f, ref = _model(fmt, X, y, C)
    assert nb.score_path(model, f) == nb.NB_PATH_TENSOR
    compare(to_np(nb.score(model, f)), ref)
    off = to_np(nb.score(model, f, recheck=nb.NB_RECHECK_OFF))
    assert off["n_rechecked"] == 0          # the fast path computes every row


def test_streams_with_rows_of_their_own():
    """Calls of a few tiles on several streams, each with other rows, heavy ones in other places
    and in other numbers: each gives the bits of the call alone."""
    C, F, n = 9, 520, 1024
    X, y = _rows(1, n, F, C, np.zeros(n, bool), False)
    model, _, _ = _model("u8", X, y, C)
    rng = np.random.default_rng(4)
    inputs = []
    for k, heavy in enumerate([0, 1, 130, 700, 800, 1000]):
        h = np.zeros(n, bool)
        h[rng.permutation(n)[:heavy]] = True
        f, _ = stored(_rows(50 + k, n, F, C, h, False)[0], "u8")
        inputs.append((f, to_np(nb.score(model, f))))
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in inputs]
    outs = []
    for _ in range(20):
        for s, (f, ref) in zip(streams, inputs):
            with torch.cuda.stream(s):
                outs.append((nb.score(model, f, stream=s), ref))
    torch.cuda.synchronize()
    for o, ref in outs:
        got = to_np(o)
        assert (got["label"] == ref["label"]).all() and got["n_rechecked"] == ref["n_rechecked"]
        for k in ("margin", "lp"):
            assert (got[k].view(np.uint32) == ref[k].view(np.uint32)).all(), k
