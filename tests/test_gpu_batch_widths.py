"""Batches of u8 rows at the widths of each lane layout of the two-class kernel and with a
partial last vector: the same bits as each group alone, and the oracle's decisions."""
import numpy as np
import pytest
import torch

from tests._common import compare, count_matrix, oracle_mn, stored, to_np

pytestmark = pytest.mark.gpu

nb = pytest.importorskip("paper_1905_13746_gb300")


@pytest.mark.parametrize("fmt", ["u8", "u8ovf"])
@pytest.mark.parametrize("F", [1, 17, 256, 257, 500, 1003, 2000])
def test_groups_of_any_width(fmt, F):
    Cs, clip = [2, 2, 3], 255 if fmt == "u8" else 65535
    models, groups = [], []
    for i, C in enumerate(Cs):
        X, y, _ = count_matrix(7 * F + i, 1000, F, C=C, clip=clip, mu=7.5)
        f, vals = stored(X, fmt)
        models.append((nb.fit(f, torch.from_numpy(y).cuda(), C), vals, y))
    for k, n in enumerate([1, 33, 0, 64, 700, 2, 31, 900]):
        X, _, _ = count_matrix(900 + 13 * k + F, max(n, 1), F, C=Cs[k % 3], clip=clip, mu=7.5)
        f, v = stored(X[:n], fmt)
        groups.append((k % 3, f, v))
    batch = nb.Batch([m for m, _, _ in models], nb.NB_U8, max(f.ld for _, f, _ in groups), 8)
    outs = [batch.outputs(s, f.n) for s, f, _ in groups]
    batch.score([(s, f, o) for (s, f, _), o in zip(groups, outs)])
    torch.cuda.synchronize()
    for (s, f, v), o in zip(groups, outs):
        if not f.n:
            continue
        got, alone = to_np(dict(o, n_rechecked=torch.zeros(1))), to_np(nb.score(models[s][0], f))
        assert (got["label"] == alone["label"]).all()
        for k in ("margin", "lp"):
            assert (got[k].view(np.uint32) == alone[k].view(np.uint32)).all(), k
        compare(got, oracle_mn(models[s][1], models[s][2], Cs[s], v)[1])
