"""The FP64 recheck at the edges of its feature batches and class blocks, and FP8
rows narrower than a lane group.

Files of all classes come from one profile, so that margins are tiny and the
scorers mark most rows; the rechecked rows must match the FP64 oracle (labels
equal, log posteriors within 1e-5).  A warp takes 32 x 8 features of two classes
or 32 x 2 of eight at a time.
"""
import numpy as np
import pytest
import torch

from _common import compare, count_matrix, oracle_mn, stored, to_np

import synth

pytestmark = pytest.mark.gpu

nb = pytest.importorskip("paper_1905_13746_gb300")


@pytest.mark.parametrize("fmt", ["u8ovf", "u16", "f32", "bf16", "fp8"])
@pytest.mark.parametrize("C,F", [(2, 1), (2, 33), (2, 255), (2, 257), (2, 1000), (3, 63), (9, 65),
                                 (33, 100), (70, 40)])
def test_near_ties_of_one_profile(fmt, C, F):
    p = np.repeat(synth.dirichlet_profiles(5, 1, F, 2.0), C, axis=0)
    n = 40 * C + 400
    labels = (np.arange(n) % C).astype(np.int32)
    X, y, _ = count_matrix(17 + F, n, F, C=C, mu=4.0, sigma=1.0, p=p, labels=labels,
                           clip=16 if fmt == "fp8" else 255)
    f, vals = stored(X, fmt)
    model = nb.fit(f, torch.from_numpy(y).cuda(), C)
    res = to_np(nb.score(model, f))
    _, ref = oracle_mn(vals, y, C, vals)
    compare(res, ref)


@pytest.mark.parametrize("F", [5, 16, 17, 64, 100, 256, 384, 500])
def test_narrow_fp8_rows_of_counts_need_no_recheck(F):
    """Lanes without a vector of their own do not send a row to FP64."""
    X, y, _ = count_matrix(50 + F, 800, F, clip=16)
    f, vals = stored(X, "fp8")
    model = nb.fit(f, torch.from_numpy(y).cuda(), 2)
    _, ref = oracle_mn(vals, y, 2, vals)
    for cfg in [(nb.NB_VARIANT_AUTO, 0, 0, 0), (nb.NB_VARIANT_PIPELINED, 2, 16, 1),
                (nb.NB_VARIANT_PIPELINED, 2, 16, 2), (nb.NB_VARIANT_REGISTER, 0, 0, 0)]:
        model.set_tile_config(*cfg)
        res = to_np(nb.score(model, f, recheck=nb.NB_RECHECK_OFF))
        assert res["n_rechecked"] == 0, cfg     # no row the fast path cannot compute
        compare(to_np(nb.score(model, f)), ref)
