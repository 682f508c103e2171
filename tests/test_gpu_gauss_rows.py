"""The CUDA-core Gaussian scorer's staged rows and tables: rows on 16-byte boundaries and
on none, features one short of, at and one past a staged slice, class blocks with and
without padding, in each of the lane layouts.

Rows that the bound does not settle go to FP64, so labels equal the FP64 oracle's and
log posteriors lie within the library's 1e-5."""
import pytest
import torch

import oracle
import synth
from tests._common import compare, to_np

pytestmark = pytest.mark.gpu

nb = pytest.importorskip("paper_1905_13746_gb300")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    nb.build()
    nb.lib()


# classes: one padded 4-class block, 8-class blocks (padded and full), 16-class ones
@pytest.mark.parametrize("C,F", [(2, 31), (4, 129), (3, 192), (6, 33), (40, 32), (20, 191),
                                 (16, 193), (24, 575), (32, 577), (64, 65)])
@pytest.mark.parametrize("ld_extra,offset", [(0, 0), (1, 1)])
def test_gaussian_rows_on_any_boundary(C, F, ld_extra, offset):
    n = 1027
    w = synth.gaussian_workload(77 + C + F, F=F, C=C, n_fit_per_class=12,
                                n_score_per_class=(n + C - 1) // C)
    Xf, yf, Xs = w["X_fit"], w["y_fit"], w["X_score"][:n]
    model = nb.fit(torch.from_numpy(Xf).cuda(), torch.from_numpy(yf).cuda(), C,
                   kind=nb.NB_GAUSSIAN)
    model.set_tile_config(nb.NB_VARIANT_REGISTER, 0, 0, 0)
    ld = (F + 3) // 4 * 4 + ld_extra
    # what lies between the rows is no number: it must not reach a sum
    buf = torch.full((n * ld + offset,), float("nan"), device="cuda")
    X = buf[offset:].view(n, ld)[:, :F]
    X.copy_(torch.from_numpy(Xs))
    assert nb.score_path(model, X, nb.NB_RECHECK_LP) == nb.NB_PATH_GENERAL
    compare(to_np(nb.score(model, X)), oracle.score(Xs, oracle.gauss_fit(Xf, yf, C)))
