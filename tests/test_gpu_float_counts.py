"""Two-class scoring of F32, U16 and BF16 counts: the exact fixed-point sums of
the log-posterior mode and the scorer for rows of any alignment.

Labels must equal the FP64 oracle's and log posteriors lie within the library's
1e-5; a row of counts needs no FP64 recheck unless its margin is within the
weight quantisation (2^-22 of the largest weight per count), which only rows
with next to no margin can be: at most 1% of the rows here.
"""
import numpy as np
import pytest
import torch

from _common import compare, count_matrix, oracle_mn, to_np

pytestmark = pytest.mark.gpu

nb = pytest.importorskip("paper_1905_13746_gb300")

DT = {"f32": (torch.float32, 4), "u16": (torch.uint16, 2), "bf16": (torch.bfloat16, 2)}


def _features(X, fmt, pad, shift=0):
    """X in storage fmt with a row pitch of F + pad elements, shift elements past a 256-byte base."""
    n, F = X.shape
    ld = F + pad
    dtype, _ = DT[fmt]
    flat = torch.zeros(n * ld + shift, dtype=torch.float32)
    flat[shift:].view(n, ld)[:, :F] = torch.from_numpy(X.astype(np.float32))
    dev = (flat.to(torch.int32) if fmt == "u16" else flat).to(dtype).cuda()
    t = dev[shift:].view(n, ld)[:, :F]
    vals = flat[shift:].view(n, ld)[:, :F].to(torch.bfloat16 if fmt == "bf16" else torch.float32)
    return nb.Features(t), vals.double().numpy()


@pytest.mark.parametrize("fmt", ["f32", "u16", "bf16"])
@pytest.mark.parametrize("F,pad,shift", [
    (1, 0, 0), (31, 0, 0), (33, 2, 0), (127, 0, 1), (129, 0, 0), (1003, 0, 0), (1024, 0, 0),
    (1024, 1, 0), (1024, 0, 1), (4097, 3, 0)])
def test_counts_at_any_alignment(fmt, F, pad, shift):
    n = 1500
    X, y, _ = count_matrix(31 + F, n, F, clip=256 if fmt == "bf16" else 65535)
    f, vals = _features(X, fmt, pad, shift)
    model = nb.fit(f, torch.from_numpy(y).cuda(), 2)
    _, ref = oracle_mn(vals, y, 2, vals)
    res = to_np(nb.score(model, f))
    compare(res, ref)
    if F >= 31:
        assert res["n_rechecked"] <= n // 100, res["n_rechecked"]
    for mode in (nb.NB_RECHECK_LABEL, nb.NB_RECHECK_OFF):
        r = to_np(nb.score(model, f, recheck=mode))
        if mode == nb.NB_RECHECK_LABEL:
            compare(r, ref, check_lp=False)
        assert np.allclose(r["margin"], ref["margin"], rtol=1e-3, atol=1e-2)


@pytest.mark.parametrize("pad", [0, 1])
def test_values_that_are_no_counts_keep_the_float_path(pad):
    """Fractions, negative zeros and counts of 2^23 and more: same definition, FP64 where the
    FP32 bound does not settle it."""
    n, F = 900, 64
    X, y, _ = count_matrix(77, n, F)
    f, _ = _features(X, "f32", pad)
    model = nb.fit(f, torch.from_numpy(y).cuda(), 2)
    Z = X.astype(np.float32)
    Z[0::9, 3] += 0.25
    Z[1::9, 5] = 9_000_000.0
    Z[2::9, 0] = -0.0
    Z[3::9] *= np.float32(1.0 / 4096)
    fz, vals = _features(Z, "f32", pad)
    _, ref = oracle_mn(X.astype(np.float64), y, 2, vals)
    compare(to_np(nb.score(model, fz)), ref)
    compare(to_np(nb.score(model, fz, recheck=nb.NB_RECHECK_LABEL)), ref, check_lp=False)
