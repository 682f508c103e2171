"""FP8 and BF16 many-class rows of 2^17 and more counts: FP64, the same bits alone, in a
batch and in a captured graph.

Up to 1,024 such rows are listed by the scoring pass and recomputed a block per row, the
rest by the recheck's scan.  The margin is then the FP64 one rounded once to FP32 (2^-24 of
it), up to the FP64 sums' own rounding: F additions of terms that make up at most T max
|log theta| on each of two sides, 2^-53 each.
"""
import ctypes

import numpy as np
import pytest
import torch

from _common import compare, oracle_mn, stored, to_np
from test_gpu_heavy_rows import _heavy

pytestmark = pytest.mark.gpu

nb = pytest.importorskip("paper_1905_13746_gb300")


def _bits(a, b):
    assert (a["label"] == b["label"]).all()
    for k in ("margin", "lp"):
        assert (a[k].view(np.uint32) == b[k].view(np.uint32)).all(), k


def _case(fmt, n, F, C, every):
    X, y = _heavy(fmt, n, F, C, every, seed=2)
    y[:C] = np.arange(C)
    f, vals = stored(X, fmt)
    model = nb.fit(f, torch.from_numpy(y).cuda(), C)
    assert nb.score_path(model, f) == nb.NB_PATH_TENSOR
    return model, f, vals, oracle_mn(vals, y, C, vals)


@pytest.mark.parametrize("fmt,F,C", [("bf16", 704, 16), ("bf16", 705, 33), ("bf16", 1100, 64),
                                     ("fp8", 800, 3), ("fp8", 1001, 64)])
@pytest.mark.parametrize("n,every", [(301, 7), (1100, 1)])
def test_heavy_rows_are_fp64_alone_and_in_a_batch(fmt, F, C, n, every):
    model, f, vals, (m, ref) = _case(fmt, n, F, C, every)
    res = to_np(nb.score(model, f))
    compare(res, ref)
    heavy = vals.sum(1) >= 1 << 17
    assert heavy.sum() >= len(range(0, n, every))
    tol = 2.0 ** -24 * ref["margin"] + 4 * F * 2.0 ** -53 * vals.sum(1) * np.abs(m["log_theta"]).max()
    assert (np.abs(res["margin"].astype(np.float64) - ref["margin"]) <= tol)[heavy].all()
    # rows past the list are left to the recheck's scan, and counted, in every mode
    off = to_np(nb.score(model, f, recheck=nb.NB_RECHECK_OFF))
    assert off["n_rechecked"] == max(0, int(heavy.sum()) - 1024)
    batch = nb.Batch([model], f.dtype_code, f.ld, 1)
    out = batch.outputs(0, n)
    batch.score([(0, f, out)])
    _bits(res, to_np(dict(out, n_rechecked=torch.zeros(1))))


def _node_types(graph):
    """cudaGraphNodeType of each node of a captured graph."""
    rt = ctypes.CDLL("libcudart.so.%s" % torch.version.cuda.split(".")[0])
    g, n = ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t(0)
    assert rt.cudaGraphGetNodes(g, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert rt.cudaGraphGetNodes(g, nodes, ctypes.byref(n)) == 0
    types = []
    for k in nodes:
        t = ctypes.c_int(-1)
        assert rt.cudaGraphNodeGetType(ctypes.c_void_p(k), ctypes.byref(t)) == 0
        types.append(t.value)
    return types


@pytest.mark.parametrize("fmt", ["bf16", "fp8"])
def test_a_captured_call_holds_no_memory_nodes_and_the_same_bits(fmt):
    """A graph with allocation nodes has one executable form at a time and is no child graph."""
    model, f, _, _ = _case(fmt, 500, 800, 8, 5)
    ref = to_np(nb.score(model, f))
    out = nb.score(model, f)
    for t in out.values():
        t.zero_()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph, stream=torch.cuda.Stream()):
        nb.score(model, f, out=out)
    types = _node_types(graph)
    assert types and not {10, 11} & set(types), types     # memory allocation and free
    for _ in range(2):
        graph.replay()
    torch.cuda.synchronize()
    _bits(ref, to_np(out))
