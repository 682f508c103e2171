"""A thread that has read from the library ends while another captures a graph: the
page-locked buffer that it gives back must not spoil the capture."""
import threading
import time

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

nb = pytest.importorskip("paper_1905_13746_gb300")


def test_a_reader_ends_during_a_capture():
    rng = np.random.default_rng(0)
    X = torch.from_numpy(rng.integers(0, 9, (200, 32)).astype(np.uint8)).cuda()
    y = torch.from_numpy((np.arange(200) % 2).astype(np.int32)).cuda()
    model = nb.fit(X, y, 2)
    expected = model.params()
    got, read, end = [], threading.Event(), threading.Event()

    def reader():
        got.append(model.params())
        read.set()
        end.wait(30)

    threads = [threading.Thread(target=reader) for _ in range(3)]
    for t in threads:
        t.start()
    read.wait(30)
    time.sleep(0.2)
    t = torch.zeros(1000, device="cuda")
    side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        graph.capture_begin(capture_error_mode="global")
        t.add_(1)
        end.set()
        for k in threads:
            k.join()
        time.sleep(0.5)       # the threads' own storage goes after Python's part
        t.add_(1)
        graph.capture_end()
    graph.replay()
    torch.cuda.synchronize()
    assert (t == 2).all()
    for p in got:
        assert all(np.array_equal(a, b) for a, b in zip(p, expected) if a is not None)
