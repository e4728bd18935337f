"""The library's scratch pool: calls from several threads and streams at once,
and a capture, give the results of calls one after another."""

import threading

import numpy as np
import pytest

from paper_2101_01160_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _pair(n, seed):
    s = inputs.random_celloff_snapshots(n, 40, 3.0, seed=seed, max_step=3.0)
    return [torch.from_numpy(s[k]).cuda() for k in ("cell0", "ox0", "oy0", "cell1", "ox1", "oy1")]


def test_threads_and_streams(mdlg):
    sizes = [50_000, 120_001, 300_000, 77_777]
    data = [_pair(n, n) for n in sizes]
    ref = [[t.cpu() for t in mdlg.mdlg_bin(*d, 40, 3.0, 61, 4)] for d in data]
    torch.cuda.synchronize()
    bad = []

    def work(i):
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            for _ in range(30):
                out = mdlg.mdlg_bin(*data[i], 40, 3.0, 61, 4, stream=st)
                st.synchronize()
                if not all(torch.equal(a.cpu(), b) for a, b in zip(out, ref[i])):
                    bad.append(i)

    th = [threading.Thread(target=work, args=(i,)) for i in range(len(sizes))]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not bad


def test_capture(mdlg):
    d = _pair(200_000, 5)
    ref = [t.clone() for t in mdlg.mdlg_bin(*d, 40, 3.0, 61, 4)]
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out = mdlg.mdlg_bin(*d, 40, 3.0, 61, 4)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    for a, b in zip(out, ref):
        assert torch.equal(a, b)
