"""The bounded waits of the training kernels, without a GPU fault: one completion
signal is withheld (mlp_train_selftest, limit 20 ms), the CTA's waits run out, it
waits for the products and copies that it issued, and the call reports
MD_E_TIMEOUT.  The signal is that of the first, a middle and the last product of
the chain, in clusters of four and of two, and that of a stage of the weight
gradients that is waited for in the loop (640 rows) or behind it (128).
Afterwards the same model gives the gradient that it gave before."""

import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

LO, HI = np.array([0.02, 1.0, 0.05, 0.5]), np.array([0.30, 20.0, 1.0, 2.0])


@pytest.mark.parametrize("B", [128, 640, 4992])
def test_training_waits_run_out_and_are_reported(mdlg, B):
    r = np.random.default_rng(B)
    n = sum(256 * (4 if k == 0 else 256) + 256 for k in range(4)) + 81 * 257
    m = mdlg.MLP(r.uniform(-0.1, 0.1, n), (LO + HI) / 2, (HI - LO) / 2, n_hidden=4, n_classes=81)
    X = torch.tensor(LO + (HI - LO) * r.uniform(size=(B, 4)), dtype=torch.float32, device="cuda")
    T = torch.softmax(torch.tensor(r.standard_normal((B, 81)), dtype=torch.float32), 1).cuda().contiguous()
    g0, l0 = m.grad(X, T)
    w0 = m.get_params()
    m.status()
    for where in (1, 3, 4, 5, 8, -1):
        t0 = time.perf_counter()
        assert m.train_selftest(X, T, where) == mdlg.MD_E_TIMEOUT, where
        assert time.perf_counter() - t0 < 2.0
        g, l = m.grad(X, T)
        m.status()
        assert torch.equal(g, g0) and torch.equal(l, l0), where
    assert np.array_equal(m.get_params(), w0)
    for where, limit in ((0, 0.02), (9, 0.02), (-2, 0.02), (1, 0.0), (1, 3.0)):
        assert m.train_selftest(X, T, where, limit) == mdlg.MD_E_ARG
    m.close()
