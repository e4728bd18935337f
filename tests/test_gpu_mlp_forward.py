"""The fused forward pass at the edges of its tiles and of its staging: fewest
and most classes (the staged rows then end where the next tile's inputs
begin), class counts that are no multiple of a load, shallow and deep
networks, ragged batches, several tiles per slot, an unaligned output.  A
small batch against the FP64 oracle with the bar of BF16 weights and
activations (relative 3e-2 on every class); a row's result must not depend on
the batch around it, bit for bit."""

import numpy as np
import pytest

from paper_2101_01160_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SHIFT = np.array([0.15, 10.0, 0.5, 1.5], dtype=np.float32)
SCALE = np.array([0.1, 6.0, 0.3, 0.8], dtype=np.float32)


@pytest.mark.parametrize("n_hidden,n_classes", [(2, 9), (4, 81), (3, 96), (2, 97), (5, 112)])
def test_forward_edges(mdlg, orc, n_hidden, n_classes):
    sizes = [4] + [256] * n_hidden + [n_classes]
    params = orc.mlp_pack(*inputs.mlp_init(sizes, 7)).astype(np.float32)
    m = mdlg.MLP(params, SHIFT, SCALE, n_hidden=n_hidden, n_classes=n_classes)
    M = 2 * 2 * 152 * 128 + 77          # the first slots of a full grid take a third tile
    X = torch.from_numpy(inputs.surrogate_queries(M, 1)).cuda()
    small = {n: m.forward(X[:n].contiguous()).cpu().numpy() for n in (1, 127, 129, 300)}
    ref = orc.mlp_forward(sizes, X[:300].cpu().numpy().astype(np.float64), params.astype(np.float64), SHIFT, SCALE)
    assert np.max(np.abs(small[300] - ref) / (ref + 1e-4)) < 3e-2
    for n, p in small.items():
        assert np.array_equal(p, small[300][:n])
    buf = torch.zeros(300 * n_classes + 1, device="cuda")
    m.forward(X[:300].contiguous(), out=buf[1:].view(300, n_classes))
    assert np.array_equal(buf[1:].view(300, n_classes).cpu().numpy(), small[300]) and buf[0] == 0
    big = m.forward(X)
    assert np.array_equal(big[:300].cpu().numpy(), small[300])
    for at in (38_900, M - 200):
        assert torch.equal(big[at:at + 200], m.forward(X[at:at + 200].contiguous()))
    m.status()
