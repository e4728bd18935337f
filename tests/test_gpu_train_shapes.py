"""The training chain at the edges of its tiling: one and many row blocks, both
cluster sizes, every count of gradient splits, the smallest and largest depth
and class counts.  The gradient is compared with a plain 64-bit evaluation of
the same network (bar of the oracle test: BF16 operands, relative 2e-2 per
parameter block), the update with Adam's formula on the returned gradient."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

LO, HI = np.array([0.02, 1.0, 0.05, 0.5]), np.array([0.30, 20.0, 1.0, 2.0])
SHIFT, SCALE = (LO + HI) / 2, (HI - LO) / 2


def _net(nh, ncls, seed):
    r = np.random.default_rng(seed)
    sizes = [4] + [256] * nh + [ncls]
    out = []
    for a, b in zip(sizes[:-1], sizes[1:]):
        out += [r.uniform(-1, 1, (b, a)).astype(np.float32) * np.float32(np.sqrt(6.0 / a)),
                r.uniform(-0.1, 0.1, b).astype(np.float32)]
    return out


@pytest.mark.parametrize("B,nh,ncls", [(128, 2, 2), (128, 4, 81), (384, 3, 33), (640, 15, 112), (4864, 2, 81),
                                       (4992, 4, 81), (8192, 4, 80)])
def test_gradient_and_update(mdlg, B, nh, ncls):
    w = _net(nh, ncls, B + nh)
    m = mdlg.MLP(np.concatenate([v.reshape(-1) for v in w]), SHIFT, SCALE, n_hidden=nh, n_classes=ncls)
    g = torch.Generator().manual_seed(B)
    X = (torch.tensor(LO) + torch.tensor(HI - LO) * torch.rand(B, 4, generator=g, dtype=torch.float64)).float().cuda()
    T = torch.softmax(2.0 * torch.randn(B, ncls, generator=g), 1).cuda()
    T[:, 0] *= (torch.arange(B, device="cuda") % 3 > 0)          # zero targets, rows that do not sum to one
    T = T.contiguous()
    p = [torch.tensor(v).double().cuda().requires_grad_() for v in w]
    a = (X.double() - torch.tensor(SHIFT, device="cuda").float().double()) / torch.tensor(SCALE, device="cuda").float().double()
    for k in range(0, 2 * nh, 2):
        a = torch.nn.functional.silu(a @ p[k].T + p[k + 1])
    lp = torch.log_softmax(a @ p[-2].T + p[-1], 1)
    Td = T.double()
    loss = (torch.where(Td > 0, Td * Td.clamp_min(1e-300).log(), Td) - Td * lp).sum(1).mean()
    ref = [v.cpu().numpy().reshape(-1) for v in torch.autograd.grad(loss, p)]
    got, l = m.grad(X, T)
    m.status()
    got = got.cpu().numpy()
    assert abs(l.item() - loss.item()) < 1e-2 * abs(loss.item()) + 1e-4
    off = 0
    for u in ref:
        v = got[off:off + u.size].astype(np.float64)
        off += u.size
        deep = 2e-2 * max(1.0, nh / 4.0)       # the bar is that of four hidden layers; it grows with depth
        assert np.linalg.norm(v - u) <= deep * np.linalg.norm(u) + 1e-9, (off, np.linalg.norm(v - u) / np.linalg.norm(u))
    assert off == got.size
    # the same gradient again (nothing is left in the workspace), then one Adam step with it
    again, _ = m.grad(X, T)
    assert torch.equal(again.cpu(), torch.from_numpy(got))
    before = m.get_params()
    m.train_step(X, T, 1e-2)
    after = m.get_params()
    step = before - 1e-2 * np.sign(got) * (np.abs(got) / (np.abs(got) + 1e-8))   # first step: m / c1 = g, v / c2 = g^2
    assert np.max(np.abs(after - step)) < 2e-5
    m.status()
    m.close()
