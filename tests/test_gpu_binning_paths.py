"""mdlg_bin at the edges of its paths: one cluster against the one-wave grid,
vector against scalar loads, the FP32-pair moments against the FP64 fallbacks
(displacements near half the box, tiny ones, cell edges far from 1).  Counts
equal the oracle's; moments are compared with extended precision.

Moment bar: the pairs carry at least 45 bits (1e-13 relative), a displacement
that goes through FP64 positions carries eps = 2^-51 L of absolute error,
which changes its square by at most 2 |d| eps + eps^2 and its fourth power by
at most 4 |d|^3 eps (1 + eps/|d|)^3; FP64 sums of n terms add 1e-13."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _snapshots(n, ncell, h, step, f64, seed):
    rng = np.random.default_rng(seed)
    ft = np.float64 if f64 else np.float32
    out = []
    X = rng.uniform(0.0, ncell, (2, n))
    for k in range(2):
        if k:
            X = np.mod(X + step * rng.standard_normal((2, n)), ncell)
        c = np.floor(X - rng.uniform(-0.2, 0.2, (2, n)))
        off = ((X - c) * h).astype(ft)
        c = np.mod(c, ncell).astype(np.int64)
        out += [(c[1] * ncell + c[0]).astype(np.int32), off[0], off[1]]
    if n > 3:   # unmoved particles, and one displaced by exactly half the box
        for a in range(3):
            out[3 + a][:2] = out[a][:2]
        out[3][2] = (out[0][2] // ncell) * ncell + (out[0][2] + ncell // 2) % ncell
        out[4][2], out[5][2] = out[1][2], out[2][2]
    return out


def _reference(a, ncell, h):
    ld = np.longdouble
    L = ld(ncell) * ld(h)
    ref, bar = np.zeros(2, ld), np.zeros(2)
    eps = 2.0 ** -51 * float(L)
    for ax in range(2):
        c0, c1 = (a[0] % ncell, a[3] % ncell) if ax == 0 else (a[0] // ncell, a[3] // ncell)
        d = (c1.astype(ld) - c0.astype(ld)) * ld(h) + (a[4 + ax].astype(ld) - a[1 + ax].astype(ld))
        d = d - L * np.rint(d / L)
        ref += [np.sum(d * d), np.sum(d ** 4)]
        q = np.abs(d).astype(np.float64)
        slow = (q < 2.1 ** -20 * h) | (q > 0.48 * float(L)) | (h < 1e-15) | (h > 1e15)
        q = q[slow]
        bar += [np.sum(2 * q * eps + eps ** 2), np.sum((q + eps) ** 4 - q ** 4)]
    return ref.astype(np.float64), bar


@pytest.mark.parametrize("n,shift,f64", [(511, 0, False), (513, 1, False), (4097, 0, True), (32768, 1, False),
                                         (32769, 0, False), (32771, 1, False), (300_003, 0, False),
                                         (100_001, 0, True), (100_001, 1, True)])
@pytest.mark.parametrize("ncell,h,step", [(33, 3.069181818, 0.7), (4, 2.75, 0.9), (333, 3.003003003, 1e-8),
                                          (540, 2.7, 30.0), (21, 3.1e-17, 0.4), (21, 2.9e20, 0.4)])
def test_bin_paths(mdlg, orc, n, shift, f64, ncell, h, step):
    h = h if f64 else float(np.float32(h))
    a = _snapshots(n, ncell, h, step, f64, seed=n + ncell)
    dev = []
    for v in a:   # `shift` elements into the buffer: arrays that are not 16-byte aligned
        b = torch.empty(n + shift, dtype=torch.from_numpy(v).dtype, device="cuda")
        b[shift:] = torch.from_numpy(v)
        dev.append(b[shift:])
    keys = ("cell0", "ox0", "oy0", "cell1", "ox1", "oy1")
    for lx, W in ((101, 4), (3, 1)):
        outs = [mdlg.mdlg_bin(*dev, ncell, h, lx, W, noalloc=f) for f in (False, True)]
        rh, ro, _ = orc.bin_celloff(dict(zip(keys, a)), ncell, h, ncell * h, lx, W)
        ref, bar = _reference(a, ncell, h)
        for hist, ovf, mom in outs:
            assert np.array_equal(hist.cpu().numpy().astype(np.int64), rh) and int(ovf.item()) == ro
            m = mom.cpu().numpy()
            assert np.all(np.abs(m - ref) <= 2e-13 * np.abs(ref) + bar), (m, ref, bar)
        assert torch.equal(outs[0][2], outs[1][2])
