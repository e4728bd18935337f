"""The f_eq stage's kernels at the edges of their tiles (feq_bootstrap: class
tiles, resample chunks, kept and recomputed resamples) against the oracle:
the same draws and the same rounding, so equal bits."""

import numpy as np
import pytest

from paper_2101_01160_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _batch(mdlg, W, windows, every=20, R=3, block_windows=1):
    params, cat = [], [[], [], [], []]
    for r in range(R):
        n = 900 + 131 * r
        L = inputs.box_length(n, 0.05 + 0.04 * r)
        st = inputs.lattice_gas_state(n, L, 5.0 + 6.0 * r, seed=11 + r)
        params.append(mdlg.make_params(n, L, W=W, lg_every=(every,), lx=(2 * int(round(L)) + 1,),
                                       block_windows=block_windows))
        for a, f in zip(cat, ("x", "y", "vx", "vy")):
            a.append(getattr(st, f))
    s = mdlg.System(params, *[np.concatenate(a) for a in cat])
    s.step(every * windows)
    return s, params


@pytest.mark.parametrize("W,windows,block_windows,sym,B", [
    (1, 1, 1, True, 2), (4, 33, 1, False, 63), (4, 7, 2, True, 65), (10, 40, 1, False, 130),
    (10, 40, 1, True, 200), (4, 32, 1, False, 700), (10, 5, 3, True, 2000)])
def test_bootstrap_tiles(mdlg, orc, W, windows, block_windows, sym, B):
    s, params = _batch(mdlg, W, windows, block_windows=block_windows)
    sig = mdlg.feq_bootstrap(s, 0, 0, symmetrize=sym, n_resamples=B, seed=5)
    for r, p in enumerate(params):
        h, w = mdlg.hist_blocks(s, r, 0, 0)
        ref = orc.bootstrap_feq(h.astype(np.int64), w, W, float(p.n), sym=sym, B=B, seed=5, rep=r)
        assert np.array_equal(sig[r], ref), (r, np.max(np.abs(sig[r] - ref)))
    s.close()


def _wsg_weights(lam):
    """Poisson weights of the window in extended precision, from the mode by
    the ratio w(c+1)/w(c) = lam/(c+1), normalised by their own sum."""
    lo, hi = max(0, int(lam - 14 * np.sqrt(lam) - 30)), int(lam + 14 * np.sqrt(lam) + 40)
    c = np.arange(lo, hi + 1)
    m = int(lam) - lo
    r = np.longdouble(lam) / np.arange(lo + 1, hi + 1).astype(np.longdouble)
    w = np.ones(c.size, np.longdouble)
    w[m + 1:] = np.cumprod(r[m:])
    w[:m] = np.cumprod(1 / r[:m][::-1])[::-1]
    return c, (w / w.sum()).astype(np.float64)


@pytest.mark.parametrize("lam", [0.0, 15.9, 39.99, 40.0, 44.5, 79.1, 333.0, 2.0e4, 1.0e5, 9.9e5])
def test_wsg_strided_window(mdlg, lam):
    """feq_wsg and disp_pdf_models on both sides of the strided window's line.
    Bar 1e-13: the weights' exponents carry up to 2^-53 * 200 below c = 16
    and the 1D factors a few 2^-53."""
    from math import erf, exp, pi, sqrt

    c, w = _wsg_weights(lam) if lam > 0 else (np.array([0]), np.array([1.0]))
    a2 = 0.21
    var = a2 * (c + 1.0) / (lam + 1.0)

    def f(u):
        return np.array([sqrt(v / (2 * pi)) * (exp(-(u - 1) ** 2 / (2 * v)) - 2 * exp(-u * u / (2 * v)) + exp(-(u + 1) ** 2 / (2 * v)))
                         + 0.5 * (u - 1) * (erf((u - 1) / sqrt(2 * v)) - erf(u / sqrt(2 * v)))
                         + 0.5 * (u + 1) * (erf((u + 1) / sqrt(2 * v)) - erf(u / sqrt(2 * v))) for v in var])

    F = [f(float(u)) for u in range(-4, 5)]
    ref = np.array([[np.sum(w * F[x] * F[y]) for x in range(9)] for y in range(9)]).reshape(-1)
    got = mdlg.feq_wsg(a2, lam, W=4).cpu().numpy()
    assert np.max(np.abs(got - ref)) < 1e-13
    if lam <= 1e5:
        nb, width, mu2 = 33, 0.3, 1.7
        s2 = np.sqrt(2 * mu2 * (c + 1.0) / (lam + 1.0))
        edge = (np.arange(nb + 1) - nb // 2) * width
        E = np.array([np.sum(w * np.array([erf(e / s) for s in s2])) for e in edge]) * 0.5
        _, pw = mdlg.disp_pdf_models(mu2, lam, width, nb)
        assert np.max(np.abs(pw.cpu().numpy() - np.diff(E))) < 1e-13


@pytest.mark.parametrize("W,sym", [(1, True), (4, False), (4, True), (10, False), (10, True)])
def test_feq_batch_rows(mdlg, orc, W, sym):
    """Every part of a feq_batch row against the integer histogram and the
    single-distribution oracle at the row's own a^2 and lambda."""
    s, params = _batch(mdlg, W, 35, every=15)
    P, G, Wg, st = mdlg.feq_batch(s, 0, 0, symmetrize=sym)
    for r, p in enumerate(params):
        h, ov, nw = s.hist_raw(r, 0, 0)
        ref = h / (float(p.n) * nw)
        if sym:
            ref = orc.symmetrize(ref, W)
        assert np.max(np.abs(P[r] - ref)) <= 4 * 2.0 ** -53
        a2, lam = st[r, 2], st[r, 3]
        assert np.max(np.abs(G[r] - orc.feq_gaussian(a2, 0.0, 0.0, W))) < 1e-12
        bar = 1e-12 + 4e-15 * lam          # the oracle's weights lose lambda * log(lambda) * 2^-53
        assert np.max(np.abs(Wg[r] - orc.feq_wsg(a2, lam, 0.0, 0.0, W))) < bar
        ok = P[r] > 0
        assert abs(st[r, 4] - np.max(np.abs(P[r] - G[r]))) < 1e-15
        assert abs(st[r, 6] - np.max(np.abs(P[r] - Wg[r]))) < 1e-15
        kl = np.sum(P[r][ok] * np.log(P[r][ok] / Wg[r][ok]))
        assert abs(st[r, 7] - kl) < 1e-12 * max(1.0, abs(kl)) and abs(st[r, 13] - P[r].sum()) < 1e-14
        assert st[r, 8] == nw and st[r, 10] == ov
    s.close()
