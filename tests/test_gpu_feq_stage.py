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
