"""The bounded wait of the slab engine's exchange, without a GPU fault: one CTA
leaves before it posts its word (md_slab_selftest, limit 20 ms), the others give
up, and the call reports MD_E_TIMEOUT.  Neither the slabs nor the global launch
behind them may touch the state: afterwards it is as before, and the same system
runs on with the bits of one that was never interrupted."""

import time

import numpy as np
import pytest

from paper_2101_01160_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _system(mdlg, prec, n):
    L = inputs.box_length(n, 0.1)
    st = inputs.lattice_gas_state(n, L, 5.0, seed=3)
    p = mdlg.make_params(n, L, precision=prec, skin=0.3, lg_every=(20,), lx=(int(L),))
    return mdlg.System(p, st.x, st.y, st.vx, st.vy)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("first", [0, 40])   # on the created state, and behind a slab launch
def test_exchange_wait_runs_out_and_is_reported(mdlg, prec, first):
    ends = []
    for interrupted in (True, False):
        s = _system(mdlg, prec, 20_000)
        if first:
            s.step(first)
        for _ in range(2 if interrupted else 0):
            step, count = s.info().step, s.info().n_rebuilds
            t0 = time.perf_counter()
            assert s.slab_selftest(0.02) == mdlg.MD_E_TIMEOUT
            assert time.perf_counter() - t0 < 2.0
            assert (s.info().step, s.info().n_rebuilds) == (step, count)
        s.step(60)
        s.step(3)
        ends.append([np.array(v) for v in s.get_state()] + [s.hist_raw()[0]])
        s.close()
    for u, v in zip(*ends):
        assert np.array_equal(u, v)


def test_slab_selftest_rejects(mdlg):
    s = _system(mdlg, 1, 20_000)
    for lim in (0.0, -1.0, 5.0):
        assert s.slab_selftest(lim) == mdlg.MD_E_ARG
    s.close()
    s = _system(mdlg, 1, 2000)       # its slabs are one cluster
    assert s.slab_selftest() == mdlg.MD_E_ARG
    s.close()
