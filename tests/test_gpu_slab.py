"""The slab engine (md_step of a single replica in shared memory) against the
global engine on the same system: equal bits of the state, the snapshots, the
histograms and the rebuild count, moment sums to 4 ulp per window count,
through rebuilds, at the edges of its plan (fewest rows, one slab, odd counts),
over split calls and readouts in between, and where a slab outgrows its room,
at the start and in flight (the global engine then runs the rest)."""

import numpy as np
import pytest

from paper_2101_01160_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _observe(s):
    out = [np.array(v) for v in s.get_state()]
    out += [t.cpu().numpy() for t in s.get_snapshot(0)]
    for k in range(2):
        for d in range(2):
            h, o, w = s.hist_raw(0, k, d)
            out += [h, np.array([o, w])]
    return out, [s.feq_measured(0, k, 0)[2] for k in range(2)], s.info()


def _check(a, b, rebuilds=True):
    for u, v in zip(a[0], b[0]):
        assert np.array_equal(u, v)
    for x, y in zip(a[1], b[1]):
        assert abs(x.mu2 - y.mu2) <= 1e-14 * y.mu2 and abs(x.mu4 - y.mu4) <= 1e-14 * y.mu4
    assert a[2].step == b[2].step


def _pair(mdlg, p, st, calls, between=None):
    res = []
    for slab in (False, True):
        s = mdlg.System(p, *st)
        s.tune(256, 1, 0 if slab else 2)
        for n in calls:
            s.step(n)
            if between:
                between(s)
        s.sync()
        res.append(_observe(s))
        s.close()
    return res


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,phi,T,skin,calls", [
    (40, 0.3, 2.0, 0.3, (16, 33)), (203, 0.2, 5.0, 0.2, (200,)), (1024, 0.0784, 20.0, 0.5, (400,)),
    (5003, 0.30, 1.0, 0.25, (3, 77, 16, 104)), (20_001, 0.02, 15.0, 0.5, (150,)),
    (99_856, 0.0784, 20.0, 0.5, (100, 20)), (200_000, 0.25, 8.0, 0.4, (60,))])
def test_slab_matches_global(mdlg, prec, n, phi, T, skin, calls):
    L = inputs.box_length(n, phi)
    st = inputs.lattice_gas_state(n, L, T, seed=n)
    p = mdlg.make_params(n, L, precision=prec, skin=skin, lg_every=(25, 40), lx=(int(L), int(L / 2)))
    a, b = _pair(mdlg, p, (st.x, st.y, st.vx, st.vy), calls)
    _check(b, a)
    assert b[2].n_rebuilds >= 2


@pytest.mark.parametrize("prec", [0, 1])
def test_slab_readouts_and_forces(mdlg, orc, prec):
    """Readouts between the calls leave the trajectory alone, and the forces
    of a slab launch's last step are the global engine's."""
    n, L = 6000, inputs.box_length(6000, 0.12)
    st = inputs.lattice_gas_state(n, L, 12.0, seed=2)
    p = mdlg.make_params(n, L, precision=prec, skin=0.3, lg_every=(20, 50), lx=(int(L), 31))
    f = []

    def between(s):
        s.get_raw()
        f.append(s.step_forces(20))
        s.energy()

    a, b = _pair(mdlg, p, (st.x, st.y, st.vx, st.vy), (20, 30, 90), between)
    _check(b, a)
    half = len(f) // 2
    for u, v in zip(f[:half], f[half:]):
        assert np.array_equal(u[0], v[0]) and np.array_equal(u[1], v[1])


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("kind", ["start", "flight"])
def test_slab_overflow_goes_on_globally(mdlg, prec, kind):
    """All particles in a narrow band of rows (the planned room is a few times
    the mean density): present at the start, or reached in flight by streaming
    towards the band's rows."""
    n, L = 4000, inputs.box_length(4000, 0.05)
    st = inputs.lattice_gas_state(n, L, 1.0, seed=4)
    vy = st.vy.copy()
    if kind == "start":
        k = np.arange(n)
        x = (k % 200 + 0.5) * (L / 200)
        y = 20.0 + 1.3 * (k // 200)
        steps = (60, 40)
    else:
        x, y = st.x, st.y
        d = np.mod(y, L) - L / 2
        vy = vy - 30.0 * np.sign(d) * np.minimum(1.0, np.abs(d) / 20.0)
        steps = (700, 600)
    p = mdlg.make_params(n, L, precision=prec, skin=0.4, lg_every=(50, 80), lx=(int(L), 31))
    p.nbr_max = 200
    a, b = _pair(mdlg, p, (x, y, st.vx, vy), steps)
    _check(b, a)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,phi,skin", [(300, 0.6, 2.2), (8100, 0.0784, 0.5), (8700, 0.0784, 0.5)])
def test_slab_long_lists_and_cluster_edge(mdlg, prec, n, phi, skin):
    """Lists of more than 64 entries, and sizes on both sides of the one up to
    which FP32 slabs form a cluster: equal bits on both engines."""
    L = inputs.box_length(n, phi)
    st = inputs.lattice_gas_state(n, L, 3.0, seed=n)
    p = mdlg.make_params(n, L, precision=prec, skin=skin, lg_every=(25, 40), lx=(int(L), int(L / 2)))
    p.nbr_max = 200
    a, b = _pair(mdlg, p, (st.x, st.y, st.vx, st.vy), (40, 60))
    _check(b, a)
