"""One replica handed from engine to engine: the slots' order, the step's
velocity bound and the rebuild count belong to the system, whichever engine ran
last.  Every walk gives the bits of the global engine alone."""

import itertools

import numpy as np
import pytest

from paper_2101_01160_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SLAB, GLOBAL, RESIDENT = (256, 1, 0), (256, 1, 2), (0, 0, 4)


def _make(mdlg, n, prec, phi=0.1, T=12.0, skin=0.3):
    L = inputs.box_length(n, phi)
    st = inputs.lattice_gas_state(n, L, T, seed=n)
    p = mdlg.make_params(n, L, precision=prec, skin=skin, lg_every=(20, 50), lx=(int(L), 31))
    return mdlg.System(p, st.x, st.y, st.vx, st.vy)


def _observe(s):
    out = [np.array(v) for v in s.get_state()] + [t.cpu().numpy() for t in s.get_snapshot(1)]
    return out + [s.hist_raw(0, k, d)[0] for k in range(2) for d in range(2)]


@pytest.mark.parametrize("n", [4000, 12_000])   # slabs as one cluster, slabs as a grid; one and several resident slabs
def test_walks_over_the_engines(mdlg, n):
    """All orders of three of slab, resident, global and readout, each step a
    call of 40 steps, then the slab engine."""
    ref = {}
    for k in range(1, 5):
        s = _make(mdlg, n, mdlg.MD_FP32_CELLOFF)
        s.tune(*GLOBAL)
        s.step(40 * k)
        ref[k] = _observe(s)
        s.close()
    for walk in itertools.product("SRGO", repeat=3):
        s = _make(mdlg, n, mdlg.MD_FP32_CELLOFF)
        k = 1
        for op in walk + ("S",):
            if op == "O":
                s.get_raw()
                continue
            s.tune(*{"S": SLAB, "R": RESIDENT, "G": GLOBAL}[op])
            s.step(40)
            k += 1
        for u, v in zip(_observe(s), ref[k - 1]):
            assert np.array_equal(u, v), walk
        s.close()


def _count(s):
    return s.info().n_rebuilds


@pytest.mark.parametrize("prec", [0, 1])
def test_rebuild_count_does_not_depend_on_the_engine(mdlg, prec):
    """Readouts, short calls, a changed shape, a checkpoint and a new state
    between slab calls: the count after each is the global engine's."""
    runs = []
    for shape in (GLOBAL, SLAB):
        s = _make(mdlg, 5000, prec)
        c = [_count(s)]
        s.tune(*shape)
        for n in (40, 3, 60, 17, 1, 1, 90):
            s.step(n)
            c.append(_count(s))
            s.get_raw()
            c.append(_count(s))
        s.step(50)
        s.energy()
        s.forces()
        s.step(5)
        c.append(_count(s))
        s.tune(128, 1, shape[2])
        s.get_raw()
        s.step(30)
        c.append(_count(s))
        ck = s.checkpoint()
        c.append(_count(s))
        s.step(70)
        s.restore(ck)
        s.step(20)
        c.append(_count(s))
        st = s.get_state()
        s.set_state(*st)
        s.step(64)
        c.append(_count(s))
        runs.append((c, _observe(s)))
        s.close()
    assert runs[0][0] == runs[1][0]
    assert runs[0][0][-1] > 10
    for u, v in zip(runs[0][1], runs[1][1]):
        assert np.array_equal(u, v)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("between", [16, 17, 18])
def test_velocity_bound_of_earlier_steps_is_not_used(mdlg, prec, between):
    """Hot steps on the global engine, slab steps, then a cold state: the
    maxima of the hot steps (each above half the skin) must not make the cold
    steps rebuild, whichever slot of three they were left in."""
    n, L = 4000, inputs.box_length(4000, 0.05)
    hot, cold = inputs.lattice_gas_state(n, L, 20.0, seed=1), inputs.lattice_gas_state(n, L, 0.05, seed=1)
    p = mdlg.make_params(n, L, precision=prec, skin=0.008, lg_every=(20,), lx=(int(L),))
    runs = []
    for shape in (GLOBAL, SLAB):
        s = mdlg.System(p, hot.x, hot.y, hot.vx, hot.vy)
        s.tune(*shape)
        s.step(4)
        s.step(between)
        s.set_state(cold.x, cold.y, cold.vx, cold.vy)
        c = _count(s)
        s.step(1)
        c = (c, _count(s))
        s.step(5)
        runs.append((c, _count(s), s.get_state()))
        s.close()
    assert runs[0][:2] == runs[1][:2] and runs[1][0][0] == runs[1][0][1]
    for u, v in zip(runs[0][2], runs[1][2]):
        assert np.array_equal(u, v)


@pytest.mark.parametrize("prec", [0, 1])
def test_list_limit_is_reported_by_every_engine(mdlg, prec):
    """A hexagonal cluster that contracts: its lists outgrow the default
    capacity (24 entries here) in flight.  Before that the call succeeds, after
    it md_sync reports MD_E_LIMIT, whichever engine runs."""
    n, L = 3000, inputs.box_length(3000, 0.04)
    a, c = 1.22, L / 2
    hexes = np.array([(a * (i + 0.5 * (j % 2)), a * np.sqrt(0.75) * j) for i in range(-9, 10) for j in range(-10, 11)])
    hexes = hexes[np.hypot(*hexes.T) < 5.6]
    g = np.stack(np.meshgrid(*[(np.arange(70) + 0.5) * (L / 70)] * 2), -1).reshape(-1, 2)
    g = g[np.hypot(*(g - c).T) > 16.0][:n - len(hexes)]
    x, y = np.concatenate([hexes + c, g]).T.copy()
    vx, vy = np.concatenate([-5.0 * hexes, np.zeros_like(g)]).T.copy()
    p = mdlg.make_params(len(x), L, precision=prec, skin=0.3, lg_every=(20,), lx=(int(L),))
    codes = []
    for shape in (GLOBAL, SLAB):
        s = mdlg.System(p, x, y, vx, vy)
        s.tune(*shape)
        for k in range(10):
            s.step(16)
            try:
                s.sync()
                codes.append(0)
            except mdlg.MDError as e:
                codes.append(e.code)
                break
        s.close()
    half = len(codes) // 2
    assert codes[:half] == codes[half:] and codes[-1] == mdlg.MD_E_LIMIT and half >= 3, codes


def _slab_runs(s, n=50):
    """Whether a call of n steps runs the slab engine."""
    from torch.profiler import ProfilerActivity, profile

    for _ in range(2):   # (the first profile of a process may record nothing)
        s.sync()
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            s.step(n)
            s.sync()
            torch.cuda.synchronize()
        names = [e.name for e in prof.events() if "k_md_" in e.name]
    if not names:
        pytest.skip("the profiler records no kernels here")
    return any("k_md_slab" in v for v in names)


def test_tuner_cache_of_a_system_without_a_slab_plan(mdlg):
    """520,000 particles have no slab plan, 270,000 have one and share the
    tuner's key: the second system, tuned without trials, keeps the slab engine."""
    big, small = (_make(mdlg, n, mdlg.MD_FP32_CELLOFF, 0.0784, 20.0, 0.5) for n in (520_000, 270_000))
    best = big.autotune(16)
    assert not _slab_runs(big)
    assert small.autotune(16) == best and small.info().step == 0
    assert _slab_runs(small)
    big.close()
    small.close()


def test_refused_tune_changes_nothing(mdlg):
    s = _make(mdlg, 5000, mdlg.MD_FP32_CELLOFF)
    for bad in ((100, 1, 1), (256, 9, 2), (256, 1, 5)):
        with pytest.raises(mdlg.MDError):
            s.tune(*bad)
        assert _slab_runs(s)
    s.tune(*GLOBAL)
    for bad in ((100, 1, 0), (256, 9, 0)):
        with pytest.raises(mdlg.MDError):
            s.tune(*bad)
        assert not _slab_runs(s)
    s.close()


@pytest.mark.parametrize("n,prec,enter,stay", [(4000, 1, 16, 8), (20_000, 1, 32, 20), (20_000, 0, 16, 8)])
def test_short_calls_leave_the_slab_engine(mdlg, n, prec, enter, stay):
    """Calls too short to pay for a slab launch run on the global engine, also
    behind a slab call, with the bits of the global engine alone."""
    runs = []
    for shape in (GLOBAL, SLAB):
        s = _make(mdlg, n, prec)
        s.tune(*shape)
        ran = []
        for k in (enter - 1, enter, stay, stay - 1, stay, 1, 1, 100, 1):
            ran.append(_slab_runs(s, k))
        runs.append((ran, _count(s), _observe(s)))
        s.close()
    assert not any(runs[0][0])
    # (_slab_runs makes two calls of each)
    assert runs[1][0] == [False, True, True, False, False, False, False, True, False]
    assert runs[0][1] == runs[1][1]
    for u, v in zip(runs[0][2], runs[1][2]):
        assert np.array_equal(u, v)


@pytest.mark.parametrize("prec", [0, 1])
def test_state_without_room_leaves_the_slab_engine(mdlg, prec):
    """All particles in a band of rows that outgrows the slabs' room: found at
    the first synchronisation, the next 32 calls go to the global engine at once,
    then one tries again, then 64; a new state gets its chance at once."""
    n, L = 4000, inputs.box_length(4000, 0.05)
    st = inputs.lattice_gas_state(n, L, 1.0, seed=4)
    k = np.arange(n)
    p = mdlg.make_params(n, L, precision=prec, skin=0.4, lg_every=(50,), lx=(int(L),))
    p.nbr_max = 200
    s = mdlg.System(p, (k % 200 + 0.5) * (L / 200), 20.0 + 1.3 * (k // 200), 0.05 * st.vx, 0.05 * st.vy)
    s.tune(*SLAB)
    s.step(32)
    s.sync()
    assert not _slab_runs(s, 32)              # two calls
    for _ in range(29):
        s.step(32)
    assert not _slab_runs(s, 1)
    s.step(32)                                # the 32nd
    s.step(32)                                # the try
    s.sync()
    for _ in range(32):
        s.step(32)
    assert not _slab_runs(s, 32)
    s.set_state(st.x, st.y, st.vx, st.vy)
    assert _slab_runs(s, 32)
    s.close()


def test_tuner_compares_engines_on_one_state(mdlg):
    """FP64 on a fresh lattice start, where a global step costs half of what it
    costs later (16,384 particles: 10 us against 19; slab 11): the slab engine,
    the faster one from then on, is chosen."""
    L = inputs.box_length(16_384, 0.0784)
    st = inputs.lattice_gas_state(16_384, L, 20.0, seed=5)
    p = mdlg.make_params(16_384, L, precision=mdlg.MD_FP64, lg_every=(400,), lx=(int(L),))
    s = mdlg.System(p, st.x, st.y, st.vx, st.vy)
    s.autotune(50)
    assert _slab_runs(s)
    s.close()


@pytest.mark.parametrize("prec", [0, 1])
def test_moment_sums_of_the_engines(mdlg, prec):
    """The engines group the FP64 moment terms differently.  Every grouping adds a
    term to others at most 5 times inside a warp, once per window, and at most 2 +
    8 times in the readout (157 warps or fewer slabs over 256 threads), each
    addition within 2^-53 of its result; all terms are positive."""
    st = []
    for shape in (GLOBAL, SLAB):
        s = _make(mdlg, 5000, prec)
        s.tune(*shape)
        s.step(100)
        s.step(100)
        st.append([s.feq_measured(0, k, 0)[2] for k in range(2)])
        s.close()
    for a, b in zip(*st):
        assert a.n_windows == b.n_windows > 0
        bar = 2 * (15 + a.n_windows) * 2.0 ** -53
        assert abs(a.mu2 - b.mu2) <= bar * a.mu2 and abs(a.mu4 - b.mu4) <= bar * a.mu4
