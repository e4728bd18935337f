"""The workloads by which the framework's speed is judged.

Each case is one call sequence of a user's program through the public binding
(``paper_2101_01160_gb300.mdlg``): MD runs with the fused MDLG sampling and
their f_eq readout, the f_eq stage with its bootstrap error bars, the
standalone snapshot analyses, and the surrogate's inference and training.
``listed()`` holds the sizes of the configured workloads and ``draw`` gives
others of the same ranges.  Inputs are synthetic and made from the seed alone.
"""

import math

import numpy as np
import torch

from paper_2101_01160_gb300 import mdlg

DT = 5e-4          # MD time step of every configured workload
RC = 2.5           # LJ cutoff
LAYERS = 4         # hidden layers of the surrogate
BOX_LO = (0.02, 1.0, 0.05, 0.5)    # the surrogate's training box (phi, T, dt_lg, dx)
BOX_HI = (0.30, 20.0, 1.0, 2.0)


def listed():
    return [
        # The paper's tiny system as a first run or a test of a user: one
        # FP64 replica, 400 steps, one sampling window, its f_eq and the final
        # state read back.  Every step is latency.
        dict(name="md_tiny_f64", kind="md", n_rep=1, n=1024, phi=0.0784, T=20.0, f64=True, steps=400,
             lg="400", dx="1", skin=0.5),
        # One large FP32 system sampled over a sweep of intervals and lattices.
        dict(name="md_large_f32", kind="md", n_rep=1, n=262144, phi=0.0784, T=20.0, f64=False, steps=200,
             lg="100,200", dx="0.5,1,2", skin=0.5),
        # The same system in FP64: the precision study and the plain method.
        dict(name="md_large_f64", kind="md", n_rep=1, n=262144, phi=0.0784, T=20.0, f64=True, steps=40,
             lg="40", dx="1", skin=0.5),
        # The batched ensemble: 256 uneven FP32 replicas, 5.7M particles.
        dict(name="md_ensemble", kind="md", n_rep=256, n=0, phi=0.0, T=0.0, f64=False, steps=100,
             lg="100", dx="1", skin=0.0),
        # The f_eq stage of that ensemble with block-bootstrap error bars.
        dict(name="feq_ensemble", kind="feq", n_rep=256, n_lo=4096, n_hi=65536, windows=32, every=100, W=4,
             resamples=200),
        # Binning a snapshot pair of 64 replicas of the paper's standard system.
        dict(name="bin_6m_f32", kind="bin", n=6390784, ncell=333, h=1000.0 / 333, lx=250, W=4, f64=False),
        # Binning a small FP64 pair: one analysis call in a loop over frames.
        dict(name="bin_small_f64", kind="bin", n=2047, ncell=33, h=101.283 / 33, lx=101, W=4, f64=True),
        # The displacement PDF of a large snapshot pair (Fig. 2).
        dict(name="disp_16m_f32", kind="disp", n=16777216, ncell=333, h=1000.0 / 333, nbins=64, f64=False),
        # Local fields of an ensemble window and their collision operator.
        dict(name="fields_6m_f32", kind="fields", n=6390784, ncell=333, h=1000.0 / 333, lx=250, W=4, f64=False),
        # Surrogate inference: a large map of state points, and one small query set.
        dict(name="mlp_forward_1m", kind="mlp_forward", n=1048576),
        dict(name="mlp_forward_577", kind="mlp_forward", n=577),
        # Sixteen Adam steps of the surrogate's training at its batch size.
        dict(name="mlp_train_512", kind="mlp_train", batch=512, steps=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["md", "md", "md_batch", "feq", "bin", "disp", "fields", "mlp_forward", "mlp_train"])
    if kind == "md":
        f64 = rng.random() < 0.5
        every = rng.choice([20, 25, 40, 50])
        return dict(kind="md", n_rep=1, n=_log(rng, 1000, 262144), phi=round(rng.uniform(0.02, 0.2), 4),
                    T=round(rng.uniform(1.0, 20.0), 3), f64=f64, steps=2 * every,
                    lg=rng.choice(["%d" % every, "%d,%d" % (every, 2 * every)]), dx=rng.choice(["1", "0.5,2"]),
                    skin=0.5)
    if kind == "md_batch":
        every = rng.choice([25, 40, 50])
        return dict(kind="md", n_rep=_log(rng, 4, 128), n=0, phi=0.0, T=0.0, f64=False, steps=2 * every,
                    lg="%d" % every, dx="1", skin=0.0)
    if kind == "feq":
        lo = _log(rng, 1024, 4096)
        return dict(kind="feq", n_rep=_log(rng, 3, 256), n_lo=lo, n_hi=8 * lo, windows=rng.randrange(5, 41),
                    every=rng.choice([40, 60, 100]), W=rng.choice([2, 3, 4, 4, 6, 10]),
                    resamples=rng.choice([50, 200, 400]))
    if kind in ("bin", "disp", "fields"):
        ncell = rng.randrange(9, 541)
        h = round(rng.uniform(2.7, 3.3), 4)
        c = dict(kind=kind, n=_log(rng, 1000, 6000000), ncell=ncell, h=h, f64=rng.random() < 0.3)
        if kind == "disp":
            c["nbins"] = rng.choice([32, 64, 101, 400])
        else:
            c["lx"] = rng.randrange(7, 301)
            c["W"] = rng.choice([1, 2, 3, 4, 4, 4, 6]) if kind == "bin" else rng.choice([2, 3, 4])
        return c
    if kind == "mlp_forward":
        return dict(kind=kind, n=_log(rng, 1, 1000000))
    return dict(kind=kind, batch=128 * _log(rng, 1, 64), steps=rng.randrange(3, 9))


# ---------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _gas(n, L, T, gen):
    """A homogeneous gas without overlaps: a square lattice, each site moved
    as far as keeps neighbours 0.95 apart; Maxwell velocities with zero mean
    and the exact kinetic temperature."""
    m = math.isqrt(n - 1) + 1
    a = L / m
    j = max(0.05, 0.5 * (a - 0.95))
    k = torch.arange(n, device="cuda")
    u = torch.rand((2, n), dtype=torch.float64, device="cuda", generator=gen)
    x = torch.remainder((k % m + 0.5) * a + (2.0 * u[0] - 1.0) * j, L)
    y = torch.remainder((k // m + 0.5) * a + (2.0 * u[1] - 1.0) * j, L)
    v = torch.randn((2, n), dtype=torch.float64, device="cuda", generator=gen)
    v = v - v.mean(dim=1, keepdim=True)
    v = v * torch.sqrt((2 * n - 2) * T / (v * v).sum())
    return x, y, v[0], v[1]


def _replicas(case):
    """(n, phi, T, skin) of every replica."""
    if case["kind"] == "md" and case["n_rep"] == 1:
        return [(case["n"], case["phi"], case["T"], case["skin"])]
    lo, hi = (case["n_lo"], case["n_hi"]) if case["kind"] == "feq" else (4096, 65536)
    r = np.random.default_rng(7)
    u, phi, T = r.uniform(size=case["n_rep"]), r.uniform(0.02, 0.30, case["n_rep"]), r.uniform(1.0, 20.0, case["n_rep"])
    return [(int(lo * (hi / lo) ** u[i]), float(phi[i]), float(T[i]), max(0.2, 0.7 * math.sqrt(T[i] / 20.0)))
            for i in range(case["n_rep"])]


def _md_inputs(case, seed):
    lg = [int(v) for v in case["lg"].split(",")]
    dx = [float(v) for v in case["dx"].split(",")]
    return _md_state(case, seed, lg, dx, case["f64"], 4, 1)


def _md_state(case, seed, lg, dx, f64, W, block_windows):
    gen = _gen(seed)
    params, parts = [], []
    for n, phi, T, skin in _replicas(case):
        L = math.sqrt(n * math.pi / (4.0 * phi))
        parts.append(_gas(n, L, T, gen))
        params.append(mdlg.make_params(n, L, dt=DT, rc=RC, skin=skin,
                                       precision=mdlg.MD_FP64 if f64 else mdlg.MD_FP32_CELLOFF, W=W, lg_every=lg,
                                       lx=[max(1, int(round(L / d))) for d in dx], block_windows=block_windows))
    state = [torch.cat([p[k] for p in parts]) for k in range(4)]
    return params, state


_TUNED = set()


def _system(params, state):
    """A system in the launch shape that a program keeps: the autotuner's for
    a single system (its trials, once per size, run on a system of their
    own), the full-occupancy global shape for a batch."""
    if len(params) > 1:
        s = mdlg.System(params, *state)
        s.tune(256, 1, 3)
        return s
    p = params[0]
    key = (p.n, p.precision, p.box_L, p.skin)
    if key not in _TUNED:
        trial = mdlg.System(params, *state)
        trial.autotune(50)
        trial.close()
        _TUNED.add(key)
    s = mdlg.System(params, *state)
    s.autotune(50)
    return s


def _pairs(case, seed):
    """Three consecutive snapshots (cell, ox, oy) of uniform particles with
    Gaussian displacements, in the cell + offset encoding with offsets as
    stale as a Verlet list leaves them."""
    gen = _gen(seed)
    n, nc, h = case["n"], case["ncell"], case["h"]
    ft = torch.float64 if case["f64"] else torch.float32
    L = nc * h
    step = 0.4 * (L / case["lx"]) if "lx" in case else 1.6
    X = torch.rand((2, n), dtype=torch.float64, device="cuda", generator=gen) * L
    out = []
    for k in range(3 if case["kind"] == "fields" else 2):
        if k:
            X = torch.remainder(X + step * torch.randn((2, n), dtype=torch.float64, device="cuda", generator=gen), L)
        s = (torch.rand((2, n), dtype=torch.float64, device="cuda", generator=gen) - 0.5) * (0.3 * h)
        c = torch.floor((X - s) / h)
        off = (X - c * h).to(ft)
        c = torch.remainder(c, nc).to(torch.int32)
        out.append((c[1] * nc + c[0], off[0].contiguous(), off[1].contiguous()))
    return out


def _mlp_weights(seed):
    r = np.random.default_rng(seed)
    sizes = [4] + [256] * LAYERS + [81]
    out = []
    for a, b in zip(sizes[:-1], sizes[1:]):
        lim = math.sqrt(6.0 / a)
        out += [r.uniform(-lim, lim, (b, a)).astype(np.float32), r.uniform(-0.1, 0.1, b).astype(np.float32)]
    return out


def _mlp(seed):
    lo, hi = np.array(BOX_LO), np.array(BOX_HI)
    w = np.concatenate([v.reshape(-1) for v in _mlp_weights(seed)])
    return mdlg.MLP(w, (lo + hi) / 2, (hi - lo) / math.sqrt(12.0), n_hidden=LAYERS, n_classes=81)


def _queries(n, gen):
    lo = torch.tensor(BOX_LO, device="cuda")
    hi = torch.tensor(BOX_HI, device="cuda")
    return lo + (hi - lo) * torch.rand((n, 4), device="cuda", generator=gen)


def _targets(X):
    """Displacement distributions of the queries' ballistic width."""
    v = torch.arange(-4, 5, device="cuda", dtype=torch.float32)
    a2 = (X[:, 1] * X[:, 2] ** 2 / X[:, 3] ** 2).clamp(0.02, 4.0)[:, None] + 1.0 / 6.0
    g = torch.exp(-v * v / (2.0 * a2))
    g = g / g.sum(dim=1, keepdim=True)
    return (g[:, :, None] * g[:, None, :]).reshape(-1, 81).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "md":
        params, state = _md_inputs(case, seed)
        s = _system(params, state)
        nlg, ndx = len(case["lg"].split(",")), len(case["dx"].split(","))
        outs = [[torch.zeros((len(params), 3 * s.nb + mdlg.FEQB_STATS), dtype=torch.float64, device="cuda")
                 for _ in range(ndx)] for _ in range(nlg)]
        return dict(kind=kind, s=s, steps=case["steps"], outs=outs)
    if kind == "feq":
        params, state = _md_state(case, seed, [case["every"]], [1.0], False, case["W"], 1)
        s = _system(params, state)
        s.step(case["every"] * case["windows"])
        s.sync()
        out = torch.zeros((len(params), 3 * s.nb + mdlg.FEQB_STATS), dtype=torch.float64, device="cuda")
        return dict(kind=kind, s=s, out=out, resamples=case["resamples"], seed=seed)
    if kind in ("bin", "disp", "fields"):
        p = _pairs(case, seed)
        st = dict(case, p=p)
        if kind == "fields":
            st["field"], _ = mdlg.site_occupation(*p[0], *p[1], case["ncell"], case["h"], case["lx"], case["W"])
        return st
    if kind == "mlp_forward":
        return dict(kind=kind, m=_mlp(seed), X=_queries(case["n"], _gen(seed)))
    X = _queries(case["batch"] * case["steps"], _gen(seed))
    return dict(kind=kind, m=_mlp(seed), X=X, T=_targets(X), batch=case["batch"], steps=case["steps"],
                loss=torch.zeros(case["steps"], device="cuda"))


def run(st):
    kind = st["kind"]
    if kind == "md":
        # advance, evaluate the f_eq stage on the device, read the state: the
        # small systems' as the host arrays a program stores, else the encoded one
        s = st["s"]
        s.step(st["steps"])
        for k, row in enumerate(st["outs"]):
            for d, out in enumerate(row):
                mdlg.feq_batch(s, k, d, True, out=out)
        state = s.get_state() if s.n_total <= 16384 else s.get_raw()
        return dict(state=list(state), feq=st["outs"])
    if kind == "feq":
        out = mdlg.feq_batch(st["s"], 0, 0, True, out=st["out"])
        sigma = mdlg.feq_bootstrap(st["s"], 0, 0, True, st["resamples"], st["seed"])
        return dict(feq=out, sigma=sigma)
    if kind == "bin":
        hist, ovf, mom = mdlg.mdlg_bin(*st["p"][0], *st["p"][1], st["ncell"], st["h"], st["lx"], st["W"])
        return dict(hist=hist, ovf=ovf, mom=mom)
    if kind == "disp":
        hist, outside = mdlg.disp_hist(*st["p"][0], *st["p"][1], st["ncell"], st["h"], 0.2, st["nbins"])
        return dict(hist=hist, outside=outside)
    if kind == "fields":
        field, ovf = mdlg.site_occupation(*st["p"][1], *st["p"][2], st["ncell"], st["h"], st["lx"], st["W"])
        omega = mdlg.collision(st["field"], field, st["W"], scale=1.0 / 64)
        return dict(field=field, ovf=ovf, omega=omega)
    if kind == "mlp_forward":
        return st["m"].forward(st["X"])
    b, m = st["batch"], st["m"]
    for i in range(st["steps"]):
        m.train_step(st["X"][i * b:(i + 1) * b], st["T"][i * b:(i + 1) * b], 1e-3, loss=st["loss"][i:i + 1])
    return dict(params=m.get_params(), loss=st["loss"])


# ---------------------------------------------------------------- work
def work(case):
    kind = case["kind"]
    if kind == "md":
        b = f = 0.0
        size = 8 if case["f64"] else 4
        for n, phi, _, _ in _replicas(case):
            pairs = math.pi * RC * RC * phi * 4.0 / math.pi     # neighbours within rc
            f += case["steps"] * n * (18.0 * pairs + 12.0)
            b += n * 2.0 * (4 * size + 4)                       # positions, velocities, cells
        return {"bytes": b, "flops": f}
    if kind == "feq":
        nb = (2 * case["W"] + 1) ** 2
        blocks = min(32, case["windows"])
        return {"bytes": case["n_rep"] * (32.0 * nb * 4 + (4 * nb + 16) * 8),
                "flops": case["n_rep"] * case["resamples"] * (nb * (blocks + 4.0) + 8.0 * blocks)}
    if kind in ("bin", "disp", "fields"):
        snap = case["n"] * 2.0 * (4 + 2 * (8 if case["f64"] else 4))
        if kind == "bin":
            return {"bytes": snap + 4.0 * (2 * case["W"] + 1) ** 2, "flops": 20.0 * case["n"]}
        if kind == "disp":
            return {"bytes": snap + 8.0 * case["nbins"], "flops": 12.0 * case["n"]}
        q = (2 * case["W"] + 1) ** 2 * case["lx"] ** 2
        return {"bytes": snap + q * (4.0 + 4.0 + 8.0), "flops": 20.0 * case["n"]}
    macs = 4 * 256 + (LAYERS - 1) * 256 * 256 + 256 * 81
    if kind == "mlp_forward":
        return {"bytes": case["n"] * 4.0 * 85 + 4.0 * macs, "flops": 2.0 * macs * case["n"]}
    return {"bytes": case["steps"] * (case["batch"] * 4.0 * 85 + 24.0 * macs),
            "flops": case["steps"] * 6.0 * macs * case["batch"]}


# ---------------------------------------------------------------- 64-bit values
def _exact_md(case, seed):
    """The final state of a small system by a plain velocity Verlet over all
    pairs (kick, drift, kick) in 64 bits."""
    params, (x, y, vx, vy) = _md_inputs(case, seed)
    L = params[0].box_L
    n = case["n"]

    def force():
        dx, dy = x[:, None] - x[None, :], y[:, None] - y[None, :]
        dx, dy = dx - L * torch.round(dx / L), dy - L * torch.round(dy / L)
        r2 = dx * dx + dy * dy
        r2.fill_diagonal_(1e30)
        i2 = 1.0 / r2
        s6 = i2 ** 3
        f = torch.where(r2 < RC * RC, 24.0 * s6 * (2.0 * s6 - 1.0) * i2, torch.zeros((), dtype=r2.dtype, device="cuda"))
        return (f * dx).sum(1), (f * dy).sum(1)

    fx, fy = force()
    for _ in range(case["steps"]):
        vx, vy = vx + 0.5 * DT * fx, vy + 0.5 * DT * fy
        x, y = x + DT * vx, y + DT * vy
        fx, fy = force()
        vx, vy = vx + 0.5 * DT * fx, vy + 0.5 * DT * fy
    assert x.numel() == n
    state = [v.cpu().numpy() for v in (torch.remainder(x, L), torch.remainder(y, L), vx, vy)]
    nlg, ndx = len(case["lg"].split(",")), len(case["dx"].split(","))
    return dict(state=state, feq=[[None] * ndx for _ in range(nlg)])


def _wrap(d, n):
    d = torch.remainder(d, n)
    return torch.where(d > n // 2, d - n, d)


def _exact_bin(case, p):
    nc, h = case["ncell"], case["h"]
    m2 = m4 = 0.0
    for ax in range(2):
        c0, c1 = (q[0] % nc if ax == 0 else q[0] // nc for q in (p[0], p[1]))
        d = _wrap(c1.long() - c0.long(), nc).double() * h + (p[1][1 + ax].double() - p[0][1 + ax].double())
        d = d - nc * h * torch.round(d / (nc * h))
        m2, m4 = m2 + (d * d).sum(), m4 + (d ** 4).sum()
    return dict(hist=None, ovf=None, mom=torch.stack([m2, m4]))


def _site(case, q, ax):
    nc, h = case["ncell"], case["h"]
    dxl = nc * h / case["lx"]
    c = q[0] % nc if ax == 0 else q[0] // nc
    return torch.remainder(torch.floor((c.double() * h + q[1 + ax].double()) / dxl).long(), case["lx"])


def _exact_fields(case, p):
    lx, W = case["lx"], case["W"]
    side = 2 * W + 1
    fields = []
    for a, b in ((p[0], p[1]), (p[1], p[2])):
        s0, s1 = [_site(case, a, k) for k in (0, 1)], [_site(case, b, k) for k in (0, 1)]
        v = [_wrap(s1[k] - s0[k], lx) for k in (0, 1)]
        ok = (v[0].abs() <= W) & (v[1].abs() <= W)
        at = ((v[1] + W) * side + v[0] + W) * lx * lx + s1[1] * lx + s1[0]
        fields.append(torch.bincount(at[ok], minlength=side * side * lx * lx).reshape(side * side, lx, lx))
    xi = torch.empty_like(fields[0])
    for i in range(side * side):
        vx, vy = i % side - W, i // side - W
        xi[i] = torch.roll(fields[1][i], shifts=(-vy, -vx), dims=(0, 1)) - fields[0][i]
    return dict(field=None, ovf=None, omega=xi.double() / 64)


def _forward64(w, X):
    lo, hi = torch.tensor(BOX_LO, device="cuda").double(), torch.tensor(BOX_HI, device="cuda").double()
    shift = ((lo + hi) / 2).float().double()
    scale = torch.tensor((np.array(BOX_HI) - np.array(BOX_LO)) / math.sqrt(12.0), device="cuda").float().double()
    a = (X.double() - shift) / scale
    for k in range(0, len(w) - 2, 2):
        a = torch.nn.functional.silu(a @ w[k].T + w[k + 1])
    return torch.log_softmax(a @ w[-2].T + w[-1], dim=1)


def _exact_train(case, seed):
    w = [torch.tensor(v, device="cuda").double().requires_grad_() for v in _mlp_weights(seed)]
    mom = [(torch.zeros_like(v), torch.zeros_like(v)) for v in w]
    X = _queries(case["batch"] * case["steps"], _gen(seed))
    T = _targets(X).double()
    losses = []
    for i in range(case["steps"]):
        sl = slice(i * case["batch"], (i + 1) * case["batch"])
        t = T[sl]
        loss = (torch.where(t > 0, t * torch.log(t.clamp_min(1e-300)), torch.zeros_like(t)) - t * _forward64(w, X[sl])).sum(1).mean()
        losses.append(float(loss))
        g = torch.autograd.grad(loss, w)
        with torch.no_grad():
            for v, d, (m, s) in zip(w, g, mom):
                m.mul_(0.9).add_(0.1 * d)
                s.mul_(0.999).add_(0.001 * d * d)
                v -= 1e-3 * (m / (1 - 0.9 ** (i + 1))) / (torch.sqrt(s / (1 - 0.999 ** (i + 1))) + 1e-8)
    return dict(params=torch.cat([v.detach().reshape(-1) for v in w]).cpu().numpy(), loss=np.array(losses))


def exact(case, seed):
    kind = case["kind"]
    if kind == "md":
        # larger or FP32 systems: the trajectory of all pairs is out of reach
        # or the state comes back in the encoding of the system's own cells
        small = case["n_rep"] == 1 and case["f64"] and case["n"] <= 1500
        return _exact_md(case, seed) if small else None
    if kind in ("bin", "fields"):
        p = _pairs(case, seed)
        return _exact_bin(case, p) if kind == "bin" else _exact_fields(case, p)
    if kind == "mlp_forward":
        w = [torch.tensor(v, device="cuda").double() for v in _mlp_weights(seed)]
        X = _queries(case["n"], _gen(seed))
        return torch.cat([torch.exp(_forward64(w, X[i:i + 65536])) for i in range(0, case["n"], 65536)])
    if kind == "mlp_train":
        return _exact_train(case, seed)
    return None     # counts (disp), or statistics of a whole MD run (feq)
