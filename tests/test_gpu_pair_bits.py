"""The FP64 pair force, bit for bit: pairs of particles too far apart for a third,
so that each force is one pair's, compared with the same operations in exact
rational arithmetic, each rounded once.  1 / r^2 is rounded correctly (0.5 ulp);
a reciprocal that is a little less accurate differs in some of the pairs."""

from fractions import Fraction as F

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

M = 36           # pairs per edge
L = 8.0 * M


def _state(seed):
    """M^2 pairs, both particles of one in one MD cell, r from 0.85 to 2.45."""
    r = np.random.default_rng(seed)
    h = L / np.floor(L / 3.0)
    k = np.arange(M * M)
    cell = np.stack([np.round((k % M) * 8.0 / h), np.round((k // M) * 8.0 / h)])
    a = r.uniform(0.15, 0.35, (2, M * M))
    phi, d = r.uniform(0.05, np.pi / 2 - 0.05, M * M), r.uniform(0.85, 2.45, M * M)
    b = a + d * np.stack([np.cos(phi), np.sin(phi)])
    x, y = np.concatenate([cell * h + a, cell * h + b], axis=1)
    v = 0.1 * r.standard_normal((2, x.size))
    return x, y, v[0], v[1]


def _force(oi, oj):
    """Force on i (lj_pair_acc): fused where the kernel fuses."""
    rn = lambda v: F(float(v))
    rx, ry = (rn(F(v) - F(u)) for u, v in zip(oi, oj))
    r2 = rn(rx * rx + rn(ry * ry))
    if r2 >= F(6.25):
        return 0.0, 0.0
    ir2 = rn(1 / r2)
    s6 = rn(rn(ir2 * ir2) * ir2)
    fr = rn(rn(rn(24 * s6) * rn(2 * s6 - 1)) * ir2)
    return float(-fr * rx), float(-fr * ry)


@pytest.mark.parametrize("engine", ["readout", "global", "slab"])
def test_fp64_pair_forces_bit_for_bit(mdlg, engine):
    x, y, vx, vy = _state(3)
    n = x.size
    p = mdlg.make_params(n, L, precision=mdlg.MD_FP64, skin=0.5, lg_every=(100,), lx=(int(L),))
    s = mdlg.System(p, x, y, vx, vy)
    if engine == "slab":       # the last of 16 steps: positions of a system that stopped before it
        t = mdlg.System(p, x, y, vx, vy)
        t.step(15)
        raw = t.get_raw()
        t.close()
        fx, fy = s.step_forces(16)
    else:
        raw = s.get_raw()
        fx, fy = s.forces()[:2] if engine == "readout" else s.step_forces(1)
    cell, ox, oy = (v.cpu().numpy() for v in raw)
    s.close()
    h = n // 2
    assert np.array_equal(cell[:h], cell[h:])
    want = np.array([_force((ox[i], oy[i]), (ox[(i + h) % n], oy[(i + h) % n])) for i in range(n)])
    bad = np.flatnonzero((want[:, 0] != fx) | (want[:, 1] != fy))
    assert bad.size == 0, (bad.size, n, np.max(np.abs(want[:, 0] / fx - 1)[bad]))
