"""The moment sums of mdlg_bin over many particles per thread.  All particles have
the same displacement, so what an addition rounds off has one sign and does not
average out over threads.

Bar, relative: a displacement's square q and its fourth power are held as pairs
of FP32 values (q, r) and (u, v) with |r| <= 3 2^-24 q and |v| <= 3 2^-24 u, each
low part rounded once to 2^-24 of itself; r enters the fourth power twice, so a
term is off by at most 3 2^-48 (square) and 9 2^-48 (fourth power).  The sums keep
what their additions round off to below 2^-48 and may add one 2^-48."""

from fractions import Fraction

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("h,dc,o0,o1", [(3.0071, (2, 0), (0.5, 1.25), (2.75, 2.640625)),
                                        (2.8819, (-3, 1), (2.1, 0.3), (0.9, 1.7)),
                                        (2.9455, (1, -1), (0.7, 2.2), (2.85, 1.1))])
def test_moments_of_many_equal_displacements(mdlg, h, dc, o0, o1):
    n, ncell, f32 = 1 << 25, 333, torch.float32
    c = torch.arange(n, device="cuda") % (ncell * ncell)
    cx, cy = c % ncell, c // ncell
    c1 = torch.remainder(cy + dc[1], ncell) * ncell + torch.remainder(cx + dc[0], ncell)
    off = [torch.full((n,), v, dtype=f32, device="cuda") for v in o0 + o1]
    hist, ovf, mom = mdlg.mdlg_bin(c.int(), off[0], off[1], c1.int(), off[2], off[3], ncell, h, 250, 6)
    assert int(hist.sum()) + int(ovf) == n
    d = [dc[a] * Fraction(h) + Fraction(float(off[2 + a][0])) - Fraction(float(off[a][0])) for a in range(2)]
    for got, p, bar in zip(mom.tolist(), (2, 4), (4 * 2.0 ** -48, 10 * 2.0 ** -48)):
        want = n * (d[0] ** p + d[1] ** p)
        assert abs(Fraction(got) - want) <= bar * want, (p, float(abs(Fraction(got) - want) / want))
