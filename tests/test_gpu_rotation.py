"""The orientation of a sphere that turns at a given spin, bit for bit the
rotation formula with every operation rounded once: the series of sin|w|/|w| and
(1 - cos|w|)/|w|^2 below |w| = 0.1, whose quotients are divisions."""
from fractions import Fraction

import pytest

from paper_2202_01631_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# spins where products with the rounded reciprocals of the divisors give another
# last bit, the ends of the range, and a few in between
SPINS = [float.fromhex(s) for s in
         ("0x1.e6a140eadb23cp-5", "0x1.05a0b739a22bdp-4", "0x1.4c06fb60a4e93p-4", "0x1.782012e1d24c3p-4",
          "0x1.69322a423d1aep-4", "0x1.81d435f2c6044p-4", "0x1.3b1c3552eea29p-4", "0x1.8f178536814e2p-4")]
SPINS += [1e-12, 3.7e-5, 0.0123, 0.0999]


def _fma(a, b, c):
    return float(Fraction(a) * Fraction(b) + Fraction(c))   # rounded once


def _dot(a, b):
    return _fma(a[0], b[0], _fma(a[1], b[1], a[2] * b[2]))


def _cross(a, b):
    return [_fma(a[i], b[j], -(a[j] * b[i])) for i, j in ((1, 2), (2, 0), (0, 1))]


def _rotated(m, w):
    w2 = _dot(w, w)
    assert w2 < 0.01
    s1 = c1 = 1.0
    for k in (4, 3, 2, 1, 0):
        s1 = _fma(-w2 / ((2 * k + 2) * (2 * k + 3)), s1, 1.0)
        c1 = _fma(-w2 / ((2 * k + 3) * (2 * k + 4)), c1, 1.0)
    c1 *= 0.5
    cw = _fma(-w2, c1, 1.0)
    wxm, wm = _cross(w, m), _dot(w, m) * c1
    r = [_fma(w[a], wm, _fma(wxm[a], s1, m[a] * cw)) for a in range(3)]
    sc = _fma(-0.5, _dot(r, r), 1.5)
    return [v * sc for v in r]


@pytest.fixture(scope="module")
def lbdp():
    from paper_2202_01631_gb300 import build
    build.build()
    import torch
    torch.cuda.init()
    from paper_2202_01631_gb300 import lbdp as mod
    return mod


@pytest.mark.parametrize("axis", [(0, 0, 1), (0.6, -0.48, 0.64)])
def test_spinning_sphere(lbdp, axis):
    params = dict(W.BASE_PARAMS, nx=20, ny=20, nz=20, periodic=(1, 1, 1), E=0.0)
    for w in SPINS:
        spin = [w * a for a in axis]
        box = lbdp.Box(precision="fp32", **params)
        box.add_particle(pos=(9.7, 10.2, 9.9), R=3.2, m_hat=(1.0, 0.0, 0.0), omega=spin, fixed=1)
        m = list(box.particles()[0]["m_hat"])
        for _ in range(3):
            m = _rotated(m, spin)
        box.step(3)
        assert list(box.particles()[0]["m_hat"]) == m, w
        box.close()
