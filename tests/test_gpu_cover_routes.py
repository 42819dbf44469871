"""Covering launched beside the end of the boundary transport, covering launched
after it, and one kernel after the other on one stream give the same bits while
spheres cover and uncover nodes in most steps."""
import numpy as np
import pytest

from paper_2202_01631_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SPHERES = [dict(pos=(6.3, 9.7, 7.6), R=3.5, m_hat=(0.2, 0.4, -1.0), alpha=1e-2, mu_plus=0.1, mu_minus=-0.1,
                theta_c_deg=60.0, vel=(0.06, 0.02, 0.05), omega=(0.0, 0.01, 0.0)),
           dict(pos=(18.1, 5.2, 8.4), R=2.6, m_hat=(1.0, 0.1, 0.3), vel=(-0.05, 0.04, 0.03)),
           dict(pos=(16.6, 12.9, 19.3), R=4.2, m_hat=(0.0, 1.0, 0.2), alpha=2e-2, vel=(0.03, -0.06, 0.04), fixed=1)]


@pytest.fixture(scope="module")
def lbdp():
    from paper_2202_01631_gb300 import build
    build.build()
    import torch
    torch.cuda.init()
    from paper_2202_01631_gb300 import lbdp as mod
    return mod


# kz_scalars grids: 1 x 3 x 28 = 84 and 1 x 3 x 14 blocks (early), 2 x 3 x 28 =
# 168 blocks (after)
@pytest.mark.parametrize("precision,nx,planes,steps",
                         [("fp32", 26, 1, 21), ("fp32", 26, 2, 200), ("fp32", 40, 1, 21), ("fp64", 26, 1, 21)])
def test_cover_routes(lbdp, precision, nx, planes, steps):
    params = dict(W.BASE_PARAMS, nx=nx, ny=20, nz=28, periodic=(1, 1, 1), E=0.3, phi_b=1.0, k_d=2e-3)
    shape = (28, 20, nx)
    z = np.arange(28)[:, None, None]
    boxes = []
    for _ in range(2):
        rng = np.random.default_rng(11)
        b = lbdp.Box(precision=precision, **params)
        b.set_fields(rho=1.0 + 0.005 * rng.uniform(-1, 1, shape), u=0.005 * rng.uniform(-1, 1, (3,) + shape),
                     psi=np.tanh((z - 14.3) / 2.0) + 0.1 * rng.uniform(-1, 1, shape),
                     phi=1.0 + 0.05 * rng.uniform(-1, 1, shape))
        for s in SPHERES:
            b.add_particle(**s)
        b.set_planes(0, planes)
        boxes.append(b)
    start = boxes[0].mask().copy()
    boxes[0].step(steps)
    lbdp.lb_profile_step(boxes[1].h, steps)
    a, b = boxes
    assert np.count_nonzero(a.mask() != start) > 10
    assert np.array_equal(a.populations(), b.populations()) and np.array_equal(a.mask(), b.mask())
    fa, fb = a.fields(), b.fields()
    assert all(np.array_equal(fa[k], fb[k]) for k in fa)
    for pa, pb in zip(a.particles(), b.particles()):
        assert all(np.array_equal(pa[k], pb[k]) for k in pa)
