"""Steps run as captured CUDA graphs give the bits of plain launches: a small
box with spheres, whose graph is captured after 128 steps, and a batch, whose
graph is captured once four of them have run or are asked for at once."""
import numpy as np
import pytest

from paper_2202_01631_gb300 import workloads as W

pytestmark = pytest.mark.gpu

PARAMS = dict(W.BASE_PARAMS, nx=24, ny=20, nz=28, periodic=(1, 1, 0), E=0.3, phi_b=1.0, k_d=2e-3)
SPHERE = dict(pos=(11.3, 9.7, 13.6), R=4.5, m_hat=(0.2, 0.4, -1.0), alpha=1e-2, mu_plus=0.1, mu_minus=-0.1,
              theta_c_deg=60.0, vel=(0.02, 0.0, 0.01), fixed=1)


@pytest.fixture(scope="module")
def lbdp():
    from paper_2202_01631_gb300 import build
    build.build()
    import torch
    torch.cuda.init()
    from paper_2202_01631_gb300 import lbdp as mod
    return mod


def _fill(box):
    rng = np.random.default_rng(7)
    shape = (PARAMS["nz"], PARAMS["ny"], PARAMS["nx"])
    z = np.arange(shape[0])[:, None, None]
    box.set_fields(rho=1.0 + 0.005 * rng.uniform(-1, 1, shape), u=0.005 * rng.uniform(-1, 1, (3,) + shape),
                   psi=np.tanh((z - 14.3) / 2.0) + 0.1 * rng.uniform(-1, 1, shape),
                   phi=1.0 + 0.05 * rng.uniform(-1, 1, shape))
    box.add_particle(**SPHERE)


def _same(a, b):
    assert np.array_equal(a.populations(), b.populations()) and np.array_equal(a.mask(), b.mask())
    fa, fb = a.fields(), b.fields()
    assert all(np.array_equal(fa[k], fb[k]) for k in fa)
    pa, pb = a.particles()[0], b.particles()[0]
    assert all(np.array_equal(pa[k], pb[k]) for k in pa)


@pytest.mark.parametrize("precision,calls", [("fp32", [61, 70, 40, 16, 13]), ("fp64", [200]), ("fp16", [135, 65])])
def test_box_with_sphere(lbdp, precision, calls):
    plain, graph = (lbdp.Box(precision=precision, **PARAMS) for _ in range(2))
    _fill(plain)
    _fill(graph)
    for _ in range(200):
        plain.step(1)   # shorter than a graph: plain launches
    for n in calls:
        graph.step(n)
    _same(plain, graph)


@pytest.mark.parametrize("calls", [[40], [5, 7, 9, 3, 11, 5]])
def test_batch(lbdp, calls):
    batch = lbdp.Batch(precision="fp32", arena_bytes=1 << 28, graph_steps=4)
    try:
        boxes = [batch.add_box(**PARAMS) for _ in range(2)]
        for k, b in enumerate(boxes):
            _fill(b)
            batch.set_steps(b, 40 - 9 * k)
        for n in calls:
            batch.run(n)
        alone = [lbdp.Box(precision="fp32", **PARAMS) for _ in range(2)]
        for k, b in enumerate(alone):
            _fill(b)
            b.step(40 - 9 * k)
            _same(b, boxes[k])
    finally:
        batch.close()
