"""Steps where a CUDA graph cannot be captured, and boxes that change after theirs
was: the bits of plain launches all the same."""
import numpy as np
import pytest
import torch

from paper_2202_01631_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CUDA_STREAM_LEGACY = 1   # the legacy default stream by its name: it cannot be captured
PARAMS = dict(W.BASE_PARAMS, nx=24, ny=20, nz=28, periodic=(1, 1, 0), E=0.3, phi_b=1.0, k_d=2e-3)
SPHERE = dict(pos=(11.3, 9.7, 9.6), R=3.5, m_hat=(0.2, 0.4, -1.0), alpha=1e-2, mu_plus=0.1, mu_minus=-0.1,
              theta_c_deg=60.0, vel=(0.02, 0.0, 0.01))


@pytest.fixture(scope="module")
def lbdp():
    from paper_2202_01631_gb300 import build
    build.build()
    torch.cuda.init()
    from paper_2202_01631_gb300 import lbdp as mod
    return mod


def _fill(box, spheres=1):
    rng = np.random.default_rng(7)
    shape = box.shape
    z = np.arange(shape[0])[:, None, None]
    box.set_fields(rho=1.0 + 0.005 * rng.uniform(-1, 1, shape), u=0.005 * rng.uniform(-1, 1, (3,) + shape),
                   psi=np.tanh((z - 14.3) / 2.0) + 0.1 * rng.uniform(-1, 1, shape),
                   phi=1.0 + 0.05 * rng.uniform(-1, 1, shape))
    for _ in range(spheres):
        box.add_particle(**SPHERE)


def _same(a, b):
    assert np.array_equal(a.populations(), b.populations()) and np.array_equal(a.mask(), b.mask())
    fa, fb = a.fields(), b.fields()
    assert all(np.array_equal(fa[k], fb[k]) for k in fa)
    for pa, pb in zip(a.particles(), b.particles()):
        assert all(np.array_equal(pa[k], pb[k]) for k in pa)


def _plain(box, steps):
    for _ in range(steps):
        box.step(1)   # shorter than a graph


@pytest.mark.parametrize("spheres", [0, 1])
def test_box_on_the_legacy_stream(lbdp, spheres):
    box = lbdp.Box(precision="fp32", stream=CUDA_STREAM_LEGACY, **PARAMS)
    ref = lbdp.Box(precision="fp32", **PARAMS)
    for b in (box, ref):
        _fill(b, spheres)
    for n in (200, 60, 5):
        box.step(n)
    _plain(ref, 265)
    _same(box, ref)


@pytest.mark.parametrize("calls", [(40,), (5, 12, 9, 8, 6)])
def test_batch_on_the_legacy_stream(lbdp, calls):
    batch = lbdp.Batch(precision="fp32", arena_bytes=1 << 28, graph_steps=4, stream=CUDA_STREAM_LEGACY)
    try:
        boxes = [batch.add_box(**PARAMS) for _ in range(2)]
        for k, b in enumerate(boxes):
            _fill(b, k)
            batch.set_steps(b, 40 - 9 * k)
        for n in calls:
            batch.run(n)
        for k, b in enumerate(boxes):
            ref = lbdp.Box(precision="fp32", **PARAMS)
            _fill(ref, k)
            _plain(ref, 40 - 9 * k)
            _same(b, ref)
    finally:
        batch.close()


def test_batch_refuses_whole_graphs_under_capture(lbdp):
    stream = torch.cuda.Stream()
    batch = lbdp.Batch(precision="fp32", arena_bytes=1 << 28, graph_steps=4, stream=stream.cuda_stream)
    try:
        box = batch.add_box(**PARAMS)
        _fill(box)
        batch.set_steps(box, 50)
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
            for n in (4, 15, 50):
                with pytest.raises(lbdp.LbError):
                    batch.run(n)
        assert batch.steps_left(box) == 50
        batch.run(50)
        ref = lbdp.Box(precision="fp32", **PARAMS)
        _fill(ref)
        _plain(ref, 50)
        _same(box, ref)
    finally:
        batch.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_box_changed_after_its_graph_was_captured(lbdp, precision):
    """Chunk lengths on either side of the 152 blocks up to which covering starts
    early (2 x 3 x 28 and 2 x 3 x 14), a second, larger sphere, a checkpoint."""
    params = dict(PARAMS, nx=40, nz=28, ny=20)
    boxes = [lbdp.Box(precision=precision, **params) for _ in range(2)]
    for b in boxes:
        _fill(b)
    captured, plain = boxes

    def both(what):
        for b in boxes:
            what(b)
        captured.step(131)   # whole graphs and a few plain steps, the parity changing
        _plain(plain, 131)
        _same(captured, plain)

    both(lambda b: None)
    both(lambda b: b.set_planes(0, 1))
    both(lambda b: b.set_planes(1, 2))
    both(lambda b: b.add_particle(pos=(29.6, 10.4, 16.2), R=4.6, m_hat=(1.0, 0.1, 0.3), alpha=1e-2, omega=(0.0, 0.01, 0.0)))
    blobs = [b.save_state() for b in boxes]
    both(lambda b: b.set_planes(0, 0))
    both(lambda b: b.load_state(blobs[boxes.index(b)]))
    assert len(captured.particles()) == 2
