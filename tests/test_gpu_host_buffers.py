"""lb_set_fields has read its arrays when it returns: one pinned buffer filled
anew for each box gives the bits of a buffer per box, also while the stream
still works on steps queued before."""
import numpy as np
import pytest
import torch

from paper_2202_01631_gb300 import workloads as W

pytestmark = pytest.mark.gpu

N = 48
PARAMS = dict(W.BASE_PARAMS, nx=N, ny=N, nz=N, periodic=(1, 1, 1), E=0.3, phi_b=1.0, k_d=2e-3)
SPHERE = dict(pos=(23.3, 24.7, 22.6), R=4.5, m_hat=(0.2, 0.4, -1.0), alpha=1e-2, mu_plus=0.1, mu_minus=-0.1)


@pytest.fixture(scope="module")
def lbdp():
    from paper_2202_01631_gb300 import build
    build.build()
    torch.cuda.init()
    from paper_2202_01631_gb300 import lbdp as mod
    return mod


def _values(k):
    rng = np.random.default_rng(100 + k)
    return dict(rho=1.0 + 0.005 * rng.uniform(-1, 1, N ** 3), u=0.01 * rng.uniform(-1, 1, 3 * N ** 3),
                psi=rng.uniform(-1, 1, N ** 3), phi=1.0 + 0.1 * rng.uniform(-1, 1, N ** 3))


@pytest.mark.parametrize("spheres", [0, 1])
@pytest.mark.parametrize("member", [False, True])
def test_pinned_buffer_written_again(lbdp, member, spheres):
    stream = torch.cuda.Stream()
    batch = lbdp.Batch(precision="fp32", arena_bytes=1 << 30, stream=stream.cuda_stream) if member else None

    def make():
        return batch.add_box(**PARAMS) if member else lbdp.Box(precision="fp32", stream=stream.cuda_stream, **PARAMS)

    try:
        busy = make()
        pinned = {k: torch.empty(v.size, dtype=torch.float64, pin_memory=True).numpy()
                  for k, v in _values(0).items()}
        boxes = []
        for k in range(8):
            box = make()
            for name, v in _values(k).items():
                pinned[name][:] = v
            busy.step(400)   # the copies wait behind these
            lbdp.lb_set_fields(box.h, **pinned)
            for v in pinned.values():
                v[:] = np.nan
            for _ in range(spheres):
                box.add_particle(**SPHERE)
            boxes.append(box)
        for k, box in enumerate(boxes):
            ref = lbdp.Box(precision="fp32", **PARAMS)
            ref.set_fields(**_values(k))
            for _ in range(spheres):
                ref.add_particle(**SPHERE)
            a, b = box.fields(), ref.fields()
            assert all(np.array_equal(a[f], b[f]) for f in a), k
            assert np.array_equal(box.populations(), ref.populations()), k
            ref.close()
            if not member:
                box.close()
        if not member:
            busy.close()
    finally:
        if member:
            batch.close()
