"""lb_tune times the chunk lengths that small boxes need: in these, blocks of one or
two planes are the fastest by a fifth or more (FP64 32^3: 128 us at one plane, 270
at four), and the library chooses them by size."""
import numpy as np
import pytest

from paper_2202_01631_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbdp():
    from paper_2202_01631_gb300 import build
    build.build()
    import torch
    torch.cuda.init()
    from paper_2202_01631_gb300 import lbdp as mod
    return mod


@pytest.mark.parametrize("precision,edge", [("fp64", 24), ("fp64", 32), ("fp32", 24)])
def test_small_boxes_keep_short_chunks(lbdp, precision, edge):
    box = lbdp.Box(precision=precision, **dict(W.BASE_PARAMS, nx=edge, ny=edge, nz=edge, periodic=(1, 1, 1), E=0.3))
    z = np.arange(edge)[:, None, None]
    box.set_fields(psi=np.broadcast_to(np.tanh((z - edge / 2) / 2.0), (edge,) * 3))
    box.add_particle(pos=(edge / 2 + 0.3, edge / 2 - 0.2, edge / 2), R=3.2, m_hat=(0.2, 0.4, -1.0))
    assert all(v <= 2 for v in box.planes().values())
    planes, ms = box.tune(reps=20)
    assert box.planes() == planes and all(v <= 3 for v in planes.values()), (planes, ms)
