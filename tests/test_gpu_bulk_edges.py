"""The bulk kernels at the edges of their tiles, halves and chunks: boxes one
node short of, equal to and one node past a 32 x 8 column tile, chunks of one
plane, of an odd number of planes and of the whole box, spheres and walls on
tile corners, at the periodic wrap and in the planes where a chunk ends.

FP64 against the oracle to 1e-10 (the bar of the parity tests); FP32 against
the same box in FP64 to 1e-4 of the largest value of each field, the bar the
FP32 mode is held to, over 12 steps.
"""
import numpy as np
import pytest

from paper_2202_01631_gb300 import workloads as W
from tests.pair_util import FIELDS, compare, make_pair, norm_rel

pytestmark = pytest.mark.gpu

# (nx, ny, nz), periodic axes, spheres (position, radius), transport scheme
BOXES = [
    ((31, 7, 9), (1, 1, 1), [], 0),
    ((32, 8, 16), (1, 1, 0), [], 1),
    ((33, 9, 5), (0, 1, 1), [], 0),
    ((65, 17, 6), (1, 0, 0), [], 0),
    ((34, 18, 15), (1, 1, 1), [((31.8, 7.6, 0.4), 3.1)], 0),          # tile corner, wrap in z
    ((33, 24, 18), (1, 1, 0), [((0.3, 15.7, 8.6), 3.4)], 1),          # wrap in x
    ((40, 19, 20), (0, 0, 0), [((32.2, 8.1, 5.1), 3.2), ((12.4, 9.7, 13.3), 3.6)], 0),
    ((24, 24, 24), (1, 1, 1), [((11.7, 12.2, 12.4), 3.0), ((12.3, 0.2, 0.7), 3.3)], 0),
]


@pytest.fixture(scope="module")
def lbdp():
    from paper_2202_01631_gb300 import build
    build.build()
    import torch
    torch.cuda.init()
    from paper_2202_01631_gb300 import lbdp as mod
    return mod


def _inputs(case):
    (nx, ny, nz), per, spheres, scheme = case
    params = dict(W.BASE_PARAMS, nx=nx, ny=ny, nz=nz, periodic=per, E=0.3, phi_b=0.5, k_d=2e-3,
                  body_force=(1e-5, -2e-5, 1e-5), scalar_scheme=scheme)
    rng = np.random.default_rng(nx * 1000 + nz)
    z = np.arange(nz)[:, None, None]
    shape = (nz, ny, nx)
    fields = dict(rho=1.0 + 0.005 * rng.uniform(-1, 1, shape), u=0.01 * rng.uniform(-1, 1, (3,) + shape),
                  psi=np.tanh((z - nz / 2 + 0.3) / 2.0) + 0.1 * rng.uniform(-1, 1, shape),
                  phi=0.5 + 0.1 * rng.uniform(-1, 1, shape))
    # an orientation that leaves no node or link midpoint on the plane between
    # the caps, where rounding alone decides the side
    parts = [dict(pos=p, R=R, m_hat=(0.3137, -0.2271, 0.9219), alpha=5e-3, mu_plus=0.1, mu_minus=-0.1,
                  theta_c_deg=65.0 + 20.0 * k) for k, (p, R) in enumerate(spheres)]
    return params, fields, parts


def _planes(nz):
    return [(0, 0), (1, 1), (2, 3), (3, 2), (nz, nz), (max(1, nz - 1), 4)]


@pytest.mark.parametrize("case", BOXES, ids=lambda c: "x".join(map(str, c[0])))
def test_fp64_matches_oracle(lbdp, case):
    params, fields, parts = _inputs(case)
    box, ref = make_pair(params, fields, parts)
    for k, (f, s) in enumerate(_planes(params["nz"])[1:]):   # every step with other chunks
        box.set_planes(f, s)
        box.step(2)
        ref.step(2)
    d = compare(box, ref)
    assert d.pop("mask_mismatch") == 0
    assert all(v <= 1e-10 for v in d.values()), d


@pytest.mark.parametrize("case", BOXES, ids=lambda c: "x".join(map(str, c[0])))
def test_fp32_matches_fp64_in_every_chunk(lbdp, case):
    params, fields, parts = _inputs(case)

    def run(precision, planes):
        b = lbdp.Box(precision=precision, **params)
        b.set_fields(**fields)
        for q in parts:
            b.add_particle(**q)
        b.set_planes(*planes)
        b.step(12)
        return b

    ref = run("fp64", (0, 0))
    first = run("fp32", (0, 0))
    fr, f0, mask = ref.fields(), first.fields(), ref.mask()
    assert np.array_equal(mask, first.mask())
    for k in FIELDS:
        assert norm_rel(f0[k], fr[k], mask) <= 1e-4, k
    pops = first.populations()
    for planes in _planes(params["nz"])[1:]:
        b = run("fp32", planes)
        fb = b.fields()
        assert all(np.array_equal(fb[k], f0[k]) for k in FIELDS), planes
        assert np.array_equal(b.populations(), pops), planes
