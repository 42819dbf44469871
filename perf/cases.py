"""The work that users of this framework have it do, as cases to be timed.

A user's program creates a box (or a batch of boxes, or a server), sets the
fields, places the spheres, and then alternates between advancing the box some
steps and reading its fields and particles.  One pass here is one such
segment: ``step(n)`` and the readout, or the submission, service and
collection of a burst of requests.  The state goes on from pass to pass, as a
simulation does.

Fields cross the library's interface in FP64 in every mode.  A program keeps
its snapshots in the precision it computes in, so the outputs here are in the
storage type of the box (``fp64`` float64, ``fp32`` float32, ``fp16``
float16, ``bf16`` bfloat16), in host buffers the program allocates once.

Initial states are what runs start from or come back to: water and oil in
layers (one rippled interface between walls, or a slab of water between two
of them in a fully periodic box), a slow smooth flow, a smooth solute field,
and Janus spheres at the interface or below it.

``exact`` advances the same state in FP64 with plain torch operations.
"""
import math
import random

import numpy as np
import torch

from paper_2202_01631_gb300 import lbdp

TYPES = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}
# Bytes of one node and step that no implementation with the state in memory
# avoids: 19 populations read and written in the storage type, psi and phi
# read and written in the field type (FP64 or FP32).
NODE_BYTES = {"fp64": 336, "fp32": 168, "fp16": 92, "bf16": 92}
# Arithmetic of one node and step, counted from the formulas with shared sums:
# chemical potentials and stress 110, force 130, collide-stream 220, transport 160.
NODE_FLOPS = 620
# the fields of a sphere's state record, as the library returns it
RECORD = ("pos", "vel", "omega", "m_hat", "force", "torque")


def _box(name, edge, precision, steps, layout="interface", walls="z", spheres=1, radius=8.0, theta=90.0, ratio=1.0,
         mobility=0.1, scheme=0, push=0.0):
    nx, ny, nz = edge
    c = dict(form="box", nx=nx, ny=ny, nz=nz, precision=precision, steps=steps, layout=layout, walls=walls,
             spheres=spheres, radius=radius, theta=theta, ratio=ratio, mobility=mobility, scheme=scheme, push=push)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest box the serving mix holds (edge 24): one sphere, a short
        # segment between readouts; launches and kernel latency count
        _box("slab24_fp32", (24, 24, 24), "fp32", 50, layout="slab", walls="", radius=3.0, theta=75.0, ratio=2.0),
        # the 32^3 FP64 configuration that method checks run on
        _box("plain32_fp64", (32, 32, 32), "fp64", 50, layout="bulk", radius=4.0, mobility=0.0),
        # a binary fluid with solute and no sphere: interface relaxation,
        # calibration of the free energy
        _box("fluid64_fp32", (64, 64, 64), "fp32", 100, layout="slab", walls="", spheres=0, ratio=2.0),
        # a driven channel with odd edges, walls on two axes, two spheres
        _box("channel_fp32", (75, 53, 101), "fp32", 50, walls="yz", spheres=2, radius=5.0, theta=60.0, ratio=0.5,
             push=2e-6),
        # the 128^3 interface study (contact angle x solubility x mobility)
        _box("interface128_fp32", (128, 128, 128), "fp32", 50, theta=60.0, ratio=2.0),
        # the same with the lattice-Boltzmann transport of psi and phi
        _box("interface128_lb_fp32", (128, 128, 128), "fp32", 50, theta=120.0, scheme=1),
        # the same with 16-bit population storage
        _box("interface128_fp16", (128, 128, 128), "fp16", 50, theta=90.0, ratio=0.5),
        # FP64 reference runs of the precision studies, periodic on every axis
        _box("slab96_fp64", (96, 96, 96), "fp64", 20, layout="slab", walls="", radius=6.0, theta=110.0, ratio=3.0,
             mobility=-0.1),
        # the benchmark box: 256^3, eight spheres R = 6 below the interface
        _box("precision256_fp32", (256, 256, 256), "fp32", 40, layout="bulk", spheres=8, radius=6.0),
        # a parameter sweep: uneven periodic boxes advanced together
        dict(name="batch48_fp32", form="batch", boxes=48, lo=32, hi=96, precision="fp32", steps=20),
        # a burst of requests at the server: admission, upload, stepping until
        # each is done, readout
        dict(name="serve10_fp32", form="serve", boxes=10, lo=24, hi=64, precision="fp32", steps=40),
    ]


def draw(rng):
    kind = rng.choice(["box"] * 5 + ["batch", "serve"])
    if kind == "batch":
        precision = rng.choice(["fp32", "fp32", "fp64", "fp16"])
        lo = rng.randint(24, 48)
        most, hi = (12, 64) if precision == "fp64" else (44, 90)
        return dict(form="batch", boxes=rng.randint(4, most), lo=lo, hi=rng.randint(lo, hi), precision=precision,
                    steps=rng.randint(8, 20))
    if kind == "serve":
        return dict(form="serve", boxes=rng.randint(2, 12), lo=24, hi=rng.randint(32, 64),
                    precision=rng.choice(["fp32", "fp32", "bf16"]), steps=rng.randint(20, 40))
    precision = rng.choice(["fp32", "fp32", "fp32", "fp64", "fp16", "bf16"])
    top = 144.0 if precision == "fp64" else 224.0
    size = math.exp(rng.uniform(math.log(24.0), math.log(top)))   # edge of the cube of the same volume
    asp = [rng.uniform(0.8, 1.25) for _ in range(3)]
    scale = (asp[0] * asp[1] * asp[2]) ** (-1.0 / 3.0)
    nx, ny, nz = (max(24, int(round(size * a * scale))) for a in asp)
    layout = rng.choice(["interface", "slab", "bulk"])
    walls = "" if layout == "slab" else rng.choice(["z", "z", "yz"])
    small = min(nx, ny, nz)
    rmax = min(8.0, small / 8.0)
    spheres = rng.choice([0, 1, 1, 2]) if small < 64 else rng.choice([0, 1, 2, 4])
    steps = max(10, min(50, int((3e7 if precision == "fp64" else 3e8) / (nx * ny * nz))))
    return _box("", (nx, ny, nz), precision, steps, layout=layout, walls=walls, spheres=spheres,
                radius=round(rng.uniform(min(3.0, rmax), rmax), 2), theta=round(rng.uniform(60.0, 120.0), 1),
                ratio=rng.choice([0.5, 1.0, 2.0]), mobility=rng.choice([-0.1, 0.0, 0.1]),
                scheme=1 if rng.random() < 0.25 else 0, push=rng.choice([0.0, 1e-6]))


# ---------------------------------------------------------------------------
# inputs (from the case and the seed alone)
# ---------------------------------------------------------------------------
def _unit(r):
    v = [r.gauss(0.0, 1.0) for _ in range(3)]
    n = math.sqrt(sum(a * a for a in v))
    return tuple(a / n for a in v)


def _boxes(case):
    """The boxes of a case; the sizes and lengths of a batch or a burst are the case's own."""
    if case["form"] == "box":
        return [case]
    r, out = random.Random("%(form)s %(boxes)d %(lo)d %(hi)d %(steps)d" % case), []
    for _ in range(case["boxes"]):
        edge = r.randint(case["lo"], case["hi"])
        one = _box("", (edge,) * 3, case["precision"], case["steps"],
                   radius=r.uniform(min(4.0, edge / 8.0), min(8.0, edge / 8.0)), theta=r.uniform(60.0, 120.0),
                   ratio=r.uniform(0.5, 2.0), mobility=r.uniform(-0.1, 0.1))
        if case["form"] == "batch":
            one.update(layout="slab", walls="")
        else:   # requests differ in length too
            one.update(steps=int(round(case["steps"] * math.exp(r.uniform(-0.7, 0.7)))),
                       spheres=1 if edge < 40 else r.randint(1, 2))
        out.append(one)
    return out


def _specs(case, seed):
    """[(parameters, particles, steps, seed of the fields)] of the boxes of a case."""
    r = random.Random(seed)
    return [_spec(c, r) for c in _boxes(case)]


def _spec(c, r):
    n = (c["nx"], c["ny"], c["nz"])
    phi_b = 0.0 if c["ratio"] == 1.0 else 1.0
    params = dict(nx=n[0], ny=n[1], nz=n[2], periodic=tuple(0 if a in c["walls"] else 1 for a in "xyz"),
                  tau=1.0, rho0=1.0, body_force=(c["push"], 0.0, 0.0), thermo_force=1, A=0.0625, kappa=0.04,
                  M_psi=0.1, C=0.0625, M_phi=1.6, E=phi_b * (c["ratio"] - 1) / ((c["ratio"] + 1) * math.tanh(1.0)),
                  phi_b=phi_b, k_d=1e-3, scalar_scheme=c["scheme"])
    z0 = n[2] / 4.0 if c["layout"] == "slab" else n[2] / 2.0   # the (lower) interface
    parts = []
    for _ in range(100000):
        if len(parts) == c["spheres"]:
            break
        R = c["radius"]
        pos = [r.uniform(0.0, n[0] - 1e-6), r.uniform(0.0, n[1] - 1e-6), z0 + 0.3 + r.uniform(-0.3, 0.3) * R]
        if c["layout"] == "bulk":
            pos[2] = r.uniform(min(n[2] * 0.08 + R + 3.0, z0 - R), max(n[2] * 0.23, R + 4.0))
        for a in range(3):
            if not params["periodic"][a]:
                pos[a] = min(max(pos[a], R + 4.0), n[a] - 1.0 - R - 4.0)
        near = False
        for q in parts:
            d = [pos[a] - q["pos"][a] for a in range(3)]
            d = [d[a] - n[a] * round(d[a] / n[a]) if params["periodic"][a] else d[a] for a in range(3)]
            near = near or math.sqrt(sum(x * x for x in d)) < 2.0 * R + 8.0
        if not near:
            parts.append(dict(pos=tuple(pos), R=R, m_hat=_unit(r), alpha=1e-3, mu_plus=c["mobility"],
                              mu_minus=c["mobility"], theta_c_deg=c["theta"], rho_p=1.0))
    assert len(parts) == c["spheres"], "the spheres do not fit"
    return params, parts, c["steps"], r.getrandbits(40)


def _fields(params, seed, device="cuda"):
    """rho, u, psi, phi of the initial state as FP64 tensors [nz][ny][nx]."""
    r = random.Random(seed)
    n = (params["nx"], params["ny"], params["nz"])
    ax = [torch.arange(n[a], dtype=torch.float64, device=device) for a in range(3)]
    x, y, z = ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]

    def wave(c, a):
        k = r.randint(1, 2)
        return torch.sin(2.0 * math.pi * k * c / n[a] + r.uniform(0.0, 2.0 * math.pi))

    fade = 1.0   # no flow at walls
    for c, a in ((x, 0), (y, 1), (z, 2)):
        if not params["periodic"][a]:
            fade = fade * torch.sin(math.pi * (c + 0.5) / n[a])
    ripple = 0.5 * wave(x, 0) * wave(y, 1)
    if params["periodic"][2]:
        psi = torch.tanh((z - n[2] / 4.0 - ripple) / 2.0) - torch.tanh((z - 3.0 * n[2] / 4.0 + ripple) / 2.0) - 1.0
    else:
        psi = torch.tanh((z - n[2] / 2.0 - ripple) / 2.0)
    phi = params["phi_b"] + params["E"] * torch.tanh(psi) + 0.05 * wave(x, 0) * wave(y, 1) * wave(z, 2)
    rho = 1.0 + 0.001 * wave(x, 0) * wave(y, 1) * wave(z, 2)
    full = (n[2], n[1], n[0])
    u = torch.stack([(0.002 * wave(y, 1) * wave(z, 2) * fade).expand(full),
                     (0.002 * wave(z, 2) * wave(x, 0) * fade).expand(full),
                     (0.002 * wave(x, 0) * wave(y, 1) * fade).expand(full)])
    return rho.expand(full).contiguous(), u, psi.expand(full).contiguous(), phi.expand(full).contiguous()


# ---------------------------------------------------------------------------
# what a user's program holds, and one pass
# ---------------------------------------------------------------------------
class _Host:
    """FP64 host buffers the library reads into, and the program's snapshots."""

    def __init__(self, nodes, parts, dtype, flow=True):
        names = ("rho", "u", "psi", "phi") if flow else ("psi", "phi")
        size = {k: (3 if k == "u" else 1) * nodes for k in names}
        self.raw = {k: torch.empty(v, dtype=torch.float64, pin_memory=True) for k, v in size.items()}
        self.out = {k: torch.empty(v, dtype=dtype) for k, v in size.items()}
        for k in names:
            self.raw[k].zero_()
            self.out[k].zero_()
        self.np = {k: v.numpy() for k, v in self.raw.items()}
        self.dtype, self.parts = dtype, parts

    def snapshot(self, states):
        """Fields in the run's precision; the state record and the motion of every sphere."""
        for k, v in self.raw.items():
            self.out[k].copy_(v)
        got = dict(self.out)
        if self.parts:
            for name, keys in (("particles", RECORD), ("motion", RECORD[1:3])):
                a = np.array([[s[k] for k in keys] for s in states])
                got[name] = torch.from_numpy(a).to(self.dtype)
        return got


def _setup(box, params, parts, seed):
    rho, u, psi, phi = (t.cpu().numpy() for t in _fields(params, seed))
    box.set_fields(rho=rho, u=u, psi=psi, phi=phi)
    for d in parts:
        box.add_particle(**d)


def _granules(params, precision):
    return lbdp.lb_device_bytes(lbdp.box_params(precision, None, **params)) + 4096


def prepare(case, seed):
    specs = _specs(case, seed)
    prec, dtype = case["precision"], TYPES[case["precision"]]
    nodes = [p["nx"] * p["ny"] * p["nz"] for p, _, _, _ in specs]
    parts = sum(len(q) for _, q, _, _ in specs)
    if case["form"] == "box":
        params, q, _, fseed = specs[0]
        box = lbdp.Box(precision=prec, **params)
        _setup(box, params, q, fseed)
        box.sync()
        return dict(case=case, box=box, host=_Host(nodes[0], parts, dtype))
    arena = sum(_granules(p, prec) for p, _, _, _ in specs)
    if case["form"] == "batch":
        batch = lbdp.Batch(precision=prec, arena_bytes=arena)
        boxes = []
        for params, q, _, fseed in specs:
            boxes.append(batch.add_box(**params))
            _setup(boxes[-1], params, q, fseed)
        batch.sync()
        host = _Host(sum(nodes), parts, dtype)
        return dict(case=case, batch=batch, boxes=boxes, host=host, nodes=nodes)
    host = _Host(sum(nodes), parts, dtype, flow=False)
    server = lbdp.Server(precision=prec, arena_bytes=arena)
    requests, at = [], 0
    for (params, q, steps, fseed), N in zip(specs, nodes):
        _, _, psi, phi = (t.cpu().numpy() for t in _fields(params, fseed))
        requests.append(dict(box=params, particles=q, psi=psi, phi=phi, steps=steps,
                             out_psi=host.np["psi"][at:at + N], out_phi=host.np["phi"][at:at + N]))
        at += N
    return dict(case=case, server=server, requests=requests, host=host)


def run(state):
    case, host = state["case"], state["host"]
    if case["form"] == "box":
        box = state["box"]
        box.step(case["steps"])
        lbdp.lb_read_fields(box.h, **host.np)
        return host.snapshot(box.particles() if host.parts else [])
    if case["form"] == "batch":
        batch, boxes = state["batch"], state["boxes"]
        for b in boxes:
            batch.set_steps(b, case["steps"])
        batch.run(case["steps"])
        states, at, total = [], 0, host.np["rho"].size
        u = host.np["u"].reshape(-1)
        for b, N in zip(boxes, state["nodes"]):
            lbdp.lb_read_fields(b.h, host.np["rho"][at:at + N], u[3 * at:3 * (at + N)], host.np["psi"][at:at + N],
                                host.np["phi"][at:at + N])
            states += b.particles()
            at += N
        assert at == total
        return host.snapshot(states)
    server = state["server"]
    ids = [server.submit(**r) for r in state["requests"]]
    done = {}
    while len(done) < len(ids):
        server.pump(0.0)
        for r in server.poll():
            if r["status"] != lbdp.LB_OK:
                raise lbdp.LbError(r["status"], "request")
            done[r["id"]] = r
    return host.snapshot([s for i in ids for s in done[i]["particles"]])


def work(case):
    nb, out = NODE_BYTES[case["precision"]], TYPES[case["precision"]].itemsize
    fields = 2 if case["form"] == "serve" else 6
    nodes = [(c["nx"] * c["ny"] * c["nz"], c["steps"]) for c in _boxes(case)]
    done = sum(n * t for n, t in nodes)
    return dict(bytes=done * nb + sum(n for n, _ in nodes) * fields * out, flops=done * NODE_FLOPS)


# ---------------------------------------------------------------------------
# the same in 64 bits, with torch alone
# ---------------------------------------------------------------------------
_C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
      (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
      (0, -1, 1)]
_W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
_OPP = [0] + [i + 1 if i % 2 else i - 1 for i in range(1, 19)]


def _cdot(i, v):
    """c_i . v for v of three tensors; None when c_i is zero."""
    s = None
    for a in range(3):
        if _C[i][a]:
            t = v[a] if _C[i][a] > 0 else -v[a]
            s = t if s is None else s + t
    return s


def _wetting_h(theta):
    lo, hi, want = -1.0, 1.0, math.cos(math.radians(theta))
    for _ in range(100):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if 0.5 * ((1 + mid) ** 1.5 - (1 - mid) ** 1.5) < want else (lo, mid)
    return 0.5 * (lo + hi)


class _Exact:
    """One box, FP64, one plain tensor operation after the other."""

    def __init__(self, params, parts, fields):
        self.p = params
        self.n = (params["nx"], params["ny"], params["nz"])
        nx, ny, nz = self.n
        self.N = nx * ny * nz
        self.dev = fields[2].device
        self.axes = [torch.arange(k, device=self.dev) for k in self.n]
        node = torch.arange(self.N, device=self.dev)
        self.xyz = (node % nx, (node // nx) % ny, node // (nx * ny))
        self.nb, self.wall = [node], [None]   # neighbour (itself beyond a wall), and where a wall is
        for i in range(1, 19):
            c, out = [], torch.zeros(self.N, dtype=torch.bool, device=self.dev)
            for a in range(3):
                v = self.xyz[a] + _C[i][a]
                if not params["periodic"][a]:
                    out |= (v < 0) | (v >= self.n[a])
                c.append(v % self.n[a])
            self.nb.append(torch.where(out, node, c[0] + nx * (c[1] + ny * c[2])))
            self.wall.append(out if bool(out.any()) else None)
        self.rho0 = params["rho0"]
        rho, u, psi, phi = fields
        self.psi, self.phi, self.u = psi.reshape(-1).clone(), phi.reshape(-1).clone(), u.reshape(3, -1).clone()
        self.mask = torch.zeros(self.N, dtype=torch.int64, device=self.dev)
        self.f = self._feq(rho.reshape(-1), self.u)
        self.cvec = torch.tensor(_C, dtype=torch.float64, device=self.dev)
        self.wvec = torch.tensor(_W, dtype=torch.float64, device=self.dev)
        self.np = len(parts)
        arr = lambda k: np.array([q[k] for q in parts], dtype=np.float64)   # noqa: E731
        if self.np:
            self.X, self.m, self.R = arr("pos"), arr("m_hat"), arr("R")
            self.m /= np.linalg.norm(self.m, axis=1)[:, None]
            self.M = arr("rho_p") * 4.0 / 3.0 * math.pi * self.R ** 3
            self.I = 0.4 * self.M * self.R ** 2
            self.V, self.imp, self.load = (np.zeros((self.np, 6)) for _ in range(3))
            self.alpha, self.mup, self.mum = arr("alpha"), arr("mu_plus"), arr("mu_minus")
            self.Hk = np.array([_wetting_h(q["theta_c_deg"]) * math.sqrt(params["kappa"] * params["A"])
                                / params["kappa"] for q in parts])
            self.mask = self._owners(self._around(4))
            inside = self.mask != 0
            self.f[:, inside] = 0.0
            self.u[:, inside] = 0.0
            self.psi[inside] = 0.0
            self.phi[inside] = 0.0

    def _t(self, a):
        return torch.as_tensor(a, device=self.dev)

    def _feq(self, rho, u):
        uu = (u * u).sum(0)
        f = torch.empty((19, self.N if rho.numel() == self.N else rho.numel()), dtype=torch.float64, device=self.dev)
        f[0] = _W[0] * rho * (1.0 - 1.5 * uu)
        for i in range(1, 19):
            cu = _cdot(i, u)
            f[i] = _W[i] * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu)
        return f

    def _around(self, more):
        """Nodes within R + more of any sphere's centre, per axis (a superset of what is asked of them)."""
        got = []
        for k in range(self.np):
            ax = []
            for a in range(3):
                lo, hi = math.floor(self.X[k, a] - self.R[k]) - more, math.ceil(self.X[k, a] + self.R[k]) + more
                v = torch.arange(lo, hi + 1, device=self.dev)
                ax.append(torch.unique(v % self.n[a]) if self.p["periodic"][a] else v[(v >= 0) & (v < self.n[a])])
            got.append((ax[0][None, None, :] + self.n[0] * (ax[1][None, :, None] + self.n[1] * ax[2][:, None, None])).reshape(-1))
        return torch.unique(torch.cat(got))

    def _offset(self, nodes, X):
        """x - X, nearest image, for nodes [M] and centres [M][3] (or one of them)."""
        d = []
        for a in range(3):
            v = self.xyz[a][nodes].double() - X[..., a]
            if self.p["periodic"][a]:
                L = float(self.n[a])
                v = torch.where(v > 0.5 * L, v - L, torch.where(v < -0.5 * L, v + L, v))
            d.append(v)
        return torch.stack(d, 1)

    def _owners(self, nodes):
        mask = torch.zeros_like(self.mask)
        for k in reversed(range(self.np)):
            d = self._offset(nodes, self._t(self.X[k]))
            mask[nodes[(d * d).sum(1) < self.R[k] ** 2]] = k + 1
        return mask

    def _links(self):
        """Links from fluid nodes into spheres: node, direction, sphere."""
        near = self._around(2)
        near = near[self.mask[near] == 0]
        n, i, k = [], [], []
        for d in range(1, 19):
            s = self.mask[self.nb[d][near]]
            if self.wall[d] is not None:
                s = torch.where(self.wall[d][near], 0, s)
            at = torch.nonzero(s)[:, 0]
            n.append(near[at])
            i.append(torch.full_like(at, d))
            k.append(s[at] - 1)
        return torch.cat(n), torch.cat(i), torch.cat(k)

    def step(self):
        p, N, nb, fluid = self.p, self.N, self.nb, self.mask == 0
        A, kap, C, E, tau = p["A"], p["kappa"], p["C"], p["E"], p["tau"]
        psi, phi, f = self.psi, self.phi, self.f
        stop = [None]   # no fluid neighbour that way
        for i in range(1, 19):
            b = self.mask[nb[i]] != 0 if self.np else None
            w = self.wall[i]
            stop.append(b if w is None else w if b is None else b | w)
        if self.np:
            ln, li, lk = self._links()
            c, w6 = self.cvec[li], 6.0 * self.wvec[li]
            r = self._offset(ln, self._t(self.X)[lk]) + 0.5 * c
            nh = r / r.norm(dim=1, keepdim=True)
        # chemical potentials and stress
        lap = torch.zeros_like(psi)
        g = torch.zeros((3, N), dtype=torch.float64, device=self.dev)
        for i in range(1, 19):
            d = psi[nb[i]] - psi
            if stop[i] is not None:
                d = torch.where(stop[i], 0.0, d)
            if self.np:
                at = li == i
                d[ln[at]] = self._t(self.Hk)[lk[at]] * (c[at] * nh[at]).sum(1)
            lap += 6.0 * _W[i] * d
            for a in range(3):
                if _C[i][a]:
                    g[a] += 3.0 * _W[i] * _C[i][a] * d
        phi0 = p["phi_b"] + E * torch.tanh(psi)
        dph = phi - phi0
        mps = A * (psi ** 3 - psi) - kap * lap - C * E * dph / torch.cosh(psi) ** 2
        mph = C * dph
        iso = psi * mps + phi * mph - (0.25 * A * psi ** 4 - 0.5 * A * psi ** 2 + 0.5 * C * dph * dph) - 0.5 * kap * (g * g).sum(0)
        # spheres: link sums, implicit velocity update
        if self.np:
            bn, inv = torch.unique(ln, return_inverse=True)
            gp = torch.zeros((bn.numel(), 3), dtype=torch.float64, device=self.dev)
            for i in range(1, 19):
                v = torch.where(stop[i][bn], phi[bn], phi[nb[i][bn]])
                gp += 3.0 * _W[i] * v[:, None] * self.cvec[i]
            gp = gp[inv]
            mu = torch.where((self._t(self.m)[lk] * r).sum(1) <= 0.0, self._t(self.mum)[lk], self._t(self.mup)[lk])
            vs = mu[:, None] * (gp - nh * (nh * gp).sum(1, keepdim=True))
            gl = g[:, ln].T
            dP = c * (2.0 * f[li, ln] - w6 * self.rho0 * (c * vs).sum(1))[:, None]
            dP = dP + w6[:, None] * (iso[ln][:, None] * c + kap * gl * (gl * c).sum(1, keepdim=True))
            g6 = torch.cat([c, torch.linalg.cross(r, c)], 1)
            F0 = torch.zeros((self.np, 6), dtype=torch.float64, device=self.dev)
            F0.index_add_(0, lk, torch.cat([dP, torch.linalg.cross(r, dP)], 1))
            Z = torch.zeros((self.np, 6, 6), dtype=torch.float64, device=self.dev)
            Z.index_add_(0, lk, (w6 * self.rho0)[:, None, None] * g6[:, :, None] * g6[:, None, :])
            rhs, Z = F0.cpu().numpy() + self.imp, Z.cpu().numpy()
            for k in range(self.np):
                Md = np.array([self.M[k]] * 3 + [self.I[k]] * 3)
                self.V[k] = np.linalg.solve(np.diag(Md) + Z[k], Md * self.V[k] + rhs[k])
                self.load[k] = rhs[k] - Z[k] @ self.V[k]
            self.imp = np.zeros((self.np, 6))
            V = self._t(self.V)[lk]
            cub = (c * (V[:, :3] + torch.linalg.cross(V[:, 3:].contiguous(), r) + vs)).sum(1)
        # force
        F = torch.zeros((3, N), dtype=torch.float64, device=self.dev)
        for i in range(1, 19):
            def at(v):
                return v[nb[i]] if stop[i] is None else torch.where(stop[i], v, v[nb[i]])
            gi, pi = [at(g[a]) for a in range(3)], at(iso)
            ks = kap * _cdot(i, gi)
            for a in range(3):
                F[a] -= 3.0 * _W[i] * (ks * gi[a] + (_C[i][a] * pi if _C[i][a] else 0.0))
        for a in range(3):
            F[a] += p["body_force"][a]
        # streaming, collision
        fl = torch.empty_like(f)
        fl[0] = f[0]
        for j in range(1, 19):
            i = _OPP[j]
            fl[j] = f[j][nb[i]] if stop[i] is None else torch.where(stop[i], f[i], f[j][nb[i]])
        if self.np:
            fl[self._t(np.array(_OPP))[li], ln] = f[li, ln] - w6 * self.rho0 * cub
        rho = torch.where(fluid, fl.sum(0), 1.0)
        u = 0.5 * F
        for i in range(1, 19):
            for a in range(3):
                if _C[i][a]:
                    u[a] += _C[i][a] * fl[i]
        u /= rho
        uF, omf = (u * F).sum(0), 1.0 - 0.5 / tau
        feq = self._feq(rho, u)
        for i in range(19):
            S = -3.0 * uF
            if i:
                cF = _cdot(i, F)
                S = S + 3.0 * cF + 9.0 * _cdot(i, u) * cF
            fl[i] += (feq[i] - fl[i]) / tau + omf * _W[i] * S
        fl *= fluid
        u *= fluid
        self.f, self.u = fl, u
        # transport
        dps, dpf = torch.zeros_like(psi), torch.zeros_like(phi)
        lb = p["scalar_scheme"] == 1
        for i in range(1, 7 if lb else 19):
            cu0, ui = _cdot(i, u), [u[a][nb[i]] for a in range(3)]
            cu1 = _cdot(i, ui)
            for acc, s, mu_, mob in ((dps, psi, mps, p["M_psi"]), (dpf, phi, mph, p["M_phi"])):
                sn = s[nb[i]]
                t = mob * (mu_[nb[i]] - mu_)
                if lb:
                    t = t - 0.5 * sn * cu1
                    other = 0.5 * s * cu0
                else:
                    ub = 0.5 * (cu0 + cu1)
                    t = 6.0 * _W[i] * (t - torch.where(ub > 0, ub * s, ub * sn))
                    other = 0.0
                acc += t if stop[i] is None else torch.where(stop[i], other, t)
        carried = np.zeros(2)
        if self.np:
            wl = torch.where(li < 7, 1.0, 0.0).double() if lb else w6
            for k, (acc, s) in enumerate(((dps, psi), (dpf, phi))):
                out = wl * cub * s[ln]
                acc.index_add_(0, ln, -out)
                carried[k] = float(out.sum())
            pairs = torch.unique(ln * 64 + lk)   # a node next to a sphere: production on the cap
            pn, pk = pairs // 64, pairs % 64
            cap = (self._t(self.m)[pk] * self._offset(pn, self._t(self.X)[pk])).sum(1) <= 0.0
            dpf.index_add_(0, pn, torch.where(cap, self._t(self.alpha)[pk], 0.0))
        self.psi = (psi + dps) * fluid
        self.phi = (phi + dpf - p["k_d"] * (phi - phi0)) * fluid
        if self.np:
            self._move(carried)

    def _move(self, short):
        near = [self._around(4)]
        for k in range(self.np):
            X = self.X[k] + self.V[k, :3]
            for a in range(3):
                if self.p["periodic"][a]:
                    X[a] += self.n[a] if X[a] < 0 else -self.n[a] if X[a] >= self.n[a] else 0.0
            self.X[k] = X
            w = self.V[k, 3:]
            ang = math.sqrt(float(w @ w))
            if ang > 0.0:
                e, m = w / ang, self.m[k]
                m = m * math.cos(ang) + np.cross(e, m) * math.sin(ang) + e * float(e @ m) * (1.0 - math.cos(ang))
                self.m[k] = m / np.linalg.norm(m)
        near.append(self._around(4))
        old, new = self.mask, self._owners(torch.unique(torch.cat(near)))
        changed = torch.nonzero(old != new)[:, 0]
        for n in changed.tolist():
            o, q = int(old[n]), int(new[n])
            one = torch.tensor([n], device=self.dev)
            k = (q or o) - 1
            d = self._offset(one, self._t(self.X[k]))[0].cpu().numpy()
            if q:
                j = (self.cvec.T @ self.f[:, n]).cpu().numpy()
                self.imp[k] += np.concatenate([j, np.cross(d, j)])
                short += np.array([float(self.psi[n]), float(self.phi[n])])
                self.f[:, n], self.u[:, n], self.psi[n], self.phi[n] = 0.0, 0.0, 0.0, 0.0
            else:
                m = torch.tensor([int(self.nb[i][n]) for i in range(1, 19)
                                  if self.wall[i] is None or not bool(self.wall[i][n])], device=self.dev)
                m = m[(old[m] == 0) & (new[m] == 0)]
                rb, pb, hb = float(self.f[:, m].sum(0).mean()), float(self.psi[m].mean()), float(self.phi[m].mean())
                ub = self.V[k, :3] + np.cross(self.V[k, 3:], d)
                self.f[:, n] = self._feq(self._t(np.array([rb])), self._t(ub)[:, None])[:, 0]
                self.u[:, n], self.psi[n], self.phi[n] = self._t(ub), pb, hb
                self.imp[k] -= np.concatenate([rb * ub, np.cross(d, rb * ub)])
                short -= np.array([pb, hb])
        self.mask = new
        fluid = new == 0
        count = float(fluid.sum())
        self.psi = torch.where(fluid, self.psi + short[0] / count, 0.0)
        self.phi = torch.where(fluid, self.phi + short[1] / count, 0.0)


def exact(case, seed):
    flow = case["form"] != "serve"
    got = {k: [] for k in (("rho", "u", "psi", "phi") if flow else ("psi", "phi"))}
    body = {"particles": [], "motion": []}
    for params, parts, steps, fseed in _specs(case, seed):
        fields = _fields(params, fseed, "cuda" if torch.cuda.is_available() else "cpu")
        if not flow:   # a request starts from rest
            fields = (torch.ones_like(fields[0]), torch.zeros_like(fields[1])) + fields[2:]
        s = _Exact(params, parts, fields)
        for _ in range(steps):
            s.step()
        for k in got:
            got[k].append((s.f.sum(0) if k == "rho" else getattr(s, k).reshape(-1)).cpu())
        if parts:
            V, load = s.V.reshape(-1, 2, 3), s.load.reshape(-1, 2, 3)
            body["particles"].append(np.stack([s.X, V[:, 0], V[:, 1], s.m, load[:, 0], load[:, 1]], 1))
            body["motion"].append(V)
        del s
    out = {k: torch.cat(v) for k, v in got.items()}
    out.update({k: torch.from_numpy(np.concatenate(v)) for k, v in body.items() if v})
    return out
