"""Performance cases of the colloid-in-liquid-crystal solver and of its learned warm start.

A case is a dict of plain values; ``prepare`` builds what a program holds before the call (solver handles, device
tensors, the network), ``run`` makes one pass through the public entry points, ``exact`` gives the same outputs from
plain 64-bit torch.  Fields that come from an FP32 box are returned as FP32, and what comes from the BF16 network as
BF16: the precision that the handle or the network holds them in.  FP64 boxes return FP64.
"""
from __future__ import annotations

import functools
import math
import random

import numpy as np
import torch

import paper_1102_2193_gb300 as P
from paper_1102_2193_gb300.surrogate import LAYERS, UNet

# Constants of the flow-coupled workloads and those of the relaxations (flow frozen).
COUPLED = dict(rho0=1.0, tau=2.5, A0=0.01, gamma=3.0, K=0.01, xi=0.7, Gamma=0.5)
RELAX = dict(rho0=1.0, tau=2.5, A0=1.0, gamma=3.0, K=0.065, xi=0.7, Gamma=0.5)
LOOPS = 512  # rows of the defect-loop table that the analysis returns (zeros after the last loop)


def listed():
    return [
        # the smallest box: a 32^3 FP64 nematic with a planar colloid, stepped between two samples of the fields
        # (validation runs in FP64; launches and latency set its time)
        box("nematic32_f64", 32, 32, 32, precision="f64", steps=20, colloids=1, radius=4.0, planar=True),
        # two colloids of both anchorings in a small cholesteric box of odd, ragged sides
        box("two_colloids_37x29x23", 37, 29, 23, steps=20, pitch=18.5, colloids=2, radius=4.2),
        # microrheology: a mobile planar colloid pulled between walls, sampled every 50 steps
        box("micro64_mobile", 64, 64, 64, walls=True, steps=50, colloids=1, radius=8.0, planar=True, mobile=True),
        # the headline workload: 128^3 cholesteric, pitch 32, a weakly normal colloid of radius 8
        box("chol128_R8", 128, 128, 128, steps=20, pitch=32.0, colloids=1, radius=8.0),
        # the largest box: fields far larger than L2, large planar colloids
        box("nematic256x192x160", 256, 192, 160, steps=4, colloids=2, radius=20.0, planar=True),
        # odd width between walls: the general (one node per thread) path on a mid-size box
        box("walled_95x77x63", 95, 77, 63, walls=True, steps=10, pitch=31.0, colloids=1, radius=9.5),
        # FP64 storage of a coupled cholesteric with a strongly anchored colloid
        box("chol64_f64", 64, 64, 64, precision="f64", steps=5, pitch=32.0, colloids=1, radius=8.0, strong=True),
        # a parameter sweep: uneven boxes advanced together
        dict(name="sweep16_32to96", kind="batch", boxes=16, lo=32, hi=96, geometry=4, steps=10),
        # relaxation towards the defect structure, flow frozen, residual checked every 100 steps
        dict(name="relax96", kind="relax", n=96, pitch=32.0, radius=4.0, precision="f32", steps=200, every=100),
        # analysis of a stored state: defect loops and labels, diagnostics, density, velocity
        dict(name="analyse128", kind="analyse", nx=128, ny=128, nz=128, radius=8.0, precision="f32"),
        # inference of the warm start on a 128^3 box
        dict(name="warm_infer128", kind="infer", S=128, radius=12.0, pitch=32.0),
        # one training step of the warm start on a 64^3 box
        dict(name="warm_train64", kind="train", S=64, radius=10.0, pitch=32.0),
    ]


def box(name, nx, ny, nz, walls=False, precision="f32", steps=10, pitch=0.0, colloids=1, radius=5.0, planar=False,
        strong=False, mobile=False):
    """One box stepped ``steps`` times, then its order parameter and velocity read."""
    c = dict(name=name, kind="step", nx=nx, ny=ny, nz=nz, walls=walls, precision=precision, steps=steps, pitch=pitch,
             colloids=colloids, radius=radius, planar=planar, strong=strong, mobile=mobile)
    return {k: v for k, v in c.items() if v is not None}


def draw(rng):
    """Another case of the same ranges: sides log-uniform, odd ones among them."""
    def side(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step", "step", "step", "mobile", "f64", "batch", "relax", "analyse", "infer", "train"])
    if kind in ("step", "mobile", "f64"):
        hi = 200 if kind == "step" else 96
        n = [side(24, hi) for _ in range(3)]
        if rng.random() < 0.6:
            n[0] += n[0] % 2
        nodes = n[0] * n[1] * n[2]
        walls = kind == "mobile" or rng.random() < 0.3
        most = {"f64": 2e6, "step": 3e7, "mobile": 1e7}[kind]
        return box(None, *n, walls=walls, precision="f64" if kind == "f64" else "f32",
                   steps=max(2, min(50, int(most / nodes))), pitch=rng.choice([0.0, round(rng.uniform(16, 48), 2)]),
                   colloids=1 if kind == "mobile" else rng.choice([1, 1, 2]),
                   radius=round(rng.uniform(2.5, 0.18 * min(n)), 2), planar=rng.random() < 0.5,
                   strong=rng.random() < 0.3, mobile=kind == "mobile")
    if kind == "batch":
        return dict(kind="batch", boxes=rng.randint(3, 16), lo=24, hi=rng.choice([48, 72, 96]),
                    geometry=rng.randrange(10**6), steps=rng.randint(4, 10))
    if kind == "relax":
        n = side(32, 96)
        return dict(kind="relax", n=n, pitch=round(n / rng.randint(1, 3), 3), radius=round(rng.uniform(3, 0.15 * n), 2),
                    precision="f32" if n > 48 else rng.choice(["f32", "f64"]), steps=rng.randint(20, 200),
                    every=rng.choice([50, 100]))
    if kind == "analyse":
        n = [side(32, 136) for _ in range(3)]
        return dict(kind="analyse", nx=n[0], ny=n[1], nz=n[2], radius=round(rng.uniform(2.5, 0.2 * min(n)), 2),
                    precision=rng.choice(["f32", "f64"]))
    S = 4 * rng.randint(4, 28 if kind == "infer" else 16)
    return dict(kind=kind, S=S, radius=round(rng.uniform(3, S / 4), 2), pitch=float(S))


# ---------------------------------------------------------------------------
# inputs (made on the GPU from the seed)
# ---------------------------------------------------------------------------
def generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def grid_axes(nx, ny, nz):
    ax = [torch.arange(n, dtype=torch.float64, device="cuda") for n in (nz, ny, nx)]
    return torch.meshgrid(*ax, indexing="ij")  # z, y, x


def uniaxial(order, n):
    """Q = order (n n - I/3), components xx, xy, xz, yy, yz."""
    return torch.stack([order * (n[0] * n[0] - 1 / 3), order * n[0] * n[1], order * n[0] * n[2],
                        order * (n[1] * n[1] - 1 / 3), order * n[1] * n[2]])


def start_q(nx, ny, nz, pitch, seed, amp=1e-3):
    """Bulk order 1/2: a helix of the pitch along z, or a tilted nematic (pitch 0), with seeded noise."""
    z, y, x = grid_axes(nx, ny, nz)
    if pitch > 0:
        ph = 2 * math.pi / pitch * z
        n = (torch.cos(ph), torch.sin(ph), torch.zeros_like(ph))
    else:
        d = np.array([0.3, 0.2, 1.0])
        n = [torch.full_like(z, float(v)) for v in d / np.linalg.norm(d)]
    q = uniaxial(0.5, n)
    return q + amp * (2 * torch.rand(q.shape, dtype=torch.float64, device="cuda", generator=generator(seed)) - 1)


def texture_q(nx, ny, nz, seed, modes=6, core=0.35):
    """A smooth periodic texture with disclination lines: the director turns by pi around the zeros of a random
    complex field of few Fourier modes, and the order falls to zero there, as in a relaxed defect structure."""
    g = random.Random(seed)
    z, y, x = grid_axes(nx, ny, nz)
    re, im = torch.zeros_like(z), torch.zeros_like(z)
    for _ in range(modes):
        k = [g.randint(-3, 3) for _ in range(3)]
        ph = 2 * math.pi * (k[0] * x / nx + k[1] * y / ny + k[2] * z / nz) + g.uniform(0, 2 * math.pi)
        a = g.uniform(0.5, 1.0)
        re, im = re + a * torch.cos(ph), im + a * torch.sin(ph)
    r = torch.sqrt(re * re + im * im)
    half = 0.5 * torch.atan2(im, re)
    n = (torch.cos(half), torch.sin(half), torch.zeros_like(half))
    q = uniaxial(0.5 * r / torch.sqrt(r * r + core * core), n)
    return q + 1e-4 * (2 * torch.rand(q.shape, dtype=torch.float64, device="cuda", generator=generator(seed)) - 1)


def colloids_of(c):
    """(position, radius, planar, w, mobile, external force) of the case's colloids; w = inf is strong anchoring."""
    n = (c["nx"], c["ny"], c["nz"])
    w = math.inf if c["strong"] else 0.02
    fr = [(0.487, 0.513, 0.479)] if c["colloids"] == 1 else [(0.281, 0.262, 0.292), (0.763, 0.741, 0.728)]
    force = (1e-4, 4e-5, 0.0) if c["mobile"] else (0.0, 0.0, 0.0)
    return [dict(X=tuple(f * (L - 1) for f, L in zip(fr[k], n)), a0=c["radius"], planar=c["planar"] ^ (k == 1),
                 w=math.inf if k == 1 else w, mobile=c["mobile"], F=force) for k in range(c["colloids"])]


def sweep_of(c):
    """The boxes of a sweep: cubic sides in steps of 8, one centred colloid each, the phase, anchoring and w drawn."""
    g = random.Random(c["geometry"])
    out = []
    for _ in range(c["boxes"]):
        L = g.randrange(c["lo"], c["hi"] + 1, 8)
        pitch = g.choice([0.0, float(L), L / 2.0])
        out.append(dict(nx=L, ny=L, nz=L, walls=False, precision="f32", pitch=pitch, colloids=1,
                        radius=g.uniform(3.0, 0.28 * L), planar=g.random() < 0.5, strong=False, mobile=False))
    return out


def params_of(pitch, base, flow=True):
    return dict(base, q0=2 * math.pi / pitch if pitch > 0 else 0.0, flow=flow)


def add_colloids(solver, cols):
    for k in cols:
        solver.add_colloid(k["X"], k["a0"], P.LC_PLANAR if k["planar"] else P.LC_NORMAL, k["w"], mobile=k["mobile"],
                           F_ext=k["F"])


def storage(c):
    return (P.LC_FP64, torch.float64) if c.get("precision") == "f64" else (P.LC_FP32, torch.float32)


def field(nc, c):
    return torch.empty((nc, c["nz"], c["ny"], c["nx"]), dtype=torch.float64, device="cuda")


def analyse_box(c):
    return dict(c, walls=False, pitch=0.0, colloids=1, planar=True, strong=False, mobile=False)


def relax_box(c):
    return dict(nx=c["n"], ny=c["n"], nz=c["n"], walls=False, precision=c["precision"], pitch=c["pitch"], colloids=1,
                radius=c["radius"], planar=False, strong=False, mobile=False)


def random_f(c, seed):
    """Populations around rest with the deviations of a slow flow."""
    w = torch.tensor(W, dtype=torch.float64, device="cuda").reshape(19, 1, 1, 1)
    d = torch.rand((19, c["nz"], c["ny"], c["nx"]), dtype=torch.float64, device="cuda", generator=generator(seed + 1))
    return w * (1.0 + 1e-2 * (d - 0.3))


def net_inputs(c, seed):
    """Solid map and helix start of a relaxation box, and a target near it."""
    S = c["S"]
    z, y, x = grid_axes(S, S, S)
    m = (S - 1) / 2
    r2 = (x - m) ** 2 + (y - m) ** 2 + (z - m) ** 2
    solid = torch.where(r2 < c["radius"] ** 2, 0.0, -1.0).to(torch.float64).reshape(-1).contiguous()
    q = start_q(S, S, S, c["pitch"], seed, amp=0.02).reshape(5, -1).contiguous()
    shell = torch.exp(-((torch.sqrt(r2) - c["radius"]) / 4.0) ** 2).reshape(1, -1)
    bump = 0.2 * (torch.rand((5, 1), dtype=torch.float64, device="cuda", generator=generator(seed + 1)) - 0.5)
    return solid, q, (q + bump * shell).contiguous()


def net_weights(seed):
    """Weights of a trained size: He-scaled convolutions, small biases, a small head."""
    g = np.random.default_rng(seed)
    st = {}
    for name, cin, cout, taps, relu, _ in LAYERS:
        w = g.standard_normal((cout, taps, cin)) * (math.sqrt(2.0 / (cin * taps)) if relu else 0.05)
        if name == "c0a":
            w[:, :, 9:] = 0.0
        st[name] = dict(w=w.astype(np.float32), b=(0.02 * g.standard_normal(cout)).astype(np.float32))
    return st


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
def prepare(case, seed):
    with torch.cuda.stream(work_stream()):
        return build(dict(case), seed)


def run(st):
    with torch.cuda.stream(work_stream()):
        return one_pass(st)


@functools.cache
def work_stream():
    """The program's stream: the solver (which takes no legacy default stream), the network and torch share it."""
    return torch.cuda.Stream()


def build(c, seed):
    prec, dt = storage(c)
    st = dict(c=c, dt=dt)
    if c["kind"] == "step":
        s = P.Solver(c["nx"], c["ny"], c["nz"], wall_z=c["walls"], precision=prec, **params_of(c["pitch"], COUPLED))
        s.set_Q(start_q(c["nx"], c["ny"], c["nz"], c["pitch"], seed))
        add_colloids(s, colloids_of(c))
        st.update(s=s, q=field(5, c), u=field(3, c))
    elif c["kind"] == "batch":
        specs = sweep_of(c)
        B = P.Batch([dict(grid=(b["nx"], b["ny"], b["nz"]), params=params_of(b["pitch"], COUPLED)) for b in specs],
                    precision=prec)
        for k, (s, b) in enumerate(zip(B.boxes, specs)):
            s.set_Q(start_q(b["nx"], b["ny"], b["nz"], b["pitch"], seed * 64 + k))
            add_colloids(s, colloids_of(b))
        st.update(B=B, q=[field(5, b) for b in specs], u=[field(3, b) for b in specs])
    elif c["kind"] == "relax":
        b = relax_box(c)
        s = P.Solver(b["nx"], b["ny"], b["nz"], precision=prec, **params_of(c["pitch"], RELAX, flow=False))
        s.set_Q(start_q(b["nx"], b["ny"], b["nz"], c["pitch"], seed))
        add_colloids(s, colloids_of(b))
        st.update(s=s, q=field(5, b))
    elif c["kind"] == "analyse":
        b = analyse_box(c)
        s = P.Solver(b["nx"], b["ny"], b["nz"], precision=prec, **params_of(0.0, COUPLED))
        add_colloids(s, colloids_of(b))
        s.set_Q(texture_q(b["nx"], b["ny"], b["nz"], seed))
        s.set_f(random_f(b, seed))
        st.update(s=s, u=field(3, b), rho=field(1, b),
                  labels=torch.empty((b["nz"], b["ny"], b["nx"]), dtype=torch.int32, device="cuda"))
    else:
        net = UNet(S=c["S"])
        net.load(net_weights(7 if c["kind"] == "infer" else seed))
        solid, q, target = net_inputs(c, seed)
        st.update(net=net, solid=solid, q=q, target=target)
    return st


def one_pass(st):
    c, dt = st["c"], st["dt"]
    if c["kind"] == "step":
        s = st["s"]
        s.step(c["steps"])
        out = dict(Q=s.get_fields(P.LC_Q, st["q"]).to(dt), u=s.get_fields(P.LC_U, st["u"]).to(dt))
        if c["mobile"]:
            f = s.forces(0)
            out["colloid"] = [np.asarray(f[k]).astype(np.float32) for k in ("F", "V", "X")]
        return out
    if c["kind"] == "batch":
        st["B"].step(c["steps"])
        return [dict(Q=s.get_fields(P.LC_Q, q).to(dt), u=s.get_fields(P.LC_U, u).to(dt))
                for s, q, u in zip(st["B"].boxes, st["q"], st["u"])]
    if c["kind"] == "relax":
        n, r = st["s"].relax(tol=1e-12, max_steps=c["steps"], check_every=c["every"])
        return dict(steps=n, residual=r, Q=st["s"].get_fields(P.LC_Q, st["q"]).to(dt))
    if c["kind"] == "analyse":
        s = st["s"]
        d = s.defects(0.435)
        k = min(LOOPS, d["n_comp"])
        loops = {n: np.zeros((LOOPS,) + d[n].shape[1:], t) for n, t in
                 (("root", np.int64), ("size", np.int64), ("centroid", np.float32), ("gyration", np.float32))}
        for n, a in loops.items():
            a[:k] = d[n][:k]
        labels = s.defect_labels(0.435, st["labels"])
        g = s.diag()
        return dict(n_defect=d["n_defect"], n_comp=d["n_comp"], **loops, labels=labels, fluid=g["n_fluid"],
                    low=g["n_defect"], mass=g["mass"], energy=g["free_energy"], momentum=g["momentum"].astype(np.float32),
                    rho=s.get_fields(P.LC_RHO, st["rho"]).to(dt), u=s.get_fields(P.LC_U, st["u"]).to(dt))
    net = st["net"]
    net.set_input(st["solid"], st["q"], c["radius"], c["pitch"], 0.02)
    if c["kind"] == "infer":
        net.forward()
        return dict(y=net.y[:, :5].bfloat16(), q=net.predict_soa().bfloat16())
    net.set_target(st["target"])
    net.forward()
    loss = net.loss_and_grad()
    net.backward()
    net.adam(lr=1e-4)
    return dict(loss=torch.tensor(loss, dtype=torch.bfloat16), y=net.y[:, :5].bfloat16(),
                grads={n: [net.params[n]["gw"].bfloat16(), net.params[n]["gb"].bfloat16()] for n in net.params})


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def work(case):
    """Bytes and operations of one pass.  A coupled step reads and writes the 19 populations and the 5 components of
    Q once per node (Q alone with the flow frozen) and takes about 1100 operations per node (700 with the flow
    frozen: stress and molecular field 400, collision 300, Q update 400); the fields read out are written in FP64."""
    c = dict(case)
    if c["kind"] in ("step", "batch"):
        boxes = [c] if c["kind"] == "step" else sweep_of(c)
        nodes = sum(b["nx"] * b["ny"] * b["nz"] for b in boxes)
        size = 8 if storage(c)[0] == P.LC_FP64 else 4
        return dict(bytes=nodes * (c["steps"] * 2 * 24 * size + 8 * 8), flops=nodes * c["steps"] * 1100)
    if c["kind"] == "relax":
        size = 8 if c["precision"] == "f64" else 4
        return dict(bytes=c["n"] ** 3 * (c["steps"] * 2 * 5 * size + 40), flops=c["n"] ** 3 * c["steps"] * 700)
    if c["kind"] == "analyse":
        nodes = c["nx"] * c["ny"] * c["nz"]
        size = 8 if c["precision"] == "f64" else 4
        return dict(bytes=nodes * (24 * size + 4 + 4 * 8), flops=nodes * 700)
    n = [c["S"] ** 3 / 8 ** k for k in range(3)]
    fl = sum(2.0 * n[lvl] * cin * cout * taps for _, cin, cout, taps, _, lvl in LAYERS)
    by = c["S"] ** 3 * (8 + 40 + 40)  # solid map and start in, proposal out
    return dict(bytes=by + (n[0] * 40 if c["kind"] == "train" else 0), flops=fl * (3 if c["kind"] == "train" else 1))


# ---------------------------------------------------------------------------
# exact: the model in plain 64-bit torch
# ---------------------------------------------------------------------------
C19 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
       (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
       (0, -1, 1)]
W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
FACES = [(1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]


def opposite(q):
    return 0 if q == 0 else (q + 1 if q % 2 else q - 1)


def at(a, e):
    """a(r + e), periodic; e = (ex, ey, ez), the last three axes of a are z, y, x."""
    if e == (0, 0, 0):
        return a
    return torch.roll(a, shifts=(-e[2], -e[1], -e[0]), dims=(-3, -2, -1))


def sym(q):
    return [[q[0], q[1], q[2]], [q[1], q[3], q[4]], [q[2], q[4], -q[0] - q[3]]]


def dot3(a, b):
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]


class Reference:
    """One box in 64 bits: fields [component][z][y][x] as torch tensors, colloids as numpy records."""

    def __init__(self, nx, ny, nz, walls, prm, cols, q):
        self.L, self.walls, self.prm = (nx, ny, nz), walls, prm
        self.Q = q.to(torch.float64).clone()
        dev = q.device
        self.f = torch.zeros((19, nz, ny, nx), dtype=torch.float64, device=dev)
        ax = [torch.arange(n, dtype=torch.float64, device=dev) for n in (nz, ny, nx)]
        z, y, x = torch.meshgrid(*ax, indexing="ij")
        self.pos = (x, y, z)
        self.cols = [dict(k, X=np.array(k["X"]), V=np.zeros(3), Om=np.zeros(3)) for k in cols]
        self.owner = self.solid_map()
        self.solid = self.owner >= 0
        g = prm["gamma"]
        self.S0 = 0.25 + 0.75 * math.sqrt(1 - 8 / (3 * g))
        self.resid = 0.0

    def offset(self, X, shift=(0.0, 0.0, 0.0)):
        """Minimum-image displacement of the nodes (moved by shift) from X."""
        out = []
        for a in range(3):
            d = self.pos[a] + shift[a] - float(X[a])
            if a < 2 or not self.walls:
                h = 0.5 * self.L[a]
                d = torch.where(d >= h, d - self.L[a], torch.where(d < -h, d + self.L[a], d))
            out.append(d)
        return out

    def solid_map(self):
        owner = torch.full(self.pos[0].shape, -1, dtype=torch.int64, device=self.Q.device)
        for k, c in enumerate(self.cols):
            d = self.offset(c["X"])
            owner[d[0] ** 2 + d[1] ** 2 + d[2] ** 2 < c["a0"] ** 2] = k
        return owner

    def beyond(self, e):
        """Nodes whose neighbour r + e lies beyond a wall."""
        m = torch.zeros_like(self.solid)
        if self.walls and e[2]:
            m[-1 if e[2] > 0 else 0] = True
        return m

    def surface(self, e, owner, idx):
        """Q0 and its weight for the fluid nodes idx whose neighbour r + e belongs to colloid owner (-1: a wall)."""
        q = self.Q[:, idx[0], idx[1], idx[2]]
        if owner < 0:
            n = [torch.zeros_like(q[0]), torch.zeros_like(q[0]), torch.ones_like(q[0])]
            return uniaxial(self.S0, n), q, 1.0
        c = self.cols[owner]
        d = [v[idx] for v in self.offset_at(c["X"], e)]
        r = torch.sqrt(dot3(d, d))
        s = [v / r for v in d]
        n = s
        if c["planar"]:
            m = torch.stack([torch.stack(row) for row in sym(q)]).permute(2, 0, 1)
            nf = torch.linalg.eigh(m)[1][:, :, 2].T
            ns = dot3(nf, s)
            p = [nf[a] - ns * s[a] for a in range(3)]
            pn = torch.sqrt(dot3(p, p))
            n = [v / pn for v in p]
        w = 1.0 if math.isinf(c["w"]) else c["w"] / (self.prm["K"] + c["w"])
        return uniaxial(self.S0, n), q, w

    def offset_at(self, X, e):
        """Displacement of the solid nodes r + e from X (the node index wraps before the minimum image is taken)."""
        return [at(v, e) for v in self.offset(X)]

    def stress(self):
        """Derivatives, molecular field, stress, free-energy density and the surface term at fluid nodes."""
        p = self.prm
        A0, g, K, q0, xi = p["A0"], p["gamma"], p["K"], p["q0"], p["xi"]
        nb, self.face_solid, surf = [], [], 0.0
        for e in FACES:
            v = at(self.Q, e).clone()
            own, out = at(self.owner, e), self.beyond(e)
            closed = ((own >= 0) | out) & ~self.solid
            for k in ([-1] if self.walls else []) + list(range(len(self.cols))):
                idx = torch.nonzero(closed & (out if k < 0 else (own == k) & ~out), as_tuple=True)
                if idx[0].numel() == 0:
                    continue
                s0, q, w = self.surface(e, k, idx)
                qs = q + w * (s0 - q)
                v[:, idx[0], idx[1], idx[2]] = qs
                if k >= 0 and w < 1.0:
                    t = sum((a ** 2).sum() for row in sym(qs - s0) for a in row)
                    surf = surf + 0.5 * self.cols[k]["w"] * t
            nb.append(v)
            self.face_solid.append((closed, own, out))
        dq = [0.5 * (nb[2 * a] - nb[2 * a + 1]) for a in range(3)]
        lap = sum(nb[1:], nb[0]) - 6 * self.Q
        Q, D, Lp = sym(self.Q), [sym(d) for d in dq], sym(lap)
        S2 = [[dot3(Q[a], Q[b]) for b in range(3)] for a in range(3)]
        C = [[D[(a + 1) % 3][(a + 2) % 3][b] - D[(a + 2) % 3][(a + 1) % 3][b] for b in range(3)] for a in range(3)]
        t2 = S2[0][0] + S2[1][1] + S2[2][2]
        t3 = sum(Q[a][b] * S2[a][b] for a in range(3) for b in range(3))
        cb = -A0 * (1 - g / 3) - A0 * g * t2 - 4 * K * q0 * q0
        H = [[cb * Q[a][b] + A0 * g * (S2[a][b] - (t2 / 3 if a == b else 0.0)) + K * Lp[a][b]
              - 2 * K * q0 * (C[a][b] + C[b][a]) for b in range(3)] for a in range(3)]
        grad = [[sum(D[a][i][j] * D[b][i][j] for i in range(3) for j in range(3)) for b in range(3)] for a in range(3)]
        qc = sum(Q[a][b] * C[a][b] for a in range(3) for b in range(3))
        fe = (0.5 * A0 * (1 - g / 3) * t2 - A0 * g / 3 * t3 + 0.25 * A0 * g * t2 ** 2
              + 0.5 * K * (grad[0][0] + grad[1][1] + grad[2][2]) + 2 * K * q0 * qc + 2 * K * q0 * q0 * t2)
        A = [[sum(Q[a][i] * H[i][b] for i in range(3)) for b in range(3)] for a in range(3)]
        qh = A[0][0] + A[1][1] + A[2][2]
        Pm = [[None] * 3 for _ in range(3)]
        for a in range(3):
            for b in range(3):
                g1, g2 = (b + 1) % 3, (b + 2) % 3  # eps(m, b, g) d_a Q_gn Q_mn over g, m, n
                e2 = dot3(D[a][g1], Q[g2]) - dot3(D[a][g2], Q[g1])
                v = 2 * xi * Q[a][b] * qh - xi * (A[a][b] + A[b][a]) - 2 * xi / 3 * H[a][b]
                v = v - K * grad[a][b] - 2 * K * q0 * e2 + A[a][b] - A[b][a]
                Pm[a][b] = v + (fe + 2 * xi / 3 * qh if a == b else 0.0)
        return H, Pm, fe, surf

    def body_force(self, Pm):
        """Face divergence of the stress, and each colloid's LC force and torque."""
        F = [torch.zeros_like(self.pos[0]) for _ in range(3)]
        acc = [np.zeros(6) for _ in self.cols]
        for d, e in enumerate(FACES):
            ax, sg = d // 2, 1.0 if d % 2 == 0 else -1.0
            closed, own, out = self.face_solid[d]
            for a in range(3):
                pi = Pm[a][ax]
                F[a] = F[a] + sg * torch.where(closed, pi, 0.5 * (pi + at(pi, e)))
            for k, c in enumerate(self.cols):
                idx = torch.nonzero(closed & (own == k) & ~out, as_tuple=True)
                ff = [-sg * Pm[a][ax][idx] for a in range(3)]
                r = [v[idx] for v in self.offset(c["X"], [0.5 * v for v in e])]
                tq = [r[1] * ff[2] - r[2] * ff[1], r[2] * ff[0] - r[0] * ff[2], r[0] * ff[1] - r[1] * ff[0]]
                acc[k] += np.array([float(v.sum()) for v in ff + tq])
        return [torch.where(self.solid, 0.0, v) for v in F], acc

    def moments(self, F):
        drho = self.f.sum(0)
        m = [sum(c[a] * self.f[q] for q, c in enumerate(C19) if c[a]) for a in range(3)]
        rho = self.prm["rho0"] + drho
        u = [(m[a] + 0.5 * F[a]) / rho for a in range(3)]
        for c_id, c in enumerate(self.cols):
            d, sel = self.offset(c["X"]), self.owner == c_id
            ur = self.rigid(c, d)
            u = [torch.where(sel, ur[a], u[a]) for a in range(3)]
        return drho, rho, u

    @staticmethod
    def rigid(c, d):
        V, w = c["V"], c["Om"]
        return [V[0] + w[1] * d[2] - w[2] * d[1], V[1] + w[2] * d[0] - w[0] * d[2], V[2] + w[0] * d[1] - w[1] * d[0]]

    def update_q(self, H, u):
        xi, Gam = self.prm["xi"], self.prm["Gamma"]
        un, qn, fl = [], [], []
        for d, e in enumerate(FACES):
            out = self.beyond(e)
            un.append([torch.where(out, 0.0, at(v, e)) for v in u])
            qn.append(at(self.Q, e))
            fl.append(~(at(self.solid, e) | out))
        Wm = [[0.5 * (un[2 * b][a] - un[2 * b + 1][a]) for b in range(3)] for a in range(3)]
        adv = torch.zeros_like(self.Q)
        for d in range(6):
            ax = d // 2
            uf = 0.5 * (u[ax] + un[d][ax])
            own = uf > 0 if d % 2 == 0 else ~(uf > 0)
            flux = torch.where(fl[d], uf, 0.0) * torch.where(own, self.Q, qn[d])
            adv = adv + (flux if d % 2 == 0 else -flux)
        Q = sym(self.Q)
        Qt = [[Q[a][b] + (1 / 3 if a == b else 0.0) for b in range(3)] for a in range(3)]
        Ds = [[0.5 * (Wm[a][b] + Wm[b][a]) for b in range(3)] for a in range(3)]
        Om = [[0.5 * (Wm[a][b] - Wm[b][a]) for b in range(3)] for a in range(3)]
        tr = sum(Q[a][b] * Ds[a][b] for a in range(3) for b in range(3))
        S = [[sum(xi * (Ds[a][i] * Qt[i][b] + Qt[a][i] * Ds[i][b]) + Om[a][i] * Q[i][b] - Q[a][i] * Om[i][b]
                  for i in range(3)) - 2 * xi * Qt[a][b] * tr for b in range(3)] for a in range(3)]
        tr = (S[0][0] + S[1][1] + S[2][2]) / 3
        ij = [(0, 0), (0, 1), (0, 2), (1, 1), (1, 2)]
        inc = torch.stack([Gam * H[a][b] + S[a][b] - adv[k] - (tr if a == b else 0.0)
                           for k, (a, b) in enumerate(ij)])
        inc = torch.where(self.solid, 0.0, inc)
        t = sum((v ** 2).sum() for row in sym(inc) for v in row)
        self.resid = math.sqrt(float(t) / float((~self.solid).sum()))
        return self.Q + inc

    def collide_stream(self, F, drho, rho, u):
        om, pref, rho0 = 1 / self.prm["tau"], 1 - 0.5 / self.prm["tau"], self.prm["rho0"]
        usq, uF = dot3(u, u), dot3(u, F)
        post = torch.empty_like(self.f)
        for q, c in enumerate(C19):
            cu = sum(c[a] * u[a] for a in range(3) if c[a]) if q else torch.zeros_like(usq)
            cF = sum(c[a] * F[a] for a in range(3) if c[a]) if q else torch.zeros_like(usq)
            eq = W[q] * (drho + rho * (3 * cu + 4.5 * cu * cu - 1.5 * usq))
            post[q] = self.f[q] - om * (self.f[q] - eq) + pref * W[q] * (3 * (cF - uF) + 9 * cu * cF)
        acc = [np.zeros(18) for _ in self.cols]
        new = torch.empty_like(self.f)
        for q, c in enumerate(C19):
            back = tuple(-v for v in c)
            own, out = at(self.owner, back), self.beyond(back)
            bounced = post[opposite(q)]
            for k, col in enumerate(self.cols):
                idx = torch.nonzero((own == k) & ~out & ~self.solid, as_tuple=True)
                if idx[0].numel() == 0:
                    continue
                d = [v[idx] for v in self.offset(col["X"], [0.5 * v for v in back])]
                ub = self.rigid(col, d)
                cub = sum(c[a] * ub[a] for a in range(3))
                corr = 6 * W[q] * rho0 * cub
                inc = bounced[idx]
                bounced = bounced.clone()
                bounced[idx] = inc + corr
                # the link r -> r - c carries the opposite population into the colloid
                mag = 2 * inc + corr
                dp = [back[a] * mag for a in range(3)]
                tq = [d[1] * dp[2] - d[2] * dp[1], d[2] * dp[0] - d[0] * dp[2], d[0] * dp[1] - d[1] * dp[0]]
                acc[k][:6] += np.array([float(v.sum()) for v in dp + tq])
                zk = 6 * W[q] * rho0
                rc = [d[1] * back[2] - d[2] * back[1], d[2] * back[0] - d[0] * back[2], d[0] * back[1] - d[1] * back[0]]
                for m, (a, b) in enumerate([(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]):
                    acc[k][6 + m] += zk * back[a] * back[b] * idx[0].numel()
                    acc[k][12 + m] += zk * float((rc[a] * rc[b]).sum())
            new[q] = torch.where(((own >= 0) | out), bounced, at(post[q], back))
        self.f = torch.where(self.solid, 0.0, new)
        return acc

    def step(self, flow=True):
        """One coupled step; False when a node would change between solid and fluid."""
        H, Pm, _, _ = self.stress()
        F, flc = self.body_force(Pm)
        if not flow:
            self.Q = self.update_q(H, [torch.zeros_like(F[0])] * 3)
            return True
        drho, rho, u = self.moments(F)
        newQ = self.update_q(H, u)
        fhyd = self.collide_stream(F, drho, rho, u)
        self.Q = newQ
        moved = False
        for c, lc, hy in zip(self.cols, flc, fhyd):
            c["total"] = lc[:3] + hy[:3]
            if not c["mobile"]:
                continue
            moved = True
            M = self.prm["rho0"] * 4 / 3 * math.pi * c["a0"] ** 3
            inertia = 0.4 * M * c["a0"] ** 2
            full = lambda s: np.array([[s[0], s[1], s[2]], [s[1], s[3], s[4]], [s[2], s[4], s[5]]])  # noqa: E731
            c["V"] = c["V"] + np.linalg.solve(M * np.eye(3) + full(hy[6:12]), c["total"] + np.array(c["F"]))
            c["Om"] = c["Om"] + np.linalg.solve(inertia * np.eye(3) + full(hy[12:18]), lc[3:] + hy[3:6])
            c["X"] = c["X"] + c["V"]
        return not moved or bool(torch.equal(self.solid_map(), self.owner))

    def velocity(self):
        _, Pm, _, _ = self.stress()
        F, _ = self.body_force(Pm)
        return torch.stack(self.moments(F)[2])


def reference_box(b, prm, q):
    return Reference(b["nx"], b["ny"], b["nz"], b["walls"], prm, colloids_of(b), q)


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "step":
        R = reference_box(c, params_of(c["pitch"], COUPLED), start_q(c["nx"], c["ny"], c["nz"], c["pitch"], seed))
        for _ in range(c["steps"]):
            if not R.step():
                return None  # re-discretised: no closed restatement here
        out = dict(Q=R.Q, u=R.velocity())
        if c["mobile"]:
            k = R.cols[0]
            out["colloid"] = [k["total"], k["V"], k["X"]]
        return out
    if c["kind"] == "batch":
        out = []
        for k, b in enumerate(sweep_of(c)):
            q = start_q(b["nx"], b["ny"], b["nz"], b["pitch"], seed * 64 + k)
            R = reference_box(b, params_of(b["pitch"], COUPLED), q)
            for _ in range(c["steps"]):
                R.step()
            out.append(dict(Q=R.Q, u=R.velocity()))
        return out
    if c["kind"] == "relax":
        b = relax_box(c)
        R = reference_box(b, params_of(c["pitch"], RELAX), start_q(b["nx"], b["ny"], b["nz"], c["pitch"], seed))
        for _ in range(c["steps"]):
            R.step(flow=False)
        return dict(steps=c["steps"], residual=np.float64(R.resid), Q=R.Q)
    if c["kind"] == "analyse":
        return exact_analyse(c, seed)
    return exact_net(c, seed)


def exact_analyse(c, seed):
    b = analyse_box(c)
    R = reference_box(b, params_of(0.0, COUPLED), texture_q(b["nx"], b["ny"], b["nz"], seed))
    R.f = random_f(b, seed) - torch.tensor(W, dtype=torch.float64, device="cuda").reshape(19, 1, 1, 1)
    fluid = ~R.solid
    _, Pm, fe, surf = R.stress()
    F, _ = R.body_force(Pm)
    _, rho, u = R.moments(F)
    m = torch.stack([sum(cc[a] * R.f[q] for q, cc in enumerate(C19) if cc[a])[fluid].sum() for a in range(3)])
    return dict(n_defect=None, n_comp=None, root=None, size=None, centroid=None, gyration=None, labels=None,
                fluid=int(fluid.sum()), low=None, mass=np.float64(float(rho[fluid].sum())),
                energy=np.float64(float(fe[fluid].sum() + surf)), momentum=m,
                rho=torch.where(fluid, rho, 1.0).unsqueeze(0), u=torch.stack(u))


def exact_net(c, seed):
    """The network in 64 bits on its BF16 weights and inputs (activations unrounded)."""
    S = c["S"]
    solid, q, target = net_inputs(c, seed)
    st = net_weights(7 if c["kind"] == "infer" else seed)
    p = {}
    for n, s in st.items():
        p[n] = [torch.tensor(s["w"], device="cuda").bfloat16().double(), torch.tensor(s["b"], device="cuda").double()]
        for t in p[n]:
            t.requires_grad_(c["kind"] == "train")
    ones = torch.ones(S ** 3, dtype=torch.float64, device="cuda")
    x = torch.stack([(solid >= 0).double(), *q, ones * c["radius"] / 32, ones * c["pitch"] / 64, ones * 0.4]
                    + [0 * ones] * 7).bfloat16().double()

    def conv(a, name, relu=True):
        s = round(a.shape[1] ** (1 / 3))
        w, bias = p[name]
        g = a.reshape(-1, s, s, s)
        taps = [(0, 0, 0)] if w.shape[1] == 1 else [(t % 3 - 1, t // 3 % 3 - 1, t // 9 - 1) for t in range(27)]
        y = sum(w[:, t] @ at(g, e).reshape(a.shape[0], -1) for t, e in enumerate(taps)) + bias[:, None]
        return torch.relu(y) if relu else y

    def pool(a, s):
        return a.reshape(-1, s // 2, 2, s // 2, 2, s // 2, 2).mean(dim=(2, 4, 6)).reshape(a.shape[0], -1)

    def up(a, s):
        g = a.reshape(-1, s, s, s)
        for d in (1, 2, 3):
            g = g.repeat_interleave(2, dim=d)
        return g.reshape(a.shape[0], -1)

    c0 = conv(conv(x, "c0a"), "c0b")
    c1 = conv(conv(pool(c0, S), "c1a"), "c1b")
    c2 = conv(conv(pool(c1, S // 2), "c2a"), "c2b")
    c3 = conv(torch.cat([up(c2, S // 4), c1]), "c3")
    y = conv(conv(torch.cat([up(c3, S // 2), c0]), "c4"), "head", relu=False)[:5]
    if c["kind"] == "infer":
        return dict(y=y.T, q=q + y)
    fluid = (solid < 0).double()
    loss = (((q + y - target) * fluid) ** 2).sum() / (5 * fluid.sum())
    loss.backward()
    return dict(loss=loss.detach(), y=y.detach().T, grads={n: [t.grad for t in p[n]] for n in p})
