"""The workloads this library's speed is judged by, and what each should return.

Every case is one call sequence of a user's program through the public entry
points (``clbm.Solver``, ``clbm.Batch``, the ``clbm_*`` functions, ``net.Net``):

* a solve of one lattice: initial fields on the device in, a run of steps, the
  macroscopic fields out (and, where a program monitors convergence, the
  residual and a wall Nusselt number);
* a batched solve of many lattices (the data generation and the settling
  studies of the warm start);
* the warm-start network: one gradient pass, one inference.

Fields and numbers leave in the precision the lattice is stored in (FP64
fields are what the library writes; an FP32 or 16-bit state carries no more
than its own digits, and that is how such results are kept and trained on).

``exact`` evaluates the same schemes in FP64 with plain torch operations.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_1801_04577_gb300 import clbm
from paper_1801_04577_gb300 import inputs as I
from paper_1801_04577_gb300 import net as N

STORED = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
# floating-point operations of one node update (collision, Eq. 4-10 and 23-24) and the
# nodes' share of walls left out
FLOPS_PER_UPDATE = 250


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # The paper's heated cavity at the size of its quick checks: a few thousand nodes, so
        # the time of a step is latency.  Monitored by its residual.
        dict(name="cavity64_f32", kind="cavity", n=64, Ra=1e4, precision="f32", rounding=0, steps=200),
        # The same flow as an accuracy reference, at an odd size, in FP64: residual and Nusselt number.
        dict(name="cavity101_f64", kind="cavity", n=101, Ra=1e5, precision="f64", rounding=0, steps=100),
        # A lattice that fits in L2: development runs, parameter scans.
        dict(name="rb512_f32", kind="rb", nx=512, ny=256, precision="f32", rounding=0, steps=200),
        # The headline Rayleigh-Benard lattice, FP32 storage, out of HBM.
        dict(name="rb4096_f32", kind="rb", nx=4096, ny=2048, precision="f32", rounding=0, steps=20),
        # The same in the recommended 16-bit format (stochastic rounding).
        dict(name="rb4096_f16_sr", kind="rb", nx=4096, ny=2048, precision="f16", rounding=1, steps=20),
        # FP64 reference runs of a large lattice.
        dict(name="rb2048_f64", kind="rb", nx=2048, ny=1024, precision="f64", rounding=0, steps=10),
        # Curved walls at their true position: masked lattice, listed links, half of the box solid.
        dict(name="annulus2048_f32", kind="annulus", n=2048, ratio=2.6, interpolated=True, precision="f32",
             rounding=0, steps=20),
        # A ragged box with an obstacle and mixed wall conditions, 16-bit round to nearest.
        dict(name="channel1021_bf16", kind="channel", nx=1021, ny=509, precision="bf16", rounding=0, steps=50),
        # Many cavities of uneven size and walls in one batch, fixed number of steps.
        dict(name="batch_mixed_f32", kind="batch_mixed", n=64, hmin=32, hmax=512, precision="f32", steps=200),
        # The warm start's training data: equal small cavities with obstacles, FP32.
        dict(name="batch_obstacles64_f32", kind="batch_obstacles", n=256, G=64, precision="f32", steps=1000),
        # One gradient pass of the warm-start network at its default size.
        dict(name="net_gradients_g64", kind="net_gradients", G=64, base=24, levels=4, batch=32),
        # Inference of the study's deeper network on the larger grid.
        dict(name="net_forward_g128", kind="net_forward", G=128, base=16, levels=5, batch=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["cavity", "rb", "rb", "annulus", "channel", "batch_mixed", "batch_obstacles",
                       "net_gradients", "net_forward"])
    precision = rng.choice(["f32", "f32", "f16", "bf16", "f64"])
    rounding = rng.randrange(2) if precision in ("f16", "bf16") else 0
    if kind == "cavity":
        return dict(kind=kind, n=_log_int(rng, 24, 300), Ra=10.0 ** rng.uniform(3, 5), precision=precision,
                    rounding=rounding, steps=rng.choice([51, 100, 200]))
    if kind == "rb":
        hi = 2048 if precision == "f64" else 4096
        nx, ny = _log_int(rng, 100, hi), _log_int(rng, 60, hi // 2)
        return dict(kind=kind, nx=nx, ny=ny, precision=precision, rounding=rounding,
                    steps=10 if precision == "f64" else rng.choice([1, 20, 33]) if nx * ny > 500000 else 200)
    if kind == "annulus":
        return dict(kind=kind, n=_log_int(rng, 100, 1500), ratio=rng.choice([2.0, 2.6, 4.0]),
                    interpolated=rng.random() < 0.5, precision=precision, rounding=rounding, steps=20)
    if kind == "channel":
        return dict(kind=kind, nx=_log_int(rng, 40, 2000), ny=_log_int(rng, 30, 1000), precision=precision,
                    rounding=rounding, steps=50 if precision != "f64" else 20)
    if kind == "batch_mixed":
        return dict(kind=kind, n=rng.randint(8, 64), hmin=32, hmax=_log_int(rng, 64, 400),
                    precision=rng.choice(["f32", "f32", "f16"]), steps=200)
    if kind == "batch_obstacles":
        return dict(kind=kind, n=_log_int(rng, 16, 256), G=rng.choice([32, 48, 64, 96]),
                    precision="f32", steps=rng.choice([200, 400]))
    levels = rng.randint(3, 5)
    return dict(kind=kind, G=rng.choice([32, 64, 96, 128] if kind == "net_forward" else [32, 48, 64, 96]),
                base=rng.choice([8, 16, 24]), levels=levels, batch=rng.randint(1, 32))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _generator(seed):
    return torch.Generator(device=_device()).manual_seed(int(seed) * 7919 + 13)


def _flow_fields(nx, ny, seed, periodic_x, hot_left):
    """(ux, uy, T): the conduction profile between the walls with smooth thermal disturbances and
    a divergence-free circulation that vanishes at the walls, as a run that is resumed or
    started from a prediction has them, plus the small noise that convection grows from."""
    g, dev = _generator(seed), _device()
    r = torch.rand(16, generator=g, device=dev, dtype=torch.float64).cpu().numpy()
    x = ((torch.arange(nx, device=dev, dtype=torch.float64) + 0.5) / nx)[None, :]
    y = ((torch.arange(ny, device=dev, dtype=torch.float64) + 0.5) / ny)[:, None]
    amp, m = 0.01 + 0.03 * r[0], 1 + int(3 * r[1])
    sy, dsy = torch.sin(math.pi * y) ** 2, math.pi * torch.sin(2 * math.pi * y)
    if periodic_x:
        sx = torch.sin(2 * math.pi * (m * x + r[2]))
        dsx = 2 * math.pi * m * torch.cos(2 * math.pi * (m * x + r[2]))
    else:
        sx, dsx = torch.sin(math.pi * x) ** 2, math.pi * torch.sin(2 * math.pi * x)
    h = min(nx, ny)
    ux = (amp / math.pi) * sx * dsy * (h / ny)
    uy = -(amp / math.pi) * dsx * sy * (h / nx)
    T = (1.0 - x + 0 * y) if hot_left else (1.0 - y + 0 * x)
    T = T + 0.1 * (r[3] - 0.5) * torch.sin(math.pi * y) * torch.cos(2 * math.pi * (x + r[4]))
    T = T + 1e-3 * (2 * torch.rand(ny, nx, generator=g, device=dev, dtype=torch.float64) - 1)
    return ux.contiguous(), uy.contiguous(), T.contiguous()


def _workload(case):
    k = case["kind"]
    if k == "cavity":
        return I.natural_convection_cavity(case["n"], case["Ra"])
    if k == "rb":
        return I.rayleigh_benard(case["nx"], case["ny"], noise=0.0)
    if k == "annulus":
        return I.annulus(case["n"], case["ratio"], Ra=1e5, interpolated=case["interpolated"])
    return I.obstacle_channel(case["nx"], case["ny"])


def _batch_workloads(case, seed):
    """The lattices of a batch: the sizes and walls of uneven cavities are the case's, the obstacles
    of equal ones the seed's."""
    if case["kind"] == "batch_mixed":
        return I.random_cavities(case["n"], hmin=case["hmin"], hmax=case["hmax"])
    return I.obstacle_cavities(case["n"], case["G"], seed=I.SURROGATE_SEED + 31 * int(seed))


def _fields(case, w, seed):
    p = w.params
    ux, uy, T = _flow_fields(p.nx, p.ny, seed, p.periodic_x, case["kind"] not in ("rb", "annulus"))
    if case["kind"] in ("annulus", "batch_mixed"):
        T = 0.5 + 0.5 * (T - 0.5)
    if w.geom.solid is not None:
        s = torch.from_numpy(w.geom.solid != 0).to(T.device)
        ux, uy, T = (torch.where(s, torch.full_like(a, v), a) for a, v in ((ux, 0.0), (uy, 0.0), (T, p.T0)))
    return ux, uy, T


def _net_inputs(case, seed):
    """A batch of problem descriptions (fluid mask, wall markers, log Ra, Pr, source) and smooth
    targets, and a parameter vector of a network some way into its training."""
    G, n, dev = case["G"], case["batch"], _device()
    g = _generator(seed)
    u = torch.rand(n, 16, generator=g, device=dev, dtype=torch.float32)
    c = (torch.arange(G, device=dev, dtype=torch.float32) + 0.5) / G
    X, Y = c[None, None, :], c[None, :, None]
    w, h = 0.06 + 0.19 * u[:, 0:1, None], 0.06 + 0.19 * u[:, 1:2, None]
    inside = ((X - 0.2 - 0.5 * u[:, 2:3, None]).abs() < 0.5 * w) & ((Y - 0.2 - 0.5 * u[:, 3:4, None]).abs() < 0.5 * h)
    mask = (~inside).to(torch.float32)
    x = torch.zeros(n, 5, G, G, device=dev)
    x[:, 0] = mask
    x[:, 1, :, 0], x[:, 1, :, G - 1] = 1.0, -1.0
    x[:, 1] *= mask
    x[:, 2] = (u[:, 4] * 2 - 1)[:, None, None]
    x[:, 3] = (u[:, 5] * 2 - 1)[:, None, None]
    x[:, 4] = torch.where(u[:, 6] < 0.5, torch.zeros_like(u[:, 6]), u[:, 7])[:, None, None]
    k = 1.0 + 2.0 * u[:, 8:9, None]
    t = torch.stack([(0.5 - X + 0.1 * torch.sin(6.2832 * Y * k)).expand(n, G, G),
                     0.3 * torch.sin(3.1416 * X * k) * torch.sin(6.2832 * Y),
                     -0.3 * torch.sin(6.2832 * X) * torch.sin(3.1416 * Y * k)], 1) * mask[:, None]
    p = []
    for ci, co, ks in N.layer_shapes(G, 5, 3, case["base"], case["levels"]):
        a = math.sqrt(6.0 / (ci * ks * ks))
        p.append((2 * torch.rand(co * ci * ks * ks, generator=g, device=dev) - 1) * a)
        p.append((2 * torch.rand(co, generator=g, device=dev) - 1) * 0.05)
    return x.contiguous(), t.contiguous(), mask.contiguous(), torch.cat(p).to(torch.float32)


# ---------------------------------------------------------------------------
# A program's set-up and its pass
# ---------------------------------------------------------------------------
_streams = {}


def _stream():
    """The one stream that the program's work runs on."""
    dev = torch.cuda.current_device()
    if dev not in _streams:
        _streams[dev] = torch.cuda.Stream()
    return _streams[dev]


def _monitored(case):
    """What the program follows beside the fields: the residual of a run towards its steady state,
    and the wall Nusselt number where it is the result (FP64 reference runs)."""
    seen = ["residual"] if case["kind"] in ("cavity", "annulus") and case["precision"] in ("f32", "f64") else []
    return ["nusselt"] + seen if seen and case["precision"] == "f64" else seen


def prepare(case, seed):
    k, stream = case["kind"], _stream()
    s = {"case": case, "stream": stream}
    if k.startswith("net"):
        x, t, mask, p = _net_inputs(case, seed)
        torch.cuda.synchronize()
        s["net"] = N.Net(case["G"], 5, 3, case["base"], case["levels"], case["batch"], seed=1,
                         stream=stream.cuda_stream)
        s["net"].set_params(p.cpu().numpy())
        s.update(x=x, t=t, mask=mask, y=torch.empty(case["batch"], 3, case["G"], case["G"], device=x.device),
                 grad=torch.empty(s["net"].nparam, device=x.device))
    elif k.startswith("batch"):
        ws = _batch_workloads(case, seed)
        s["batch"] = clbm.Batch(ws, case["precision"], stream=stream.cuda_stream)
        s["views"] = [s["batch"].view(i) for i in range(len(ws))]
        s["init"] = [_fields(case, w, 1000 * int(seed) + i) for i, w in enumerate(ws)]
        s["out"] = [torch.empty(3, w.params.ny, w.params.nx, dtype=torch.float64, device="cuda") for w in ws]
    else:
        w = _workload(case)
        s["which"], s["length"] = 4 if k == "annulus" else 0, w.length
        s["fields"] = _fields(case, w, seed)
        s["solver"] = clbm.Solver(w.params, w.geom, case["precision"], stream.cuda_stream, None, case["rounding"])
        s["out"] = [torch.empty(w.params.ny, w.params.nx, dtype=torch.float64, device="cuda") for _ in range(4)]
    torch.cuda.synchronize()
    return s


def run(s):
    case = s["case"]
    k = case["kind"]
    with torch.cuda.stream(s["stream"]):
        if k == "net_forward":
            s["net"].forward(s["x"], s["y"])
            return [s["y"]]
        if k == "net_gradients":
            loss = N.C.c_double()
            N._check(N.load().clbm_net_gradients(s["net"].h, s["x"].data_ptr(), s["t"].data_ptr(),
                                                 s["mask"].data_ptr(), case["batch"], s["grad"].data_ptr(),
                                                 N.C.byref(loss)), s["net"].h, "gradients")
            return [np.float32(loss.value), s["grad"]]
        dt = STORED[case["precision"]]
        if k.startswith("batch"):
            for v, (ux, uy, T) in zip(s["views"], s["init"]):
                clbm.clbm_init_fields(v, ux=ux, uy=uy, T=T, on_device=True)
            conv, _, steps = s["batch"].solve(0.0, case["steps"], case["steps"] // 2)
            for v, o in zip(s["views"], s["out"]):
                clbm.clbm_moments(v, ux=o[0], uy=o[1], T=o[2], on_device=True)
            return [torch.cat([o.reshape(-1) for o in s["out"][j::8]]).to(dt) for j in range(8)] + [conv, steps]
        solver, (ux, uy, T), out = s["solver"], s["fields"], s["out"]
        clbm.clbm_init_fields(solver.ctx, ux=ux, uy=uy, T=T, on_device=True)
        solver.step(case["steps"])
        clbm.clbm_moments(solver.ctx, *out, on_device=True)
        res = [o.to(dt) for o in out]
        for what in _monitored(case):
            v = solver.nusselt(s["which"], s["length"], 1.0) if what == "nusselt" else solver.residual()
            res.append(torch.tensor(v, dtype=torch.float64).to(dt))
        return res


def _net_convs(case):
    """(ci, co, k, pixels per sample) of every convolution."""
    G, L = case["G"], case["levels"]
    sides = [G >> l for l in range(L - 1) for _ in (0, 1)] + [G >> (L - 1)] * 2
    sides += [G >> l for l in range(L - 2, -1, -1) for _ in (0, 1)] + [G]
    return [(ci, co, k, h * h) for (ci, co, k), h in zip(N.layer_shapes(G, 5, 3, case["base"], L), sides)]


def work(case):
    k = case["kind"]
    if k.startswith("net"):
        n, convs = case["batch"], _net_convs(case)
        macs = [ci * co * ks * ks * px * n for ci, co, ks, px in convs]
        params = sum(ci * co * ks * ks + co for ci, co, ks, _ in convs)
        io = 8 * n * case["G"] ** 2 * 4
        if k == "net_forward":
            return {"bytes": io + 4 * params, "flops": 2 * sum(macs)}
        # backward: a weight gradient for every layer, an input gradient for all but the first
        return {"bytes": io + 4 * n * case["G"] ** 2 + 8 * params, "flops": 2 * (3 * sum(macs) - macs[0])}
    if k == "batch_obstacles":
        nodes = case["n"] * case["G"] ** 2
        fields = (3 * 8 + 3 * STORED[case["precision"]].itemsize) * nodes
    elif k == "batch_mixed":
        nodes = sum(w.params.nx * w.params.ny for w in _batch_workloads(case, 0))
        fields = (3 * 8 + 3 * STORED[case["precision"]].itemsize) * nodes
    else:
        nx, ny = (case["n"], case["n"]) if "n" in case else (case["nx"], case["ny"])
        share = 1.0
        if k == "annulus":
            share = math.pi / 4 * (1 - 1 / case["ratio"] ** 2)
        nodes = nx * ny * share
        fields = (3 * 8 + 4 * STORED[case["precision"]].itemsize) * nx * ny
    return {"bytes": fields, "flops": FLOPS_PER_UPDATE * nodes * case["steps"]}


# ---------------------------------------------------------------------------
# The same results in FP64 from plain torch operations
# ---------------------------------------------------------------------------
_EX, _EY = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
_OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)


class _Lattice:
    """Cascaded D2Q9 / D2Q5 lattices of one size, each with its own rates and walls, advanced
    together in FP64: populations f [9][n][ny][nx] and g [5][n][ny][nx], post-collision."""

    def __init__(self, ws, dev):
        p0 = ws[0].params
        self.n, self.ny, self.nx, self.dev = len(ws), p0.ny, p0.nx, dev
        col = lambda name: torch.tensor([getattr(w.params, name) for w in ws], dtype=torch.float64,  # noqa: E731
                                        device=dev).view(-1, 1, 1)
        self.s_nu, self.s_b, self.s4 = col("s_nu"), col("s_b"), col("s_4")
        self.l1, self.rho0, self.T0 = col("lambda1"), col("rho0"), col("T0")
        self.gb, self.Fx, self.Fy, self.Q, self.cT2 = (col(a) for a in ("gbeta", "Fvx", "Fvy", "Q", "cT2"))
        self.s3 = torch.where(col("s_3") > 0, col("s_3"), (16 - 8 * self.s_nu) / (8 - self.s_nu))
        self.l2 = torch.where(col("lambda2") > 0, col("lambda2"), 12 * (self.l1 - 2) / (self.l1 - 12))
        solid = np.stack([np.zeros((self.ny, self.nx), bool) if w.geom.solid is None else w.geom.solid != 0 for w in ws])
        self.solid = torch.from_numpy(solid).to(dev)
        self.walls = [self._walls(ws, solid, j) for j in range(9)]
        self.geoms = [w.geom for w in ws]

    def _walls(self, ws, solid, j):
        """Nodes whose population j comes from a wall: flat index, the two nodes behind (-1: none),
        wall fraction q and (axis directions) condition and n.e."""
        if j == 0:
            return None
        n, ny, nx = solid.shape
        p = ws[0].params
        b, y, x = np.nonzero(~solid)

        def node(yy, xx, bb):
            """(flat index, box side beyond which it lies or -1); flat -1 where there is no fluid node."""
            side = np.full(len(yy), -1)
            if p.periodic_y:
                yy = yy % ny
            else:
                side = np.where(yy < 0, 2, np.where(yy >= ny, 3, side))
            if p.periodic_x:
                xx = xx % nx
            else:
                side = np.where(xx < 0, 0, np.where(xx >= nx, 1, side))
            inside = side < 0
            flat = (bb * ny + np.where(inside, yy, 0)) * nx + np.where(inside, xx, 0)
            return np.where(inside & ~solid.reshape(-1)[flat], flat, -1), side

        src, side = node(y - _EY[j], x - _EX[j], b)
        at = src < 0
        b, y, x, side = b[at], y[at], x[at], side[at]
        own = (b * ny + y) * nx + x
        i2, _ = node(y + _EY[j], x + _EX[j], b)
        i3, _ = node(y + 2 * _EY[j], x + 2 * _EX[j], b)
        i3 = np.where(i2 < 0, -1, i3)
        q = np.full(len(own), 0.5)
        ne, cond = np.ones(len(own)), np.zeros((len(own), 3))
        for k, w in enumerate(ws):
            g, mine = w.geom, b == k
            if j <= 4:
                for sd in range(4):
                    m = mine & (side == sd)
                    if m.any():
                        cond[m] = g.tbc[g.side_tbc[sd]]
            if g.n_links:
                sel = g.link_dir == _OPP[j]
                where = np.full(ny * nx, -1)
                where[g.link_node[sel]] = np.nonzero(sel)[0]
                m = mine & (side < 0)
                link = where[own[m] - k * ny * nx]
                has = link >= 0
                idx = np.nonzero(m)[0][has]
                q[idx] = g.link_q_or_half()[link[has]]
                if j <= 4:
                    ne[idx] = np.asarray(g.link_ne)[link[has]]
                    cond[idx] = np.asarray(g.tbc, np.float64)[np.asarray(g.link_tbc)[link[has]]]
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(self.dev)  # noqa: E731
        return dict(own=t(own), i2=t(i2), i3=t(i3), q=t(q), ne=t(ne), b1=t(cond[:, 0]), b2=t(cond[:, 1]),
                    b3=t(cond[:, 2]), lat=t(b), half=bool((q == 0.5).all()))

    # -- moments -----------------------------------------------------------
    @staticmethod
    def _forward(am, a0, ap, u):
        c0, s = am + a0 + ap, ap - am
        return c0, s - u * c0, (ap + am) - 2 * u * s + u * u * c0

    @staticmethod
    def _inverse(c0, c1, c2, u):
        r1, r2 = c1 + u * c0, c2 + 2 * u * c1 + u * u * c0
        return 0.5 * (r2 - r1), c0 - r2, 0.5 * (r2 + r1)

    def _from_central(self, k, ux, uy):
        """Populations of the nine central moments k[m][n]."""
        rows = [self._inverse(k[m][0], k[m][1], k[m][2], uy) for m in range(3)]  # e_y = -1, 0, 1
        f = [None] * 9
        for e, (a, b, c) in zip((-1, 0, 1), ((7, 4, 8), (3, 0, 1), (6, 2, 5))):
            f[a], f[b], f[c] = self._inverse(rows[0][e + 1], rows[1][e + 1], rows[2][e + 1], ux)
        return f

    def _thermal(self, t00, t10, t01, t20, t02, ux, uy):
        qx1, qy1 = t10 + ux * t00, t01 + uy * t00
        qx2, qy2 = t20 + 2 * ux * t10 + ux * ux * t00, t02 + 2 * uy * t01 + uy * uy * t00
        return [t00 - qx2 - qy2, 0.5 * (qx2 + qx1), 0.5 * (qy2 + qy1), 0.5 * (qx2 - qx1), 0.5 * (qy2 - qy1)]

    def collide(self, f, g):
        T = sum(g[1:], g[0]) + 0.5 * self.Q
        Fx, Fy = self.Fx, self.Fy + self.rho0 * self.gb * (T - self.T0)
        rho = sum(f[1:], f[0])
        ux = ((f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7]) + 0.5 * Fx) / rho
        uy = ((f[2] - f[4]) + (f[5] - f[7]) + (f[6] - f[8]) + 0.5 * Fy) / rho
        rows = [self._forward(f[a], f[b], f[c], ux) for a, b, c in ((7, 4, 8), (3, 0, 1), (6, 2, 5))]
        k = [list(self._forward(rows[0][m], rows[1][m], rows[2][m], uy)) for m in range(3)]
        a, b = k[2][0] - rho / 3, k[0][2] - rho / 3
        plus, minus = 0.5 * (1 - self.s_b) * (a + b), 0.5 * (1 - self.s_nu) * (a - b)
        post = [[rho, k[0][1] + Fy, rho / 3 + plus - minus],
                [k[1][0] + Fx, (1 - self.s_nu) * k[1][1], (1 - self.s3) * k[1][2] + (1 - 0.5 * self.s3) * Fx / 3],
                [rho / 3 + plus + minus, (1 - self.s3) * k[2][1] + (1 - 0.5 * self.s3) * Fy / 3,
                 (1 - self.s4) * k[2][2] + self.s4 * rho / 9]]
        fs = self._from_central(post, ux, uy)
        s, sx, sy = T - 0.5 * self.Q, g[1] - g[3], g[2] - g[4]
        t10, t01 = sx - ux * s, sy - uy * s
        t20 = g[1] + g[3] - 2 * ux * sx + ux * ux * s
        t02 = g[2] + g[4] - 2 * uy * sy + uy * uy * s
        src = (1 - 0.5 * self.l2) * self.cT2 * self.Q + self.l2 * self.cT2 * T
        gs = self._thermal(s + self.Q, (1 - self.l1) * t10, (1 - self.l1) * t01, (1 - self.l2) * t20 + src,
                           (1 - self.l2) * t02 + src, ux, uy)
        return fs, gs

    def init(self, ux, uy, T):
        z = torch.zeros(self.n, self.ny, self.nx, dtype=torch.float64, device=self.dev)
        ux, uy, T = z + ux, z + uy, z + T
        r = z + self.rho0
        f = self._from_central([[r, z, r / 3], [z, z, z], [r / 3, z, r / 9]], ux, uy)
        g = self._thermal(T, z, z, self.cT2 * T, self.cT2 * T, ux, uy)
        self.f, self.g = self.collide(f, g)

    # -- one step ----------------------------------------------------------
    def _T_at(self, T, idx):
        return T.reshape(-1)[idx.clamp(min=0)]

    @staticmethod
    def _wall_T(w, T1, T2, have2):
        """T on the wall from b1 dT/dn + b2 T = b3, the profile quadratic through the wall and the
        fluid nodes at q and 1 + q (linear where the second is missing)."""
        q, p = w["q"], 1 + w["q"]
        two = (w["b3"] * q * p * w["ne"] + w["b1"] * (p * p * T1 - q * q * T2)) / (
            w["b1"] * (1 + 2 * q) + w["b2"] * q * p * w["ne"])
        one = (w["b3"] * q * w["ne"] + w["b1"] * T1) / (w["b1"] + w["b2"] * q * w["ne"])
        return torch.where(have2, two, one)

    def step(self):
        f, g = self.f, self.g
        T = sum(g[1:], g[0]) - 0.5 * self.Q
        fn, gn = [], []
        for j in range(9):
            shift = lambda a: torch.roll(a, (_EY[j], _EX[j]), (1, 2)) if j else a  # noqa: E731, B023
            fj, gj = shift(f[j]), shift(g[j]) if j < 5 else None
            w = self.walls[j]
            if w is not None and len(w["own"]):
                own, q, i = w["own"], w["q"], _OPP[j]
                have2 = w["i2"] >= 0
                fi = f[i].reshape(-1)[own]
                val = fi
                if not w["half"]:
                    near = 2 * q * fi + (1 - 2 * q) * f[i].reshape(-1)[w["i2"].clamp(min=0)]
                    far = fi / (2 * q) + (2 * q - 1) / (2 * q) * f[j].reshape(-1)[own]
                    val = torch.where(q < 0.5, torch.where(have2, near, fi), torch.where(q > 0.5, far, fi))
                fj = fj.clone().reshape(-1)
                fj[own] = val
                fj = fj.view_as(T)
                if j < 5:
                    T1, T2 = self._T_at(T, own), self._T_at(T, w["i2"])
                    Tw = self._wall_T(w, T1, T2, have2)
                    Tm = Tw
                    if not w["half"]:
                        m, p, p2, have3 = 2 * q - 1, 1 + q, 2 + q, w["i3"] >= 0
                        T3 = self._T_at(T, w["i3"])
                        a = torch.where(have2, 3 / (4 * q * p) * Tw + 3 * m / (4 * q) * T1 - m / (4 * p) * T2,
                                        Tw + (T1 - Tw) * m / (2 * q))
                        b = torch.where(have2 & have3, 15 / (4 * p * p2) * Tw + 5 * m / (4 * p) * T2 - 3 * m / (4 * p2) * T3,
                                        torch.where(have2, Tw + (T2 - Tw) * m / (2 * p), Tw))
                        Tm = torch.where(q == 0.5, Tw, torch.where((q > 0.5) | (w["b1"] != 0), a, b))
                    gj = gj.clone().reshape(-1)
                    gj[own] = -g[i].reshape(-1)[own] + self.cT2.reshape(-1)[w["lat"]] * Tm
                    gj = gj.view_as(T)
            fn.append(fj)
            if j < 5:
                gn.append(gj)
        fs, gs = self.collide(fn, gn)
        masked = bool(self.solid.any())
        self.f = [torch.where(self.solid, a, b) if masked else b for a, b in zip(f, fs)]
        self.g = [torch.where(self.solid, a, b) if masked else b for a, b in zip(g, gs)]

    # -- results -----------------------------------------------------------
    def fields(self):
        f, g = self.f, self.g
        T = sum(g[1:], g[0]) - 0.5 * self.Q
        Fy = self.Fy + self.rho0 * self.gb * (T - self.T0)
        rho = sum(f[1:], f[0])
        ux = ((f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7]) - 0.5 * self.Fx) / rho
        uy = ((f[2] - f[4]) + (f[5] - f[7]) + (f[6] - f[8]) - 0.5 * Fy) / rho
        return [torch.where(self.solid, torch.zeros_like(a), a) for a in (rho, ux, uy, T)]

    def nusselt(self, which, length):
        """length x mean dT/dn over a box side (0..3) or the listed links of condition which - 4."""
        T = sum(self.g[1:], self.g[0]) - 0.5 * self.Q
        tot, cnt = 0.0, 0
        for j in range(1, 5):
            w = self.walls[j]
            if which < 4:
                if {0: 1, 1: 3, 2: 2, 3: 4}[which] != j:
                    continue
                y, x = (w["own"] // self.nx) % self.ny, w["own"] % self.nx
                at = {0: x == 0, 1: x == self.nx - 1, 2: y == 0, 3: y == self.ny - 1}[which]
            else:
                geom = self.geoms[0]
                listed = torch.zeros(self.ny * self.nx, dtype=torch.bool)
                sel = (geom.link_dir == _OPP[j]) & (np.asarray(geom.link_tbc) == which - 4)
                listed[torch.from_numpy(np.asarray(geom.link_node)[sel]).long()] = True
                at = listed.to(self.dev)[w["own"]]
            w = {k: v[at] for k, v in w.items() if torch.is_tensor(v)}
            have2 = w["i2"] >= 0
            T1, T2, q = self._T_at(T, w["own"]), self._T_at(T, w["i2"]), w["q"]
            Tw = self._wall_T(w, T1, T2, have2)
            p = 1 + q
            grad = torch.where(have2, ((1 + 2 * q) * Tw - p * p * T1 + q * q * T2) / (q * p * w["ne"]),
                               (Tw - T1) / (q * w["ne"]))
            tot, cnt = tot + float(grad.sum()), cnt + int(at.sum())
        return length * tot / cnt


def _exact_single(case, seed):
    w = _workload(case)
    lat = _Lattice([w], _device())
    ux, uy, T = _fields(case, w, seed)
    lat.init(ux[None], uy[None], T[None])
    before = None
    for t in range(case["steps"]):
        if t == case["steps"] - 1:
            before = lat.fields()
        lat.step()
    now = lat.fields()
    out = [a[0] for a in now]
    for what in _monitored(case):
        if what == "nusselt":
            v = lat.nusselt(4 if case["kind"] == "annulus" else 0, w.length)
        else:
            v = max(float((a - b).norm()) / max(float(a.norm()), 1e-30) for a, b in zip(now[1:], before[1:]))
        out.append(torch.tensor(v, dtype=torch.float64))
    return out


def _exact_batch(case, seed):
    ws = _batch_workloads(case, seed)
    out = [None] * 10
    # equal lattices are advanced together; of unequal ones the first eighth of the outputs is given
    groups = [list(range(len(ws)))] if case["kind"] == "batch_obstacles" else [[i] for i in range(0, len(ws), 8)]
    fields = {}
    for ids in groups:
        lat = _Lattice([ws[i] for i in ids], _device())
        lat.init(*(torch.stack(a) for a in zip(*(_fields(case, ws[i], 1000 * int(seed) + i) for i in ids))))
        for _ in range(case["steps"]):
            lat.step()
        f = torch.stack(lat.fields()[1:], 1)  # [lattice][ux, uy, T][ny][nx]
        for k, i in enumerate(ids):
            fields[i] = f[k]
    for j in range(8):
        mine = range(j, len(ws), 8)
        if all(i in fields for i in mine):
            out[j] = torch.cat([fields[i].reshape(-1) for i in mine])
    return out


def _exact_net(case, seed):
    x, t, mask, p = (a.double() for a in _net_inputs(case, seed))
    L = case["levels"]
    p.requires_grad_(case["kind"] == "net_gradients")
    off, layers = 0, []
    for ci, co, k in N.layer_shapes(case["G"], 5, 3, case["base"], L):
        n = ci * co * k * k
        layers.append((p[off:off + n].view(co, ci, k, k), p[off + n:off + n + co], k // 2))
        off += n + co
    it = iter(layers)

    def conv(a, act=True):
        w, b, pad = next(it)
        a = F.conv2d(a, w, b, padding=pad)
        return F.relu(a) if act else a

    skips = []
    for _ in range(L - 1):
        x = conv(conv(x))
        skips.append(x)
        x = F.avg_pool2d(x, 2)
    x = conv(conv(x))
    for skip in reversed(skips):
        x = conv(conv(torch.cat([F.interpolate(x, scale_factor=2, mode="nearest"), skip], 1)))
    y = conv(x, act=False)
    if case["kind"] == "net_forward":
        return [y]
    loss = (mask[:, None] * (y - t) ** 2).sum() / (mask.sum() * 3)
    loss.backward()
    return [loss.detach(), p.grad]


def exact(case, seed):
    k = case["kind"]
    if k.startswith("net"):
        return _exact_net(case, seed)
    with torch.no_grad():
        return _exact_batch(case, seed) if k.startswith("batch") else _exact_single(case, seed)
