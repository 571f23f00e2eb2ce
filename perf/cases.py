"""What a user of the library has it do, as timed cases.

The library advances regularised Herschel-Bulkley flow in a box by time steps
(``HBFlow.step``), runs the start-up / cessation study on top of them, sweeps
many cavities at once (``Batch``), offers the stages of the step one by one,
and evaluates and trains the network of the learned initial guess (``UNet``).
Every case goes through those entry points.  A step is run the way a driver
restarts one: velocity and pressure set from device arrays, one step, both
read back into device arrays.

Cases are dicts of plain values; ``prepare`` makes the inputs on the GPU from
the seed alone (seeded smooth velocity and pressure, decaying away from the
lid, so that sheared regions and unyielded plugs are both there, as in a
developed cavity).  ``exact`` restates the explicit stages, the whole step on
small 2D grids (direct solves) and the network in 64-bit torch.
"""

import math

import numpy as np
import torch

from paper_1803_00417_gb300.hbflow import FP64, MIXED, Batch, HBFlow, UNet

CHANNELS = (16, 32, 64, 128)


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def _flow(kind, n, precision, Re, nexp, Bi, Pa, dt_h=0.5, **more):
    c = {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2] if len(n) == 3 else 0, "precision": precision, "Re": Re,
         "nexp": nexp, "Bi": Bi, "Pa": Pa, "dt_h": dt_h}
    c.update(more)
    return c


def _net(kind, n):
    return {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2] if len(n) == 3 else 0}


def listed():
    return [
        # the smallest workload a user starts with: the 2D Bingham cavity in FP64; many short launches
        dict(_flow("step", (64, 64), "fp64", 1.0, 1.0, 2.0, 1e4), name="cavity2d_64_fp64"),
        # the paper's main experiment: lid stopped, steps and the yield test until the fluid rests (2D, 256^2, FP64)
        dict(_flow("cessation", (256, 256), "fp64", 1.0, 1.0, 10.0, 400.0, dt_h=0.00256, steps=3),
             name="cessation2d_256_fp64"),
        # a large 2D shear-thinning cavity in mixed precision
        dict(_flow("step", (1024, 1024), "mixed", 1000.0, 0.5, 5.0, 1e5), name="cavity2d_1024_mixed"),
        # the headline workload: the 3D shear-thickening cavity at full size, mixed precision
        dict(_flow("step", (256, 256, 256), "mixed", 100.0, 1.5, 10.0, 1e5), name="cavity3d_256_mixed"),
        # the same flow at an ordinary size with the plain FP64 method
        dict(_flow("step", (128, 128, 128), "fp64", 100.0, 1.5, 10.0, 1e5), name="cavity3d_128_fp64"),
        # a small 3D Bingham cavity (the low end of the rate-against-N study)
        dict(_flow("step", (32, 32, 32), "mixed", 1.0, 1.0, 10.0, 400.0), name="cavity3d_32_mixed"),
        # a box that is no power of two: the multigrid stops coarsening at 9 x 7 x 5 cells
        dict(_flow("step", (72, 56, 40), "mixed", 100.0, 1.0, 5.0, 1e4), name="cavity3d_72x56x40_mixed"),
        # channel flow between two walls, periodic along the other axes, driven by a body force
        dict(_flow("step", (96, 64, 64), "mixed", 10.0, 0.8, 2.0, 1e4, periodic=True), name="channel3d_96x64x64_mixed"),
        # a parameter sweep: uneven 2D cavities advanced together
        {"kind": "batch", "cavities": 16, "lo": 64, "hi": 256, "precision": "mixed", "name": "sweep2d_16_mixed"},
        # the explicit stages alone (viscosity, gradients, Godunov predictor), as a user studying the scheme calls them
        dict(_flow("predict", (128, 128, 128), "fp64", 100.0, 1.5, 10.0, 1e5), name="predict3d_128"),
        # one gradient evaluation of the initial-guess network at its training size
        dict(_net("net_gradient", (32, 32, 32)), name="net_gradient3d_32"),
        # one inference of it on the nodes of the 256^3 workload's second coarse level
        dict(_net("net_forward", (72, 72, 72)), name="net_forward3d_72"),
    ]


def _even_box(rng, d, lo, hi, cells):
    """Sizes b_a 2^k with 4 <= b_a <= 10, from lo to hi cells along an axis and at most `cells` in all: the
    hierarchy then ends on a small level, of even or odd sizes."""
    while True:
        ks = [k for k in range(1, 9) if 4 << k <= hi and 10 << k >= lo]
        k = rng.choice(ks)
        n = [rng.randint(4, 10) << k for _ in range(d)]
        if min(n) >= lo and max(n) <= hi and math.prod(n) <= cells:
            return n


def draw(rng):
    kind = rng.choice(("step", "step", "step", "step", "step", "cessation", "batch", "predict", "net_gradient",
                       "net_forward"))
    if kind == "batch":
        lo = rng.choice((16, 32, 64))
        return {"kind": kind, "cavities": rng.randint(2, 24), "lo": lo, "hi": lo * rng.choice((2, 4)),
                "precision": rng.choice(("mixed", "fp64"))}
    if kind in ("net_gradient", "net_forward"):
        d = rng.choice((2, 3))
        top = {("net_gradient", 2): 256, ("net_gradient", 3): 48, ("net_forward", 2): 512, ("net_forward", 3): 96}
        lo, hi = 16, top[kind, d]
        side = lambda: 8 * round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 8)  # noqa: E731
        return _net(kind, [side() for _ in range(d)])
    d = 2 if kind == "cessation" else rng.choice((2, 3, 3))
    precision = rng.choice(("fp64", "mixed"))
    rheo = (math.exp(rng.uniform(0.0, math.log(1000.0))), rng.uniform(0.5, 1.5), rng.uniform(0.0, 20.0), 1e4)
    if kind == "cessation":
        n = _even_box(rng, 2, 32, 320, 320 * 320)
        return _flow(kind, n, precision, 1.0, 1.0, rng.uniform(1.0, 10.0), 400.0, dt_h=0.00256, steps=3)
    if d == 2:
        n = _even_box(rng, 2, 16, 1024, 1024 * 1024)
    else:
        n = _even_box(rng, 3, 16, 256, 110 ** 3 if precision == "fp64" else 160 ** 3)
    if kind == "predict":
        return _flow(kind, n, precision, *rheo)
    return _flow(kind, n, precision, *rheo, dt_h=rng.choice((0.25, 0.5)), periodic=rng.random() < 0.25)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _sizes(case):
    return [case["nx"], case["ny"]] + ([case["nz"]] if case["nz"] else [])


def _periodic(case, d):
    # channel: walls on the last axis only
    return [bool(case.get("periodic")) and a < d - 1 for a in range(d)]


def _axes(n, centred):
    """Coordinates in the unit cube along each axis, shaped to broadcast over arrays indexed [(z,) y, x]."""
    d = len(n)
    out = []
    for a in range(d):
        m = n[a] if centred else n[a] + 1
        x = (torch.arange(m, dtype=torch.float64, device="cuda") + (0.5 if centred else 0.0)) / n[a]
        out.append(x.reshape([m if b == d - 1 - a else 1 for b in range(d)]))
    return out


def _modes(rng, axes, per, kmax=4, count=8):
    """A sum of random product modes: cos(pi k x) across walls, cos(2 pi k x + phase) along periodic axes."""
    out = 0.0
    for _ in range(count):
        term, norm = float(rng.normal()), 1.0
        for a, x in enumerate(axes):
            k = int(rng.integers(0, kmax + 1))
            norm += k * k
            term = term * torch.cos(2 * math.pi * k * x + float(rng.uniform(0, 2 * math.pi)) if per[a] else
                                    math.pi * k * x)
        out = out + term / math.sqrt(norm)
    return out


def _state(n, per, seed):
    """Seeded velocity (the curl of a smooth potential that vanishes at the walls and decays away from the top one;
    largest component 0.5) and nodal pressure, flat in the library's layout."""
    d = len(n)
    rng = np.random.default_rng(seed)
    ax = _axes(n, centred=False)  # potential on the nodes, differences at cell centres
    env = torch.exp(-(1.0 - ax[d - 1]) / float(rng.uniform(0.1, 0.25)))
    for a in range(d):
        if not per[a]:
            env = env * torch.sin(math.pi * ax[a]) ** 2
    h = 1.0 / max(n)

    def diff(f, a):
        g = f.diff(dim=d - 1 - a) / h
        for b in range(d):
            if b != a:
                m = f.shape[d - 1 - b] - 1
                g = 0.5 * (g.narrow(d - 1 - b, 0, m) + g.narrow(d - 1 - b, 1, m))
        return g

    pot = [env * (_modes(rng, ax, per) + 1.0) for _ in range(1 if d == 2 else 3)]
    if d == 2:
        u = [diff(pot[0], 1), -diff(pot[0], 0)]
    else:
        u = [diff(pot[2], 1) - diff(pot[1], 2), diff(pot[0], 2) - diff(pot[2], 0), diff(pot[1], 0) - diff(pot[0], 1)]
    u = torch.stack([torch.broadcast_to(c, tuple(reversed(n))) for c in u])
    u = (u * (0.5 / u.abs().max())).reshape(-1).contiguous()
    p = torch.broadcast_to(_modes(rng, ax, per), tuple(v + 1 for v in reversed(n)))
    p = (p * (0.1 / p.abs().max())).clone()
    for a in range(d):
        if per[a]:  # the last node along a periodic axis repeats the first
            p.narrow(d - 1 - a, n[a], 1).copy_(p.narrow(d - 1 - a, 0, 1))
    return u, p.reshape(-1).contiguous()


def _walls(d, per):
    w = np.zeros((d, 2, d))
    if not any(per):
        w[d - 1, 1, 0] = 1.0  # the lid
    return w


def _physics(case, d):
    """(K, n, tau_y, m, body force) of a case."""
    return (2.0 ** (1.0 - case["nexp"]) / case["Re"], case["nexp"], case["Bi"] / case["Re"], case["Pa"],
            [1.0 if case.get("periodic") and a == 0 else 0.0 for a in range(d)])


def _precision(case):
    return MIXED if case["precision"] == "mixed" else FP64


def _context(case):
    n = _sizes(case)
    d = len(n)
    per = _periodic(case, d)
    h = 1.0 / max(n)
    sim = HBFlow(n, h, _walls(d, per), precision=_precision(case))
    K, nexp, tau_y, m, f = _physics(case, d)
    sim.set_rheology(K, nexp, tau_y, m)
    if any(per):
        sim.set_periodic(per)
        sim.set_body_force(f)
    return sim, n, per, case["dt_h"] * h


def _net_shapes(d):
    """(c_in stored, c_in used, c_out) of the 3^d convolutions of the network, in order (the flat parameter vector's)."""
    c = CHANNELS
    convs = [(1, c[0])] + [(a, b) for a, b in ((c[0], c[0]), (c[0], c[1]), (c[1], c[1]), (c[1], c[2]), (c[2], c[2]),
                                               (c[2], c[3]), (c[3], c[3]), (c[3] + c[2], c[2]), (c[2], c[2]),
                                               (c[2] + c[1], c[1]), (c[1], c[1]), (c[1] + c[0], c[0]), (c[0], c[0]))]
    return [(max(16, a), a, b) for a, b in convs]


def _net_params(d, seed):
    """He-normal weights as the flat vector of hbf_unet_set_params: W[tap][c_out][c_in], b[c_out], ..., head."""
    rng = np.random.default_rng(seed)
    flat = []
    for stored, used, co in _net_shapes(d):
        w = np.zeros((3 ** d, co, stored), dtype=np.float32)
        w[:, :, :used] = rng.normal(size=(3 ** d, co, used)) * math.sqrt(2.0 / (3 ** d * used))
        flat += [w.ravel(), rng.uniform(-0.05, 0.05, size=co).astype(np.float32)]
    flat += [(rng.normal(size=CHANNELS[0]) * math.sqrt(1.0 / CHANNELS[0])).astype(np.float32),
             np.zeros(1, dtype=np.float32)]
    return np.concatenate(flat)


def _net_data(n, seed):
    """Input and target (smooth, max 1) and mask, one FP32 value a point, x fastest."""
    rng = np.random.default_rng(seed + 1)
    ax = _axes(n, centred=True)
    per = [False] * len(n)
    shape = tuple(reversed(n))
    xt = []
    for _ in range(2):
        f = torch.broadcast_to(_modes(rng, ax, per, kmax=6), shape)
        xt.append((f / f.abs().max()).float().reshape(-1).contiguous())
    return xt[0], xt[1], torch.ones_like(xt[0])


def _cavities(case, seed):
    """Sizes and rheologies of a sweep.  The sizes are the case's: side lengths lo, ..., hi in turn; the rheologies and
    states are the seed's."""
    rng = np.random.default_rng(seed)
    sides = []
    s = case["lo"]
    while s <= case["hi"]:
        sides += [s, s * 3 // 2] if s * 3 // 2 <= case["hi"] else [s]
        s *= 2
    out = []
    for i in range(case["cavities"]):
        n = sides[i % len(sides)]
        out.append(dict(n=[n, n], Re=float(np.exp(rng.uniform(0.0, math.log(1000.0)))), Bi=float(rng.uniform(0.0, 20.0)),
                        nexp=float(rng.uniform(0.5, 1.5)), Pa=1e4, seed=int(rng.integers(1 << 30))))
    return out


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "batch":
        cav = _cavities(case, seed)
        s["batch"] = Batch([c["n"] for c in cav], [1.0 / c["n"][0] for c in cav], [_walls(2, [False] * 2)] * len(cav),
                           precision=_precision(case))
        s["in"], s["out"] = [], []
        for i, c in enumerate(cav):
            K, nexp, tau_y, m, _ = _physics(c, 2)
            s["batch"].cavity(i).set_rheology(K, nexp, tau_y, m)
            u, p = _state(c["n"], [False] * 2, c["seed"])
            s["in"].append((u, p))
            s["out"].append({"u": torch.empty_like(u), "p": torch.empty_like(p)})
        s["batch"].set_dt([0.5 / c["n"][0] for c in cav])
        return s
    if kind in ("net_gradient", "net_forward"):
        n = _sizes(case)
        s["net"] = UNet(n, train=kind == "net_gradient")
        s["net"].set_params(_net_params(len(n), seed))
        s["x"], s["t"], s["mask"] = _net_data(n, seed)
        s["y"], s["gy"] = torch.empty_like(s["x"]), torch.empty_like(s["x"])
        return s
    s["sim"], n, per, s["dt"] = _context(case)
    s["u0"], s["p0"] = _state(n, per, seed)
    if kind == "predict":
        s["out"] = {k: torch.empty(s["sim"].field_size(k.upper()), dtype=torch.float64, device="cuda")
                    for k in ("eta", "gp", "lu", "ul", "ur", "uadv")}
    else:
        s["u"], s["p"] = torch.empty_like(s["u0"]), torch.empty_like(s["p0"])
    if kind == "cessation":
        s["record"], s["steps"] = s["sim"].get_state(with_fields=False)[0], case["steps"]
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s):
    kind = s["kind"]
    if kind == "step":
        sim = s["sim"]
        sim.set_field("U", s["u0"])
        sim.set_field("P", s["p0"])
        sim.step(s["dt"])
        return {"u": sim.get_field("U", s["u"]), "p": sim.get_field("P", s["p"])}
    if kind == "cessation":
        sim = s["sim"]
        sim.set_state(s["record"], s["u0"], s["p0"])  # the lid moves again
        info = sim.run_cessation(s["dt"], max_steps=s["steps"], damp_steps=1)
        return {"u": sim.get_field("U", s["u"]), "p": sim.get_field("P", s["p"]), "tau_ratio": info["tau_ratio"],
                "steps": info["steps"]}
    if kind == "batch":
        b = s["batch"]
        for i, (u, p) in enumerate(s["in"]):
            b.cavity(i).set_field("U", u)
            b.cavity(i).set_field("P", p)
        b.step()
        for i, o in enumerate(s["out"]):
            b.cavity(i).get_field("U", o["u"])
            b.cavity(i).get_field("P", o["p"])
        return s["out"]
    if kind == "predict":
        sim = s["sim"]
        sim.set_field("U", s["u0"])
        sim.set_field("P", s["p0"])
        sim.compute_viscosity()
        sim.predict(s["dt"])
        return {k: sim.get_field(k.upper(), v) for k, v in s["out"].items()}
    net = s["net"]
    net.forward(s["x"], s["y"])
    if kind == "net_forward":
        return s["y"]
    loss = net.loss(s["t"], s["mask"], s["gy"])
    net.zero_grads()
    net.backward(s["gy"])
    return {"y": s["y"], "loss": loss, "gy": s["gy"], "grads": net.get_grads()}


# ---------------------------------------------------------------------------
# the work of a pass
# ---------------------------------------------------------------------------
def _net_flops(n):
    """Multiply-adds of one forward pass, times two."""
    d, pts = len(n), math.prod(n)
    levels = (0, 0, 1, 1, 2, 2, 3, 3, 2, 2, 1, 1, 0, 0)
    return sum(2.0 * 3 ** d * used * co * pts / 2 ** (d * lv) for (_, used, co), lv in zip(_net_shapes(d), levels))


def work(case):
    kind = case["kind"]
    if kind in ("net_gradient", "net_forward"):
        n = _sizes(case)
        pts, params = math.prod(n), _net_params(len(n), 0).size
        if kind == "net_forward":
            return {"bytes": 8.0 * pts + 4.0 * params, "flops": _net_flops(n)}
        # forward, the gradient of the inputs and that of the weights
        return {"bytes": 20.0 * pts + 8.0 * params, "flops": 3.0 * _net_flops(n)}
    if kind == "batch":
        boxes, steps = [c["n"] for c in _cavities(case, 0)], 1
    else:
        boxes, steps = [_sizes(case)], case.get("steps", 1)
    d = len(boxes[0])
    cells = sum(math.prod(n) for n in boxes)
    nodes = sum(math.prod(v + 1 for v in n) for n in boxes)
    explicit = 250.0 if d == 2 else 900.0  # operations per cell of the viscosity, the gradients and the predictor
    if kind == "predict":
        faces = sum(math.prod(n) // n[a] * (n[a] + 1) for n in boxes for a in range(d))
        return {"bytes": 8.0 * ((3 * d + 1) * cells + nodes + (2 * d + 1) * faces), "flops": explicit * cells}
    # velocity and pressure in and out; the three solves to ten digits at one V(2,2) cycle a digit
    cycle = 300.0 if d == 2 else 1300.0
    return {"bytes": 16.0 * (d * cells + nodes), "flops": steps * (explicit + 10 * cycle) * cells}


# ---------------------------------------------------------------------------
# 64-bit torch restatement.  Arrays [..., (z,) y, x]: axis a is dim -(a + 1).
# ---------------------------------------------------------------------------
class _Box:
    def __init__(self, n, per, walls):
        self.n, self.d, self.per, self.walls, self.h = n, len(n), per, walls, 1.0 / max(n)

    def wall(self, a, side, c, hom):
        return 0.0 if hom else float(self.walls[a, side, c])

    def part(self, f, a, lo, count):
        return f.narrow(-(a + 1), lo, count)

    def pad_axis(self, f, a, g, kind, c=0, hom=False):
        m, dim = f.shape[-(a + 1)], -(a + 1)
        if self.per[a]:
            lo, hi = f.narrow(dim, m - g, g), f.narrow(dim, 0, g)
        else:
            lo, hi = f.narrow(dim, 0, g).flip(dim), f.narrow(dim, m - g, g).flip(dim)
            if kind == "dirichlet":
                lo, hi = 2.0 * self.wall(a, 0, c, hom) - lo, 2.0 * self.wall(a, 1, c, hom) - hi
            elif kind == "zero":
                lo, hi = torch.zeros_like(lo), torch.zeros_like(hi)
        return torch.cat([lo, f, hi], dim)

    def pad(self, f, g, kind, c=0, hom=False):
        for a in range(self.d):
            f = self.pad_axis(f, a, g, kind, c, hom)
        return f

    def inner(self, f, g, skip=()):
        for a in range(self.d):
            if a not in skip:
                f = self.part(f, a, g, f.shape[-(a + 1)] - 2 * g)
        return f

    def diff(self, f, a, k=1):
        m = f.shape[-(a + 1)]
        return self.part(f, a, k, m - k) - self.part(f, a, 0, m - k)

    def mean(self, f, a):
        m = f.shape[-(a + 1)]
        return 0.5 * (self.part(f, a, 1, m - 1) + self.part(f, a, 0, m - 1))

    def mask_walls(self, f, a):
        if not self.per[a]:
            f = f.clone()
            f.narrow(-(a + 1), 0, 1).zero_()
            f.narrow(-(a + 1), self.n[a], 1).zero_()
        return f

    def node_full(self, f):
        """A node array with n + 1 points, padded by one: even reflection, or the wrap that skips the repeated node."""
        for a in range(self.d):
            m, dim = f.shape[-(a + 1)], -(a + 1)
            k = m - 2  # even reflection about the end node, and the wrap, both take the second node from an end
            lo, hi = (f.narrow(dim, k, 1), f.narrow(dim, 1, 1)) if self.per[a] else (f.narrow(dim, 1, 1),
                                                                                    f.narrow(dim, k, 1))
            f = torch.cat([lo, f, hi], dim)
        return f

    # -- operators ---------------------------------------------------------
    def viscosity(self, u, K, nexp, tau_y, m):
        up = [self.pad(u[c], 1, "dirichlet", c) for c in range(self.d)]
        s = 0.0
        for i in range(self.d):
            for j in range(self.d):
                gij = self.inner(self.diff(up[j], i, 2), 1, (i,)) / (2 * self.h)
                gji = self.inner(self.diff(up[i], j, 2), 1, (j,)) / (2 * self.h)
                s = s + (0.5 * (gij + gji)) ** 2
        g = torch.sqrt(0.5 * s)
        x = m * g
        F = torch.where(x < 1e-5, m * (1 - x / 2 + x * x / 6), -torch.expm1(-x) / g.clamp_min(1e-300))
        return (2.0 ** (nexp - 1) * K * g ** nexp + 0.5 * tau_y) * F

    def face_eta(self, eta):
        return [self.mean(self.pad_axis(eta, a, 1, "neumann"), a) for a in range(self.d)]

    def stress_div(self, u, ef, hom=False):
        """div(eta (grad u + grad u^T)), u a list of components."""
        up = [self.pad(u[c], 1, "dirichlet", c, hom) for c in range(self.d)]
        out = []
        for c in range(self.d):
            acc = 0.0
            for a in range(self.d):
                nrm = self.inner(self.diff(up[c], a), 1, (a,)) / self.h
                if a == c:
                    flux = 2.0 * ef[a] * nrm
                else:
                    x = self.inner(self.diff(up[a], c, 2), 1, (a, c)) / (2 * self.h)
                    flux = ef[a] * (nrm + self.mask_walls(self.mean(x, a), a))
                acc = acc + self.diff(flux, a) / self.h
            out.append(acc)
        return out

    def grad(self, p):
        out = []
        for a in range(self.d):
            g = self.diff(p, a) / self.h
            for b in range(self.d):
                if b != a:
                    g = self.mean(g, b)
            out.append(g)
        return out

    def slopes(self, uc, a, c):
        up = self.pad_axis(uc, a, 2, "dirichlet", c)
        n = self.n[a]
        dl, dc = self.diff(up, a), 0.5 * self.diff(up, a, 2)
        lo, hi = self.part(dl, a, 0, n + 2), self.part(dl, a, 1, n + 2)
        lim = torch.where(lo * hi > 0, 2.0 * torch.minimum(lo.abs(), hi.abs()), torch.zeros_like(lo))
        df = torch.sign(dc) * torch.minimum(dc.abs(), lim)
        d4 = 4.0 / 3.0 * self.part(dc, a, 1, n) - (self.part(df, a, 2, n) + self.part(df, a, 0, n)) / 6.0
        return torch.sign(d4) * torch.minimum(d4.abs(), self.part(lim, a, 1, n))

    def to_faces(self, left, right, a, c):
        """Extrapolated cell values to the a-faces: from the cell below and from the cell above; walls take theirs."""
        m, dim = self.n[a], -(a + 1)
        if self.per[a]:
            return torch.cat([left.narrow(dim, m - 1, 1), left], dim), torch.cat([right, right.narrow(dim, 0, 1)], dim)
        w = [torch.full_like(left.narrow(dim, 0, 1), self.wall(a, s, c, False)) for s in (0, 1)]
        return (torch.cat([w[0], left.narrow(dim, 0, m - 1), w[1]], dim),
                torch.cat([w[0], right.narrow(dim, 1, m - 1), w[1]], dim))

    @staticmethod
    def riemann(l, r):
        z = torch.zeros_like(l)
        return torch.where((l > 0) & (l + r > 0), l, torch.where((r < 0) & (l + r < 0), r, z))

    @staticmethod
    def upwind(l, r, v):
        return torch.where(v > 0, l, torch.where(v < 0, r, 0.5 * (l + r)))

    def predictor(self, u, F, dt):
        """Left and right face states [a][c] and the advection velocity [a]."""
        d, h = self.d, self.h
        S = [[self.slopes(u[c], a, c) for c in range(d)] for a in range(d)]
        hats = [[None] * d for _ in range(d)]
        for b in range(d):
            fl, fr = 0.5 - u[b] * dt / (2 * h), 0.5 + u[b] * dt / (2 * h)
            pre = [self.to_faces(u[c] + fl * S[b][c], u[c] - fr * S[b][c], b, c) for c in range(d)]
            v = self.riemann(*pre[b])
            for c in range(d):
                st = v if c == b else self.upwind(*pre[c], v)
                hats[b][c] = self.mean(v, b) * self.diff(st, b) / h
        uL, uR, adv = [], [], []
        for a in range(d):
            fl, fr = 0.5 - u[a] * dt / (2 * h), 0.5 + u[a] * dt / (2 * h)
            st = []
            for c in range(d):
                com = 0.5 * dt * (F[c] - sum(hats[b][c] for b in range(d) if b != a))
                st.append(self.to_faces(u[c] + fl * S[a][c] + com, u[c] - fr * S[a][c] + com, a, c))
            uL.append([q[0] for q in st])
            uR.append([q[1] for q in st])
            adv.append(self.mask_walls(self.riemann(*st[a]), a))
        return uL, uR, adv

    def explicit(self, u, p, physics, dt):
        K, nexp, tau_y, m, f = physics
        eta = self.viscosity(u, K, nexp, tau_y, m)
        gp = self.grad(p)
        ef = self.face_eta(eta)
        lu = self.stress_div(u, ef)
        uL, uR, adv = self.predictor(u, [-gp[c] + f[c] for c in range(self.d)], dt)
        return eta, ef, gp, lu, uL, uR, adv

    def cell_lap(self, phi):
        return sum(self.diff(self.mask_walls(self.diff(self.pad_axis(phi, a, 1, "neumann"), a), a), a)
                   for a in range(self.d)) / self.h ** 2

    def node_lap(self, phi):
        """The finite-element Laplacian of a 2D node array (walls on both axes)."""
        f = self.node_full(phi)
        s = sum(f.narrow(-1, i, phi.shape[-1]).narrow(-2, j, phi.shape[-2]) for i in range(3) for j in range(3))
        return (s - 9.0 * phi) / (3.0 * self.h ** 2)

    def node_div(self, v):
        """Divergence of a 2D cell field at the nodes: existing cells only, over the dual cell's share."""
        p = [self.pad(c, 1, "zero") for c in v]
        w = self.node_share(p[0])
        return (self.mean(self.diff(p[0], 0), 1) + self.mean(self.diff(p[1], 1), 0)) / (self.h * w)

    def node_share(self, like):
        w = torch.ones_like(self.mean(self.mean(like, 0), 1))
        for a in range(self.d):
            w.narrow(-(a + 1), 0, 1).mul_(0.5)
            w.narrow(-(a + 1), self.n[a], 1).mul_(0.5)
        return w

    @staticmethod
    def direct(op, b, weights=None):
        """The solution of op(x) = b by a dense factorisation (op linear, over leading batch dims); with weights, the
        one of weighted mean zero, for the b without its weighted mean."""
        shape, n = b.shape, b.numel()
        A = torch.empty(n, n, dtype=torch.float64, device=b.device)
        for k in range(0, n, 512):
            m = min(512, n - k)
            e = torch.zeros(m, n, dtype=torch.float64, device=b.device)
            e[torch.arange(m), torch.arange(k, k + m)] = 1.0
            A[:, k:k + m] = op(e.reshape(m, *shape)).reshape(m, n).T
        r = b.reshape(n, 1).clone()
        if weights is not None:
            w = weights.reshape(n, 1)
            r -= (w * r).sum() / w.sum()
            A += A.abs().max() / n * w.T
        x = torch.linalg.solve(A, r)
        x += torch.linalg.solve(A, r - A @ x)
        if weights is not None:
            x -= (w * x).sum() / w.sum()
        return x.reshape(shape)

    def step2d(self, u, p, physics, dt):
        """One whole step between walls in 2D by direct solves."""
        eta, ef, gp, lu, uL, uR, adv = self.explicit(u, p, physics, dt)
        div = sum(self.diff(adv[a], a) for a in range(2)) / self.h
        phi = self.direct(self.cell_lap, div, torch.ones_like(div))
        mac = [adv[a] - self.mask_walls(self.diff(self.pad_axis(phi, a, 1, "neumann"), a), a) / self.h
               for a in range(2)]
        rhs = []
        for c in range(2):
            A = sum(self.mean(mac[a], a) * self.diff(self.upwind(uL[a][c], uR[a][c], mac[a]), a) / self.h
                    for a in range(2))
            rhs.append(u[c] - dt * A + dt * (-gp[c] + 0.5 * lu[c] + physics[4][c]))
        beta = 0.5 * dt
        zero = [torch.zeros_like(u[0]), torch.zeros_like(u[1])]
        wall = self.stress_div(zero, ef)  # what the walls' velocity adds

        def op(x):
            v = [x[..., 0, :, :], x[..., 1, :, :]]
            L = self.stress_div(v, ef, hom=True)
            return torch.stack([v[c] - beta * L[c] for c in range(2)], -3)

        us = self.direct(op, torch.stack([rhs[c] + beta * wall[c] for c in range(2)]))
        b = self.node_div([us[c] / dt + gp[c] for c in range(2)])
        phi = self.direct(self.node_lap, b, self.node_share(self.pad(us[0], 1, "zero")))
        gphi = self.grad(phi)
        return torch.stack([us[c] + dt * (gp[c] - gphi[c]) for c in range(2)]), phi


def _net_exact(case, seed):
    n = _sizes(case)
    d = len(n)
    flat = torch.from_numpy(_net_params(d, seed)).to("cuda", torch.float64).requires_grad_(True)
    x, t, mask = (v.double().reshape(1, 1, *reversed(n)) for v in _net_data(n, seed))
    conv = torch.nn.functional.conv2d if d == 2 else torch.nn.functional.conv3d
    at, layers = 0, []
    for stored, used, co in _net_shapes(d):
        w = flat[at:at + 3 ** d * co * stored].reshape(*(3,) * d, co, stored)[..., :used]
        at += 3 ** d * co * stored
        # taps run over (x, y(, z)) offsets, x slowest; the arrays are indexed [(z,) y, x]
        w = w.permute(d, d + 1, *reversed(range(d)))
        layers.append((w, flat[at:at + co]))
        at += co
    it = iter(layers)

    def block(h):
        for _ in range(2):
            w, b = next(it)
            h = torch.relu(conv(h, w, b, padding=1))
        return h

    pool = torch.nn.functional.avg_pool2d if d == 2 else torch.nn.functional.avg_pool3d
    h, skips = x, []
    for _ in range(3):
        h = block(h)
        skips.append(h)
        h = pool(h, 2)
    h = block(h)
    for sk in reversed(skips):
        h = block(torch.cat([torch.nn.functional.interpolate(h, scale_factor=2, mode="nearest"), sk], 1))
    wh, bh = flat[at:at + CHANNELS[0]], flat[at + CHANNELS[0]]
    y = (h * wh.reshape(1, -1, *(1,) * d)).sum(1, keepdim=True) + bh
    if case["kind"] == "net_forward":
        return y.detach().reshape(-1)
    r = (y - t) * mask
    loss = (r * r).sum() / mask.sum()
    gy, grads = torch.autograd.grad(loss, (y, flat))
    return {"y": y.detach().reshape(-1), "loss": float(loss), "gy": gy.reshape(-1), "grads": grads.cpu().numpy()}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("net_gradient", "net_forward"):
        return _net_exact(case, seed)
    if kind not in ("predict", "step"):
        return None
    n = _sizes(case)
    d = len(n)
    per = _periodic(case, d)
    if kind == "step" and (d == 3 or any(per) or 2 * math.prod(n) > 10000):
        return None  # the direct solves are dense
    box = _Box(n, per, _walls(d, per))
    u, p = _state(n, per, seed)
    u, p = u.reshape(d, *reversed(n)), p.reshape([v + 1 for v in reversed(n)])
    dt = case["dt_h"] * box.h
    if kind == "step":
        un, pn = box.step2d([u[0], u[1]], p, _physics(case, d), dt)
        return {"u": un.reshape(-1), "p": pn.reshape(-1)}
    eta, _, gp, lu, uL, uR, adv = box.explicit(list(u), p, _physics(case, d), dt)
    flat = lambda v: torch.cat([x.reshape(-1) for x in v])  # noqa: E731
    return {"eta": eta.reshape(-1), "gp": flat(gp), "lu": flat(lu), "ul": flat([x for a in uL for x in a]),
            "ur": flat([x for a in uR for x in a]), "uadv": flat(adv)}
