"""The work that a user of this library has it do, as cases that can be timed and checked.

Every case starts from a seeded relativistic double Harris sheet (the state the
library's own configurations, tests and benchmark use) and goes through the
Python binding: simulations in 2D (linear and quadratic shapes) and 3D, in both
precisions, from a 64x32 box to the full-size 2D and 3D runs; a batch of
independent instances; one step's adjoint and the gradient of a whole window;
and the load of a particle record with the diagnostics taken from it.

The library hands every floating result over in FP64 arrays. In its FP32 form
those values were computed in FP32, so they are given here as float32.
"""
import math

import numpy as np
import torch

import paper_2509_11100_gb300 as rs
from paper_2509_11100_gb300.window import ModeEnergyWindow

THETA_T, DELTA, SIGMA = 0.3, 1.0, 10.0      # temperature, sheet half-thickness, magnetisation
SCAN_LX, SCAN_DELTA, SCAN_SIGMA = (128, 192, 256, 384), (0.5, 1.0, 2.0), (1.0, 10.0, 40.0)
Q = (1.0, -1.0)                             # positrons, electrons (unit masses)
EXACT_MOST = 3.0e7                          # particle-steps that 64-bit arithmetic does in seconds
BINS = np.geomspace(1e-2, 1e4, 257)         # 256 logarithmic bins of gamma - 1


def listed():
    return [
        # the small validation run in double precision: a step is all launches and latency
        dict(name="step_64x32_f64", kind="step", shape=1, precision=64, nx=64, ny=32, nz=0, ppc=16, pred=False,
             dt=0.5, steps=10),
        # the smallest box of a tearing scan in the FP32 form
        dict(name="step_128x64_f32", kind="step", shape=1, precision=32, nx=128, ny=64, nz=0, ppc=32, pred=False,
             dt=0.5, steps=10),
        # a box whose sides are multiples of nothing, an odd number of particles a cell
        dict(name="step_251x99_f32", kind="step", shape=1, precision=32, nx=251, ny=99, nz=0, ppc=21, pred=True,
             dt=0.7, steps=6),
        # the full-size 2D reconnection run
        dict(name="step_1024x512_f32", kind="step", shape=1, precision=32, nx=1024, ny=512, nz=0, ppc=64, pred=True,
             dt=1.0, steps=6),
        # the double-precision form as a check on a medium FP32 run
        dict(name="step_256x128_f64", kind="step", shape=1, precision=64, nx=256, ny=128, nz=0, ppc=32, pred=True,
             dt=1.0, steps=3),
        # smoother (quadratic) particles
        dict(name="step_quad_512x256_f32", kind="step", shape=2, precision=32, nx=512, ny=256, nz=0, ppc=64,
             pred=False, dt=1.0, steps=3),
        # a small 3D box
        dict(name="step_3d_64x32x32_f32", kind="step", shape=1, precision=32, nx=64, ny=32, nz=32, ppc=16,
             pred=False, dt=0.5, steps=6),
        # the full-size 3D run
        dict(name="step_3d_256x128x128_f32", kind="step", shape=1, precision=32, nx=256, ny=128, nz=128, ppc=16,
             pred=False, dt=0.5, steps=3),
        # a parameter scan: uneven independent boxes advanced together, the tearing modes recorded
        dict(name="batch_8_f32", kind="batch", shape=1, precision=32, count=8, ppc=32, pred=False, dt=0.5, steps=5,
             pick=3),
        # the reverse pass of one step: gradients of fields and particles
        dict(name="adjoint_256x128_f32", kind="adjoint", shape=1, precision=32, nx=256, ny=128, nz=0, ppc=32,
             pred=False, dt=0.5, steps=1),
        # the gradient of a late mode energy in the initial state, forward and backward
        dict(name="window_128x64_f32", kind="window", shape=1, precision=32, nx=128, ny=64, nz=0, ppc=32, pred=False,
             dt=0.5, steps=10),
        # a restart from an unsorted FP64 record, with the diagnostics of the loaded state
        dict(name="load_512x256_f32", kind="load", shape=1, precision=32, nx=512, ny=256, nz=0, ppc=32, pred=False,
             dt=1.0, steps=1, shuffled=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the ranges above: sizes spread over their logarithm, odd ones among them."""
    kind = rng.choice(("step",) * 6 + ("batch", "adjoint", "window", "load"))
    precision = rng.choice((32, 32, 32, 64))
    c = dict(kind=kind, shape=1, precision=precision, nz=0, pred=rng.random() < 0.5, dt=rng.choice((0.5, 0.7, 1.0)),
             steps=1)
    if kind == "batch":
        c.update(precision=32, count=rng.randint(2, 8), ppc=_log(rng, 8, 40), dt=0.5, steps=rng.randint(2, 5),
                 pick=rng.randint(0, 9999))
        return c
    most = 6.0e7 if precision == 32 else 4.0e6
    if kind == "step":
        form = rng.choice(("2d", "2d", "3d", "3d", "quad"))
        c["steps"] = rng.randint(2, 6)
        if form == "3d":
            c.update(nx=_log(rng, 12, 256), ny=_log(rng, 10, 128), nz=_log(rng, 8, 128), ppc=_log(rng, 4, 32),
                     pred=False)
        else:
            c.update(nx=_log(rng, 32, 1024), ny=_log(rng, 20, 512), ppc=_log(rng, 4, 100))
        if form == "quad":
            c.update(shape=2, pred=False)
            most /= 3.0
    else:
        c.update(nx=_log(rng, 48, 512), ny=_log(rng, 32, 256), ppc=_log(rng, 4, 64))
        most = 4.0e6 if kind in ("adjoint", "window") else 3.0e7
        if kind == "window":
            c.update(steps=rng.randint(4, 10))
            most = 1.0e6
        if kind == "load":
            c.update(shuffled=rng.random() < 0.5)
    while 2.0 * _cells(c) * c["ppc"] > most:
        c["ppc"] = max(1, c["ppc"] // 2)
        if c["ppc"] == 1:
            c["nx"] = max(12, c["nx"] // 2)
    return c


def _cells(c):
    return c["nx"] * c["ny"] * max(1, c["nz"])


# ---------------------------------------------------------------------------
# the initial state: the double Harris sheet, made on the GPU


def _sheet(c, seed, delta=DELTA, sigma=SIGMA, pert=0.01):
    """Positions, momenta and weights of both species and the fields, FP64 on
    the GPU; momenta, weights, fields and the offsets within a cell are values
    that FP32 holds too."""
    dev = "cuda"
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    nx, ny, nz, ppc = c["nx"], c["ny"], c["nz"], c["ppc"]
    dims = (nx, ny, nz) if nz else (nx, ny)
    ncell = _cells(c)
    n = ncell * ppc
    s = THETA_T / delta ** 2                 # Gamma_d beta_d^2 (force balance and Ampere's law)
    beta = math.sqrt(0.5 * (-s * s + math.sqrt(s ** 4 + 4.0 * s * s)))
    Gd = 1.0 / math.sqrt(1.0 - beta * beta)
    B0 = math.sqrt(4.0 * THETA_T / Gd)
    nb = B0 * B0 / sigma

    def rand(*shape):
        return torch.rand(shape, generator=gen, device=dev, dtype=torch.float32)

    cell = torch.arange(n, device=dev, dtype=torch.int64).div_(ppc, rounding_mode="floor")
    x = torch.empty((n, len(dims)), device=dev, dtype=torch.float64)
    for k, d in enumerate(dims):
        x[:, k] = (cell % d).double().add_(rand(n).mul_(1.0 - 2.0 ** -20))
        cell = cell.div_(d, rounding_mode="floor")
    del cell
    y = x[:, 1].to(torch.float32)
    n1 = torch.cosh((y - 0.25 * ny).div_(delta).clamp_(-40, 40)).pow_(-2)
    n2 = torch.cosh((y - 0.75 * ny).div_(delta).clamp_(-40, 40)).pow_(-2)
    del y
    total = n1 + n2 + nb
    w = total.div(ppc).double()
    member = rand(n).mul_(total)
    drift = torch.where(member < n1, -beta, torch.where(member < n1 + n2, beta, 0.0))
    del total, member, n1, n2
    # speeds of the rest frame's Maxwell-Juettner law by its inverse distribution
    grid = np.linspace(0.0, 40.0 * THETA_T + 2.0, 8193)
    pdf = grid ** 2 * np.exp(-(np.sqrt(1.0 + grid ** 2) - 1.0) / THETA_T)
    cdf = np.concatenate([[0.0], np.cumsum(0.5 * (pdf[1:] + pdf[:-1]))])
    inverse = np.interp(np.linspace(0.0, 1.0 - 1e-7, 65536), cdf / cdf[-1], grid)
    inverse = torch.from_numpy(inverse).to(dev, torch.float32)
    species = []
    for q in Q:
        at = rand(n).mul_(65534.0)
        low = at.to(torch.int64)
        speed = torch.lerp(inverse[low], inverse[low + 1], at - low)
        del at, low
        gamma = torch.sqrt(1.0 + speed * speed)
        mu = rand(n).mul_(2.0).sub_(1.0)
        phi = rand(n).mul_(2.0 * math.pi)
        flat = speed * torch.sqrt(1.0 - mu * mu)
        uz = speed * mu
        b = drift * q
        uz = torch.where(rand(n) < -b * uz / gamma, -uz, uz)      # the flip that weights by 1 + beta v_z
        uz = torch.where(b != 0.0, Gd * (uz + b * gamma), uz)
        u = torch.empty((n, 3), device=dev, dtype=torch.float64)
        u[:, 0], u[:, 1], u[:, 2] = flat * torch.cos(phi), flat * torch.sin(phi), uz
        species.append(u)
        del speed, gamma, mu, phi, flat, uz, b
    yc = torch.arange(ny, device=dev, dtype=torch.float64) + 0.5
    xc = torch.arange(nx, device=dev, dtype=torch.float64) + 0.5
    Bx = B0 * (torch.tanh((yc - 0.25 * ny) / delta) - torch.tanh((yc - 0.75 * ny) / delta) - 1.0)
    phase = 2.0 * math.pi * rand(1).double()
    By = pert * B0 * torch.cos(2.0 * math.pi * xc / nx + phase)
    B = torch.zeros((3, max(1, nz), ny, nx), device=dev, dtype=torch.float64)
    B[0] = Bx[None, :, None]
    B[1] = By[None, None, :]
    B = B.reshape(3, ncell).float().double()
    # fields of a run under way: a little noise on E
    E = (0.01 * B0 * torch.randn((3, ncell), generator=gen, device=dev, dtype=torch.float32)).double()
    return dict(x=x, u=species, w=w, E=E, B=B)


def _config(c, ids):
    return rs.make_config(c["nx"], c["ny"], dt=c["dt"], precision=c["precision"], q=Q, m=(1.0, 1.0), track_ids=ids,
                          gamma_pred=c["pred"], nz=c["nz"] or None, shape=c["shape"])


def _simulation(c, st, ids=True, stream=None):
    sim = rs.Simulation(_config(c, ids), stream)
    for s in range(2):
        sim.load_species(s, st["x"], st["u"][s], st["w"])
    sim.set_fields(st["E"], st["B"])
    return sim


def _instances(c):
    out = []
    for i in range(c["count"]):
        k = c["pick"] + 7 * i
        lx = SCAN_LX[k % 4]
        out.append((dict(c, nx=lx, ny=lx // 2, nz=0), SCAN_DELTA[k % 3], SCAN_SIGMA[(k // 3) % 3]))
    return out


def prepare(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind == "batch":
        sims, firsts, streams = [], [], []
        for i, (ci, delta, sigma) in enumerate(_instances(c)):
            st = _sheet(ci, seed * 64 + i, delta, sigma, 1e-3)
            stream = torch.cuda.Stream()
            stream.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(stream):
                sims.append(_simulation(ci, st))
            firsts.append(st["x"])
            streams.append(stream)
            torch.cuda.synchronize()
        return dict(case=c, sims=sims, x=firsts, streams=streams, batch=rs.Batch(sims, nworkers=8))
    st = _sheet(c, seed)
    if kind == "step":
        return dict(case=c, sim=_simulation(c, st), x=st["x"])
    if kind == "load":
        if c["shuffled"]:
            gen = torch.Generator(device="cuda")
            gen.manual_seed(seed + 1)
            order = torch.randperm(st["w"].shape[0], generator=gen, device="cuda")
            st["x"], st["w"] = st["x"][order], st["w"][order]
            st["u"] = [u[order] for u in st["u"]]
        return dict(case=c, sim=rs.Simulation(_config(c, False)), st=st)
    if kind == "adjoint":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed + 1)
        n, nn = st["w"].shape[0], _cells(c)

        def up(*shape):
            return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32).double()

        grads = dict(E=up(3, nn), B=up(3, nn), u=[up(n, 3).mul_(0.1) for _ in Q], x=[up(n, 2).mul_(0.1) for _ in Q])
        return dict(case=c, sim=_simulation(c, st), st=st, up=grads)
    if kind == "window":
        host = dict(E=st["E"].cpu().numpy(), B=st["B"].cpu().numpy(), species=[])
        x, w = st["x"].cpu().numpy(), st["w"].cpu().numpy()
        for u in st["u"]:
            u = u.cpu().numpy()
            host["species"].append(dict(x=x[:, 0].copy(), y=x[:, 1].copy(), ux=u[:, 0].copy(), uy=u[:, 1].copy(),
                                        uz=u[:, 2].copy(), w=w))
        return dict(case=c, window=ModeEnergyWindow(_config(c, True), c["steps"], checkpoint_every=5), state=host)
    raise ValueError(kind)


# ---------------------------------------------------------------------------
# one pass


def _tracked(c, sim, x0):
    """Each particle's displacement since the start (the tracked trajectory),
    momentum and weight, in the order it was loaded in."""
    box = torch.tensor((c["nx"], c["ny"], c["nz"])[:x0.shape[1]], dtype=torch.float64, device="cuda")
    out = []
    for s in range(2):
        x, u, w, ids = sim.particles(s, ids=True, device=True)
        ids = ids.long()
        d = torch.empty_like(x).index_copy_(0, ids, x).sub_(x0)
        if c["precision"] == 32:
            d, u, w = d.float(), u.float(), w.float()
        box = box.to(d.dtype)
        d.sub_(torch.round(d / box).mul_(box))
        out.append([d] + [torch.empty_like(v).index_copy_(0, ids, v) for v in (u, w)])
    return out


def _give(c, v):
    return v.float() if c["precision"] == 32 else v


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "step":
        sim = state["sim"]
        for _ in range(c["steps"]):
            led, _ = sim.step()
        E, B = sim.fields(device=True)
        return dict(E=_give(c, E), B=_give(c, B), p=_tracked(c, sim, state["x"]),
                    energy=[led["W_E"], led["W_B"], led["K"]])
    if kind == "batch":
        modes, _, _ = state["batch"].run(c["steps"], component=1, nmodes=4)
        out = []
        for (ci, _, _), sim, x0, stream in zip(_instances(c), state["sims"], state["x"], state["streams"]):
            with torch.cuda.stream(stream):
                E, B = sim.fields(device=True)
                out.append([_give(c, E), _give(c, B)] + [v[1] for v in _tracked(ci, sim, x0)])
        return dict(modes=modes.astype(np.float32), out=out)
    if kind == "adjoint":
        sim, st, up = state["sim"], state["st"], state["up"]
        sim.set_fields(st["E"], st["B"])
        gE, gB = up["E"].clone(), up["B"].clone()
        gu, gx = [g.clone() for g in up["u"]], [g.clone() for g in up["x"]]
        gw = [torch.zeros_like(st["w"]) for _ in Q]
        sim.step_adjoint(gE, gB, gu, gx, gw)
        return dict(E=_give(c, gE), B=_give(c, gB), u=[_give(c, g) for g in gu], x=[_give(c, g) for g in gx],
                    w=[_give(c, g) for g in gw])
    if kind == "window":
        win = state["window"]
        loss = win.forward(state["state"])
        g = win.backward()
        as_ = np.float32 if c["precision"] == 32 else np.float64
        return dict(loss=loss, E=g["E"].astype(as_), B=g["B"].astype(as_), w=[v.astype(as_) for v in g["w"]],
                    p=[[v.astype(as_) for v in pair] for pair in g["particles"]])
    if kind == "load":
        sim, st = state["sim"], state["st"]
        for s in range(2):
            sim.load_species(s, st["x"], st["u"][s], st["w"])
        sim.set_fields(st["E"], st["B"])
        led = sim.ledger()
        out = dict(energy=[led["W_E"], led["W_B"], led["K"]], modes=sim.field_modes(1, 8, device=True).float(), p=[])
        for s in range(2):
            weight, count = sim.spectrum(s, BINS, device=True)
            start, off, u, w = sim.particles_native(s, device=True)
            out["p"].append([_give(c, weight), count, start, off, u, w])
        return out
    raise ValueError(kind)


def work(case):
    """Per step and particle: read for the deposit, read and written by the
    push; per step and node: the fields read and written, the mass matrix
    written and read. Operations: the deposit's node pairs (9 multiply-adds
    each), and the gathers and the rotation twice."""
    if case["kind"] == "batch":
        every = [work(dict(ci, kind="step")) for ci, _, _ in _instances(case)]
        return {k: sum(e[k] for e in every) for k in ("bytes", "flops")}
    cells, real = _cells(case), case["precision"] // 8
    n = 2 * cells * case["ppc"]
    dim = 3 if case["nz"] else 2
    nodes = 8 if dim == 3 else (9 if case["shape"] == 2 else 4)
    half = 14 if dim == 3 else (13 if case["shape"] == 2 else 5)
    record = (dim + 4) * real
    if case["kind"] == "load":       # the FP64 record in, the library's own form out (and once through the spectrum)
        return {"bytes": float(n * (8 * (dim + 4) + 2 * record) + cells * 96), "flops": float(n * 20)}
    step = {"bytes": float(n * 3 * record + cells * real * (12 + 2 * 9 * half)),
            "flops": float(n * (nodes * (nodes + 1) * 9 + 3 * 6 * nodes + 120))}
    times = case["steps"]
    if case["kind"] == "adjoint":    # the step forward, and its reverse with FP64 gradients in and out
        return {"bytes": step["bytes"] * 2 + n * 8.0 * 11, "flops": step["flops"] * 3}
    if case["kind"] == "window":
        return {"bytes": times * (step["bytes"] * 2 + n * 8.0 * 11), "flops": times * step["flops"] * 3}
    return {k: v * times for k, v in step.items()}


# ---------------------------------------------------------------------------
# the same in 64 bits, plain torch


class _Step:
    """One step of the scheme on FP64 tensors; species share positions' layout."""

    def __init__(self, c):
        self.c, self.dt = c, c["dt"]
        self.dims = (c["nx"], c["ny"], c["nz"]) if c["nz"] else (c["nx"], c["ny"])
        self.nn = _cells(c)
        self.td = 0.5 * c["dt"]

    # ---- the grid
    def _diff(self, F, axis, back):
        """Derivative along an axis, averaged over the edges in the other directions."""
        dim = len(self.dims)
        F = F.reshape(tuple(reversed(self.dims)))
        sh = 1 if back else -1
        at = dim - 1 - axis
        F = (F - torch.roll(F, 1, at)) if back else (torch.roll(F, -1, at) - F)
        for other in range(dim):
            if other != at:
                F = 0.5 * (F + torch.roll(F, sh, other))
        return F.reshape(-1)

    def curl(self, F, back):
        d = [[self._diff(F[k], a, back) for k in range(3)] if a < len(self.dims) else [torch.zeros_like(F[0])] * 3
             for a in range(3)]
        return torch.stack([d[1][2] - d[2][1], d[2][0] - d[0][2], d[0][1] - d[1][0]])

    # ---- the shapes: [(node index, weight)] of every node of a particle
    def shapes(self, x, shift):
        axes = []
        for k, L in enumerate(self.dims):
            s = x[:, k] - shift
            if self.c["shape"] == 2:
                base = torch.floor(s.detach() + 0.5)
                d = s - base
                ws = (0.5 * (0.5 - d) ** 2, 0.75 - d * d, 0.5 * (0.5 + d) ** 2)
                first = -1
            else:
                base = torch.floor(s.detach())
                f = s - base
                ws = (1.0 - f, f)
                first = 0
            base = base.long()
            axes.append([((base + first + a) % L, w) for a, w in enumerate(ws)])
        out = axes[-1]
        for k in range(len(self.dims) - 2, -1, -1):
            out = [(i * self.dims[k] + i2, w * w2) for i, w in out for i2, w2 in axes[k]]
        return out

    @staticmethod
    def gather(F, shape):
        Ft = F.t().contiguous()
        return sum(w[:, None] * Ft[i] for i, w in shape)

    def scatter(self, v, shape):
        out = torch.zeros((self.nn, 3), dtype=torch.float64, device=v.device)
        for i, w in shape:
            out = out.index_add(0, i, w[:, None] * v) if v.requires_grad or w.requires_grad else \
                out.index_add_(0, i, w[:, None] * v)
        return out.t()

    # ---- particles
    def particle(self, s, x, u, w, E, B):
        """What the deposit and the push share of a species."""
        node, beta = self.shapes(x, 0.0), 0.5 * Q[s] * self.dt
        Bp = self.gather(B, self.shapes(x, 0.5))
        up = u + beta * self.gather(E, node) if self.c["pred"] else u
        g = torch.sqrt(1.0 + (up * up).sum(1, keepdim=True))
        return dict(node=node, beta=beta, a=beta * Bp / g, c=Q[s] * w[:, None] / g, u=u)

    @staticmethod
    def rotate(p, v, transposed=False):
        a = -p["a"] if transposed else p["a"]
        return (v - torch.cross(a, v, dim=1) + a * (a * v).sum(1, keepdim=True)) / (1.0 + (a * a).sum(1, keepdim=True))

    def current(self, ps):
        return sum(self.scatter(p["c"] * self.rotate(p, p["u"]), p["node"]) for p in ps)

    def mass(self, ps, v, transposed=False):
        return sum(self.scatter(p["c"] * p["beta"] * self.rotate(p, self.gather(v, p["node"]), transposed), p["node"])
                   for p in ps)

    def operator(self, ps, v, transposed=False):
        return v + self.td ** 2 * self.curl(self.curl(v, False), True) + self.td * self.mass(ps, v, transposed)

    def solve(self, A, b, x):
        """GMRES to round-off."""
        norm = float(b.norm())
        if norm == 0.0:
            return torch.zeros_like(b)
        for _ in range(4):
            r = b - A(x)
            rn = float(r.norm())
            if rn < 3e-14 * norm:
                break
            V, H = [r / rn], np.zeros((61, 60))
            for j in range(60):
                z = A(V[j])
                for _ in range(2):
                    for i, v in enumerate(V):
                        h = float((v * z).sum())
                        H[i, j] += h
                        z = z - h * v
                H[j + 1, j] = float(z.norm())
                e = np.zeros(j + 2)
                e[0] = rn
                y, *_ = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)
                if np.linalg.norm(H[:j + 2, :j + 1] @ y - e) < 1e-14 * norm or H[j + 1, j] == 0.0:
                    break
                V.append(z / H[j + 1, j])
            x = x + sum(float(yi) * v for yi, v in zip(y, V))
        return x

    def right(self, ps, E, B):
        return E + self.td * self.curl(B, True) - self.td * self.current(ps)

    def push(self, ps, Et, x):
        out = []
        for p, xs in zip(ps, x):
            bar = self.rotate(p, p["u"] + p["beta"] * self.gather(Et, p["node"]))
            u1 = 2.0 * bar - p["u"]
            v1 = u1 / torch.sqrt(1.0 + (u1 * u1).sum(1, keepdim=True))
            out.append((xs + self.dt * v1[:, :len(self.dims)], u1))
        return out

    def fields(self, Et, E, B):
        return 2.0 * Et - E, B - self.dt * self.curl(Et, False)

    def forward(self, E, B, x, u, w):
        with torch.no_grad():
            ps = [self.particle(s, x[s], u[s], w[s], E, B) for s in range(2)]
            Et = self.solve(lambda v: self.operator(ps, v), self.right(ps, E, B), E)
            moved = self.push(ps, Et, x)
            E1, B1 = self.fields(Et, E, B)
        return E1, B1, [m[0] for m in moved], [m[1] for m in moved], Et

    def reverse(self, E, B, x, u, w, Et, gE, gB, gu, gx):
        """Gradients in the state before the step from those after it, and the weights'."""
        E, B, Et = (v.detach().clone().requires_grad_() for v in (E, B, Et))
        x, u, w = ([v.detach().clone().requires_grad_() for v in vs] for vs in (x, u, w))
        leaves = [E, B] + x + u + w

        def after():
            ps = [self.particle(s, x[s], u[s], w[s], E, B) for s in range(2)]
            E1, B1 = self.fields(Et, E, B)
            moved = self.push(ps, Et, x)
            L = (E1 * gE).sum() + (B1 * gB).sum()
            for s in range(2):
                L = L + (moved[s][0] * gx[s]).sum() + (moved[s][1] * gu[s]).sum()
            return L

        got = torch.autograd.grad(after(), leaves + [Et], allow_unused=True)
        with torch.no_grad():
            ps = [self.particle(s, x[s], u[s], w[s], E, B) for s in range(2)]
            lam = self.solve(lambda v: self.operator(ps, v, True), got[-1], torch.zeros_like(got[-1]))
        del ps
        ps = [self.particle(s, x[s], u[s], w[s], E, B) for s in range(2)]
        fixed = Et.detach()
        off = (lam * (self.operator(ps, fixed) - self.right(ps, E, B))).sum()
        more = torch.autograd.grad(off, leaves, allow_unused=True)
        out = []
        for v, a, b in zip(leaves, got, more):
            t = torch.zeros_like(v)
            t = t + a if a is not None else t
            out.append(t - b if b is not None else t)
        return out[0], out[1], out[2:4], out[4:6], out[6:8]


def _energies(E, B, u, w):
    K = sum(float((w[s] * ((u[s] ** 2).sum(1) / (1.0 + torch.sqrt(1.0 + (u[s] ** 2).sum(1))))).sum()) for s in range(2))
    return [0.5 * float((E ** 2).sum()), 0.5 * float((B ** 2).sum()), K]


def _modes(B1, nx, ny, count):
    F = torch.fft.rfft(B1.reshape(ny, nx), dim=1)[:, :count]
    c = torch.full((count,), 2.0, dtype=torch.float64, device=B1.device)
    c[0] = 1.0
    if nx % 2 == 0 and count > nx // 2:
        c[nx // 2] = 1.0
    return 0.5 * c / nx * (F.abs() ** 2).sum(0)


def _exact_steps(c, st):
    S = _Step(c)
    E, B, x, u, w = st["E"], st["B"], [st["x"], st["x"]], list(st["u"]), [st["w"], st["w"]]
    every = []
    for _ in range(c["steps"]):
        before = (E, B, x, u)
        E, B, x, u, Et = S.forward(E, B, x, u, w)
        every.append(before + (Et,))
        yield S, E, B, x, u, w, every


def exact(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind == "batch":
        if sum(2.0 * _cells(ci) * c["ppc"] for ci, _, _ in _instances(c)) * c["steps"] > EXACT_MOST:
            return None
        modes, out = [], []
        for i, (ci, delta, sigma) in enumerate(_instances(c)):
            rows = []
            for _, E, B, x, u, w, every in _exact_steps(ci, _sheet(ci, seed * 64 + i, delta, sigma, 1e-3)):
                rows.append(_modes(B[1], ci["nx"], ci["ny"], 4).cpu().numpy())
                every.clear()
            modes.append(np.stack(rows))
            out.append([E, B] + u)
        return dict(modes=np.stack(modes), out=out)
    parts = 2.0 * _cells(c) * c["ppc"]
    if parts * c["steps"] > EXACT_MOST:
        return None
    st = _sheet(c, seed)
    if kind == "step":
        for _, E, B, x, u, w, every in _exact_steps(c, st):
            every.clear()
        return dict(E=E, B=B, p=[[x[s] - st["x"], u[s], w[s]] for s in range(2)], energy=_energies(E, B, u, w))
    if kind == "adjoint":
        up = prepare(c, seed)["up"]
        S = _Step(c)
        args = (st["E"], st["B"], [st["x"]] * 2, st["u"], [st["w"]] * 2)
        Et = S.forward(*args)[4]
        gE, gB, gx, gu, gw = S.reverse(*args, Et, up["E"], up["B"], up["u"], up["x"])
        return dict(E=gE, B=gB, u=gu, x=gx, w=gw)
    if kind == "window":
        for S, E, B, x, u, w, every in _exact_steps(c, st):
            pass
        B1 = B[1].clone().requires_grad_()
        loss = _modes(B1, c["nx"], c["ny"], 2)[1]
        gB = torch.zeros_like(B)
        gB[1] = torch.autograd.grad(loss, B1)[0]
        gE = torch.zeros_like(E)
        gu, gx = [torch.zeros_like(v) for v in u], [torch.zeros_like(v) for v in x]
        sums = [torch.zeros_like(v) for v in w]
        for E, B, x, u, Et in reversed(every):
            gE, gB, gx, gu, gw = S.reverse(E, B, x, u, w, Et, gE, gB, gu, gx)
            sums = [a + b for a, b in zip(sums, gw)]
        return dict(loss=float(loss), E=gE, B=gB, w=sums, p=[[gu[s], gx[s]] for s in range(2)])
    if kind == "load":
        st = prepare(c, seed)["st"]
        nx, ny = c["nx"], c["ny"]
        cell = torch.floor(st["x"]).long()
        key, order = torch.sort(cell[:, 1] * nx + cell[:, 0], stable=True)
        off = (st["x"] - cell)[order].t()
        out = dict(energy=_energies(st["E"], st["B"], st["u"], [st["w"]] * 2),
                   modes=_modes(st["B"][1], nx, ny, 8), p=[])
        edges = torch.from_numpy(BINS).to("cuda")
        for u in st["u"]:
            u2 = (u * u).sum(1)
            b = torch.searchsorted(edges, u2 / (1.0 + torch.sqrt(1.0 + u2)), right=True)
            weight = torch.zeros(BINS.size + 1, dtype=torch.float64, device="cuda").index_add_(0, b, st["w"])
            out["p"].append([weight, None, None, off, u[order].t(), st["w"][order]])
        return out
    raise ValueError(kind)
