"""The work that users of this package have it do, as cases that can be timed.

Each case is one call, or one step made of a few calls, through the public
Python entry points: the time steps of the paper's experiments (G2P -> move ->
P2G) in 1D and 2D, the large mass assignment, many uneven instances at once,
the learned start and the training of its network, assignment from and into
host memory, the projections back to the particles, sampling, the cheaper
assignments, and the P1 mesh. ``listed()`` names one of each, ``draw`` gives
others over the same ranges.
"""
import math
import random

import numpy as np
import torch

import paper_1610_05258_gb300 as pm
from paper_1610_05258_gb300 import warmstart
from paper_1610_05258_gb300 import workloads as W

TWO_PI = 2.0 * math.pi


def listed():
    return [
        # 1D transport of a top-hat, one time step: the smallest call, all launches and latency
        {"name": "tophat_step", "kind": "tophat", "n": 128, "particles": 128},
        # 2D slotted disk on a jittered lattice, one step of its rotation
        {"name": "zalesak_step", "kind": "zalesak", "n": 256},
        # 2D Taylor-Green vortex, one step: G2P, midpoint move, mass assignment of u and v
        {"name": "taylor_green_step", "kind": "taylor_green", "n": 1024, "ppc": 4},
        # the largest: mass assignment of four fields on clustered particles
        {"name": "mixture_assign", "kind": "mixture", "n": 2048, "ppc": 4, "fields": 4, "start": "delta"},
        # uneven independent instances advanced together
        {"name": "batch_assign", "kind": "batch", "count": 24, "nmin": 64, "nmax": 512, "fields": 3, "sizes": 16104},
        # mass assignment started by the trained network
        {"name": "learned_assign", "kind": "learned", "n": 1024, "ppc": 4, "fields": 4},
        # mass assignment for an application that holds its particles in (pinned) host memory
        {"name": "host_assign", "kind": "host", "n": 512, "ppc": 4, "fields": 3},
        # full-mass projection from the mesh back to the particles, odd mesh side
        {"name": "project_back", "kind": "project", "n": 701, "ppc": 4, "fields": 3},
        # mesh fields sampled at many particles in no particular order
        {"name": "sample", "kind": "sample", "n": 2048, "ppc": 4, "fields": 4},
        # FLIP assignment on a ragged mesh with dense particles
        {"name": "flip_assign", "kind": "assign", "method": "flip", "n": 333, "ppc": 6, "fields": 3},
        # mass assignment on the split-square P1 mesh, Chebyshev solver, odd side
        {"name": "p1_assign", "kind": "p1", "n": 501, "ppc": 4, "fields": 2, "solver": "chebyshev"},
        # one training step of the network: forward, backward and update
        {"name": "net_train", "kind": "train", "n": 256, "batch": 8},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice([c["kind"] for c in listed()])
    if kind == "tophat":
        n = _log_int(rng, 64, 4096)
        return {"kind": kind, "n": n, "particles": n * rng.choice([1, 2, 4]) + rng.randrange(0, 7)}
    if kind == "zalesak":
        return {"kind": kind, "n": _log_int(rng, 96, 512)}
    if kind == "taylor_green":
        return {"kind": kind, "n": _log_int(rng, 200, 1024), "ppc": 4}
    if kind == "mixture":
        return {"kind": kind, "n": _log_int(rng, 128, 1500), "ppc": 4, "fields": rng.randint(1, 4),
                "start": rng.choice(["delta", "direct"])}
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(8, 24), "nmin": 64, "nmax": rng.randint(128, 512),
                "fields": rng.randint(1, 3), "sizes": rng.randrange(1 << 20)}
    if kind == "learned":
        return {"kind": kind, "n": 128 * rng.randint(2, 8), "ppc": 4, "fields": rng.randint(3, 4)}
    if kind == "host":
        return {"kind": kind, "n": _log_int(rng, 100, 700), "ppc": 4, "fields": rng.randint(1, 4)}
    if kind == "project":
        return {"kind": kind, "n": _log_int(rng, 150, 701), "ppc": rng.choice([3, 4, 6]), "fields": rng.randint(1, 4)}
    if kind == "sample":
        return {"kind": kind, "n": _log_int(rng, 200, 1800), "ppc": 4, "fields": rng.randint(1, 5)}
    if kind == "assign":
        return {"kind": kind, "method": rng.choice(["flip", "pic", "lumped", "delta"]), "n": _log_int(rng, 100, 500),
                "ppc": rng.randint(3, 8), "fields": rng.randint(1, 4)}
    if kind == "p1":
        return {"kind": kind, "n": _log_int(rng, 101, 501), "ppc": 4, "fields": rng.randint(1, 3),
                "solver": rng.choice(["cg", "chebyshev"])}
    return {"kind": "train", "n": rng.choice([128, 256]), "batch": rng.randint(2, 8)}


# ------------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda")


def _uniform(g, count, L):
    """Uniform distinct particles: the library's particle functions need
    distinct positions, so the rare coincident draws are made again."""
    x, y = _rand(g, count) * L, _rand(g, count) * L
    inv = torch.tensor(1.0 / L, dtype=torch.float32, device="cuda")
    for _ in range(8):
        q = lambda v: ((v * inv - torch.floor(v * inv)) * 4294967296.0).to(torch.int64) & 0xFFFFFFFF  # noqa: E731
        key, order = torch.sort((q(x) << 32) | q(y))
        again = order[1:][key[1:] == key[:-1]]
        if again.numel() == 0:
            break
        x[again] = _rand(g, again.numel()) * L
        y[again] = _rand(g, again.numel()) * L
    return x, y


def _waves(g, fields, x, y, L):
    """Smooth random periodic fields: a few Fourier modes of falling amplitude."""
    out = []
    for _ in range(fields):
        k = torch.randint(-6, 7, (8, 2), generator=g, device="cuda").double()
        ph = _rand(g, 8).double() * TWO_PI
        a = 1.0 / (1.0 + k.square().sum(1))
        v = torch.zeros_like(x)
        for m in range(8):
            v += (a[m] * torch.sin((k[m, 0] * x + k[m, 1] * y) * (TWO_PI / L) + ph[m])).float()
        out.append(v)
    return torch.stack(out).float().contiguous()


def _mesh_waves(g, fields, n, L):
    c = torch.arange(n, device="cuda", dtype=torch.float32) * (L / n)
    y, x = torch.meshgrid(c, c, indexing="ij")
    return _waves(g, fields, x.reshape(-1).contiguous(), y.reshape(-1).contiguous(), L)


def _batch_sizes(case):
    r = random.Random(case["sizes"])
    sides = [r.randint(case["nmin"], case["nmax"]) for _ in range(case["count"])]
    return sides, [r.randint(1, 8) * n * n for n in sides]


def prepare(case, seed):
    s = dict(case)
    kind, n = case["kind"], case.get("n", 0)
    g = _gen(seed)
    if kind == "tophat":
        cells = torch.randperm(1 << 22, generator=g, device="cuda")[: case["particles"]]
        s["px"] = ((cells.double() + 0.5) / (1 << 22)).float()
        x = torch.arange(n, device="cuda", dtype=torch.float64) / n
        s["mesh"] = ((x >= 0.25) & (x < 0.5)).float().reshape(1, n)
        s["ctx"] = pm.Context(1, n, 1.0, case["particles"], 1)
    elif kind == "zalesak":
        x, y = W.jittered_lattice(n, 2, seed=seed)
        # up to five steps along the revolution (the corners of the square have wrapped)
        a = 2.0 * math.pi * 1e-3 * (1 + seed % 5)
        X, Y = x.astype(np.float64) - 0.5, y.astype(np.float64) - 0.5
        s["px"] = torch.from_numpy(np.mod(0.5 + math.cos(a) * X - math.sin(a) * Y, 1.0).astype(np.float32)).cuda()
        s["py"] = torch.from_numpy(np.mod(0.5 + math.sin(a) * X + math.cos(a) * Y, 1.0).astype(np.float32)).cuda()
        c = np.arange(n) / n
        xx, yy = np.meshgrid(c, c, indexing="xy")
        s["mesh"] = torch.from_numpy(W.zalesak_indicator(xx.ravel(), yy.ravel())[None]).cuda()
        s["ctx"] = pm.Context(2, n, 1.0, s["px"].numel(), 1)
    elif kind == "taylor_green":
        s["px"], s["py"] = _uniform(g, case["ppc"] * n * n, TWO_PI)
        c = torch.arange(n, device="cuda", dtype=torch.float64) * (TWO_PI / n)
        y, x = torch.meshgrid(c, c, indexing="ij")
        s["mesh"] = torch.stack([torch.sin(x) * torch.cos(y), -torch.cos(x) * torch.sin(y)]).reshape(2, -1).float()
        s["ctx"] = pm.Context(2, n, TWO_PI, s["px"].numel(), 2)
    elif kind in ("mixture", "learned"):
        s["px"], s["py"], s["vals"] = warmstart.mixture_gpu(torch, n, case["ppc"], max(2, case["fields"]), seed, "cuda")
        s["vals"] = s["vals"][: case["fields"]].contiguous()
        s["ctx"] = pm.Context(2, n, TWO_PI, s["px"].numel(), case["fields"])
        if kind == "learned":
            s["net"] = pm.Net(n, case["fields"])
            warmstart.load_weights(s["net"])
    elif kind == "batch":
        sides, counts = _batch_sizes(case)
        s["xs"], s["ys"], s["vs"], s["outs"] = [], [], [], []
        for m, count in zip(sides, counts):
            x, y = _uniform(g, count, 1.0)
            s["xs"].append(x)
            s["ys"].append(y)
            s["vs"].append(_waves(g, case["fields"], x, y, 1.0))
            s["outs"].append(torch.empty(case["fields"], m * m, device="cuda"))
        s["batch"] = pm.Batch(sides, [1.0] * len(sides), counts, case["fields"])
    elif kind == "sample":
        s["px"], s["py"], _ = warmstart.mixture_gpu(torch, n, case["ppc"], 2, seed, "cuda")
        s["mesh"] = _mesh_waves(g, case["fields"], n, TWO_PI)
        s["ctx"] = pm.Context(2, n, TWO_PI, s["px"].numel(), case["fields"])
    elif kind == "train":
        s["x"] = torch.stack([_mesh_waves(g, 2, n, 1.0).reshape(2, n, n) for _ in range(case["batch"])]).contiguous()
        s["x"][:, 1] = 0.2 * s["x"][:, 1] + 0.1 * torch.randn(case["batch"], n, n, generator=g, device="cuda")
        s["target"] = (-s["x"][:, 1] + 0.05 * torch.randn(case["batch"], n, n, generator=g, device="cuda")).contiguous()
        s["net"] = pm.Net(n, case["batch"])
        s["net"].load(warmstart.init_theta(seed))
    else:  # host, project, assign, p1: uniform particles on the unit square
        F = case["fields"]
        s["px"], s["py"] = _uniform(g, case["ppc"] * n * n, 1.0)
        if kind == "project":
            s["mesh"] = _mesh_waves(g, F, n, 1.0)
        else:
            s["vals"] = _waves(g, F, s["px"], s["py"], 1.0)
        s["ctx"] = pm.Context(2, n, 1.0, s["px"].numel(), F, mesh="p1" if kind == "p1" else "q1")
        if kind == "host":
            for k in ("px", "py", "vals"):
                s[k] = s[k].cpu().pin_memory()
            s["out"] = torch.empty(F, n * n).pin_memory()
    return s


# --------------------------------------------------------------------- one pass

def run(s):
    kind = s["kind"]
    ctx = s.get("ctx")
    if kind == "tophat":
        back = ctx.interpolate(s["mesh"], s["px"])
        x = s["px"].clone()
        ctx.advect_shift(x, None, 1.0 / 256)
        return [back, x, ctx.assign_mass(x, None, back, info=False)]
    if kind == "zalesak":
        back = ctx.interpolate(s["mesh"], s["px"], s["py"])
        x, y = s["px"].clone(), s["py"].clone()
        ctx.advect_rotate(x, y, 0.5, 0.5, TWO_PI / 1000)
        return [back, x, y, ctx.assign_mass(x, y, back, info=False)]
    if kind == "taylor_green":
        dt = 0.5 * TWO_PI / s["n"]
        v = ctx.interpolate(s["mesh"], s["px"], s["py"])
        x, y = s["px"].clone(), s["py"].clone()
        ctx.advect_rk2(s["mesh"], v, x, y, dt, vals=v, factor=math.exp(-0.02 * dt))
        return [v, x, y, ctx.assign_mass(x, y, v, info=False)]
    if kind == "mixture":
        return [ctx.assign_mass(s["px"], s["py"], s["vals"], warm_start=s["start"], info=False)]
    if kind == "learned":
        return [ctx.assign_mass(s["px"], s["py"], s["vals"], net=s["net"], info=False)]
    if kind == "batch":
        s["batch"].assign_mass(s["xs"], s["ys"], s["vs"], s["outs"], info=False)
        return s["outs"]
    if kind == "host":
        return [ctx.assign_mass_host(s["px"], s["py"], s["vals"], out=s["out"])[0]]
    if kind == "project":
        return [ctx.interpolate_mass(s["mesh"], s["px"], s["py"], info=False)]
    if kind == "sample":
        return [ctx.interpolate(s["mesh"], s["px"], s["py"])]
    if kind == "assign":
        return [getattr(ctx, "assign_" + s["method"])(s["px"], s["py"], s["vals"])]
    if kind == "p1":
        return [ctx.assign_mass(s["px"], s["py"], s["vals"], solver=s["solver"], info=False)]
    s["net"].train_step(s["x"], s["target"], 2e-3, want_loss=False)
    return [s["net"].grad()]


# ------------------------------------------------------------------- least work

def work(case):
    """Inputs read and outputs written once. Operations: 2 x 2^dim per sampled
    value, about 200 per particle for a star of six neighbours (a distance, a
    circumcentre and a test per vertex), 100 per particle and field for the
    exact integrals over its two triangles; the network's products."""
    kind, n = case["kind"], case.get("n", 0)
    if kind == "train":
        px = case["batch"] * n * n
        return {"bytes": 4.0 * 3 * px + 4.0 * 19393 * 7, "flops": 3 * 2.0 * 9 * px * (64 + 1024 + 1024 + 32)}
    if kind == "batch":
        sides, counts = _batch_sizes(case)
        p, m, F = sum(counts), sum(k * k for k in sides), case["fields"]
    else:
        F = {"tophat": 1, "zalesak": 1, "taylor_green": 2}.get(kind) or case["fields"]
        m = n if kind == "tophat" else n * n
        p = case["particles"] if kind == "tophat" else (4 if kind == "zalesak" else case["ppc"]) * m
    dim = 1 if kind == "tophat" else 2
    once = 4.0 * dim * p + 4.0 * F * p + 4.0 * F * m
    if kind == "sample":
        return {"bytes": once, "flops": 8.0 * F * p}
    ops = 100.0 * F * p + (200.0 * p if dim == 2 else 0.0)
    if kind in ("tophat", "zalesak", "taylor_green"):  # the mesh in, the values and the moved positions out
        return {"bytes": once + 4.0 * F * m + 4.0 * dim * p, "flops": ops + 2.0 * 2 ** dim * F * p}
    return {"bytes": once, "flops": ops}


# ---------------------------------------------------------------- in 64 bits

def _sample64(mesh, n, L, x, y=None):
    """(Bi)linear interpolation of the mesh fields [F, n^dim] at the particles."""
    m = mesh.double()
    gx = x.double() * (n / L)
    i0 = torch.floor(gx)
    s, i0 = gx - i0, i0.long() % n
    i1 = (i0 + 1) % n
    if y is None:
        return m[:, i0] * (1 - s) + m[:, i1] * s
    gy = y.double() * (n / L)
    j0 = torch.floor(gy)
    t, j0 = gy - j0, j0.long() % n
    j1 = (j0 + 1) % n
    return torch.stack([f[j0 * n + i0] * (1 - s) * (1 - t) + f[j0 * n + i1] * s * (1 - t) +
                        f[j1 * n + i0] * (1 - s) * t + f[j1 * n + i1] * s * t for f in m])


def _mass1d64(n, x, a):
    """Mass assignment on the unit circle: int A psi_j with A linear between the
    particles (Simpson between all nodes and particles, exact there), M^-1 by FFT."""
    order = np.argsort(x)
    x, a = x[order], a[order]
    xp, ap = np.concatenate([[x[-1] - 1], x, [x[0] + 1]]), np.concatenate([[a[-1]], a, [a[0]]])
    cut = np.unique(np.concatenate([np.arange(n + 1) / n, x]))
    lo, hi = cut[:-1], cut[1:]
    cell = np.minimum((0.5 * (lo + hi) * n).astype(int), n - 1)
    b = np.zeros(n)
    for u, w in ((lo, 1 / 6), (0.5 * (lo + hi), 4 / 6), (hi, 1 / 6)):
        v, t = np.interp(u, xp, ap) * w * (hi - lo), u * n - cell
        np.add.at(b, cell, v * (1 - t))
        np.add.at(b, (cell + 1) % n, v * t)
    k = 2 * np.pi * np.arange(n) / n
    return np.fft.ifft(np.fft.fft(b) / ((4 + 2 * np.cos(k)) / (6 * n))).real


def _net64(theta, x):
    """The network's layers (3x3 periodic convolutions, ReLU after the first three)."""
    at = 0
    for k, (ci, co) in enumerate([(2, 32), (32, 32), (32, 32), (32, 1)]):
        w, at = theta[at:at + co * ci * 9].reshape(co, ci, 3, 3), at + co * ci * 9
        b, at = theta[at:at + co], at + co
        pad = torch.nn.functional.pad(x, (1, 1, 1, 1), mode="circular")
        x = sum(torch.einsum("oi,bihw->bohw", w[:, :, i, j], pad[:, :, i:i + x.shape[2], j:j + x.shape[3]])
                for i in range(3) for j in range(3)) + b[None, :, None, None]
        x = torch.relu(x) if k < 3 else x
    return x[:, 0]


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("tophat", "zalesak", "taylor_green", "sample", "train"):
        return None  # the periodic Delaunay triangulation in 64 bits would take too long here
    s = prepare(case, seed)
    if kind == "train":
        net = s.pop("net")
        theta = torch.from_numpy(net.state()[0]).cuda().double().requires_grad_()
        grad = torch.zeros_like(theta)
        for x, t in zip(s["x"], s["target"]):  # one image at a time: the 64-bit activations are large
            r = _net64(theta, x[None].double()) - t[None].double()
            grad += torch.autograd.grad(0.5 * r.square().sum() / s["target"].numel(), theta)[0]
        return [grad]
    s["ctx"] = None
    n, L = case["n"], 1.0 if kind in ("tophat", "zalesak") else TWO_PI
    back = _sample64(s["mesh"], n, L, s["px"], s.get("py"))
    if kind == "sample":
        return [back]
    if kind == "tophat":
        x = torch.remainder(s["px"].double() + 1.0 / 256, 1.0)
        out = _mass1d64(n, x.cpu().numpy(), back[0].cpu().numpy())
        return [back, x, torch.from_numpy(out).reshape(1, n)]
    if kind == "zalesak":
        a, X, Y = TWO_PI / 1000, s["px"].double() - 0.5, s["py"].double() - 0.5
        return [back, torch.remainder(0.5 + math.cos(a) * X - math.sin(a) * Y, 1.0),
                torch.remainder(0.5 + math.sin(a) * X + math.cos(a) * Y, 1.0), None]
    dt = 0.5 * L / n
    x, y = s["px"].double(), s["py"].double()
    mid = _sample64(s["mesh"], n, L, torch.remainder(x + 0.5 * dt * back[0], L), torch.remainder(y + 0.5 * dt * back[1], L))
    return [back * math.exp(-0.02 * dt), torch.remainder(x + dt * mid[0], L), torch.remainder(y + dt * mid[1], L), None]
