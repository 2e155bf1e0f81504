"""Particle sets that the triangulation's main pass gives up, by any of its
routes: lattices (along the axes, hexagonal, turned, in part), which go to the
exact pass with or without an attempt, and crowds inside a cell, which end in the
last pass; against the oracle, in batches, and for bits that do not depend on the
route."""
import numpy as np
import pytest

import oracle
from gpu_util import canon_tris, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def grid(mx, my, order="C"):
    x, y = np.meshgrid((np.arange(mx) + 0.5) / mx, (np.arange(my) + 0.5) / my, indexing="xy")
    return np.stack([x.ravel(order), y.ravel(order)], -1)


def hexagonal(m):
    x = grid(m, m).reshape(m, m, 2)
    x[1::2, :, 0] += 0.5 / m
    return x.reshape(-1, 2) % 1.0


def turned(m, a):
    """A square lattice turned about the centre and cut to the middle, in a sparse random frame."""
    g = np.random.default_rng(m)
    x = grid(m, m) - 0.5
    r = np.stack([np.cos(a) * x[:, 0] - np.sin(a) * x[:, 1], np.sin(a) * x[:, 0] + np.cos(a) * x[:, 1]], -1) + 0.5
    inside = (np.abs(r - 0.5) < 0.35).all(1)
    frame = g.uniform(0, 1, (m * m // 2, 2))
    return np.concatenate([r[inside], frame[(np.abs(frame - 0.5) >= 0.355).any(1)]])


def crowds(n, g, count, width):
    c = (g.integers(0, n, (8, 2)) + g.uniform(0.2, 0.8, (8, 2))) / n
    return np.concatenate([g.uniform(0, 1, (4 * n * n, 2))] + [q + g.normal(0, width / n, (count, 2)) for q in c]) % 1.0


CASES = {
    "square_4_per_cell": (33, lambda g: grid(66, 66)),
    "square_1_per_cell": (64, lambda g: grid(64, 64)),
    "square_9_per_cell": (22, lambda g: grid(66, 66)),
    "square_small": (20, lambda g: grid(40, 40)),
    "square_by_columns": (33, lambda g: grid(66, 66, "F")),
    "square_uneven_cells": (47, lambda g: grid(65, 65)),
    "rectangles": (35, lambda g: grid(105, 40)),
    "square_with_gaps": (36, lambda g: grid(72, 72)[g.uniform(size=5184) > 0.2]),
    "hexagonal": (24, lambda g: hexagonal(48)),
    "turned": (33, lambda g: turned(80, 0.3)),
    "crowds_in_cells": (20, lambda g: crowds(20, g, 200, 0.1)),
    "tight_crowds": (20, lambda g: crowds(20, g, 150, 0.004)),
    "crowds_over_cells": (20, lambda g: crowds(20, g, 300, 1.0)),
}


def make(name):
    n, f = CASES[name]
    xy = (f(np.random.default_rng(sum(map(ord, name)))) % 1.0).astype(np.float32)
    xy = np.unique(xy[(xy < 1).all(1)], axis=0) if "crowds" in name else xy
    return n, np.ascontiguousarray(xy[:, 0]), np.ascontiguousarray(xy[:, 1])


@pytest.mark.parametrize("name", CASES)
def test_stars(name):
    from paper_1610_05258_gb300 import Context
    n, px, py = make(name)
    c = Context(2, n, 1.0, px.size, 1)
    dpx, dpy = to_dev(torch, px, py)
    tri, off = c.triangulate(dpx, dpy)
    t, o, _ = oracle.triangulate(1.0, px, py)
    assert canon_tris(tri.cpu().numpy(), off.cpu().numpy()) == canon_tris(t, o)
    v = c.particle_volumes(dpx, dpy)
    assert abs(v.double().sum().item() - 1.0) <= 1e-6
    # the counting build takes the same decisions
    c.profile(True, count_work=True)
    assert torch.equal(c.particle_volumes(dpx, dpy), v)


def test_batch_of_lattices_and_crowds():
    from paper_1610_05258_gb300 import Batch, Context
    names = ["square_4_per_cell", "crowds_in_cells", "hexagonal", "square_1_per_cell", "turned"]
    sets = [make(q) for q in names]
    dev = [to_dev(torch, px, py) for _, px, py in sets]
    vals = [torch.stack([torch.sin(6.28 * x) + 1.0, torch.cos(12.56 * y)]) for x, y in dev]
    outs = [torch.empty(2, n * n, device="cuda") for n, _, _ in sets]
    b = Batch([n for n, _, _ in sets], [1.0] * len(sets), [px.size for _, px, _ in sets], 2)
    b.assign_mass([d[0] for d in dev], [d[1] for d in dev], vals, outs)
    for (n, px, _), (x, y), v, o in zip(sets, dev, vals, outs):
        ref, _ = Context(2, n, 1.0, px.size, 2).assign_mass(x, y, v, warm_start="direct")
        # both solve to 1e-6 of the same right-hand side: kappa (9) times that
        assert float((o - ref).norm() / ref.norm()) <= 2 * 9 * 1e-6


def test_route_leaves_no_trace():
    """A turned lattice of 290,000 particles, where blocks read the running count of ties: the
    triangles are those of another mesh, and the projection's sums, which follow the stars'
    order, give the same bits every time."""
    from paper_1610_05258_gb300 import Context
    xy = turned(600, 0.3).astype(np.float32)
    px, py = to_dev(torch, np.ascontiguousarray(xy[:, 0]), np.ascontiguousarray(xy[:, 1]))

    def triangles(n):
        tri, _ = Context(2, n, 1.0, px.numel(), 1).triangulate(px, py)
        t = tri.cpu().numpy()
        t = np.take_along_axis(t, (t.argmin(1)[:, None] + np.arange(3)) % 3, 1)
        return t[np.lexsort(t.T[::-1])]

    a = triangles(300)
    assert len(a) == 2 * px.numel()
    assert np.array_equal(a, triangles(211))
    c = Context(2, 300, 1.0, px.numel(), 1)
    mesh = torch.sin(torch.arange(90000, device="cuda") * 0.01).reshape(1, -1).float()
    first = c.interpolate_mass(mesh, px, py, info=False).clone()
    for _ in range(6):
        assert torch.equal(c.interpolate_mass(mesh, px, py, info=False), first)
