"""The triangulation's passes at the edges of their ranges, against the oracle
(exact equality of the triangles): meshes too small for the main pass's search
disc, lists that overflow or fall short (crowds beside voids, where the wide
pass searches again), regular lattices whole and in part (few and many
undecided tests per warp), rings of nearly cocircular particles, particles on
the box edge."""
import numpy as np
import pytest

import oracle
from gpu_util import canon_tris, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def crowd(n, g):
    """A crowd of 30 per cell, a background of 2, and an empty disc between."""
    x = np.concatenate([g.uniform(0.3, 0.4, (30 * n * n // 100, 2)), g.uniform(0, 1, (2 * n * n, 2))])
    d = np.hypot(x[:, 0] - 0.48, x[:, 1] - 0.35)
    return x[d > 3.2 / n]


def lattice(m, g, moved=0.0):
    i = (np.arange(m) + 0.5) / m
    x = np.stack(np.meshgrid(i, i, indexing="xy"), -1).reshape(-1, 2)
    k = g.uniform(size=len(x)) < moved
    x[k] += g.uniform(-0.3, 0.3, (int(k.sum()), 2)) / m
    return x % 1.0


def rings(n, g):
    """Rings of 5 to 9 particles within a few float roundings of a circle about another one."""
    out = []
    for j in range(0, n, 4):
        for i in range(0, n, 4):
            k = 5 + (i // 4 + j // 4) % 5
            c = (np.array([i, j]) + 2 + g.uniform(-0.5, 0.5, 2)) / n
            a = 2 * np.pi * (np.arange(k) + g.uniform(0, 0.3, k)) / k
            out += [c[None], c + 0.9 / n * np.stack([np.cos(a), np.sin(a)], -1)]
    return np.concatenate(out) % 1.0


CASES = {
    "n8": (8, lambda g: g.uniform(0, 1, (2500, 2))),
    "n9": (9, lambda g: g.uniform(0, 1, (1700, 2))),
    "n13": (13, lambda g: g.uniform(0, 1, (700, 2))),
    "n40_below_one_per_cell": (40, lambda g: g.uniform(0, 1, (900, 2))),
    "n24_dense": (24, lambda g: g.uniform(0, 1, (24 * 24 * 12, 2))),
    "crowd_and_void": (32, lambda g: crowd(32, g)),
    "lattice": (24, lambda g: lattice(48, g)),
    "lattice_mostly_moved": (24, lambda g: lattice(48, g, 0.9)),
    "lattice_half_moved": (33, lambda g: lattice(33, g, 0.5)),
    "rings": (32, lambda g: rings(32, g)),
    "box_edge": (20, lambda g: np.concatenate([g.uniform(0, 1, (1200, 2)), g.uniform(-1e-4, 1e-4, (40, 2)) % 1.0])),
}


@pytest.mark.parametrize("name", CASES)
def test_stars(name):
    from paper_1610_05258_gb300 import Context
    n, make = CASES[name]
    xy = make(np.random.default_rng(sum(map(ord, name)))).astype(np.float32)
    px, py = np.ascontiguousarray(xy[:, 0] % np.float32(1)), np.ascontiguousarray(xy[:, 1] % np.float32(1))
    c = Context(2, n, 1.0, px.size, 1)
    dpx, dpy = to_dev(torch, px, py)
    tri, off = c.triangulate(dpx, dpy)
    t, o, _ = oracle.triangulate(1.0, px, py)
    assert canon_tris(tri.cpu().numpy(), off.cpu().numpy()) == canon_tris(t, o)
    # volumes: the same stars fill the box
    v = c.particle_volumes(dpx, dpy).double().sum().item()
    assert abs(v - 1.0) <= 1e-6
