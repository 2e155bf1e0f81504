"""The right-hand side and the delta assignment where their work is cut
differently: tiles shared by 8, several and one block, 1 to 8 fields (gradients
kept per triangle or per piece), triangles of many cells and nodes (sparse
particles), particles on nodes, cell lines and the box edge. Against the oracle,
relative L2 <= 1e-5 as for every transfer."""
import numpy as np
import pytest

import oracle
from gpu_util import rel_l2, to_dev
from paper_1610_05258_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def on_lines(n, g):
    """A third of the particles moved onto cell lines, some onto nodes."""
    x = g.uniform(0, 1, (3 * n * n, 2))
    k = len(x) // 3
    x[:k, 0] = np.round(x[:k, 0] * n) / n
    x[k // 2:k // 2 + k // 4, 1] = np.round(x[k // 2:k // 2 + k // 4, 1] * n) / n
    x = np.unique((x % 1.0).astype(np.float32), axis=0)
    return x[:, 0].copy(), x[:, 1].copy()


@pytest.mark.parametrize("n,ppc,F", [(16, 12, 1), (50, 4, 4), (50, 4, 5), (33, 5, 8), (90, 0.7, 2), (120, 0.15, 1)])
def test_rhs_and_delta(n, ppc, F):
    from paper_1610_05258_gb300 import Context
    inst = W.uniform_instance(n, ppc, F=F, seed=n + F)
    c = Context(2, n, inst.L, inst.np, F)
    px, py, vals = to_dev(torch, inst.px, inst.py, inst.vals)
    b = c.mass_rhs(px, py, vals).cpu().numpy().reshape(F, -1)
    assert rel_l2(b, oracle.rhs(2, n, inst.L, inst.px, inst.py, inst.vals)) <= 1e-5
    d = c.assign_delta(px, py, vals).cpu().numpy().reshape(F, -1)
    assert rel_l2(d, oracle.delta(2, n, inst.L, inst.px, inst.py, inst.vals)) <= 1e-5


def test_particles_on_cell_lines():
    from paper_1610_05258_gb300 import Context
    n = 24
    px, py = on_lines(n, np.random.default_rng(5))
    vals = np.stack([np.sin(6.28 * px), np.cos(6.28 * py) * px]).astype(np.float32)
    c = Context(2, n, 1.0, px.size, 2)
    dx, dy, dv = to_dev(torch, px, py, vals)
    b = c.mass_rhs(dx, dy, dv).cpu().numpy().reshape(2, -1)
    assert rel_l2(b, oracle.rhs(2, n, 1.0, px, py, vals)) <= 1e-5
    d = c.assign_delta(dx, dy, dv).cpu().numpy().reshape(2, -1)
    assert rel_l2(d, oracle.delta(2, n, 1.0, px, py, vals)) <= 1e-5


@pytest.mark.parametrize("n", [144, 400, 576])
def test_shared_tiles_conserve(n):
    """81, 625 and 1296 tiles: 8, 1 and 1 blocks each; the integer sums over
    the mesh equal the particle integrals to FP32 rounding of the volumes."""
    from paper_1610_05258_gb300 import Context
    inst = W.uniform_instance(n, 3, F=2, seed=n)
    c = Context(2, n, inst.L, inst.np, 2)
    px, py, vals = to_dev(torch, inst.px, inst.py, inst.vals + 2.0)
    b = c.mass_rhs(px, py, vals).double().reshape(2, -1).sum(1)
    want = (c.particle_volumes(px, py).double()[None] * vals.double()).sum(1)
    assert ((b - want).abs() / want.abs()).max().item() <= 1e-6
