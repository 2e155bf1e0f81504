"""Sums over threads, warps and blocks of the solves: FP64 precision and range."""

import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n", [(1, 31), (2, 5)])
@pytest.mark.parametrize("solver", ["cg", "chebyshev"])
def test_reported_sum_of_cancelling_nodes(dim, n, solver):
    """One warp holds all nodes, one each: its total is exact to far below FP64,
    so the reported integral is off by its conversion (two additions), the scale
    and the node volume, 2^-53 each, whatever the nodes cancel to."""
    import torch

    import paper_1610_05258_gb300 as pmt

    N, h = n**dim, float(np.float32(1.0 / n))
    ctx = pmt.Context(dim, n, 1.0, 16, 1)
    for seed in range(20):
        b = np.random.default_rng(seed).standard_normal((1, N))
        b = (b - b.mean() + 1e-3).astype(np.float32)
        x, info = ctx.mass_solve(torch.from_numpy(b).cuda(), solver=solver)
        x = x.cpu().numpy().astype(np.float64).ravel()
        exact = math.fsum(x) * (h * h if dim == 2 else h)
        tol = 6 * 2.0**-53 * abs(exact) + 2.0**-66 * np.abs(x).sum()
        assert abs(info[0].sum_mesh - exact) <= tol, (seed, info[0].sum_mesh, exact)


@pytest.mark.parametrize("solver", ["cg", "chebyshev"])
@pytest.mark.parametrize("n", [63, 64])
def test_mesh_solve_near_the_largest_float(n, solver):
    """The sums over the threads leave FP32's range, the nodes and the result do not."""
    import torch

    import paper_1610_05258_gb300 as pmt

    t = 2 * np.pi * np.arange(n) / n
    b = (1 + 0.2 * np.sin(t)[:, None] * np.cos(2 * t)[None, :]).astype(np.float32).reshape(1, -1)
    ctx = pmt.Context(2, n, float(n), 16, 1)  # h = 1
    bd, k = torch.from_numpy(b).cuda(), 2.0**124
    ref, i0 = ctx.mass_solve(bd, solver=solver)
    got, i1 = ctx.mass_solve(bd * k, solver=solver)
    assert torch.equal(got, ref * k)
    assert i0[0].iters == i1[0].iters > 0 and i1[0].sum_mesh == i0[0].sum_mesh * k


@pytest.mark.parametrize("threads,cluster", [(256, 1), (1024, 1), (512, 4), (256, 8)])
def test_batch_near_the_largest_float(threads, cluster):
    """As above for a batch: results and reported sums scale by the power of two."""
    import torch

    import paper_1610_05258_gb300 as pmt
    from paper_1610_05258_gb300 import workloads as W

    n, k = 48, 2.0**118
    inst = W.uniform_instance(n, 4, F=1, seed=9)
    px, py, v = (torch.from_numpy(a).cuda() for a in (inst.px, inst.py, 1 + 0.1 * inst.vals))
    bt = pmt.Batch([n], [float(n)], [inst.np], 1)
    bt.set_tuning(threads, cluster)
    out = [torch.empty(1, n * n, device="cuda") for _ in range(2)]
    rep = [bt.assign_mass([px * n], [py * n], [v * s], [o])[0][0] for s, o in ((1.0, out[0]), (k, out[1]))]
    assert torch.equal(out[1], out[0] * k)
    assert rep[1].sum_mesh == rep[0].sum_mesh * k and rep[1].sum_particles == rep[0].sum_particles * k
