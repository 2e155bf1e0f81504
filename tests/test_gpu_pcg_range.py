"""Full-mass projection at field amplitudes and box sizes whose inner products
leave the range of FP32: a power-of-two factor on the field multiplies the
result by it bit for bit, and a power-of-two factor on the box leaves it alone."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F", [1, 3, 5])
@pytest.mark.parametrize("L,k", [(1.0, 70), (1.0, -60), (2.0**10, 60), (2.0**30, 17), (2.0**-20, 10), (2.0**-20, -30),
                                 (2.0**-28, 0), (2.0**-28, 80)])
def test_projection_scales_exactly_2d(L, k, F):
    import torch

    import paper_1610_05258_gb300 as pmt
    from paper_1610_05258_gb300 import workloads as W

    n = 160
    inst = W.uniform_instance(n, 4, F=1, seed=11)
    px, py = (torch.from_numpy(v).cuda() for v in (inst.px, inst.py))
    mesh = torch.from_numpy(W.mesh_field(2, n, 1.0, F=F, seed=5).astype(np.float32)).cuda().reshape(F, -1)
    ref, info0 = pmt.Context(2, n, 1.0, inst.np, F).interpolate_mass(mesh, px, py)
    got, info = pmt.Context(2, n, L, inst.np, F).interpolate_mass(mesh * 2.0**k, px * L, py * L)
    assert torch.equal(got, ref * 2.0**k)
    for a, b in zip(info0, info):
        assert a.iters == b.iters > 0 and b.rel_resid <= 1e-6
        assert b.sum_particles == pytest.approx(a.sum_particles * L * L * 2.0**k, rel=1e-12)


def test_projection_scales_exactly_1d():
    import torch

    import paper_1610_05258_gb300 as pmt

    n, N, L, k = 4096, 20000, 2.0**24, 60
    g = np.random.default_rng(3)
    px = torch.from_numpy(np.unique(g.random(N).astype(np.float32))).cuda()
    mesh = torch.from_numpy(g.standard_normal((1, n)).astype(np.float32)).cuda()
    ref, i0 = pmt.Context(1, n, 1.0, N, 1).interpolate_mass(mesh, px)
    got, i1 = pmt.Context(1, n, L, N, 1).interpolate_mass(mesh * 2.0**k, px * L)
    assert torch.equal(got, ref * 2.0**k) and i0[0].iters == i1[0].iters > 0
