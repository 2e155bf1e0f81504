"""Batches whose instances share blocks of the gather and differ in scale, at
every setting of the solve, against single contexts."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# mesh sides and particles: several instances in one block of 256 slots, blocks
# that end with an instance, instances longer than a block
SIDES = [16, 17, 16, 18, 33, 16, 64]
COUNTS = [m * m for m in (12, 13, 12, 14, 47, 23, 95)]


@pytest.mark.parametrize("threads,cluster", [(256, 1), (512, 4), (1024, 8)])
@pytest.mark.parametrize("F", [1, 3])
def test_batch_edges(threads, cluster, F):
    import torch

    import paper_1610_05258_gb300 as pmt

    rng = np.random.default_rng(11 * F + cluster)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()
    # jittered lattices: no void that a small mesh could not certify
    grid = [np.divmod(np.arange(p), round(p**0.5)) for p in COUNTS]
    xs, ys = ([dev((g[c] + 0.9 * rng.random(p)) / round(p**0.5)) for g, p in zip(grid, COUNTS)] for c in (0, 1))
    # a scale of its own for every instance and field: a maximum of the wrong
    # instance would lose the small fields in the fixed-point sums
    vs = [dev((rng.random((F, p)) + 0.5) * 10.0 ** (6 * rng.random((F, 1)) - 3)) for p in COUNTS]
    outs = [torch.zeros((F, n * n), device="cuda") for n in SIDES]
    b = pmt.Batch(SIDES, [1.0] * len(SIDES), COUNTS, F, tune=threads)
    b.set_tuning(threads, cluster, largest_first=cluster > 1)
    info = b.assign_mass(xs, ys, vs, outs)
    for k, n in enumerate(SIDES):
        one, ref = pmt.Context(2, n, 1.0, COUNTS[k], F).assign_mass(xs[k], ys[k], vs[k])
        got, want = outs[k].cpu().numpy(), one.cpu().numpy().reshape(F, -1)
        for f in range(F):
            # both meet rtol = 1e-6 on the same right-hand side, kappa = 9; each is rounded to FP32
            assert np.linalg.norm(got[f] - want[f]) <= 9 * 2.4e-6 * np.linalg.norm(want[f])
            assert info[k][f].rel_resid <= 1e-6
            assert abs(info[k][f].sum_particles - ref[f].sum_particles) <= 1e-6 * abs(ref[f].sum_particles)
