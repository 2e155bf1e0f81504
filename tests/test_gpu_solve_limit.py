"""The limit on the iterations of a mesh solve: kept, counted and reported."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("solver", ["cg", "chebyshev"])
@pytest.mark.parametrize("dim,n,F", [(1, 300, 1), (2, 64, 2), (2, 130, 3)])
def test_limit(dim, n, F, solver):
    import torch

    import paper_1610_05258_gb300 as pmt

    N, rtol = n**dim, 1e-6
    g = np.random.default_rng(n)
    b = torch.from_numpy((g.standard_normal((F, N)) + 0.3).astype(np.float32)).cuda()
    x = torch.empty_like(b)
    ctx = pmt.Context(dim, n, 1.0, 16, F)

    def solve(limit):
        o, info = ctx._opts("zero", rtol, limit, None, solver=solver), (pmt._Info * F)()
        ctx._stream()
        s = ctx.lib.pm_mass_solve(ctx.h, ctypes.c_void_p(b.data_ptr()), F, ctypes.c_void_p(x.data_ptr()),
                                  ctypes.byref(o), info)
        return s, [i.iters for i in info], [i.rel_resid for i in info]

    ok, not_converged = 0, 3  # pm_status
    s, need, res = solve(200)
    assert s == ok and max(res) <= rtol
    most = max(need)
    assert 5 < most < 40
    for limit in (2, most // 2, most - 1):
        s, its, res = solve(limit)
        # Chebyshev's step count is a bound, which the residual beats by a step or two
        if s == not_converged:
            assert max(res) > rtol
        else:
            assert s == ok and solver == "chebyshev" and limit == most - 1 and max(res) <= rtol
        assert max(its) <= limit
    s, its, res = solve(most)
    assert s == ok and its == need and max(res) <= rtol
