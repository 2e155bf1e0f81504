"""Mesh solves (single-barrier CG, Chebyshev) against the FP64 Fourier solution
at the edges of their access widths and grids."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def eigenvalues(dim, n, mesh):
    """Eigenvalues of the periodic mass matrix (Fourier modes), L = 1."""
    h, t = 1.0 / n, 2 * np.pi * np.arange(n) / n
    if dim == 1:
        return h / 6 * (4 + 2 * np.cos(t))
    if mesh == "p1":
        a, b = t[:, None], t[None, :]
        return h * h / 12 * (6 + 2 * np.cos(a) + 2 * np.cos(b) + 2 * np.cos(a + b))
    s = 4 + 2 * np.cos(t)
    return h * h / 36 * s[:, None] * s[None, :]


# sizes: the smallest, quads of a row or single nodes, one block or several,
# fewer and more nodes than threads; offset 1: arrays off the 16-byte boundary
CASES = [(1, 4, 1, "q1", 0), (1, 255, 3, "q1", 0), (1, 257, 8, "q1", 1), (1, 50001, 2, "q1", 0),
         (2, 4, 8, "q1", 0), (2, 5, 2, "p1", 0), (2, 32, 1, "q1", 0), (2, 36, 5, "p1", 1), (2, 63, 3, "q1", 0),
         (2, 256, 4, "q1", 1), (2, 401, 1, "p1", 0), (2, 1028, 2, "q1", 0), (2, 1028, 2, "p1", 0)]


@pytest.mark.parametrize("solver", ["cg", "chebyshev"])
@pytest.mark.parametrize("dim,n,F,mesh,offset", CASES)
def test_mesh_solve_edges(dim, n, F, mesh, offset, solver):
    import torch

    import paper_1610_05258_gb300 as pmt

    N, rtol = n**dim, 1e-6
    rng = np.random.default_rng(n + F)
    # fields of very different size, the last of several zero
    b = rng.standard_normal((F, N)).astype(np.float32) + np.float32(0.3)
    b *= (10.0 ** (4 * (np.arange(F) - F // 2))).astype(np.float32)[:, None]
    if F > 1:
        b[-1] = 0.0
    buf, dst = torch.zeros(F * N + 4, device="cuda"), torch.zeros(F * N + 4, device="cuda")
    bd, out = (v[offset:offset + F * N].view(F, N) for v in (buf, dst))
    bd.copy_(torch.from_numpy(b))
    ctx = pmt.Context(dim, n, 1.0, 16, F, mesh=mesh)
    x, info = ctx.mass_solve(bd, out=out, rtol=rtol, solver=solver)
    x = x.cpu().numpy().astype(np.float64)
    axes = tuple(range(1, dim + 1))
    exact = np.fft.ifftn(np.fft.fftn(b.astype(np.float64).reshape((F,) + (n,) * dim), axes=axes)
                         / eigenvalues(dim, n, mesh), axes=axes).real.reshape(F, N)
    # ||e|| / ||x|| <= kappa ||r|| / ||b||, and the rounding of the FP32 result
    # and of the residual that is compared with rtol (a few units of 2^-24)
    kappa = {1: 3.0, 2: 4.0 if mesh == "p1" else 9.0}[dim]
    for f in range(F):
        if not b[f].any():
            assert not x[f].any() and info[f].iters == 0
            continue
        assert info[f].rel_resid <= rtol
        err = np.linalg.norm(x[f] - exact[f]) / np.linalg.norm(exact[f])
        assert err <= kappa * (rtol + 4 * 2.0**-24), (f, err)
    assert not dst[:offset].any() and not dst[offset + F * N:].any()
    if N < 32:
        return
    # a limit on the iterations is kept and reported
    with pytest.raises(pmt.PMError):
        ctx.mass_solve(bd, rtol=1e-30, max_iter=2, solver=solver)
