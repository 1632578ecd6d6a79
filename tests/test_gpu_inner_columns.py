"""A handle with the inexact coarse solve takes calls of any column counts in turn, wider and narrower ones, applications and solves
(whose iterations are replayed from graphs), with the results of a handle that sees one count only.

Bar: applications to 1e-8 relative (the inner solve's bar), solutions to 10 times the tolerance."""
import pytest

from paper_2103_14921_gb300 import synth

pytestmark = pytest.mark.gpu


def test_narrower_calls_after_wider_ones():
    import torch
    from paper_2103_14921_gb300 import build, helm
    build.build()
    ctx = helm.Context(0)
    nx, ny, nz, tol = 33, 29, 21, 1e-6
    c = synth.linear_gradient(nx, ny, nz, 25.0, 1500.0, 1.0, Q=80.0)
    grid = helm.Grid(ctx, nx, ny, nz, 25.0, 5.0, c, npml=3, weights=helm.fit_weights())
    mk = lambda: helm.Oras(grid, (2, 2, 1), 2, coarse_ratio=4, coarse_iters=10, factor_prec=helm.PREC_TF32)
    o, v = mk(), torch.from_numpy(synth.random_complex((nz, ny, nx, 8), 5)).cuda()
    solve = lambda h, b: h.solve(b, tol=tol, basis_prec=helm.PREC_FP32)[0]
    rel = lambda a, b: float(torch.linalg.norm(a - b) / torch.linalg.norm(b))
    want = {n: (mk().apply(v[..., :n].contiguous()), solve(mk(), v[..., :n].contiguous())) for n in (8, 3, 4, 2)}
    for n in (8, 3, 8, 4, 4, 3):
        b = v[..., :n].contiguous()
        assert rel(solve(o, b), want[n][1]) <= 10 * tol, n
        assert rel(solve(o, b), want[n][1]) <= 10 * tol, n   # the second solve replays its iterations
        assert rel(o.apply(b), want[n][0]) <= 1e-8, n
        assert rel(o.apply(v[..., :2].contiguous()), want[2][0]) <= 1e-8, n
