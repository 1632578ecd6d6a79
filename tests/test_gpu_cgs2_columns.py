"""The fused Arnoldi step with the most coefficients its split form takes: 125 to 128 columns and bases that reach 16 vectors
(FP64) and 32 (FP32), where its shared memory is as large as it gets, and one column more (the wide form).

Bar: every column converges, and the FP64 residual of the first and the last is at or below tol.  The FP32 cases ask for
1e-12: a first cycle that stopped at 1e-6 would be 22 vectors long."""
import numpy as np
import pytest

from oracle.discretization import Problem, apply_A
from paper_2103_14921_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs,restart,prec", [(125, 30, "fp64"), (128, 30, "fp64"), (128, 40, "fp32"), (125, 33, "fp32"),
                                               (129, 30, "fp64")])
def test_many_columns_and_long_bases(nrhs, restart, prec):
    import torch
    from paper_2103_14921_gb300 import build, helm
    build.build()
    ctx = helm.Context(0)
    nx, ny, nz, tol = 22, 20, 18, 1e-6 if prec == "fp64" else 1e-12
    c = synth.linear_gradient(nx, ny, nz, 25.0, 1500.0, 0.6, Q=100.0)
    w = helm.fit_weights()
    grid = helm.Grid(ctx, nx, ny, nz, 25.0, 6.0, c, npml=4, weights=w)
    prob = Problem(nx, ny, nz, 25.0, 6.0, c, npml=4, weights=w)
    b = synth.random_complex((nz, ny, nx, nrhs), 12)
    o = helm.Oras(grid, (3, 3, 3), 1)
    x, st = o.solve(torch.from_numpy(b).cuda(), tol=tol, restart=restart,
                    basis_prec=helm.PREC_FP64 if prec == "fp64" else helm.PREC_FP32)
    assert all(s["converged"] for s in st) and min(s["iterations"] for s in st) > (16 if prec == "fp64" else 32)
    x = x.cpu().numpy()
    for r in (0, nrhs - 1):
        assert np.linalg.norm(apply_A(prob, x[..., r]) - b[..., r]) <= tol * np.linalg.norm(b[..., r])


@pytest.mark.parametrize("nrhs", [128, 30])
def test_inner_solve_with_many_columns(nrhs):
    """Sixteen inner iterations with an FP64 basis, against the same apply a few columns at a time: the same inner
    iteration per column, sums in another order (FP64 rounding through 16 steps: the 1e-8 of the same solve against the oracle)."""
    import torch
    from paper_2103_14921_gb300 import build, helm
    build.build()
    ctx = helm.Context(0)
    nx, ny, nz = 37, 33, 25
    c = synth.linear_gradient(nx, ny, nz, 25.0, 1500.0, 1.0, Q=80.0)
    grid = helm.Grid(ctx, nx, ny, nz, 25.0, 5.0, c, npml=3, weights=helm.fit_weights())
    o, few = (helm.Oras(grid, (2, 2, 2), 2, coarse_ratio=3, coarse_iters=16) for _ in range(2))
    v = torch.from_numpy(synth.random_complex((nz, ny, nx, nrhs), 9)).cuda()
    got = o.apply(v)
    for r in (0, nrhs - 3):
        want = few.apply(v[..., r:r + 3].contiguous())
        assert float(torch.linalg.norm(got[..., r:r + 3] - want)) <= 1e-8 * float(torch.linalg.norm(want))
