"""The fused Arnoldi step at the widths of its kernels: restart lengths that end in each of them (wide kernels up to 8
vectors, the split form in steps of four, more than 128 columns without it), odd column counts, both basis precisions.

Bars: the FP64 residual of the first and last column at or below tol, and with the FP64 basis the oracle's GMRES iteration
count +-1 (the repository's bar for its orthogonalisation against the oracle's modified Gram-Schmidt)."""
import numpy as np
import pytest

from oracle.discretization import Problem, apply_A, assemble_A
from oracle.krylov import gmres
from oracle.schwarz import ORAS
from paper_2103_14921_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs,restart,prec", [(3, 40, "fp32"), (16, 40, "fp32"), (5, 40, "fp64"), (130, 12, "fp32")])
def test_fused_cgs2_widths(nrhs, restart, prec):
    import torch
    from paper_2103_14921_gb300 import build, helm
    build.build()
    ctx = helm.Context(0)
    nx, ny, nz, tol = 22, 20, 18, 1e-6
    c = synth.linear_gradient(nx, ny, nz, 25.0, 1500.0, 0.6, Q=100.0)
    w = helm.fit_weights()
    grid = helm.Grid(ctx, nx, ny, nz, 25.0, 6.0, c, npml=4, weights=w)
    prob = Problem(nx, ny, nz, 25.0, 6.0, c, npml=4, weights=w)
    b = synth.random_complex((nz, ny, nx, nrhs), 12)
    o = helm.Oras(grid, (3, 3, 3), 1)   # one level, small boxes: more than 32 iterations
    x, st = o.solve(torch.from_numpy(b).cuda(), tol=tol, restart=restart,
                    basis_prec=helm.PREC_FP64 if prec == "fp64" else helm.PREC_FP32)
    x = x.cpu().numpy()
    for r in (0, nrhs - 1):
        assert st[r]["converged"]
        assert np.linalg.norm(apply_A(prob, x[..., r]) - b[..., r]) <= tol * np.linalg.norm(b[..., r])
    if prec == "fp64":
        M, A = ORAS(prob, (3, 3, 3), 1), assemble_A(prob)
        _, info = gmres(lambda v: A @ v, b[..., 0].ravel(), M.apply, tol=tol, restart=restart)
        assert abs(st[0]["iterations"] - info["iterations"]) <= 1
