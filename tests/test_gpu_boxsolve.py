"""The inexact coarse solve's one-launch box solver against the oracle's preconditioner, on coarse partitions that give
boxes of one plane, odd plane sizes, one column and ragged column chunks.

Bars: FP64 1e-8 and FP32 factors 1e-3 in relative L2, those of the same comparisons with the general sweeps (ten GMRES
steps are a smooth function of the data; FP32 factors carry their rounding through the sweeps)."""
import numpy as np
import pytest

from oracle.discretization import Problem
from oracle.schwarz import ORAS
from paper_2103_14921_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,parts,cov,nrhs", [
    ((25, 22, 9), (3, 2, 1), 1, 1),
    ((30, 17, 14), (2, 2, 3), 0, 5),      # boxes of one or two coarse planes, no coarse overlap
    ((33, 29, 21), (2, 1, 2), 2, 18),     # larger planes, a ragged second chunk of 16 columns
])
def test_small_coarse_boxes_match_oracle(dims, parts, cov, nrhs):
    import torch
    from paper_2103_14921_gb300 import build, helm
    build.build()
    ctx = helm.Context(0)
    nx, ny, nz = dims
    c = synth.linear_gradient(nx, ny, nz, 25.0, 1500.0, 2.0, Q=80.0)
    w = synth.random_weights(4)
    grid = helm.Grid(ctx, nx, ny, nz, 25.0, 5.0, c, npml=3, weights=w)
    prob = Problem(nx, ny, nz, 25.0, 5.0, c, npml=3, weights=w)
    M = ORAS(prob, parts, 2, coarse_ratio=4, coarse_solve="gmres", coarse_iters=10, coarse_overlap=cov)
    v = synth.random_complex((nz, ny, nx, nrhs), 41)
    want = M.apply(v.reshape(-1, nrhs)).reshape(v.shape)
    for prec, bar in ((helm.PREC_FP64, 1e-8), (helm.PREC_FP32, 1e-3)):
        o = helm.Oras(grid, parts, 2, coarse_ratio=4, coarse_iters=10, coarse_overlap=cov, factor_prec=prec)
        got = o.apply(torch.from_numpy(v).cuda()).cpu().numpy()
        assert np.linalg.norm(got - want) <= bar * np.linalg.norm(want)
