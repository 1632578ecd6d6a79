"""The z-marching stencil at the edges of its tiles: every vector form (two complex64 columns, one complex64 column,
complex128), column counts that leave a ragged chunk, grids smaller than a tile, one plane of halo more than the
grid, real and complex k^2, either top.

Bars.  The per-node kernel and the walk sum the same 27 products (with the coefficients formed in another order): a
sum of n terms is off by at most n eps of the sum of their moduli, in practice sqrt(n) eps, and the moduli of a
Helmholtz row sum to a few times its result on random data.  So 1e-6 (FP32, eps 6e-8) and 1e-14 (FP64, eps 1.1e-16)
in relative L2 between the two, 1e-5 and 1e-12 against the oracle as for every stencil form.
"""
import numpy as np
import pytest

from oracle.discretization import Problem, apply_A
from paper_2103_14921_gb300 import synth

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


@pytest.mark.parametrize("case", [
    # nx, ny, nz, npml, top_pml, Q, columns
    (2, 2, 2, 0, False, None, 1),
    (33, 7, 19, 2, True, None, 18),      # 9 column pairs: two chunks of 5 and 4
    (5, 41, 26, 2, False, 50.0, 13),     # odd columns, complex k^2
    (66, 34, 9, 3, False, None, 3),
    (37, 36, 21, 4, False, None, 27),    # the coarse operator's probes
    (20, 18, 25, 3, True, 80.0, 130),    # 65 pairs
])
def test_march_matches_per_node_kernel_and_oracle(case):
    import torch
    from paper_2103_14921_gb300 import build, helm
    build.build()
    ctx = helm.Context(0)
    nx, ny, nz, npml, top, Q, nrhs = case
    c = synth.linear_gradient(nx, ny, nz, 25.0, 1500.0, 2.0, Q=Q)
    w = synth.random_weights(nx)
    grid = helm.Grid(ctx, nx, ny, nz, 25.0, 5.0, c, npml=npml, top_bc=helm.TOP_PML if top else helm.TOP_DIRICHLET,
                     weights=w)
    prob = Problem(nx, ny, nz, 25.0, 5.0, c, npml=npml, top_pml=top, weights=w)
    u = synth.random_complex((nz, ny, nx, nrhs), 3000 + nx)
    want = apply_A(prob, u)
    for prec, dt, near, bar in ((helm.PREC_FP64, np.complex128, 1e-14, 1e-12), (helm.PREC_FP32, np.complex64, 1e-6, 1e-5)):
        ud = torch.from_numpy(u.astype(dt)).cuda()
        got = []
        for march in (2, 0):
            ctx.set_tuning(helm.TUNE_STENCIL_MARCH, march)
            got.append(grid.apply(ud, prec=prec).cpu().numpy().astype(np.complex128))
        ctx.set_tuning(helm.TUNE_STENCIL_MARCH, 1)
        assert _rel(got[0], got[1]) <= near
        assert _rel(got[0], want) <= bar and _rel(got[1], want) <= bar
