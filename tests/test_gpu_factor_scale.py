"""The factorisations' choice of path does not depend on the units of length, nor on the rows that pad the last panel: the
same model in millimetres, metres and kilometres, and the exact and inexact coarse operators (entries of 1e-4), whose planes
are all narrower than a panel, take the tensor-core path and give the inverses of the fully pivoted elimination.

Bars.  FP64: 1e-11 in relative Frobenius norm between the two, as in the comparison of the FP64 inverses.  TF32 sets (complex64
inverses): 1e-4, as against the oracle."""
import numpy as np
import pytest

from paper_2103_14921_gb300 import synth

pytestmark = pytest.mark.gpu

TC, CUDA_CORE = ("gj_update_tc",), ("gj_update", "gj_diag")


def _factor(ctx, make):
    """The set, and which families of factor kernels ran."""
    ctx.profile(True, only=list(TC + CUDA_CORE))
    o = make()
    ran = tuple(any(ctx.profile_query(f) is not None for f in fam) for fam in (TC, CUDA_CORE))
    ctx.profile(False)
    return o, ran


@pytest.fixture(scope="module")
def ctx():
    from paper_2103_14921_gb300 import build, helm
    build.build()
    return helm.Context(0)


@pytest.mark.parametrize("unit", [1e3, 1.0, 1e-3, 1e-6])
@pytest.mark.parametrize("prec", ["fp64", "tf32"])
def test_units_of_length(ctx, unit, prec):
    from paper_2103_14921_gb300 import helm
    nx, ny, nz = 21, 17, 4      # boxes of 12 x 17 nodes: a full panel and a partial one
    c = synth.linear_gradient(nx, ny, nz, 25.0, 1500.0, 1.0, Q=80.0) * unit
    grid = helm.Grid(ctx, nx, ny, nz, 25.0 * unit, 5.0, c, npml=2, weights=helm.fit_weights())
    p, tune, bar = (helm.PREC_FP64, helm.TUNE_BLOCK_GJ, 1e-11) if prec == "fp64" else (helm.PREC_TF32, helm.TUNE_TC_FACTOR, 1e-4)
    o, ran = _factor(ctx, lambda: helm.Oras(grid, (2, 1, 1), 2, factor_prec=p))
    assert ran == (True, False)
    got = [o.plane_inverse(b, k).cpu().numpy() for b in range(2) for k in range(nz)]
    ctx.set_tuning(tune, 0)
    o = helm.Oras(grid, (2, 1, 1), 2, factor_prec=p)
    ctx.set_tuning(tune, 2 if prec == "fp64" else 1)
    for x, y in zip(got, [o.plane_inverse(b, k).cpu().numpy() for b in range(2) for k in range(nz)]):
        assert np.linalg.norm(x - y) <= bar * np.linalg.norm(y)


@pytest.mark.parametrize("dims,f,npml,Q,iters", [
    ((28, 26, 24), 6.0, 4, 100.0, 0),      # planes of 64: pivots of 3e-7 in a block whose entries are 2e-4 at most
    ((34, 33, 24), 2.0, 8, None, 0),       # 90: 2e-7
    ((44, 40, 30), 4.0, 8, None, 0),       # 132: a full panel and four columns
    ((80, 80, 80), 4.0, 8, None, 10),      # boxes of 64 to 81
])
def test_small_coarse_operators(ctx, dims, f, npml, Q, iters):
    from paper_2103_14921_gb300 import helm
    nx, ny, nz = dims
    c = synth.linear_gradient(nx, ny, nz, 25.0, 1500.0, 0.6, Q=Q)
    grid = helm.Grid(ctx, nx, ny, nz, 25.0, f, c, npml=npml, weights=helm.fit_weights())
    parts = (3, 3, 3) if iters else (2, 2, 2)
    _, ran = _factor(ctx, lambda: helm.Oras(grid, parts, 2, coarse_ratio=4, coarse_iters=iters, factor_prec=helm.PREC_TF32))
    assert ran == (True, False)
