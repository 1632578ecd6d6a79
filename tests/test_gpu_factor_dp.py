"""FP64 plane inverses from complex64 ones and Newton steps with exact digit products on the tensor cores, against the
fully pivoted FP64 elimination: planes below one tile, at and around 128 unknowns (one panel, one row tile), ragged 64-real
column tiles, and boxes of different plane sizes in one set.

Bars.  Both are inverses in FP64 of Schur complements with condition numbers up to 1e3: each is off by a few tens of
eps times that at most, so 1e-11 in relative Frobenius norm between the two; the first plane's S_0 = D_0 is known exactly
from the oracle, and |I - D_0 G_0| / sqrt(m) <= 1e-13 (an elimination's is 1e-15 .. 1e-14)."""
import numpy as np
import pytest

from oracle.discretization import Problem
from oracle.schwarz import decompose, local_operator, plane_blocks
from paper_2103_14921_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,parts,ov,Q", [
    ((5, 3, 4), (1, 1, 1), 0, None),           # 15 unknowns
    ((16, 8, 5), (1, 1, 1), 0, 60.0),          # 128: exactly one panel and row tile
    ((43, 3, 4), (1, 1, 1), 0, None),          # 129
    ((33, 31, 6), (2, 2, 1), 1, 80.0),         # boxes of 16..18 x 16..17 nodes
    ((40, 22, 5), (1, 1, 1), 0, None),         # 880: seven panels, the last partial
    ((43, 41, 3), (1, 1, 1), 0, None),         # 1763: more 128-column tiles than SMs, two passes of four orders
    ((70, 62, 3), (2, 2, 1), 1, 80.0),         # the same with boxes of up to 36 x 32 = 1152 = 9 x 128 nodes
])
def test_newton_inverses_match_pivoted_fp64_elimination(dims, parts, ov, Q):
    from paper_2103_14921_gb300 import build, helm
    build.build()
    ctx = helm.Context(0)
    nx, ny, nz = dims
    c = synth.linear_gradient(nx, ny, nz, 25.0, 1500.0, 1.0, Q=Q)
    w = synth.random_weights(nx)
    grid = helm.Grid(ctx, nx, ny, nz, 25.0, 5.0, c, npml=1, weights=w)
    prob = Problem(nx, ny, nz, 25.0, 5.0, c, npml=1, weights=w)
    boxes = decompose(dims, parts, ov)
    got = {}
    for mode in (2, 0):
        ctx.set_tuning(helm.TUNE_BLOCK_GJ, mode)
        ctx.profile(True, only=["gj_update_tc", "gj_update"])
        o = helm.Oras(grid, parts, ov, factor_prec=helm.PREC_FP64)
        newton = ctx.profile_query("gj_update_tc") is not None and ctx.profile_query("gj_update") is None
        ctx.profile(False)
        assert newton == (mode == 2)
        got[mode] = [[o.plane_inverse(b, k).cpu().numpy() for k in range(box.dims[2])] for b, box in enumerate(boxes)]
        o.close()
    for b, box in enumerate(boxes):
        m = box.dims[0] * box.dims[1]
        D, _, _ = plane_blocks(local_operator(prob, box, "oras"), m, box.dims[2])
        D0 = D[0].toarray() if hasattr(D[0], "toarray") else np.asarray(D[0])
        assert np.linalg.norm(np.eye(m) - D0 @ got[2][b][0]) <= 1e-13 * np.sqrt(m)
        for x, y in zip(got[2][b], got[0][b]):
            assert np.linalg.norm(x - y) <= 1e-11 * np.linalg.norm(y)
