"""The tensor-core sweep with every number of pipeline stages that can be set, at column counts whose output tile fits in
the stages and (two stages, 98 columns and more) does not.

Bar: the stages only say how far loads run ahead.  Products are summed in the same order and the results moved unchanged,
so the applications are equal bit for bit."""
import pytest

from paper_2103_14921_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [8, 48, 66, 96, 98, 127, 128])
@pytest.mark.parametrize("prec", ["tf32", "bf16"])
def test_stages_do_not_change_the_result(nrhs, prec):
    import torch
    from paper_2103_14921_gb300 import build, helm
    build.build()
    ctx = helm.Context(0)
    nx, ny, nz = 30, 26, 6      # boxes of 17 x 26 nodes: three full row tiles and a partial one
    c = synth.linear_gradient(nx, ny, nz, 25.0, 1500.0, 1.0, Q=80.0)
    grid = helm.Grid(ctx, nx, ny, nz, 25.0, 5.0, c, npml=2, weights=helm.fit_weights())
    o = helm.Oras(grid, (2, 1, 1), 2, factor_prec=helm.PREC_TF32 if prec == "tf32" else helm.PREC_BF16)
    v = torch.from_numpy(synth.random_complex((nz, ny, nx, nrhs), 7)).cuda()
    want = o.apply(v)
    assert bool(torch.isfinite(torch.view_as_real(want)).all())
    for stages in (2, 3, 4, 5):
        for flow in (1, 0):
            ctx.set_tuning(helm.TUNE_TC_STAGES, stages)
            ctx.set_tuning(helm.TUNE_TC_FLOW, flow)
            assert torch.equal(o.apply(v), want), (stages, flow)
