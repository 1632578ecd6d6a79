"""A call whose working vectors do not fit the budget fails with ENOMEM, every time it is made, gives its memory back, and leaves
the handle as it was for narrower calls.

Bar: a narrower application afterwards is that of a handle without a budget, bit for bit."""
import pytest

from paper_2103_14921_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,coarse,iters", [("fp64", 4, 0), ("tf32", 4, 0), ("tf32", 4, 10), ("fp32", 0, 0)])
def test_too_wide_calls_leave_the_handle_whole(prec, coarse, iters):
    import torch
    from paper_2103_14921_gb300 import build, helm
    build.build()
    nx, ny, nz = 28, 26, 24
    p = {"fp64": helm.PREC_FP64, "fp32": helm.PREC_FP32, "tf32": helm.PREC_TF32}[prec]
    c = synth.linear_gradient(nx, ny, nz, 25.0, 1500.0, 1.0, Q=80.0)
    v = torch.from_numpy(synth.random_complex((nz, ny, nx, 64), 3)).cuda()

    def make(budget):
        ctx = helm.Context(0, budget_bytes=budget)
        g = helm.Grid(ctx, nx, ny, nz, 25.0, 5.0, c, npml=3, weights=helm.fit_weights())
        return ctx, g, helm.Oras(g, (2, 2, 2), 2, coarse_ratio=coarse, coarse_iters=iters, factor_prec=p)

    free, _, o = make(0)
    held = free.bytes_in_use
    want = o.apply(v[..., :2].contiguous())
    narrow = free.bytes_in_use - held
    o.apply(v)
    wide = free.bytes_in_use - held
    assert wide > 6 * narrow
    budget = 512 << 20
    ctx, _, o = make(budget)
    for part in (0.9, 0.5, 0.2):        # room for some of the wide call's vectors
        planes = int((budget - ctx.bytes_in_use - part * wide) / (100 * 100 * 40))   # a grid's 40 bytes a node
        filler = helm.Grid(ctx, 100, 100, planes, 25.0, 5.0,
                           torch.full((planes, 100, 100), 1500.0, dtype=torch.complex128, device="cuda"), npml=3)
        before = ctx.bytes_in_use
        assert narrow < budget - before < wide
        for _ in range(2):
            with pytest.raises(helm.HelmError) as e:
                o.apply(v)
            assert e.value.status == helm.ENOMEM
            assert ctx.bytes_in_use == before
        assert torch.equal(o.apply(v[..., :2].contiguous()), want)
        filler.close()
        o.apply(v)                      # with the room back
        o.close()
        ctx, _, o = make(budget)
