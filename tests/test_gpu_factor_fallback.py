"""The FP64 factorisation where it leaves its usual way: the third Newton step of ill-conditioned planes, the two reasons for which a
set goes to the FP64 elimination (and the third, no room), and sets that are factored in several batches of boxes.

Ill-conditioned planes come from a uniform medium without layers or loss, driven next to an eigenfrequency of its first
plane's operator (f (1 + d): condition number about 1 / d).  The numbers beside the cases are max |I - S X| of a complex64 inverse X0
and of a Newton step on it, X1, cut to 24 and 40 bits of their columns' largest entries, as numpy gives them; an elimination
by blocks leaves up to ten times as much.  The third step is taken from 3e-10 of the second on, and the set given up where
the first exceeds 1e-3.

Bars.  After a fallback the factors are those of the elimination that it names, bit for bit.  A third Newton step: the residual
|I - D_0 G_0| of the first plane at most twice the fully pivoted FP64 elimination's (both are bounded by eps times the condition
number) plus 1e-14 sqrt(m); with the exact coarse solve, applications equal to 1e-9, the bar of FP64 applications.  Batches: 1e-11 in relative Frobenius norm from the pivoted elimination, as for one batch."""
import numpy as np
import pytest

from oracle.discretization import Problem
from oracle.schwarz import decompose, local_operator, plane_blocks
from paper_2103_14921_gb300 import synth

pytestmark = pytest.mark.gpu

H, C0 = 25.0, 1500.0


@pytest.fixture(scope="module")
def helm():
    from paper_2103_14921_gb300 import build, helm
    build.build()
    return helm


def _planes(dims, f):
    """Schur complements S_0, S_1, ... of the one box of the grid, in FP64."""
    nx, ny, nz = dims
    prob = Problem(nx, ny, nz, H, f, np.full((nz, ny, nx), C0, dtype=complex), npml=0, weights=synth.random_weights(nx))
    box = decompose(dims, (1, 1, 1), 0)[0]
    D, L, U = (([np.asarray(a.toarray() if hasattr(a, "toarray") else a) if a is not None else None for a in x])
               for x in plane_blocks(local_operator(prob, box, "oras"), nx * ny, nz))
    S = [D[0]]
    for k in range(1, nz):
        S.append(D[k] - L[k] @ np.linalg.solve(S[-1], U[k - 1]))
    return S


def _eigenfrequency(dims):
    a, b = _planes(dims, 1e-9)[0], _planes(dims, 5.0)[0]
    ev = np.linalg.eigvals(-np.linalg.solve((b - a) / (2 * np.pi * 5.0 / C0) ** 2, a))
    ev = np.sort(ev.real[(abs(ev.imag) < 1e-12 * abs(ev)) & (ev.real > 0)])
    return np.sqrt(ev[1]) * C0 / (2 * np.pi)


def _cut(x, bits):
    top = np.maximum(abs(x.real), abs(x.imag)).max(axis=0)
    scale = np.exp2(bits - 2 - np.floor(np.log2(top)))
    return (np.rint(x.real * scale) + 1j * np.rint(x.imag * scale)) / scale


def _newton_residuals(S):
    """max |I - S X| of X0 and of X1."""
    x = _cut(np.linalg.inv(S.astype(np.complex64)).astype(complex), 24)
    r = np.eye(len(S)) - S @ x
    return abs(r).max(), abs(np.eye(len(S)) - S @ _cut(x + x @ r, 40)).max()


def _factor(helm, ctx, dims, f, mode):
    nx, ny, nz = dims
    grid = helm.Grid(ctx, nx, ny, nz, H, f, np.full((nz, ny, nx), C0, dtype=complex), npml=0,
                     weights=synth.random_weights(nx))
    ctx.set_tuning(helm.TUNE_BLOCK_GJ, mode)
    o = helm.Oras(grid, (1, 1, 1), 0, factor_prec=helm.PREC_FP64)
    ctx.set_tuning(helm.TUNE_BLOCK_GJ, 2)
    return [o.plane_inverse(0, k).cpu().numpy() for k in range(nz)]


@pytest.mark.parametrize("dims", [(9, 8, 2), (20, 16, 2)])   # 9e-6, 2e-10 and 7e-6, 4e-10
def test_third_newton_step(helm, dims):
    nx, ny, _ = dims
    a, b = _planes(dims, 1e-9)[0], _planes(dims, 5.0)[0]
    v = np.outer(np.sin(np.pi * np.arange(1, ny + 1) / (ny + 1)), np.sin(np.pi * np.arange(1, nx + 1) / (nx + 1))).ravel()
    k2 = (v @ a @ v).real / (v @ (a - b) @ v).real * (2 * np.pi * 5.0 / C0) ** 2   # the plane's longest wave
    f = np.sqrt(k2) * C0 / (2 * np.pi) * (1 + 1e-3)
    S = _planes(dims, f)
    res = [_newton_residuals(s) for s in S]
    assert max(r[0] for r in res) < 5e-5 and max(r[1] for r in res) > 1e-10
    ctx = helm.Context(0)
    got = _factor(helm, ctx, dims, f, 2)
    assert sum(ctx.factor_fallbacks.values()) == 0
    ref = _factor(helm, ctx, dims, f, 0)
    off = [np.linalg.norm(np.eye(len(S[0])) - S[0] @ x[0]) for x in (got, ref)]
    assert off[0] <= 2 * off[1] + 1e-14 * np.sqrt(len(S[0]))


def test_third_newton_step_of_a_large_coarse_plane(helm):
    """An exact coarse problem with planes of 44 x 42 (tiles of 128 columns; 5e-5, 9e-10)."""
    import torch
    nx, ny, nz = 86, 82, 6
    ctx = helm.Context(0)
    grid = helm.Grid(ctx, nx, ny, nz, H, 4.0, synth.linear_gradient(nx, ny, nz, H, C0, 0.6), npml=2, weights=helm.fit_weights())
    v = torch.from_numpy(synth.random_complex((nz, ny, nx, 2), 31)).cuda()
    got = {}
    for mode in (2, 0):
        ctx.set_tuning(helm.TUNE_BLOCK_GJ, mode)
        got[mode] = helm.Oras(grid, (4, 4, 1), 2, coarse_ratio=2, factor_prec=helm.PREC_FP64).apply(v)
    assert sum(ctx.factor_fallbacks.values()) == 0
    assert float(torch.linalg.norm(got[2] - got[0])) <= 1e-9 * float(torch.linalg.norm(got[0]))


@pytest.mark.parametrize("d,why", [(1e-6, "accuracy"),    # 6e-2; smallest pivot 1e-5 of the block
                                   (1e-9, "pivot")])      # smallest pivot 7e-9
def test_fallback_is_counted_and_gives_the_elimination(helm, d, why):
    dims = (16, 8, 2)
    f = _eigenfrequency(dims) * (1 + d)
    assert max(_newton_residuals(s)[0] for s in _planes(dims, f)) > 3e-3
    ctx = helm.Context(0)
    ref = _factor(helm, ctx, dims, f, 1)
    n1 = ctx.factor_fallbacks      # the elimination itself may meet a weak pivot
    got = _factor(helm, ctx, dims, f, 2)
    n2 = ctx.factor_fallbacks
    extra = {k: n2[k] - 2 * n1[k] for k in n1}
    assert extra == {"pivot": int(why == "pivot"), "accuracy": int(why == "accuracy"), "room": 0}
    assert all(np.array_equal(x, y) for x, y in zip(got, ref))


def test_no_room_for_the_newton_workspace(helm):
    """A budget that holds the factors and the elimination's work matrices but not the digit slices."""
    dims = (43, 41, 3)
    m = dims[0] * dims[1]
    ctx = helm.Context(0)
    ref = _factor(helm, ctx, dims, 5.0, 1)
    tight = helm.Context(0, budget_bytes=(3 + 2) * m * m * 16 + (80 << 20))   # the digit slices alone take 270 MB
    got = _factor(helm, tight, dims, 5.0, 2)
    assert tight.factor_fallbacks == {"pivot": 0, "accuracy": 0, "room": 1}
    assert helm.lib().helm_last_error(tight._h) == b""
    assert all(np.array_equal(x, y) for x, y in zip(got, ref))


def test_batches_of_unequal_boxes(helm):
    """64 boxes of 676 to 784 unknowns a plane: more than 4 GB of workspace, so two batches, the second with corner boxes
    where the first had inner ones."""
    nx, ny, nz, parts, ov = 192, 186, 2, (8, 8, 1), 2
    c = synth.linear_gradient(nx, ny, nz, H, C0, 1.0, Q=80.0)
    ctx = helm.Context(0)
    grid = helm.Grid(ctx, nx, ny, nz, H, 5.0, c, npml=1, weights=helm.fit_weights())
    got = {}
    for mode in (2, 0):
        ctx.set_tuning(helm.TUNE_BLOCK_GJ, mode)
        o = helm.Oras(grid, parts, ov, factor_prec=helm.PREC_FP64)
        got[mode] = [o.plane_inverse(b, k).cpu() for b in range(0, 64, 3) for k in range(nz)]
        o.close()
    assert sum(ctx.factor_fallbacks.values()) == 0
    for x, y in zip(got[2], got[0]):
        assert x.shape == y.shape and float((x - y).norm()) <= 1e-11 * float(y.norm())
