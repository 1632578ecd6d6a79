"""What the framework's users have it do, as cases that can be timed: the matrix-free stencil, the preconditioner,
whole solves, and set-up plus solve for a model that has not been seen before.

    listed()            the cases, as dicts of plain values
    draw(rng)           one more case of the same ranges
    prepare(case, seed) what a program holds before the call: inputs on the GPU, the grid, the factors
    run(state)          one pass through the public entry points (paper_2103_14921_gb300.helm)
    work(case)          bytes and flops that one pass cannot do without
    exact(case, seed)   the result in 64 bits, in plain torch

A mixed-precision solution (tolerance 1e-6, factors in TF32 or BF16, a complex64 Krylov basis) holds no more than
single precision, so the wavefields are handed on as complex64, the form in which a program keeps them; FP64 solves
and FP64 operators return complex128.
"""
import math

import numpy as np
import torch

from paper_2103_14921_gb300 import helm

H = 25.0        # grid spacing, metres
NPML = 8        # absorbing-layer nodes
PML_R = 1e-3    # nominal reflection of the layers
# Mixed-grid weights of the least-squares dispersion fit over 4..30 points per wavelength (both sets sum to one).
WEIGHTS = (0.10980402724150182, 0.7336890594897049, 0.15650691326879332,
           0.4903156890122782, 0.07834855063504595, 0.0032994172647871837, 0.0)
PREC = {"fp64": helm.PREC_FP64, "fp32": helm.PREC_FP32, "tf32": helm.PREC_TF32, "bf16": helm.PREC_BF16}
ENTRY = {"fp64": 16, "fp32": 8, "tf32": 8, "bf16": 4}   # bytes of one stored factor entry


def _stencil(name, nx, ny, nz, nrhs, prec, model="gradient", q=0, top=0, f=5.0):
    return dict(name=name, kind="stencil", nx=nx, ny=ny, nz=nz, nrhs=nrhs, prec=prec, model=model, q=q, top=top, f=f)


def _solver(name, kind, nx, ny, nz, nrhs, f, parts, overlap, coarse, inner, prec, model="gradient", q=0, restart=30,
            flexible=True, nfreq=1):
    return dict(name=name, kind=kind, nx=nx, ny=ny, nz=nz, nrhs=nrhs, f=f, px=parts[0], py=parts[1], pz=parts[2],
                overlap=overlap, coarse=coarse, inner=inner, prec=prec, model=model, q=q, restart=restart,
                flexible=flexible, nfreq=nfreq)


def listed():
    return [
        # one wavefield on the smallest grid (a residual check, a time-slice product): latency
        _stencil("stencil_48_c64_r1", 48, 48, 48, 1, "fp32", f=3.0),
        # the operator of the mixed-precision solver at the headline size: 16 sources on 112^3
        _stencil("stencil_112_c64_r16", 112, 112, 112, 16, "fp32"),
        # the same for the attenuating survey: complex k^2, 128 sources, the largest batch of one call
        _stencil("stencil_160x160x80_q_c64_r128", 160, 160, 80, 128, "fp32", q=100, f=4.0),
        # a cut-out of a model: odd sizes, absorbing top, a source count that is no multiple of 16
        _stencil("stencil_101x93x77_c64_r10", 101, 93, 77, 10, "fp32", model="layered", top=1),
        # the FP64 operator: true residuals of a 16-source solve
        _stencil("stencil_112_c128_r16", 112, 112, 112, 16, "fp64"),
        # the FP64 two-level preconditioner on its own (a program that brings its own Krylov method)
        _solver("precond_48x44x40_fp64_r4", "precond", 48, 44, 40, 4, 4.0, (2, 2, 2), 2, 4, 0, "fp64", "layered"),
        # the plain method in FP64, one source, one level, GMRES(30): set-up and solve of a new small model
        _solver("new_48_plain_fp64_r1", "new", 48, 48, 48, 1, 3.0, (2, 2, 2), 2, 0, 0, "fp64", flexible=False),
        # the headline: 16 sources on 112^3, TF32 factors resident, FGMRES(30) to 1e-6
        _solver("solve_112_tf32_r16", "solve", 112, 112, 112, 16, 5.0, (4, 4, 4), 2, 4, 0, "tf32"),
        # the attenuating survey: 128 sources in one batch, planes of about 36 x 36 nodes
        _solver("solve_96x96x64_q_tf32_r128", "solve", 96, 96, 64, 128, 4.0, (3, 3, 2), 2, 4, 0, "tf32", q=100),
        # folded and faulted layers, BF16 factors, the coarse problem solved inexactly (10 inner iterations)
        _solver("solve_fold_128x128x64_bf16_r32", "solve", 128, 128, 64, 32, 5.0, (6, 6, 3), 3, 4, 10, "bf16", "fold"),
        # two neighbouring frequencies of one model, set-up included, the second started from the first
        _solver("sweep_96_tf32_r8", "new", 96, 96, 96, 8, 4.9, (4, 4, 4), 2, 4, 0, "tf32", nfreq=2),
        # a request of the service on a model it has not seen: boxes of about 24 nodes, FGMRES(15), inner iterations
        _solver("request_80_tf32_r4", "new", 80, 80, 80, 4, 4.0, (3, 3, 3), 2, 4, 10, "tf32", "layered", restart=15),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _columns(rng, most):
    """A source count up to `most`: over the logarithm, odd ones among them."""
    return max(1, min(most, _log(rng, 1, max(1, most))))


def draw(rng):
    model = rng.choice(("gradient", "layered", "fold"))
    q = rng.choice((0, 0, 100))
    f = round(rng.uniform(2.0, 6.0), 2)
    kind = rng.choice(("stencil", "stencil", "precond", "solve", "solve", "new"))
    if kind == "stencil":
        prec = rng.choice(("fp32", "fp32", "fp64"))
        nx, ny, nz = _log(rng, 32, 200), _log(rng, 32, 200), _log(rng, 32, 128)
        most = max(1, min(128, (22_000_000 if prec == "fp64" else 250_000_000) // (nx * ny * nz)))
        nrhs = rng.choice((_columns(rng, most), _columns(rng, most), max(1, most // 16 * 16)))
        c = _stencil("", nx, ny, nz, nrhs, prec, model, q, rng.choice((0, 0, 1)), f)
    elif kind == "precond" or (kind == "new" and rng.random() < 0.3):
        n = [_log(rng, 28, 48) for _ in range(3)]
        parts = [2 if v > 32 else rng.choice((1, 2)) for v in n]
        parts[rng.randrange(2)] = 2
        c = _solver("", kind, *n, _columns(rng, 8 if kind == "precond" else 2), f, parts, rng.choice((1, 2, 3)),
                    rng.choice((0, 4)), 0, "fp64", model, q, flexible=rng.choice((True, False)))
    else:
        n = [_log(rng, 44, 100) for _ in range(3)]
        parts = [max(2, round(v / rng.uniform(22.0, 30.0))) for v in n]
        cells = n[0] * n[1] * n[2]
        inner = rng.choice((0, 10))
        nrhs = _columns(rng, min(64, max(1, (20_000_000 if kind == "solve" else 8_000_000) // cells)))
        c = _solver("", kind, *n, nrhs, f, parts, rng.choice((2, 2, 3)), 4, inner,
                    rng.choice(("tf32", "tf32", "bf16", "fp32")), model, q, rng.choice((15, 30)))
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs


def _generator(seed):
    return np.random.default_rng([2103, int(seed)])


def _velocity(case, rng):
    """complex128 [nz, ny, nx] on the GPU: wave speeds of the case's model, made from rng."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    z = (torch.arange(nz, device="cuda", dtype=torch.float64) + 1) * H
    if case["model"] == "gradient":
        c = (rng.uniform(1450.0, 1550.0) + rng.uniform(0.55, 0.65) * z)[:, None, None].expand(nz, ny, nx)
    else:
        layers = int(rng.integers(4, 8))
        tops = torch.tensor(np.sort(rng.uniform(0.1, 0.9, layers - 1)) * nz * H, device="cuda")
        speeds = torch.tensor(np.sort(rng.uniform(1500.0, 4500.0, layers)), device="cuda")
        depth = z[:, None, None].expand(nz, ny, nx)
        if case["model"] == "fold":
            x = (torch.arange(nx, device="cuda", dtype=torch.float64) * H)[None, None, :]
            y = (torch.arange(ny, device="cuda", dtype=torch.float64) * H)[None, :, None]
            lx, ly = rng.uniform(1500.0, 4000.0, 2)
            depth = depth - rng.uniform(40.0, 120.0) * torch.sin(2 * math.pi * x / lx) * torch.cos(2 * math.pi * y / ly)
        c = speeds[torch.bucketize(depth.contiguous(), tops)]
        if case["model"] == "fold":
            side = (x - rng.uniform(0.3, 0.7) * nx * H) + rng.uniform(0.5, 1.5) * (z[:, None, None] - 0.5 * nz * H) + 0 * y
            c = torch.where(side > 0, c * 1.15, c)
    c = c.to(torch.complex128)
    return (c * (1.0 - 0.5j / case["q"]) if case["q"] else c).contiguous()


def _field(case, rng, dtype):
    """Random wavefields [nz, ny, nx, nrhs] on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 31)))
    return torch.randn((case["nz"], case["ny"], case["nx"], case["nrhs"]), generator=g, device="cuda", dtype=dtype)


def _sources(case, rng):
    """complex128 [nz, ny, nx, nrhs]: one unit point source per column, inside the absorbing layers."""
    nx, ny, nz, n = case["nx"], case["ny"], case["nz"], case["nrhs"]
    b = torch.zeros((nz, ny, nx, n), dtype=torch.complex128, device="cuda")
    k, j, i = (torch.tensor(rng.integers(lo, hi, n), device="cuda")
               for lo, hi in ((2, min(8, nz - NPML)), (NPML, ny - NPML), (NPML, nx - NPML)))
    b[k, j, i, torch.arange(n, device="cuda")] = 1.0 / H ** 3
    return b


def _grid(case, c):
    return helm.Grid(helm.Context(0), case["nx"], case["ny"], case["nz"], H, case["f"], c, npml=NPML, pml_R=PML_R,
                     top_bc=helm.TOP_PML if case.get("top") else helm.TOP_DIRICHLET, weights=WEIGHTS)


def prepare(case, seed):
    rng = _generator(seed)
    c = _velocity(case, rng)
    s = {"case": case}
    if case["kind"] == "stencil":
        s["u"] = _field(case, rng, torch.complex128 if case["prec"] == "fp64" else torch.complex64)
        s["grid"] = _grid(case, c)
        return s
    if case["kind"] == "new":   # a model that has not been seen: wave speeds and sources only
        s["c"], s["b"], s["ctx"] = c, _sources(case, rng), helm.Context(0)
        return s
    s["b"] = _field(case, rng, torch.complex128) if case["kind"] == "precond" else _sources(case, rng)
    s["oras"] = helm.Oras(_grid(case, c), (case["px"], case["py"], case["pz"]), case["overlap"],
                          coarse_ratio=case["coarse"], factor_prec=PREC[case["prec"]], coarse_iters=case["inner"])
    return s


# ------------------------------------------------------------------ one pass


def run(state):
    case = state["case"]
    if case["kind"] == "stencil":
        return state["grid"].apply(state["u"], prec=PREC[case["prec"]])
    if case["kind"] == "precond":
        return state["oras"].apply(state["b"])
    basis = helm.PREC_FP64 if case["prec"] == "fp64" else helm.PREC_FP32
    if case["kind"] == "solve":
        x, _ = state["oras"].solve(state["b"], tol=1e-6, restart=case["restart"], flexible=case["flexible"],
                                   basis_prec=basis)
    else:
        x, _, _ = helm.frequency_sweep(
            state["ctx"], case["nx"], case["ny"], case["nz"], H, [case["f"] + 0.1 * i for i in range(case["nfreq"])],
            state["c"], state["b"], (case["px"], case["py"], case["pz"]), case["overlap"], npml=NPML, pml_R=PML_R,
            weights=WEIGHTS, coarse_ratio=case["coarse"], factor_prec=PREC[case["prec"]], coarse_iters=case["inner"],
            tol=1e-6, restart=case["restart"], flexible=case["flexible"], basis_prec=basis)
    return x if case["prec"] == "fp64" else x.to(torch.complex64)


def _planes(case):
    """[(unknowns of one z-plane, planes)] of every box."""
    dims = []
    for a, p in (("nx", "px"), ("ny", "py"), ("nz", "pz")):
        n, parts = case[a], case[p]
        cuts = [t * n // parts for t in range(parts + 1)]
        dims.append([min(n, hi + case["overlap"]) - max(0, lo - case["overlap"]) for lo, hi in zip(cuts, cuts[1:])])
    return [(x * y, z) for x in dims[0] for y in dims[1] for z in dims[2]]


def work(case):
    n, nrhs = case["nx"] * case["ny"] * case["nz"], case["nrhs"]
    if case["kind"] == "stencil":
        # u in, y out, k^2 once; 27 complex multiply-adds per value
        return {"bytes": n * (2 * nrhs + 1) * (16 if case["prec"] == "fp64" else 8), "flops": 27 * 8 * n * nrhs}
    entries = sum(m * m * z for m, z in _planes(case))
    if case["kind"] == "new":
        # c and b in, x out, each frequency's plane inverses written and read; their inversion and one local solve
        return {"bytes": n * 16 * (1 + nrhs * (1 + case["nfreq"])) + 2 * case["nfreq"] * entries * ENTRY[case["prec"]],
                "flops": case["nfreq"] * (8 * sum(m ** 3 * z for m, z in _planes(case)) + 16 * entries * nrhs)}
    # b in, x out, every plane inverse at least once; forward and backward products of one local solve
    return {"bytes": n * 32 * nrhs + entries * ENTRY[case["prec"]], "flops": 16 * entries * nrhs}


# ------------------------------------------------------------------ the result in 64 bits


def _tables(case, c, f):
    """Per axis the coefficients [n, 3] of the stretched second difference of the absorbing layers."""
    omega, c_ref, depth = 2 * math.pi * f, float(c.real.max()), NPML * H
    out = []
    for a, n in enumerate((case["nx"], case["ny"], case["nz"])):
        def xi(s):
            low = (NPML - s).clip(0) if a < 2 or case.get("top") else 0 * s
            d = np.maximum(low, (s - (n - 1 - NPML)).clip(0)) * H
            return 1 + 1j * (1.5 * c_ref / depth * math.log(1 / PML_R)) * (d / depth) ** 2 / omega
        node, half = xi(np.arange(n) * 1.0), xi(np.arange(n + 1) - 0.5)
        cm, cp = 1 / (node * half[:-1]), 1 / (node * half[1:])
        out.append(torch.tensor(np.stack([cm, -(cm + cp), cp], 1), device="cuda"))
    return out


def _second_difference(u, axis, t):
    """t[i, 0] u[i - 1] + t[i, 1] u[i] + t[i, 2] u[i + 1] along an axis, zero past both ends."""
    n = u.shape[axis]
    shape = [1] * u.dim()
    shape[axis] = n
    t = [t[:, d].reshape(shape) for d in range(3)]
    y = t[1] * u
    y.narrow(axis, 1, n - 1).add_(t[0].narrow(axis, 1, n - 1) * u.narrow(axis, 0, n - 1))
    y.narrow(axis, 0, n - 1).add_(t[2].narrow(axis, 0, n - 1) * u.narrow(axis, 1, n - 1))
    return y


def _plain(n):
    return torch.tensor([1.0, -2.0, 1.0], dtype=torch.complex128, device="cuda").expand(n, 3)


def _coefficients():
    _, w2, w3, m1, m2, m3, m4 = WEIGHTS
    return w2 / 6 + w3 / 2, w3 / 4, m1 + 6 * m2 + 12 * m3 + 8 * m4, m2 + 4 * m3 + 4 * m4, m3 + 2 * m4, m4


def _operator(case, c, f, u):
    """The 27-point operator in 64 bits: h^-2 [sum D + a2 sum DD + a3 DDD] u + [m0 + m1 sum P + m2 sum PP + m3 PPP] k^2 u."""
    a2, a3, m0, m1, m2, m3 = _coefficients()

    def product(w, tabs, k0, k1, k2, k3):
        x = _second_difference(w, 2, tabs[0])
        y = _second_difference(w, 1, tabs[1])
        xy = _second_difference(x, 1, tabs[1])
        s = x.add_(y)
        out = k0 * w + k1 * s + k2 * xy
        return out.add_(_second_difference(k1 * w + k2 * s + k3 * xy, 0, tabs[2]))

    k2c = ((2 * math.pi * f / c) ** 2)[..., None]
    lap = product(u, _tables(case, c, f), 0.0, 1.0, a2, a3)
    return lap.div_(H * H).add_(product(k2c * u, [_plain(n) for n in (case["nx"], case["ny"], case["nz"])], m0, m1, m2, m3))


def _direct(case, c, f, b):
    """A x = b by elimination of the z-planes (dense blocks)."""
    a2, a3, m0, m1, m2, m3 = _coefficients()
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    m = nx * ny
    tx, ty, tz = _tables(case, c, f)
    eye = torch.eye(m, dtype=torch.complex128, device="cuda").reshape(ny, nx, m)

    def blocks(x, y, k0, k1, k2, k3):
        dx, dy = _second_difference(eye, 1, x), _second_difference(eye, 0, y)
        dxy, s = _second_difference(dx, 0, y), dx + dy
        return [(p * eye + q * s + r * dxy).reshape(m, m) for p, q, r in ((k0, k1, k2), (k1, k2, k3))]

    s0, s1 = blocks(tx, ty, 0.0, 1.0, a2, a3)
    t0, t1 = blocks(_plain(nx), _plain(ny), m0, m1, m2, m3)
    k2c = ((2 * math.pi * f / c) ** 2).reshape(nz, m)

    def block(k, d):
        p = -2.0 if d == 0 else 1.0
        a = (tz[k, d + 1] * s1 + (s0 if d == 0 else 0)) / (H * H)
        return a + (p * t1 + (t0 if d == 0 else 0)) * k2c[k + d][None, :]

    b = b.reshape(nz, m, -1)
    e, y = [], []
    for k in range(nz):
        s, r = block(k, 0), b[k]
        if k:
            low = block(k, -1)
            s, r = s - low @ e[-1], r - low @ y[-1]
        up = block(k, 1) if k + 1 < nz else s.new_zeros((m, 0))
        z = torch.linalg.solve(s, torch.cat([up, r], 1))
        e.append(z[:, :up.shape[1]].contiguous())
        y.append(z[:, up.shape[1]:].contiguous())
    for k in range(nz - 2, -1, -1):
        y[k] = y[k] - e[k] @ y[k + 1]
    return torch.stack(y).reshape(nz, ny, nx, -1)


def exact(case, seed):
    rng = _generator(seed)
    c = _velocity(case, rng)
    if case["kind"] == "stencil":
        u = _field(case, rng, torch.complex128 if case["prec"] == "fp64" else torch.complex64)
        parts = [_operator(case, c, case["f"], p.to(torch.complex128)) for p in u.split(16, dim=3)]
        return torch.cat(parts, 3)
    # the tolerance, not the arithmetic, bounds a mixed solve; the dense elimination is quick on small grids only
    if case["kind"] != "new" or case["prec"] != "fp64" or case["nfreq"] != 1 or case["nx"] * case["ny"] > 2400:
        return None
    return _direct(case, c, case["f"], _sources(case, rng))[None]
