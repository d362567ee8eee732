"""What the library's users have it do, as timed cases.

The flow changes the density every substep, so nearly every pass is one substep's share of the
work: the new density is set (face coefficients, scalings, weights) and the pressure equation
div((1/rho) grad p) = f is solved to its tolerance on a context that the program keeps.  Grid
sizes, tolerances, precisions and methods are those of the library's own workloads (32^3 to 512^3
boxes, the 256 x 128 x 128 duct, grids of uneven sizes in one batch, request sizes of the serving
loop) or odd sizes of the same range.

Inputs follow the workloads' recipe, made on the GPU from the seed: a gas of temperature T = a few
random Fourier modes plus Gaussian hot spots 1.5 cells wide, rho = 1 / T with the stated ratio of
the largest to the smallest density, and f = the discrete divergence of a random low-wavenumber
velocity field.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1601_05448_gb300 as vdp

TWO_PI = 2.0 * math.pi
FFT_SIZES = (32, 48, 64, 96, 128, 192, 256, 512)   # line lengths of the spectral passes
DUCT_X = (32, 48, 64, 96, 128, 256)                # duct rows: twice the length is transformed
DEFAULT_X = (16, 24, 32, 40, 48, 56, 64, 80, 96, 112)  # row lengths that FP64 sweeps take, any ny and nz
BATCH_SIZES = (64, 96, 128, 192)


def listed():
    return [
        # the smallest request of the serving loop: launches and host latency
        _step("step_32_mixed", (32, 32, 32), "mixed", "fixed", 1e-8, 4.0),
        # a small box of unequal sides, FP64 throughout
        _step("step_64x48x32_fp64", (64, 48, 32), "fp64", "fixed", 1e-10, 3.0),
        # the library's defaults (FP64, Jacobi CG) on a small grid with odd sides
        _step("default_40x37x29_fp64", (40, 37, 29), "fp64", "jacobi", 1e-10, 3.0),
        # ... and on a grid that neither the FFT lengths nor the coarsening cover
        _step("default_112x100x90_fp64", (112, 100, 90), "fp64", "jacobi", 1e-10, 4.0),
        # a middle request of the serving loop
        _step("step_96_mixed", (96, 96, 96), "mixed", "fixed", 1e-9, 6.0),
        # a strong density contrast, where the preconditioned iteration is the robust choice
        _step("cg_spectral_128_fp64", (128, 128, 128), "fp64", "spectral", 1e-10, 10.0),
        # a grid with no FFT length: the multigrid preconditioner
        _step("cg_multigrid_160_mixed", (160, 160, 160), "mixed", "mg", 1e-8, 4.0),
        # the inflow-outflow duct
        _step("duct_256x128x128_fp64", (256, 128, 128), "fp64", "fixed", 1e-10, 4.0, duct=True),
        # one whole projection substep, from the pressure of the substep before
        dict(_step("project_256_fp64", (256, 256, 256), "fp64", "fixed", 1e-10, 4.0), kind="project"),
        # the largest request of the serving loop
        _step("step_256_mixed", (256, 256, 256), "mixed", "fixed", 1e-8, 4.0),
        # the largest grid
        _step("step_512_mixed", (512, 512, 512), "mixed", "fixed", 1e-8, 7.6),
        # independent grids of uneven sizes advanced together
        {"name": "batch_8_mixed", "kind": "batch", "members": 8, "choice": 1, "tol": 1e-8},
    ]


def _step(name, shape, precision, method, tol, ratio, duct=False):
    nx, ny, nz = shape
    return {"name": name, "kind": "step", "nx": nx, "ny": ny, "nz": nz, "precision": precision,
            "method": method, "tol": tol, "ratio": ratio, "duct": duct}


def draw(rng):
    kind = rng.choice(("fixed", "fixed", "fixed", "spectral", "mg", "jacobi", "duct", "project", "batch"))
    if kind == "batch":
        return {"kind": "batch", "members": rng.randint(3, 8), "choice": rng.randrange(1 << 20),
                "tol": _log_uniform(rng, 1e-10, 1e-8)}
    precision = rng.choice(("mixed", "fp64"))
    tol = _log_uniform(rng, 1e-10, 1e-8)
    ratio = rng.uniform(2.0, 8.0 if kind in ("fixed", "duct", "project") else 10.0)
    if kind == "jacobi":
        precision, tol = "fp64", 1e-10
        nx = _nearest(_log_uniform(rng, 16, 112), DEFAULT_X)
        ny, nz = (round(_log_uniform(rng, 9, 100)) for _ in range(2))
    elif kind == "mg":
        k = rng.randint(3, 5)
        nx, ny, nz = (rng.choice((3, 4, 5, 6, 7)) * 2 ** k for _ in range(3))
    else:
        top = 512 if precision == "mixed" and kind == "fixed" else 256
        n = _log_uniform(rng, 32, top)
        nx, ny, nz = (_nearest(n * math.exp(rng.uniform(-0.4, 0.4)), FFT_SIZES) for _ in range(3))
        if kind == "duct":
            nx = _nearest(n, DUCT_X)
        while nx * ny * nz > (512 * 512 * 256 if top == 512 else 256 ** 3):
            nx, ny, nz = sorted((nx, ny, nz))
            nz = _nearest(0.6 * nz, FFT_SIZES)
        if kind == "duct" and nx not in DUCT_X:
            nx = 256
    c = _step("", (nx, ny, nz), precision, "fixed" if kind in ("duct", "project") else kind, tol,
              round(ratio, 3), kind == "duct")
    del c["name"]
    if kind == "project":
        c["kind"] = "project"
    return c


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _nearest(v, sizes):
    return min(sizes, key=lambda s: abs(math.log(s / v)))


# ---- inputs --------------------------------------------------------------------------------------

def _lengths(case):
    # the duct is longer in x, with cells of equal size; boxes are cubes
    if case.get("duct"):
        return (TWO_PI * case["nx"] / case["ny"], TWO_PI, TWO_PI * case["nz"] / case["ny"])
    return (TWO_PI, TWO_PI, TWO_PI)


def _modes(shape, kv, coefs, offset):
    """Re sum_m coefs[m] exp(2 pi i k_m . (index + offset) / n) on the (nz, ny, nx) grid."""
    nz, ny, nx = shape
    spec = torch.zeros(shape, dtype=torch.complex128, device="cuda")
    phase = np.exp(1j * TWO_PI * (kv @ (np.asarray(offset) / np.array([nx, ny, nz]))))
    at = [torch.from_numpy(kv[:, d] % n).cuda() for d, n in ((2, nz), (1, ny), (0, nx))]
    spec.index_put_(at, torch.from_numpy(coefs * phase).cuda(), accumulate=False)
    return torch.fft.ifftn(spec).real.mul(float(nx * ny * nz))


def _wavevectors(shape, kmax):
    nz, ny, nx = shape
    r = np.arange(-kmax, kmax + 1)
    k = np.stack(np.meshgrid(r, r, r, indexing="ij"), axis=-1).reshape(-1, 3)
    n2 = (k * k).sum(axis=1)
    # half the modes (the real part supplies the other half), below the grid's Nyquist limit
    keep = (n2 >= 1) & (n2 <= kmax * kmax) & (2 * np.abs(k) < np.array([nx, ny, nz])).all(axis=1)
    k = k[keep]
    first = (k[:, 0] > 0) | ((k[:, 0] == 0) & ((k[:, 1] > 0) | ((k[:, 1] == 0) & (k[:, 2] > 0))))
    return k[first]


def _density(shape, ratio, rng):
    nz, ny, nx = shape
    kv = _wavevectors(shape, 8)
    kv = kv[rng.choice(len(kv), size=min(16, len(kv)), replace=False)]
    amp = rng.uniform(0.5, 1.0, len(kv)) * np.exp(1j * rng.uniform(0.0, TWO_PI, len(kv)))
    F = _modes(shape, kv, amp, (0.5, 0.5, 0.5))
    F *= 0.3 / F.abs().max()
    # hot spots: amplitudes (multiples of 2^-10, so that sums are exact in any order) on cells,
    # convolved with a Gaussian of 1.5 cells
    n = nx * ny * nz
    spots = max(8, round(20000 * n / 256 ** 3))
    cell = torch.from_numpy(rng.integers(0, n, spots)).cuda()
    a = torch.from_numpy(rng.integers(512, 2049, spots) / 1024.0).cuda()
    H = torch.zeros(n, dtype=torch.float64, device="cuda").index_put_((cell,), a, accumulate=True).view(shape)
    hat = torch.fft.rfftn(H)
    for axis, m in enumerate(shape):
        k = torch.arange(hat.shape[axis], dtype=torch.float64, device="cuda")
        k = torch.minimum(k, m - k) * (TWO_PI / m)
        g = torch.exp(-0.5 * (1.5 * k) ** 2) * (1.5 * math.sqrt(TWO_PI))
        hat *= g.view([-1 if d == axis else 1 for d in range(3)])
    g = F + torch.fft.irfftn(hat, s=shape)
    lo, hi = g.min(), g.max()
    return 1.0 / (1.0 + (ratio - 1.0) * ((g - lo) / (hi - lo)))


def _velocity(shape, d, rng):
    """Random velocity along d (0: x) on the low d-faces: modes |k| <= 4, zero mean, unit variance."""
    kv = _wavevectors(shape, 4)
    if not len(kv):
        kv = np.array([[1, 0, 0]])
    offset = [0.5, 0.5, 0.5]
    offset[d] = 0.0
    u = _modes(shape, kv, rng.standard_normal(len(kv)) + 1j * rng.standard_normal(len(kv)), offset)
    u -= u.mean()
    return u / u.std()


def _problem(nx, ny, nz, lengths, ratio, rng):
    shape = (nz, ny, nx)
    rho = _density(shape, ratio, rng)
    f = torch.zeros(shape, dtype=torch.float64, device="cuda")
    for d, (n, length) in enumerate(zip((nx, ny, nz), lengths)):
        u = _velocity(shape, d, rng)
        f += (torch.roll(u, -1, 2 - d) - u) * (n / length)
    return rho, f


def _members(case):
    rng = np.random.default_rng(case["choice"])
    return [(int(rng.choice(BATCH_SIZES)), float(rng.uniform(2.0, 10.0))) for _ in range(case["members"])]


def _inputs(case, seed):
    rng = np.random.default_rng(seed)
    if case["kind"] == "batch":
        return [_problem(n, n, n, (TWO_PI,) * 3, ratio, rng) for n, ratio in _members(case)]
    dims = (case["nx"], case["ny"], case["nz"])
    if case["kind"] == "step":
        return _problem(*dims, _lengths(case), case["ratio"], rng)
    # a projection substep: momenta on the faces, RHS^div on the cells
    shape = dims[::-1]
    rho = _density(shape, case["ratio"], rng)
    m = [_velocity(shape, d, rng) + rng.uniform(-1.0, 1.0) for d in range(3)]
    div = 0.1 + 0.05 * _velocity(shape, 0, rng)
    return rho, m, div


PRESSURE_COEFFICIENT = 0.5 * 1e-3  # C_pre[0] dt


def _solver(case):
    opts = {"fixed": {"method": vdp.VDP_METHOD_FIXED_POINT},
            "spectral": {"precond": vdp.VDP_PRECOND_SPECTRAL},
            "mg": {"precond": vdp.VDP_PRECOND_MG},
            "jacobi": {}}[case["method"]]
    if case.get("duct"):
        opts = dict(opts, lengths=_lengths(case), bc_x=vdp.VDP_BC_DUCT)
    return vdp.Solver(case["nx"], case["ny"], case["nz"], TWO_PI, precision=case["precision"], **opts)


def prepare(case, seed):
    """The context (or batch and contexts) and this substep's fields, all on the GPU."""
    if case["kind"] == "batch":
        problems = _inputs(case, seed)
        solvers = [vdp.Solver(n, n, n, TWO_PI, precision="mixed", method=vdp.VDP_METHOD_FIXED_POINT)
                   for n, _ in _members(case)]
        return {"case": case, "batch": vdp.Batch("mixed", persistent=False), "solvers": solvers,
                "problems": problems, "p": [torch.empty_like(f) for _, f in problems]}
    solver = _solver(case)
    if case["kind"] == "step":
        rho, f = _inputs(case, seed)
        return {"case": case, "solver": solver, "rho": rho, "f": f, "p": torch.empty_like(f)}
    rho, m, div = _inputs(case, seed)
    # the substep before: its pressure is this one's initial guess.  Its fields are this one's,
    # shifted by one cell along x, with slightly weaker momenta
    before = torch.empty_like(div)
    solver.set_density(torch.roll(rho, 1, 2).contiguous())
    solver.project([torch.roll(a, 1, 2).mul_(0.98) for a in m], torch.roll(div, 1, 2).contiguous(),
                   PRESSURE_COEFFICIENT, case["tol"], before)
    solver.set_options(use_guess=1)
    return {"case": case, "solver": solver, "rho": rho, "m": m, "div": div, "before": before,
            "p": torch.empty_like(div), "m_work": [torch.empty_like(a) for a in m]}


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        batch = state["batch"]
        for s, (rho, f), p in zip(state["solvers"], state["problems"], state["p"]):
            s.set_density(rho)
            batch.add(s, f, p, case["tol"])
        batch.run_to_completion()
        for s in state["solvers"]:
            batch.remove(s)
        return state["p"]
    solver, p = state["solver"], state["p"]
    if case["kind"] == "step":
        solver.set_density(state["rho"])
        solver.solve(state["f"], p, case["tol"])
        return p
    # the momentum predictor leaves new momenta and the last pressure in the program's arrays
    for work, a in zip(state["m_work"], state["m"]):
        work.copy_(a)
    p.copy_(state["before"])
    solver.set_density(state["rho"])
    solver.project(state["m_work"], state["div"], PRESSURE_COEFFICIENT, case["tol"], p)
    return {"p": p, "mx": state["m_work"][0], "my": state["m_work"][1], "mz": state["m_work"][2]}


def work(case):
    """Fields read and written once (FP64); arithmetic of the iterations that the method needs for
    the tolerance: a 7-point operator per iteration and, where the method has one, the constant-
    coefficient inverse (two real transforms) or a V-cycle."""
    if case["kind"] == "batch":
        one = [_solve_flops(n ** 3, "fixed", 0.5 * (2 + r), case["tol"]) for n, r in _members(case)]
        return {"bytes": 24.0 * sum(n ** 3 for n, _ in _members(case)), "flops": float(sum(one))}
    n = case["nx"] * case["ny"] * case["nz"]
    fields = 3 if case["kind"] == "step" else 10  # rho, f, p; or rho, m in and out, RHS^div, p in and out
    return {"bytes": 8.0 * fields * n, "flops": _solve_flops(n, case["method"], case["ratio"], case["tol"])}


def _solve_flops(n, method, ratio, tol):
    digits = math.log(1.0 / tol)
    transform = 5.0 * n * math.log2(n)
    r = math.sqrt(ratio)
    if method == "fixed":  # the error falls by about 0.18 an iteration
        return digits / 1.7 * (transform + 16.0 * n)
    if method == "spectral":
        return digits / math.log((r + 1) / (r - 1)) * (transform + 26.0 * n)
    if method == "mg":
        return digits / 1.4 * (60.0 + 26.0) * n
    return digits * 0.2 * n ** (1.0 / 3.0) * r * 26.0 * n


# ---- the same results in 64 bits, by torch alone -------------------------------------------------------

def exact(case, seed):
    if case["kind"] == "batch":
        return [_pressure(rho, f, (TWO_PI,) * 3, False) for rho, f in _inputs(case, seed)]
    if case["kind"] == "step":
        rho, f = _inputs(case, seed)
        return _pressure(rho, f, _lengths(case), case["duct"])
    rho, m, div = _inputs(case, seed)
    c, h = PRESSURE_COEFFICIENT, [TWO_PI / n for n in (case["nx"], case["ny"], case["nz"])]
    f = -div
    for d, a in enumerate(m):
        u = a / (0.5 * (rho + torch.roll(rho, 1, 2 - d)))
        f += (torch.roll(u, -1, 2 - d) - u) / h[d]
    p = _pressure(rho, f / c, _lengths(case), False)
    out = {"p": p}
    for d, a in enumerate(m):
        out["m" + "xyz"[d]] = a - c * (p - torch.roll(p, 1, 2 - d)) / h[d]
    return out


def _pressure(rho, f, lengths, duct):
    """CG on the 7-point operator, preconditioned by the FFT inverse of the constant one."""
    nz, ny, nx = rho.shape
    h = [length / n for length, n in zip(lengths, (nx, ny, nz))]
    b = [2.0 / (rho + torch.roll(rho, 1, 2 - d)) / h[d] ** 2 for d in range(3)]
    if duct:
        b[0][:, :, 0] = 0.0

    def minus_a(p):
        out = torch.zeros_like(p)
        for d in range(3):
            flux = b[d] * (p - torch.roll(p, 1, 2 - d))
            out += flux
            out -= torch.roll(flux, -1, 2 - d)
        return out

    nxt = 2 * nx if duct else nx
    lam = 0.0
    for axis, (n, hd, count) in enumerate(((nz, h[2], nz), (ny, h[1], ny), (nxt, h[0], nxt // 2 + 1))):
        k = torch.arange(count, dtype=torch.float64, device="cuda")
        e = 4.0 * torch.sin(math.pi * k / n) ** 2 / hd ** 2
        lam = lam + e.view([-1 if d == axis else 1 for d in range(3)])
    lam[0, 0, 0] = 1.0

    def inverse(r):
        if duct:
            r = torch.cat((r, torch.flip(r, (2,))), 2)
        hat = torch.fft.rfftn(r) / lam
        hat[0, 0, 0] = 0.0
        return torch.fft.irfftn(hat, s=(nz, ny, nxt))[:, :, :nx]

    g = f.mean() - f  # minus_a(p) = g
    norm = g.norm()
    p = torch.zeros_like(g)
    r, q, rz = g.clone(), None, None
    for _ in range(100):
        z = inverse(r)
        new = (r * z).sum()
        q = z.clone() if q is None else z + (new / rz) * q
        rz = new
        aq = minus_a(q)
        alpha = rz / (q * aq).sum()
        p += alpha * q
        r -= alpha * aq
        if float(r.norm() / norm) < 2e-14:
            break
    return p - p.mean()
