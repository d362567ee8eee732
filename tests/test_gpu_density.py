"""The density form of the inner iteration (face coefficients computed from the density in the
sweep): the returned pressure must meet the tolerance on the operator evaluated by numpy, on row
lengths from one warp to one row per block, rows that leave threads idle, unequal spacings, the
duct's end faces, and densities and boxes whose coefficients lie outside the FP32 range."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1601_05448_gb300 as vdp  # noqa: E402
import vdp_inputs as V  # noqa: E402

DEV = "cuda:0"
FIXED = {"method": vdp.VDP_METHOD_FIXED_POINT}
SPECTRAL = {"precond": vdp.VDP_PRECOND_SPECTRAL}


def residual(rho, f, p, lengths, duct):
    """||(f - <f>) - A p|| / ||f - <f>|| by the flux form."""
    r = f - f.mean()
    norm = np.linalg.norm(r)
    for axis, n, L in zip((2, 1, 0), rho.shape[::-1], lengths):
        h = L / n
        flux = 2.0 / (np.roll(rho, 1, axis) + rho) / h ** 2 * (p - np.roll(p, 1, axis))
        if duct and axis == 2:
            flux[:, :, 0] = 0.0
        r = r - (np.roll(flux, -1, axis) - flux)
    return np.linalg.norm(r) / norm


@pytest.mark.parametrize("opts", [FIXED, SPECTRAL], ids=["fixed", "spectral"])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("shape,lengths,duct,unit", [
    ((32, 32, 32), (1.0, 1.0, 1.0), False, 1.0), ((512, 32, 48), (4.0, 1.0, 1.0), False, 1.0),
    ((48, 96, 32), (1.0, 3.0, 0.5), False, 1.0), ((96, 48, 32), (3.0, 1.0, 1.0), True, 1.0),
    ((256, 32, 32), (2.0, 1.0, 1.0), True, 1.0), ((64, 32, 48), (1e-8, 1e-8, 1e-8), False, 1e-30),
    ((64, 32, 48), (1e8, 1e8, 1e8), False, 1e30)])
def test_density_form(shape, lengths, duct, unit, precision, opts):
    nx, ny, nz = shape
    rng = np.random.default_rng(nx + ny + nz)
    rho = unit * V.density_modes((nz, ny, nx), rng, amplitude=0.5)
    f = rng.standard_normal((nz, ny, nx)) + 0.3
    tol = 1e-9 if precision == "mixed" else 1e-10
    p = torch.empty(f.shape, dtype=torch.float64, device=DEV)
    with vdp.Solver(nx, ny, nz, lengths[1], precision=precision, lengths=lengths,
                    bc_x=vdp.VDP_BC_DUCT if duct else vdp.VDP_BC_PERIODIC, **opts) as s:
        s.set_density(torch.from_numpy(rho).to(DEV))
        fd = torch.from_numpy(f).to(DEV)
        st = s.solve(fd, p, tol)
        timed = torch.empty_like(p)
        s.solve_timed(fd, timed, tol)
    assert st.ok and torch.equal(p, timed)
    # the library's residual is evaluated on the same coefficients: 1 % for its own rounding
    assert residual(rho, f, p.cpu().numpy(), lengths, duct) <= 1.01 * tol


def test_method_chosen_after_the_density():
    """Spectral CG selected when the density is already set has no FP32 density and runs in the
    scaled form; setting the density again, or another precision, gives the same pressure."""
    prob = V.smooth_problem((32, 48, 64), seed=81)
    nz, ny, nx = prob.shape
    rho, f = torch.from_numpy(prob.rho).to(DEV), torch.from_numpy(prob.f).to(DEV)
    out = []
    with vdp.Solver(nx, ny, nz, prob.L, precision="mixed") as s:
        s.set_density(rho)
        s.set_options(**SPECTRAL)
        for change in (lambda: None, lambda: s.set_density(rho), lambda: s.set_options(precision="mixed_bf16"),
                       lambda: s.set_options(precision="mixed", **FIXED), lambda: s.set_options(precision="mixed_bf16"),
                       lambda: s.set_options(precision="fp64"),
                       lambda: s.set_options(precision="mixed", method=vdp.VDP_METHOD_CG, precond=vdp.VDP_PRECOND_MG),
                       lambda: s.set_options(precond=vdp.VDP_PRECOND_JACOBI)):
            change()
            p = torch.empty_like(f)
            assert s.solve(f, p, 1e-10).ok
            out.append(p)
    for p in out[1:]:  # two pressures whose residuals are 1e-10: the condition number of the
        # preconditioned operator is at most the density ratio (3), of L_h on this grid below 2e3
        assert float((p - out[0]).norm() / out[0].norm()) <= 2 * 3 * 2e3 * 1e-10
