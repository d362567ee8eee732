"""Densities and boxes at the ends of what is accepted: face coefficients near and past the ends of the
binary64 range (spacings and densities that the seeded quotient takes one by one, whose quotient it does
not), and densities whose cells the FP32 density of the FP64 solves does not hold together."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1601_05448_gb300 as vdp  # noqa: E402

DEV = "cuda:0"


# box length, density, and the binary exponent of 2 / (rho_l + rho_r) / h^2 at unit density (h = L / 8)
@pytest.mark.parametrize("L,scale", [
    (1e90, 1e120), (1e90, 1e124), (1e90, 1e130), (1e90, 1e135), (1e100, 1e150), (1e115, 1e70), (1e115, 1e100),
    (1e-90, 1e-120), (1e-90, 1e-124), (1e-100, 1e-102), (1e-115, 1e-70), (1e-115, 1e-72)])
def test_operator_near_the_ends_of_the_range(L, scale):
    shape = (8, 8, 8)
    rng = np.random.default_rng(5)
    rho = scale * np.exp(rng.uniform(-1.0, 1.0, shape))
    p = rng.standard_normal(shape)
    out = torch.empty(shape, dtype=torch.float64, device=DEV)
    with vdp.Solver(8, 8, 8, L) as s:
        s.set_density(torch.from_numpy(rho).to(DEV))
        s.apply(torch.from_numpy(p).to(DEV), out)
    # the flux form in extended precision, which holds every coefficient
    r, q, h2 = rho.astype(np.longdouble), p.astype(np.longdouble), (np.longdouble(L) / 8) ** 2
    ref, mag = np.zeros_like(q), np.zeros_like(q)
    for axis in range(3):
        b = 2 / (np.roll(r, 1, axis) + r) / h2
        flux = b * (q - np.roll(q, 1, axis))
        ref += np.roll(flux, -1, axis) - flux
        size = b * (abs(q) + abs(np.roll(q, 1, axis)))
        mag += np.roll(size, -1, axis) + size
    # coefficients within 3 roundings, six products and eleven additions of the magnitudes; below the
    # normal range a rounding is half of 2^-1074, six coefficients' times |p| differences below 8
    assert np.all(abs(out.cpu().numpy() - ref) <= 20 * 2.0 ** -53 * mag + np.longdouble(2.0) ** -1074 * 64)


SPECTRAL = {"precond": vdp.VDP_PRECOND_SPECTRAL}


def relative_residual(s, f, p):
    a = torch.empty_like(p)
    s.apply(p, a)
    return float((f - a).norm() / f.norm())


# factor of one cell's density, and the cell: the first one sets the scale of the FP32 density.  A light
# cell is one more isolated eigenvalue of the preconditioned operator, so CG takes a few more iterations
@pytest.mark.parametrize("cell", [(0, 0, 0), (31, 17, 5)])
@pytest.mark.parametrize("factor", [1e-12, 1e-17, 1e-18, 1e-19, 1e-30, 1e-36, 1e-40, 1e-60, 1e-300])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_one_cell_of_another_density(factor, cell, precision):
    rng = np.random.default_rng(6)
    base = np.exp(rng.uniform(-0.5, 0.5, (32, 32, 32)))
    rho = base.copy()
    rho[cell] *= factor
    f = torch.from_numpy(rng.standard_normal(rho.shape)).to(DEV)
    f -= f.mean()
    p = torch.empty_like(f)
    with vdp.Solver(32, 32, 32, 1.0, precision=precision, **SPECTRAL) as s:
        for r in (rho, base, rho):  # and from one form to the other
            s.set_density(torch.from_numpy(r).to(DEV))
            st = s.solve(f, p, 1e-8)
            # 1 %: the check's own rounding, here of coefficients near 2e3 in all but one cell
            assert st.iters < 40 and relative_residual(s, f, p) <= 1.01e-8
