"""Face coefficients near and past the ends of the binary64 range: spacings and densities that the
seeded quotient takes one by one, whose quotient it does not."""
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
