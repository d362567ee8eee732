"""The coefficients that vdp_set_density builds, through vdp_apply: a seeded reciprocal replaces
the FP64 division over the middle of the binary64 range and the division itself runs outside it,
so densities on both sides of that line are compared with the flux form evaluated by numpy."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1601_05448_gb300 as vdp  # noqa: E402

DEV = "cuda:0"


def flux_form(rho, p, L):
    """A p and the sum of the magnitudes of its terms, in numpy's extended precision."""
    rho, p = rho.astype(np.longdouble), p.astype(np.longdouble)
    out, mag = np.zeros_like(p), np.zeros_like(p)
    for axis, n in zip((2, 1, 0), rho.shape[::-1]):
        h = np.longdouble(L) / n
        b = 2 / (np.roll(rho, 1, axis) + rho) / (h * h)
        d = b * (p - np.roll(p, 1, axis))
        out += np.roll(d, -1, axis) - d
        m = b * (abs(p) + abs(np.roll(p, 1, axis)))
        mag += np.roll(m, -1, axis) + m
    return out, mag


# (nx, ny, nz): a single pair of rows, odd sides, more than one block per plane; densities scaled
# into the seeded range (1, 1e-150, 1e120) and out of it on both sides (the range is 2^-822 .. 2^822)
@pytest.mark.parametrize("shape", [(8, 1, 1), (8, 3, 5), (40, 37, 3), (512, 4, 2)])
@pytest.mark.parametrize("scale", [1.0, 1e-150, 1e120, 1e-260, 1e260])
def test_operator_of_any_density(shape, scale):
    nx, ny, nz = shape
    rng = np.random.default_rng(nx + 10 * ny + 100 * nz)
    rho = scale * np.exp(rng.uniform(-3.0, 3.0, (nz, ny, nx)))
    p = rng.standard_normal((nz, ny, nx))
    out = torch.empty(p.shape, dtype=torch.float64, device=DEV)
    # one element further than the 16-byte boundary: the set-up takes any 8-byte aligned rho
    pad = torch.empty(rho.size + 1, dtype=torch.float64, device=DEV)
    shifted = pad[1:].view(rho.shape)
    shifted.copy_(torch.from_numpy(rho))
    for r in (torch.from_numpy(rho).to(DEV), shifted):
        with vdp.Solver(nx, ny, nz, 2.0) as s:
            s.set_density(r)
            s.apply(torch.from_numpy(p).to(DEV), out)
        ref, mag = flux_form(rho, p, 2.0)
        # coefficients within 3 roundings, six products and eleven additions of the magnitudes
        assert np.all(abs(out.cpu().numpy() - ref) <= 20 * 2.0 ** -53 * mag)


def test_rejected_density_changes_nothing():
    rng = np.random.default_rng(3)
    rho = np.exp(rng.uniform(-1.0, 1.0, (32, 32, 32)))
    f = rng.standard_normal(rho.shape)
    f -= f.mean()
    f = torch.from_numpy(f).to(DEV)
    for opts in ({}, {"method": vdp.VDP_METHOD_FIXED_POINT}, {"precond": vdp.VDP_PRECOND_MG}):
        with vdp.Solver(32, 32, 32, 1.0, precision="mixed", **opts) as s:
            s.set_density(torch.from_numpy(rho).to(DEV))
            a, b = torch.empty_like(f), torch.empty_like(f)
            s.solve(f, a, 1e-9)
            for bad in (0.0, -1.0, np.nan, np.inf):
                broken = 2.0 * rho
                broken[31, 31, 31] = bad
                with pytest.raises(vdp.VdpError) as e:
                    s.set_density(torch.from_numpy(broken).to(DEV))
                assert e.value.status == vdp.VDP_EDENSITY
            s.solve(f, b, 1e-9)
        assert torch.equal(a, b)
