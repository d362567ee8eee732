"""The resident solve (one cooperative launch) against the host-polled schedule of separate kernels:
the same units, sums and arithmetic, so the same bits, iteration and sweep counts -- on every line
length of the Y and Z passes, row lengths from 16 to 256 cells, odd sides and single planes, the
duct, an initial guess, and solves that stop at the iteration cap."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1601_05448_gb300 as vdp  # noqa: E402
import vdp_inputs as V  # noqa: E402

DEV = "cuda:0"
FIXED = {"method": vdp.VDP_METHOD_FIXED_POINT}
SPECTRAL = {"precond": vdp.VDP_PRECOND_SPECTRAL}


def both(shape, opts, precision, tol, duct=False, guess=False, max_iter=20000):
    nx, ny, nz = shape
    rng = np.random.default_rng(7 * nx + 3 * ny + nz)
    rho = torch.from_numpy(V.density_modes((nz, ny, nx), rng, amplitude=0.5)).to(DEV)
    f = torch.from_numpy(rng.standard_normal((nz, ny, nx))).to(DEV)
    start = torch.from_numpy(rng.standard_normal((nz, ny, nx))).to(DEV)
    out = []
    for steps in (0, 16):
        with vdp.Solver(nx, ny, nz, 1.0, precision=precision, lengths=(2.0, 1.0, 1.0), steps_per_sync=steps,
                        bc_x=vdp.VDP_BC_DUCT if duct else vdp.VDP_BC_PERIODIC, use_guess=int(guess),
                        max_iter=max_iter, **opts) as s:
            s.set_density(rho)
            p = start.clone()
            out.append((p, s.solve(f, p, tol, check=False)))
    (p, a), (q, b) = out
    assert a.launches == 2 and b.launches > 2
    assert torch.equal(p, q)
    assert (a.status, a.iters, a.outer_iters, a.sweeps, a.rel_res, a.rhs_mean) == \
        (b.status, b.iters, b.outer_iters, b.sweeps, b.rel_res, b.rhs_mean)
    return a


@pytest.mark.parametrize("opts", [FIXED, SPECTRAL], ids=["fixed", "spectral"])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("shape,duct", [((32, 32, 32), False), ((48, 96, 64), False), ((64, 128, 48), False),
                                        ((128, 32, 192), False), ((256, 48, 32), False), ((192, 32, 48), False),
                                        ((32, 256, 32), False), ((96, 32, 128), True), ((32, 64, 256), True)])
def test_spectral_solves_equal_the_launches(shape, duct, precision, opts):
    assert both(shape, opts, precision, 1e-9, duct).ok


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("shape", [(8, 1, 1), (16, 9, 1), (40, 37, 29), (24, 5, 100), (256, 20, 33), (112, 100, 90)])
def test_default_solves_equal_the_launches(shape, precision):
    both(shape, {}, precision, 1e-9 if precision == "mixed" else 1e-10)


def test_guess_and_iteration_cap():
    for opts in ({}, FIXED, SPECTRAL):
        both((32, 48, 32), opts, "fp64", 1e-10, guess=True)
        assert both((32, 48, 32), opts, "mixed", 1e-10, max_iter=3).status == vdp.VDP_ENOTCONV
