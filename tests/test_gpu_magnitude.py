"""Right sides of any magnitude: what a solve holds in FP32 (norms, inner variables, the spectral passes)
is scaled by powers of two where it would leave the FP32 range, so the relative residual that the library
reports is the one of the pressure, and a scaled right side gives the scaled pressure."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1601_05448_gb300 as vdp  # noqa: E402
import vdp_inputs as V  # noqa: E402

DEV = "cuda:0"
FIXED = {"method": vdp.VDP_METHOD_FIXED_POINT}
SPECTRAL = {"precond": vdp.VDP_PRECOND_SPECTRAL}
# 2^-200 .. 2^200; 2^-83 is 1e-25, 2^-50 1e-15, 2^64 2e19, 2^67 1.5e20, 2^80 1.2e24
POWERS = (-200, -100, -83, -63, -50, -31, 41, 64, 67, 80, 200)


@pytest.mark.parametrize("precision,opts", [("mixed", {}), ("mixed", FIXED), ("mixed", SPECTRAL), ("fp64", FIXED),
                                            ("fp64", SPECTRAL)], ids=str)
@pytest.mark.parametrize("L", [1.0, 1e-8])
def test_pressure_scales_with_the_right_side(precision, opts, L):
    prob = V.smooth_problem((32, 32, 48), seed=61)
    nz, ny, nx = prob.shape
    f = torch.from_numpy(prob.f).to(DEV)
    f -= f.mean()
    with vdp.Solver(nx, ny, nz, L, precision=precision, **opts) as s:
        s.set_density(torch.from_numpy(prob.rho).to(DEV))
        one, p, a = (torch.empty_like(f) for _ in range(3))
        st1 = s.solve(f, one, 1e-9)
        for k in POWERS:
            # a power of two rounds nothing anywhere: the same pressure times it, bit for bit, from the
            # same iterations, but for terms that FP32 flushed to zero without the scaling
            st = s.solve(f * 2.0 ** k, p, 1e-9)
            assert (st.iters, st.outer_iters) == (st1.iters, st1.outer_iters)
            assert float((p * 2.0 ** -k - one).norm() / one.norm()) <= 1e-12
            s.apply(p * 2.0 ** -k, a)
            assert float((f - a).norm() / f.norm()) <= 1.01e-9  # 1 %: the check's own rounding


@pytest.mark.parametrize("precision,opts", [("mixed", FIXED), ("fp64", FIXED), ("fp64", SPECTRAL)], ids=str)
@pytest.mark.parametrize("k", [-90, 70])
def test_initial_guess_and_launches(precision, opts, k):
    """The same from an initial guess, and in the separate launches."""
    prob = V.smooth_problem((32, 48, 32), seed=62)
    nz, ny, nx = prob.shape
    f = torch.from_numpy(prob.f).to(DEV) * 2.0 ** k
    f -= f.mean()
    out = []
    for steps in (0, 16):
        with vdp.Solver(nx, ny, nz, prob.L, precision=precision, use_guess=1, steps_per_sync=steps, **opts) as s:
            s.set_density(torch.from_numpy(prob.rho).to(DEV))
            p = 1e-3 * f
            s.solve(f, p, 1e-9)
            a = torch.empty_like(p)
            s.apply(p, a)
            assert float(((f - a) * 2.0 ** -k).norm() / (f * 2.0 ** -k).norm()) <= 1.01e-9
            out.append(p)
    assert torch.equal(*out)
