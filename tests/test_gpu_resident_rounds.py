"""What bounds a resident launch: rounds of the separate launches (residual, preconditioner, stencil, flat
sweep, each where the solve is in its phase).  So a batch's max_pairs means one iteration to every member,
and a solve ends by its own rules and not by the launch's bound."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1601_05448_gb300 as vdp  # noqa: E402
import vdp_inputs as V  # noqa: E402

DEV = "cuda:0"
FIXED = {"method": vdp.VDP_METHOD_FIXED_POINT}
SPECTRAL = {"precond": vdp.VDP_PRECOND_SPECTRAL}


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("opts", [FIXED, SPECTRAL], ids=["fixed", "spectral"])
@pytest.mark.parametrize("pairs", [1, 3])
def test_a_pair_is_a_round(opts, precision, pairs):
    prob = V.smooth_problem((32, 48, 32), seed=91)
    nz, ny, nx = prob.shape
    f = torch.from_numpy(prob.f).to(DEV)
    p = torch.empty_like(f)
    with vdp.Solver(nx, ny, nz, prob.L, precision=precision, **opts) as s, vdp.Batch(precision, persistent=False) as b:
        s.set_density(torch.from_numpy(prob.rho).to(DEV))
        st = s.solve(f, p, 1e-9)
        assert st.launches == 2  # resident
        # the mean, an iteration each (fixed point: its sweep is followed by the correction in the same
        # round; CG: update and correction are both flat sweeps), the last residual with the gauge
        rounds = 1 + st.iters + (st.outer_iters - 1 if opts is SPECTRAL else 0) + 1
        b.add(s, f, p, 1e-9)
        runs = 1
        while b.run(pairs):
            runs += 1
        assert runs == -(-rounds // pairs)


@pytest.mark.parametrize("opts", [FIXED, SPECTRAL], ids=["fixed", "spectral"])
def test_unattainable_tolerance_ends_at_the_iteration_limit(opts):
    """Inner solves of an iteration each: five sweeps an iteration with spectral CG."""
    prob = V.smooth_problem((32, 32, 32), seed=92)
    f = torch.from_numpy(prob.f).to(DEV)
    p = torch.empty_like(f)
    with vdp.Solver(32, 32, 32, prob.L, precision="mixed", max_iter=3000, inner_tol=0.9, **opts) as s:
        s.set_density(torch.from_numpy(prob.rho).to(DEV))
        st = s.solve(f, p, 1e-30, check=False)
    assert st.launches == 2 and st.status == vdp.VDP_ENOTCONV
    assert abs(float(p.mean())) <= 1e-14 * float(p.abs().max())
