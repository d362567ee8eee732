"""Options that a program sets on a context while its solve is queued in a batch are for its later
solves: the queued one finishes as it was added -- as one resident launch, as the context's device-side
loop, or in the shared launches."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1601_05448_gb300 as vdp  # noqa: E402
import vdp_inputs as V  # noqa: E402

DEV = "cuda:0"
FIXED = {"method": vdp.VDP_METHOD_FIXED_POINT}
SPECTRAL = {"precond": vdp.VDP_PRECOND_SPECTRAL}


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("shape,opts", [((32, 32, 32), FIXED), ((48, 32, 64), SPECTRAL), ((128, 128, 96), FIXED),
                                        ((128, 128, 96), SPECTRAL), ((40, 32, 32), {"precond": vdp.VDP_PRECOND_MG}),
                                        ((24, 20, 16), {})])
@pytest.mark.parametrize("started", [False, True])
def test_options_of_a_queued_member(shape, opts, precision, started):
    tol = 1e-9
    prob = V.smooth_problem(shape, seed=71)
    other = V.smooth_problem((32, 32, 32), seed=72)
    rho, f = (torch.from_numpy(a).to(DEV) for a in (prob.rho, prob.f))
    g = torch.from_numpy(other.f).to(DEV)
    alone, p, q = torch.empty_like(f), torch.full_like(f, 2.0), torch.empty_like(g)
    nz, ny, nx = shape
    with vdp.Solver(nx, ny, nz, prob.L, precision=precision, **opts) as s, \
            vdp.Solver(32, 32, 32, other.L, precision=precision, **FIXED) as t, \
            vdp.Batch(precision, persistent=False) as b:
        s.set_density(rho)
        t.set_density(torch.from_numpy(other.rho).to(DEV))
        iters = s.solve(f, alone, tol).iters
        b.add(s, f, p, tol)
        if started:
            assert b.run(2) == 1
        s.set_options(steps_per_sync=8)
        b.run(1)
        if opts in (FIXED, SPECTRAL):
            s.set_options(spec_slab=16, steps_per_sync=0)
            b.run(1)
            s.set_options(method=vdp.VDP_METHOD_CG if opts is FIXED else vdp.VDP_METHOD_FIXED_POINT, damping=0.7)
        b.add(t, g, q, tol)  # the device tables are built again
        b.run_to_completion(max_pairs=8)
        assert s.stats().ok and s.stats().iters == iters
        assert torch.equal(p, alone)
