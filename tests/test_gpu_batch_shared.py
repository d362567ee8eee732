"""Members with the spectral passes or the V-cycle in a batch's shared launches (steps_per_sync > 0):
both forms of the inner solve, both methods, the duct, and Jacobi members besides; every result is the
one of the solve alone, bit for bit."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1601_05448_gb300 as vdp  # noqa: E402
import vdp_inputs as V  # noqa: E402

DEV = "cuda:0"
FIXED = {"method": vdp.VDP_METHOD_FIXED_POINT}
SPECTRAL = {"precond": vdp.VDP_PRECOND_SPECTRAL}
MG = {"precond": vdp.VDP_PRECOND_MG}
DUCT = {"bc_x": vdp.VDP_BC_DUCT}
# shape, options at creation, options after the density (a density set before the method: scaled form)
ALL = [((32, 32, 32), FIXED, {}), ((48, 64, 32), SPECTRAL, {}), ((64, 32, 48), {**FIXED, **DUCT}, {}),
       ((32, 48, 64), {}, SPECTRAL), ((32, 32, 48), FIXED, SPECTRAL), ((40, 32, 32), MG, {}), ((16, 16, 24), {}, {}),
       ((12, 20, 40), {"precond": vdp.VDP_PRECOND_CHEB}, {})]


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("members", [ALL, ALL[:1], ALL[1:2], [ALL[0], ALL[2]], [ALL[1], ALL[3]], [ALL[0], ALL[6]],
                                     [ALL[5], ALL[7]], 3 * ALL[:4]], ids=range(8))
def test_members_in_shared_launches_equal_alone(members, precision):
    made = []
    for k, (shape, opts, later) in enumerate(members):
        prob = V.smooth_problem(shape, seed=100 + k)
        nz, ny, nx = shape
        s = vdp.Solver(nx, ny, nz, prob.L, precision=precision, steps_per_sync=8, **opts)
        s.set_density(torch.from_numpy(prob.rho).to(DEV))
        if later:
            s.set_options(**later)
        f = torch.from_numpy(prob.f).to(DEV)
        alone = torch.empty_like(f)
        made.append((s, f, alone, torch.full_like(f, 3.0), s.solve(f, alone, 1e-9).iters))
    with vdp.Batch(precision, persistent=False) as b:
        for s, f, _, p, _ in made:
            b.add(s, f, p, 1e-9)
        b.run_to_completion(max_pairs=5)
    for s, f, alone, p, iters in made:
        assert s.stats().ok and s.stats().iters == iters
        assert torch.equal(p, alone)
        s.close()
