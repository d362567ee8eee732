"""The bounded waits of the resident solve: with a barrier that expects one block more than the launch
has, every wait runs out after the limit, the kernel returns, the run reports VDP_ETIMEOUT, and the
members then finish with exactly the results they have alone."""
import time

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1601_05448_gb300 as vdp  # noqa: E402
import vdp_inputs as V  # noqa: E402

DEV = "cuda:0"
FIXED = {"method": vdp.VDP_METHOD_FIXED_POINT}
SPECTRAL = {"precond": vdp.VDP_PRECOND_SPECTRAL}


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("first_run", [0, 3])
def test_resident_members_recover_from_a_lost_arrival(precision, first_run):
    members = []
    for shape, opts, guess in (((32, 32, 32), FIXED, 0), ((48, 32, 64), SPECTRAL, 0), ((32, 48, 32), FIXED, 1),
                               ((16, 16, 24), {}, 0)):
        prob = V.smooth_problem(shape, seed=81)
        nz, ny, nx = shape
        s = vdp.Solver(nx, ny, nz, prob.L, precision=precision, use_guess=guess, **opts)
        s.set_density(torch.from_numpy(prob.rho).to(DEV))
        f = torch.from_numpy(prob.f).to(DEV)
        alone = torch.zeros_like(f)
        s.solve(f, alone, 1e-9)
        members.append((s, f, alone, torch.zeros_like(f), guess))
    with vdp.Batch(precision, persistent=False) as b:
        b.set_wait_limit(0.05)
        for s, f, _, p, _ in members:
            b.add(s, f, p, 1e-9)
        if first_run:
            b.run(first_run)
        b.inject_lost_arrival()
        start = time.perf_counter()
        with pytest.raises(vdp.VdpError) as e:
            b.run(2)
        assert e.value.status == vdp.VDP_ETIMEOUT and 0.04 < time.perf_counter() - start < 5.0
        assert not any(b.done(s) for s, *_ in members)
        b.run_to_completion(max_pairs=16)
        for s, f, alone, p, guess in members:
            assert s.stats().ok
            # a solve with a guess goes on from what its pressure held
            assert torch.equal(p, alone) if not guess else float((p - alone).norm() / alone.norm()) < 1e-6
        with pytest.raises(vdp.VdpError):  # nothing is left that waits
            b.inject_lost_arrival()
    for s, f, alone, p, guess in members:  # and the contexts solve as before
        p.zero_()
        s.solve(f, p, 1e-9)
        assert torch.equal(p, alone)
        s.close()
