"""The pseudo-inverse of the coarsest multigrid level, which one cluster of blocks builds: the numbers of
cells where a thread has more than one column and a block more than sixteen rows, and matrices that it
refuses."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import multigrid as MG  # noqa: E402
import paper_1601_05448_gb300 as vdp  # noqa: E402
import vdp_inputs as V  # noqa: E402

DEV = "cuda:0"


# (nz, ny, nx) and the coarsest level's cells: around a column per thread (256), the largest (512)
@pytest.mark.parametrize("duct", [False, True])
@pytest.mark.parametrize("shape,cells", [((136, 120, 8), 255), ((136, 136, 8), 289), ((56, 56, 56), 343),
                                         ((80, 80, 40), 500), ((128, 256, 8), 512)])
def test_vcycle_with_a_large_coarsest_level(shape, cells, duct):
    levels = vdp.vdp_mg_levels(*shape[::-1])
    assert shape[0] * shape[1] * shape[2] >> 3 * (levels - 1) == cells
    rng = np.random.default_rng(sum(shape))
    rho = V.density_modes(shape, rng, amplitude=0.7)
    g = rng.standard_normal(shape)
    lengths = (2.0, 1.0, 1.5)
    ref = MG.Hierarchy.from_density(rho, 0.0, geom=(*lengths, int(duct))).vcycle(g)
    nz, ny, nx = shape
    out = torch.empty(shape, dtype=torch.float64, device=DEV)
    with vdp.Solver(nx, ny, nz, 1.0, lengths=lengths,
                    bc_x=vdp.VDP_BC_DUCT if duct else vdp.VDP_BC_PERIODIC) as s:
        s.set_density(torch.from_numpy(rho).to(DEV))
        s.mg_apply(torch.from_numpy(g).to(DEV), out)
    # FP32 against the FP64 cycle, the tolerance of every V-cycle here
    assert np.linalg.norm(out.cpu().numpy() - ref) <= 2e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("scale", [1e-36, 1e-60, 1e60])
def test_levels_that_fp32_does_not_hold_are_refused(scale):
    rng = np.random.default_rng(1)
    rho = np.exp(rng.uniform(-1.0, 1.0, (16, 16, 16)))
    g = torch.from_numpy(rng.standard_normal(rho.shape)).to(DEV)
    g -= g.mean()
    out = torch.empty_like(g)
    with vdp.Solver(16, 16, 16, 1.0, precond=vdp.VDP_PRECOND_MG) as s:
        for steps in (0, 8):
            s.set_options(steps_per_sync=steps)
            for first in (0, 1):
                s.set_density(torch.from_numpy(scale * rho).to(DEV))
                for k in (first, 1 - first):
                    with pytest.raises(vdp.VdpError) as e:
                        if k:
                            s.mg_apply(g, out)
                        else:
                            s.solve(g, out, 1e-9, check=False)
                    assert e.value.status == vdp.VDP_ECUDA
        s.set_density(torch.from_numpy(rho).to(DEV))  # and the context goes on
        s.mg_apply(g, out)
        assert bool(torch.isfinite(out).all()) and s.solve(g, out, 1e-9).ok
