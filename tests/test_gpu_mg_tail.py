"""The multigrid levels that one block takes (up to 4096 cells), against the CPU oracle's V-cycle: the
largest such level, a level just above it, sides of two and one cells, a single level besides the
coarsest, the duct's ends, and levels with more cells than the block has threads.

Tolerance: that of every V-cycle here, FP32 against the FP64 cycle, relative L2 <= 2e-5.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import multigrid as MG  # noqa: E402
import paper_1601_05448_gb300 as vdp  # noqa: E402
import vdp_inputs as V  # noqa: E402

DEV = "cuda:0"


# (nz, ny, nx)
@pytest.mark.parametrize("duct", [False, True])
@pytest.mark.parametrize("shape", [(32, 32, 32), (40, 32, 32), (64, 4, 8), (4, 64, 16), (32, 4, 64), (8, 8, 40),
                                   (24, 40, 32)])
def test_vcycle_with_levels_in_one_block(shape, duct):
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
    got = out.cpu().numpy()
    assert np.linalg.norm(got - ref) <= 2e-5 * np.linalg.norm(ref)
