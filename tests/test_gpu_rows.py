"""The D3Q19 row march (domains periodic in x whose rows are whole 16-byte
parts): the same state bit for bit as the march, which the domains of a batch
take, for rows around one and several tiles of 28 columns and of the tile's
rows, walls on y and z, a conductivity that follows the density, latent heat,
and steps in ranges of planes."""
import numpy as np
import pytest

from paper_1705_10045_gb300 import lbm
from paper_1705_10045_gb300 import workloads as W

pytestmark = pytest.mark.gpu

WALLS = dict(wall=1, wall_y=1, T_fixed_lo=1, T_lo=0.86, T_fixed_y=(0, 1), T_y=(0.0, 0.83))


@pytest.mark.parametrize("storage", [lbm.LBM_STORE_FP32, lbm.LBM_STORE_FP16])
@pytest.mark.parametrize("nx,ny,nz,kw", [
    (112, 96, 110, {}), (116, 101, 150, dict(WALLS)), (140, 130, 71, dict(chi_mode=1, chi=0.05, tau=0.8)),
    (168, 65, 100, dict(WALLS, chi_mode=1, chi=0.05, latent=0.02)), (128, 128, 128, dict(wall=1, T_fixed_hi=1, T_hi=0.78))])
def test_row_march_equals_the_march(nx, ny, nz, kw, storage):
    f = W.spinodal((nz, ny, nx), rho0=0.9, T0=0.8, noise=2e-2, seed=41)
    kw = dict(kw, nx=nx, ny=ny, nz=nz, gravity=(1e-5, -2e-5, 1e-5))
    u, eps = np.ascontiguousarray(f.u), 1.5 * f.T
    sim = lbm.Lbm(lattice=19, storage=storage, **kw)
    cut = lbm.Lbm(lattice=19, storage=storage, **kw)
    batch = lbm.LbmBatch(lattice=19, storage=storage)
    try:
        assert lbm.lbm_launch_name(sim.h, 0) == "row_march_kernel"
        sim.init(f.rho, u, eps)
        sim.step(4)
        cut.init(f.rho, u, eps)
        for _ in range(4):
            for first, count in ((nz // 2, nz - nz // 2), (0, nz // 2)):
                lbm.lbm_step_begin(cut.h, first, count)
            lbm.lbm_step_end(cut.h)
        # two stepping domains: the persistent launch
        ids = [batch.add(f.rho, u, eps, 4, **kw) for _ in range(2)]
        batch.step(4)
        want = batch.get_state(ids[0])
        assert np.array_equal(sim.get_state(), want)
        assert np.array_equal(cut.get_state(), want)
        assert sim.diagnostics()["bad"] == 0
    finally:
        sim.close()
        cut.close()
        batch.close()
