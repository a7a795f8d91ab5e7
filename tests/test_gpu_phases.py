"""FP64 steps and small D3Q19 domains run as three launches over all nodes; the
domains of a batch run the fused march.  Both use the same per-node
arithmetic, so a job alone and in a batch agree bit for bit (walls on every
axis, sides around and below the march's 32 x 8 tile, single-node axes), and
match the oracle: FP64 to 1e-10; FP32 and FP16 to the bounds derived in
test_gpu_strip.py and test_gpu_precision.py (11 steps of the 20 and 500 they
are derived for)."""
import numpy as np
import pytest

from gpu_helpers import max_abs, run_oracle
from paper_1705_10045_gb300 import lbm
from paper_1705_10045_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = {lbm.LBM_STORE_FP64: {"rho": 1e-10, "T": 1e-10, "u": 1e-10, "P": 1e-10},
       lbm.LBM_STORE_FP32: {"rho": 1e-4, "T": 1e-4, "u": 1e-4, "P": 2e-5},
       lbm.LBM_STORE_FP16: {"rho": 3e-2, "T": 1.5e-2, "u": 5e-3, "P": 5e-4}}
KEYS = ("rho", "u", "T", "P")
BOX = dict(wall=1, wall_x=1, wall_y=1, T_fixed_lo=1, T_lo=0.86, T_fixed_y=(0, 1), T_y=(0.0, 0.83))


@pytest.mark.parametrize("storage", [lbm.LBM_STORE_FP64, lbm.LBM_STORE_FP32, lbm.LBM_STORE_FP16])
@pytest.mark.parametrize("nx,ny,nz,kw", [
    (1, 1, 5, {}), (5, 1, 3, {}), (33, 9, 4, {}), (32, 8, 2, dict(wall=1, T_fixed_hi=1, T_hi=0.78)),
    (40, 21, 19, BOX), (31, 7, 12, dict(BOX, chi_mode=1, chi=0.05, latent=0.02, tau=0.8))])
def test_job_alone_equals_the_march_and_the_oracle(nx, ny, nz, kw, storage):
    f = W.spinodal((nz, ny, nx), rho0=0.9, T0=0.8, noise=2e-2, seed=91)
    kw = dict(kw, nx=nx, ny=ny, nz=nz, gravity=(1e-5, -2e-5, 1e-5))
    rho, u, eps = f.rho, np.ascontiguousarray(np.resize(f.u, (3, nz, ny, nx))), 1.5 * f.T
    sim = lbm.Lbm(lattice=19, storage=storage, **kw)
    batch = lbm.LbmBatch(lattice=19, storage=storage)
    try:
        sim.init(rho, u, eps)
        sim.step(11)
        i = batch.add(rho, u, eps, 11, **kw)
        batch.step(11)
        alone, mixed = sim.moments(), batch.moments(i)
        assert np.array_equal(sim.get_state(), batch.get_state(i))
        assert sim.diagnostics()["bad"] == 0
    finally:
        sim.close()
        batch.close()
    o = run_oracle(W.Fields(rho, u, f.T), 11, lattice=19, **kw)
    for k in KEYS:
        assert np.array_equal(alone[k], mixed[k]), k
        assert max_abs(alone[k], o[k]) <= TOL[storage][k], k
