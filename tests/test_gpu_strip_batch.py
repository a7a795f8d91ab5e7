"""D2Q9 batches of domains at and around one and several strips of 28 columns
and fewer rows than a work item, periodic and walled together: every domain
equals the job run alone bit for bit, in every CTA shape and storage format,
also after the set of stepping domains changes (and with it the rows of an
item)."""
import numpy as np
import pytest

from paper_1705_10045_gb300 import lbm
from paper_1705_10045_gb300 import workloads as W

pytestmark = pytest.mark.gpu

WALLS = dict(wall=1, T_fixed_lo=1, T_lo=0.85, wall_x=1, T_fixed_x=(0, 1), T_x=(0.0, 0.82))
SIZES = [(1, 9, {}), (27, 5, {}), (28, 40, dict(WALLS)), (29, 3, {}), (113, 70, {}), (225, 31, dict(WALLS))]


@pytest.mark.parametrize("storage", [lbm.LBM_STORE_FP64, lbm.LBM_STORE_FP32, lbm.LBM_STORE_FP16])
@pytest.mark.parametrize("variant", [0, 1, 2])
def test_strip_batch_equals_jobs_alone(storage, variant):
    batch = lbm.LbmBatch(lattice=9, storage=storage)
    jobs = []
    try:
        batch.set_variant(variant)
        for j, (nx, ny, kw) in enumerate(SIZES):
            f = W.spinodal((1, ny, nx), rho0=0.9, T0=0.8, noise=2e-2, seed=31 + j)
            kw = dict(kw, nx=nx, ny=ny, gravity=(1e-5, -2e-5, 0.0), tau=0.9)
            steps = 9 + 4 * j
            jobs.append((batch.add(f.rho, f.u, 1.5 * f.T, steps, **kw), f, kw, steps))
        batch.step(11)
        batch.step(30)
        for i, f, kw, steps in jobs:
            assert batch.status(i) == (steps, 0)
            sim = lbm.Lbm(lattice=9, storage=storage, **kw)
            try:
                sim.init(f.rho, f.u, 1.5 * f.T)
                sim.step(steps)
                assert np.array_equal(sim.get_state(), batch.get_state(i)), kw
                assert np.array_equal(lbm.lbm_diagnostics(sim.h)[5:], batch.diagnostics(i)[5:]), kw
            finally:
                sim.close()
    finally:
        batch.close()
