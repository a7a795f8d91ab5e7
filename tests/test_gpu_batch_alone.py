"""A batch request in which one domain steps takes the single-domain step, one
in which several do the persistent launch; every mix of the two, with walls
appearing and disappearing from the set of stepping domains, leaves each
domain where the job run alone ends."""
import numpy as np
import pytest

from paper_1705_10045_gb300 import lbm
from paper_1705_10045_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", [lbm.LBM_STORE_FP64, lbm.LBM_STORE_FP32, lbm.LBM_STORE_FP16])
@pytest.mark.parametrize("lattice", [9, 19])
def test_requests_of_one_and_of_several_domains_mix(lattice, storage):
    shapes = [(40, 33, 1), (40, 33, 1), (70, 20, 1)] if lattice == 9 else [(20, 16, 12), (20, 16, 12), (33, 9, 17)]
    kws = [{}, dict(wall=1, wall_x=1, T_fixed_lo=1, T_lo=0.85), {}]
    batch = lbm.LbmBatch(lattice=lattice, storage=storage)
    jobs = []
    try:
        for j, ((nx, ny, nz), kw) in enumerate(zip(shapes, kws)):
            f = W.spinodal((nz, ny, nx), rho0=0.9, T0=0.8, noise=2e-2, seed=21 + j)
            kw = dict(kw, nx=nx, ny=ny, nz=nz)
            jobs.append((batch.add(f.rho, f.u, 1.5 * f.T, 0, **kw), f, kw))
        taken = [0, 0, 0]
        for budgets, n in (((5, 0, 0), 5), ((4, 4, 4), 3), ((0, 7, 0), 9), ((6, 0, 2), 6), ((0, 0, 3), 2), ((2, 2, 0), 2)):
            for (i, _, _), s in zip(jobs, budgets):
                batch.set_budget(i, s)
            batch.step(n)
            for j, s in enumerate(budgets):
                taken[j] += min(s, n)
                assert batch.status(jobs[j][0]) == (taken[j], s - min(s, n))
        for (i, f, kw), steps in zip(jobs, taken):
            sim = lbm.Lbm(lattice=lattice, storage=storage, **kw)
            try:
                sim.init(f.rho, f.u, 1.5 * f.T)
                sim.step(steps)
                assert np.array_equal(sim.get_state(), batch.get_state(i)), kw
            finally:
                sim.close()
    finally:
        batch.close()
