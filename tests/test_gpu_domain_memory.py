"""lbm_domain_bytes is what a domain takes, whichever form steps it: the
device memory in use after a whole life of calls grows by no more than that
(and the allocator's 2 MiB granularity per allocation, at most three), and a
batch request that steps one domain by itself takes none."""
import numpy as np
import pytest

from paper_1705_10045_gb300 import lbm
from paper_1705_10045_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CASES = [(9, (1, 1000, 1100), lbm.LBM_STORE_FP64), (19, (100, 96, 104), lbm.LBM_STORE_FP64),
         (19, (72, 70, 68), lbm.LBM_STORE_FP32), (19, (72, 70, 68), lbm.LBM_STORE_FP16)]


def _free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info(0)[0]


def _job(lattice, shape, storage, seed):
    f = W.spinodal(shape, rho0=0.9, T0=0.8, noise=2e-2, seed=seed)
    kw = dict(nx=shape[2], ny=shape[1], nz=shape[0])
    return f.rho, np.ascontiguousarray(f.u[: 2 if lattice == 9 else 3]), 1.5 * f.T, kw


@pytest.mark.parametrize("lattice,shape,storage", CASES)
def test_a_domain_takes_what_domain_bytes_says(lattice, shape, storage):
    for small in (True, False):   # the first pass loads the kernels
        rho, u, eps, kw = _job(lattice, (1, 16, 16) if lattice == 9 else (16, 16, 16), storage, 3) if small else \
            _job(lattice, shape, storage, 3)
        before = _free()
        sim = lbm.Lbm(lattice=lattice, storage=storage, **kw)
        try:
            sim.init(rho, u, eps)
            sim.step(3)
            sim.moments()
            sim.diagnostics()
            used = before - _free()
        finally:
            sim.close()
    limit = lbm.lbm_domain_bytes(lbm.make_params(lattice=lattice, storage=storage, **kw))
    assert used <= limit + 3 * (2 << 20), (used, limit)


@pytest.mark.parametrize("lattice,shape,storage", CASES)
def test_stepping_alone_in_a_batch_takes_no_memory(lattice, shape, storage):
    batch = lbm.LbmBatch(lattice=lattice, storage=storage)
    try:
        rho, u, eps, kw = _job(lattice, (1, 16, 16) if lattice == 9 else (16, 16, 16), storage, 4)
        batch.add(rho, u, eps, 2, **kw)
        batch.step(2)   # loads the kernels
        batch.sync()
        rho, u, eps, kw = _job(lattice, shape, storage, 5)
        i = batch.add(rho, u, eps, 6, **kw)
        before = _free()
        batch.step(3)
        batch.step(3)
        batch.sync()
        assert batch.status(i) == (6, 0)
        assert before - _free() < 1 << 20
    finally:
        batch.close()
