"""A small domain that is read once costs little more than its read: what a
read adds to the whole life of a handle stays within four reads of a handle
that has been read before (fields of 32 x 32 nodes to the host, about 30 us
each), however the library stages them."""
import time

import numpy as np
import pytest

from paper_1705_10045_gb300 import lbm
from paper_1705_10045_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _median(v):
    return sorted(v)[len(v) // 2]


def test_reading_a_small_domain_once_costs_a_read():
    f = W.spinodal((1, 32, 32), rho0=0.9, T0=0.8, noise=2e-2, seed=5)
    u, eps = np.ascontiguousarray(f.u[:2]), 1.5 * f.T

    def life(reads):
        """Seconds from create to close, and of the last read."""
        start = time.perf_counter()
        sim = lbm.Lbm(lattice=9, nx=32, ny=32, storage=lbm.LBM_STORE_FP32)
        sim.init(f.rho, u, eps)
        sim.step(3)
        lbm.lbm_sync(sim.h)
        t = time.perf_counter()
        for _ in range(reads):
            t = time.perf_counter()
            sim.moments()
        read = time.perf_counter() - t
        sim.close()
        return time.perf_counter() - start, read

    lives = {0: [], 1: []}
    for k in range(120):
        lives[k % 2].append(life(k % 2)[0])
    again = _median([life(4)[1] for _ in range(40)])
    never, once = _median(lives[0][10:]), _median(lives[1][10:])
    assert once - never <= 4.0 * again, (never, once, again)
