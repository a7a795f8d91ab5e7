"""Conservation sums (lbm_diagnostics) against exactly rounded sums
(math.fsum) of the same node moments, formed in the arithmetic type and the
same order from the checkpointed populations: node counts around a block's
first group of nodes and beyond one group per thread.

Bound: the compensated sums and the tree over partials each stay within a few
units of 2^-53 of sum |v|; 1e-15 sum |v| (9 units) holds them."""
import math

import numpy as np
import pytest

from paper_1705_10045_gb300 import lbm
from paper_1705_10045_gb300 import workloads as W

pytestmark = pytest.mark.gpu

C9 = [(0, 0), (1, 0), (-1, 0), (0, 1), (0, -1), (1, 1), (-1, -1), (1, -1), (-1, 1)]


@pytest.mark.parametrize("storage", [lbm.LBM_STORE_FP32, lbm.LBM_STORE_FP64])
@pytest.mark.parametrize("nx,ny", [(1, 1), (255, 1), (257, 1), (1025, 1), (123, 77), (1111, 499)])
def test_sums_equal_exact_sums_of_the_node_moments(nx, ny, storage):
    f = W.spinodal((1, ny, nx), rho0=0.9, T0=0.8, noise=2e-2, seed=81)
    f.u[0], f.u[1] = 0.02, W.uniform_noise(f.rho.shape, 1e-3, 82)
    sim = lbm.Lbm(lattice=9, nx=nx, ny=ny, storage=storage)
    try:
        sim.init(f.rho, f.u, 1.5 * f.T)
        sim.step(3)
        got = lbm.lbm_diagnostics(sim.h)
        dt = np.float32 if storage == lbm.LBM_STORE_FP32 else np.float64
        s = sim.get_state()[16:].view(dt).reshape(18, -1)
    finally:
        sim.close()
    m = {q: np.zeros(s.shape[1], dt) for q in ("rho", "jx", "jy", "E")}
    for k, c in enumerate(C9):
        m["rho"] += s[k]
        m["E"] += s[9 + k]
        for a, q in enumerate(("jx", "jy")):
            if c[a]:
                m[q] = m[q] + s[k] if c[a] > 0 else m[q] - s[k]
    for i, q in ((0, "rho"), (1, "jx"), (2, "jy"), (4, "E")):
        v = m[q].astype(np.float64)
        assert abs(got[i] - math.fsum(v)) <= 1e-15 * math.fsum(np.abs(v)), q
    assert got[3] == 0.0 and got[5] == 0 and got[6] == 0 and got[7] == 3
