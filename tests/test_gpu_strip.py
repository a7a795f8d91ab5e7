"""The D2Q9 step in FP32 and FP16 storage, where a warp marches a strip of 28
columns: widths at and around one and two strips, rows fewer than the four a
warp keeps, and walls on either axis, against the FP64 oracle.

FP32 bounds (max-abs after 20 steps): a population takes about 10 rounded
operations a step, 6e-8 relative each, so in the worst case 20 x 10 x 6e-8 =
1.2e-5 relative on a density of up to 2, amplified about three times at the
interface: rho 1e-4; T is a ratio of two such sums: 1e-4; u* is a momentum
error over the smallest density (0.2): 1e-4; P = kappa p~ with kappa = 0.01
and dp~/drho of order 10: 2e-5.  FP16 bounds: the module docstring of
test_gpu_precision.py (500 steps) holds for 20."""
import numpy as np
import pytest

from gpu_helpers import max_abs, run_gpu, run_oracle
from paper_1705_10045_gb300 import lbm
from paper_1705_10045_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = {lbm.LBM_STORE_FP32: {"rho": 1e-4, "T": 1e-4, "u": 1e-4, "P": 2e-5},
       lbm.LBM_STORE_FP16: {"rho": 3e-2, "T": 1.5e-2, "u": 5e-3, "P": 5e-4}}


@pytest.mark.parametrize("storage", [lbm.LBM_STORE_FP32, lbm.LBM_STORE_FP16])
@pytest.mark.parametrize("nx,ny", [(1, 9), (2, 1), (27, 5), (28, 2), (29, 40), (57, 3), (113, 70)])
@pytest.mark.parametrize("walls", ["periodic", "y", "x", "box"])
def test_strip_edges_match_oracle(nx, ny, walls, storage):
    kw = dict(lattice=9, nx=nx, ny=ny, nz=1, gravity=(1e-5, -2e-5, 0.0), tau=0.9)
    if walls in ("y", "box"):
        if ny < 2:
            pytest.skip("a walled axis needs two nodes")
        kw.update(wall=1, T_fixed_lo=1, T_lo=0.85)
    if walls in ("x", "box"):
        if nx < 2:
            pytest.skip("a walled axis needs two nodes")
        kw.update(wall_x=1, T_fixed_x=(0, 1), T_x=(0.0, 0.82))
    f = W.spinodal((1, ny, nx), rho0=0.9, T0=0.8, noise=2e-2, seed=71)
    g = run_gpu(f, 20, storage=storage, **kw)
    o = run_oracle(f, 20, **kw)
    errs = {k: max_abs(g[k], o[k]) for k in TOL[storage]}
    assert all(np.isfinite(v) and v <= TOL[storage][k] for k, v in errs.items()), errs
    assert g["diag"]["bad"] == 0
