"""Host outputs of lbm_moments and lbm_moments_f equal the device outputs on
both sides of the size below which they come through one pinned buffer (128
KiB of fields: 3276 D2Q9 nodes as doubles, 6553 as floats), any subset of the
fields, in either order of the two calls; the fields match the oracle to the
FP64 bound."""
import numpy as np
import pytest

from gpu_helpers import max_abs, run_oracle
from paper_1705_10045_gb300 import lbm
from paper_1705_10045_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(1, 1), (13, 7), (63, 52), (3277, 1), (6553, 1), (118, 56)])
@pytest.mark.parametrize("single_first", [False, True])
def test_host_outputs_equal_device_outputs(nx, ny, single_first):
    import torch
    f = W.spinodal((1, ny, nx), rho0=0.9, T0=0.8, noise=2e-2, seed=61)
    sim = lbm.Lbm(lattice=9, nx=nx, ny=ny, storage=lbm.LBM_STORE_FP64)
    shape = {"rho": (1, ny, nx), "u": (2, 1, ny, nx), "T": (1, ny, nx), "P": (1, ny, nx)}
    try:
        sim.init(f.rho, f.u, 1.5 * f.T)
        sim.step(4)
        for single in (single_first, not single_first):
            read, dt = (lbm.lbm_moments_f, torch.float32) if single else (lbm.lbm_moments, torch.float64)
            dev = {k: torch.empty(s, dtype=dt, device="cuda") for k, s in shape.items()}
            host = {k: np.full(s, -7.0, np.float32 if single else np.float64) for k, s in shape.items()}
            read(sim.h, *dev.values())
            read(sim.h, *host.values())
            part = {k: np.full(shape[k], -7.0, host[k].dtype) for k in ("u", "P")}
            read(sim.h, u=part["u"], P=part["P"])
            for k in shape:
                assert np.array_equal(host[k], dev[k].cpu().numpy()), (single, k)
            assert np.array_equal(part["u"], host["u"]) and np.array_equal(part["P"], host["P"])
            if not single:
                o = run_oracle(f, 4, lattice=9, nx=nx, ny=ny)
                assert all(max_abs(host[k], o[k]) <= 1e-10 for k in shape)
    finally:
        sim.close()
