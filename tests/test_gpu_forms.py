"""Every form of a step against another one, at sizes where the form is really
the one that runs (lbm_launch_name; two stepping domains of a batch take the
persistent launch, one alone takes the single-domain step):

* phases against the batch's march (D3Q19) and strips (D2Q9 FP64): walls on
  every axis, single-node axes, sides below a tile, a conductivity that
  follows the density, latent heat;
* the single-domain march, which large domains take that the row march cannot
  (walls on x, rows that are no whole 16-byte parts), against the batch's, whole
  and in ranges;
* the row march on narrow and low domains, in ranges of three planes, and
  against the oracle.

States agree bit for bit; the oracle bounds are those of
test_gpu_oracle_wide.py, derived there for 500 steps (60 here)."""
import numpy as np
import pytest

from gpu_helpers import max_abs, run_oracle
from paper_1705_10045_gb300 import lbm
from paper_1705_10045_gb300 import workloads as W

pytestmark = pytest.mark.gpu

FP64, FP32, FP16 = lbm.LBM_STORE_FP64, lbm.LBM_STORE_FP32, lbm.LBM_STORE_FP16
KEYS = ("rho", "u", "T", "P")
BOX = dict(wall=1, wall_x=1, wall_y=1, T_fixed_lo=1, T_lo=0.86, T_fixed_y=(0, 1), T_y=(0.0, 0.83))
BOX9 = dict(wall=1, wall_x=1, T_fixed_lo=1, T_lo=0.86, T_fixed_x=(0, 1), T_x=(0.0, 0.83))
RICH = dict(chi_mode=1, chi=0.05, latent=0.02, tau=0.8)


def _job(lattice, nx, ny, nz, seed=61):
    f = W.spinodal((nz, ny, nx), rho0=0.9, T0=0.8, noise=2e-2, seed=seed)
    u = np.ascontiguousarray(np.resize(f.u, (2 if lattice == 9 else 3, nz, ny, nx)))
    return f.rho, u, 1.5 * f.T


def _single(lattice, storage, fields, steps, kw, ranges=None, name=None):
    """State and kernel name after `steps` steps of a handle, whole or in ranges of planes."""
    sim = lbm.Lbm(lattice=lattice, storage=storage, **kw)
    try:
        if name:
            assert lbm.lbm_launch_name(sim.h, 0) == name
        sim.init(*fields)
        if ranges is None:
            sim.step(steps)
        else:
            for _ in range(steps):
                for first, count in ranges:
                    lbm.lbm_step_begin(sim.h, first, count)
                lbm.lbm_step_end(sim.h)
        d = sim.diagnostics()
        assert d["bad"] == 0
        return sim.get_state(), d
    finally:
        sim.close()


def _together(lattice, storage, fields, steps, kw):
    """States of two equal domains of a batch, stepped by the persistent launch."""
    batch = lbm.LbmBatch(lattice=lattice, storage=storage)
    try:
        ids = [batch.add(*fields, steps, **kw) for _ in range(2)]
        batch.step(steps)
        d = [batch.diagnostics(i) for i in ids]
        return [batch.get_state(i) for i in ids], d
    finally:
        batch.close()


def _check(lattice, storage, fields, steps, kw, name, cuts=()):
    alone, d = _single(lattice, storage, fields, steps, kw, name=name)
    both, db = _together(lattice, storage, fields, steps, kw)
    for state, q in zip(both, db):
        assert np.array_equal(alone, state)
        assert q[5] == d["clamps"] and q[6] == d["bad"]
    for ranges in cuts:
        assert np.array_equal(alone, _single(lattice, storage, fields, steps, kw, ranges=ranges)[0]), ranges


@pytest.mark.parametrize("storage", [FP64, FP32, FP16])
@pytest.mark.parametrize("nx,ny,nz,kw", [
    (1, 1, 5, {}), (5, 1, 3, {}), (33, 9, 4, {}), (32, 8, 2, dict(wall=1, T_fixed_hi=1, T_hi=0.78)), (40, 21, 19, BOX),
    (31, 7, 12, dict(BOX, **RICH)), (26, 30, 9, dict(RICH, wall_y=1))])
def test_phases_equal_the_march(nx, ny, nz, kw, storage):
    kw = dict(kw, nx=nx, ny=ny, nz=nz, gravity=(1e-5, -2e-5, 1e-5))
    cuts = [[(0, 1), (1, nz - 1)], [(nz - 1, 1), (0, nz - 1)]]
    _check(19, storage, _job(19, nx, ny, nz), 11, kw, "phase_moments_kernel", cuts)


@pytest.mark.parametrize("nx,ny,kw", [(1, 7, {}), (9, 1, {}), (28, 2, dict(wall=1, T_fixed_hi=1, T_hi=0.78)),
                                      (57, 40, BOX9), (64, 33, dict(BOX9, **RICH)), (83, 29, RICH)])
def test_phases_equal_the_strips(nx, ny, kw):
    kw = dict(kw, nx=nx, ny=ny, gravity=(1e-5, -2e-5, 0.0))
    cuts = [[(ny - 1, 1), (0, ny - 1)]] if ny > 1 else []
    _check(9, FP64, _job(9, nx, ny, 1), 11, kw, "phase_moments_kernel", cuts)


@pytest.mark.parametrize("storage,nx,ny,nz,kw", [
    (FP32, 127, 99, 101, {}), (FP32, 126, 100, 111, BOX),
    (FP32, 160, 128, 120, dict(RICH, wall_x=1, T_fixed_x=(1, 0), T_x=(0.85, 0.0))),
    (FP16, 191, 128, 128, {}), (FP16, 160, 128, 120, BOX),
    (FP16, 192, 128, 128, dict(RICH, wall_x=1, T_fixed_x=(1, 0), T_x=(0.85, 0.0)))])
def test_single_march_equals_the_batch_march(storage, nx, ny, nz, kw):
    kw = dict(kw, nx=nx, ny=ny, nz=nz, gravity=(1e-5, -2e-5, 1e-5))
    cuts = [[(nz - 3, 3), (0, 3), (3, nz - 6)]]
    _check(19, storage, _job(19, nx, ny, nz), 3, kw, "fused_step_kernel", cuts)


@pytest.mark.parametrize("storage,nx,ny,nz,kw", [
    (FP32, 26, 9, 9728, {}), (FP32, 26, 8, 9728, dict(RICH, wall=1, T_fixed_lo=1, T_lo=0.86)),
    (FP32, 56, 20, 2432, dict(wall_y=1, T_fixed_y=(0, 1), T_y=(0.0, 0.83))), (FP32, 54, 7, 4864, {}),
    (FP32, 20, 18, 4864, {}),
    (FP16, 24, 16, 9728, dict(BOX, wall_x=0)), (FP16, 28, 13, 9728, {}), (FP16, 56, 14, 4864, RICH),
    (FP32, 112, 96, 110, {}), (FP16, 112, 96, 110, dict(BOX, wall_x=0))])
def test_row_march_on_narrow_domains_and_short_ranges(storage, nx, ny, nz, kw):
    kw = dict(kw, nx=nx, ny=ny, nz=nz, gravity=(1e-5, -2e-5, 1e-5))
    h = nz // 2
    cuts = [[(nz - 3, 3), (0, 3), (3, h - 3), (h, 1), (h + 1, nz - h - 4)]]
    _check(19, storage, _job(19, nx, ny, nz), 3, kw, "row_march_kernel", cuts)


def test_row_march_matches_the_oracle():
    nx, ny, nz, steps = 84, 90, 40, 60
    f = W.pool_boiling_3d(nx=nx, ny=ny, nz=nz, T=0.8, depth=10, noise=1e-4, seed=3)
    kw = dict(lattice=19, nx=nx, ny=ny, nz=nz, wall=1, T_fixed_lo=1, T_lo=0.95, gravity=(0.0, 0.0, -1e-5))
    o = run_oracle(f, steps, **kw)
    sim = lbm.Lbm(storage=FP32, **kw)
    try:
        assert lbm.lbm_launch_name(sim.h, 0) == "row_march_kernel"
        sim.init(f.rho, np.ascontiguousarray(f.u), 1.5 * f.T)
        sim.step(steps)
        g, d = sim.moments(), sim.diagnostics()
    finally:
        sim.close()
    errs = {k: max_abs(g[k], o[k]) for k in KEYS}
    assert errs["rho"] <= 2e-4 and errs["T"] <= 5e-5 and errs["u"] <= 5e-6 and errs["P"] <= 2e-5, errs
    assert d["bad"] == 0 and d["clamps"] == 0
