"""Conservation sums of FP32 moments whose magnitudes spread over far more than
the 53 bits of a double, next to each other in what one thread adds up:
exactly rounded sums (math.fsum) hold as for moments of like size.

* One thread's nodes hold 1 and then values of 1.5 x 2^-54, each too small to
  change a double sum of 1: compensation carries them, so the sum over all
  threads is the exactly rounded one (1024 (1 + 2^-52)); an uncompensated sum
  of the group ends at 1024.
* Random magnitudes from 2^-60 to 1 and both signs, more nodes than one group
  per thread.  Bound: compensated sums stay within 2 units of 2^-53 of
  sum |v| per thread, the five plain levels of the warp tree add 5, the
  partials 2: 1e-15 sum |v| (9 units).
* Values whose FP32 sum overflows, and a NaN: as in double arithmetic.
"""
import math

import numpy as np
import pytest

from paper_1705_10045_gb300 import lbm

pytestmark = pytest.mark.gpu

HEADER = 16


def _sums(nx, ny, right, left=None):
    """lbm_diagnostics of a D2Q9 FP32 state whose only populations are N of
    directions +x and -x, and g of the resting direction (1)."""
    sim = lbm.Lbm(lattice=9, nx=nx, ny=ny, storage=lbm.LBM_STORE_FP32)
    try:
        one = np.ones((1, ny, nx))
        sim.init(0.9 * one, np.zeros((2, 1, ny, nx)), 1.2 * one)
        state = sim.get_state()
        s = state[HEADER:].view(np.float32).reshape(18, -1)
        s[:] = 0
        s[9] = 1
        s[1] = right
        if left is not None:
            s[2] = left
        sim.set_state(state)
        return lbm.lbm_diagnostics(sim.h)
    finally:
        sim.close()


def test_small_values_beside_a_large_one_are_not_lost():
    n, threads = 4096, 1024   # four nodes per thread: node i belongs to thread i mod 1024
    v = np.full(n, 1.5 * 2.0**-54, np.float32)
    v[:threads] = 1
    got, want = _sums(n, 1, v), math.fsum(v.astype(np.float64))
    assert want == 1024 * (1 + 2.0**-52)
    assert got[0] == want and got[1] == want


@pytest.mark.parametrize("nx,ny", [(777, 3), (1201, 903)])
def test_wide_magnitudes_of_both_signs(nx, ny):
    rng = np.random.default_rng(7)
    n = nx * ny
    right = np.exp2(rng.uniform(-60, 0, n)).astype(np.float32)
    left = np.exp2(rng.uniform(-60, 0, n)).astype(np.float32)
    got = _sums(nx, ny, right, left)
    for i, m in ((0, right + left), (1, right - left)):   # the node's moments, rounded to FP32
        v = m.astype(np.float64)
        assert abs(got[i] - math.fsum(v)) <= 1e-15 * math.fsum(np.abs(v)), i
    assert got[4] == n


def test_sums_beyond_the_range_of_fp32_and_nan():
    v = np.full(4096, 2e38, np.float32)
    want = math.fsum(v.astype(np.float64))
    got = _sums(4096, 1, v)
    assert abs(got[0] - want) <= 1e-15 * want and abs(got[1] - want) <= 1e-15 * want
    v[:] = 1
    v[3000] = np.nan
    got = _sums(4096, 1, v)
    assert math.isnan(got[0]) and math.isnan(got[1]) and got[2] == 0 and got[4] == 4096
