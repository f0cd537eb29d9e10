"""The FP64 collision in 64-bit integers and its way out to fused multiply-adds: against the oracle
where the populations of a family differ much in size, and where they are zero, tiny or huge."""

import numpy as np
import pytest

import oracle
from paper_1401_0427_gb300 import inputs, lbm_sw

from gpu_helpers import FP64_TOL, gpu_post, oracle_params, oracle_post, rel_max

pytestmark = pytest.mark.gpu

P, W = lbm_sw.PERIODIC, lbm_sw.WALL


@pytest.mark.parametrize("kernel", [lbm_sw.KERNEL_SIMPLE, lbm_sw.KERNEL_VEC], ids=["simple", "vec"])
@pytest.mark.parametrize("s,lam", [(1.8, 8.0), (1.0, 8.0), (0.0, 8.0), (0.3, 80.0)])
def test_sizes_apart_match_the_oracle(s, lam, kernel):
    """Each population scaled by a power of two between 2^-70 and 2^3 (depths stay positive), some
    zero: integer cells and others side by side.  The tolerance is the stated FP64 bar."""
    ny, nx = 21, 70
    F0 = inputs.random_populations(13, ny, nx, seed=9700)
    k = np.floor(inputs.uniform(9701, F0.size, -70.0, 4.0)).reshape(F0.shape)
    F0 = np.where(inputs.uniform(9702, F0.size).reshape(F0.shape) < 0.5, F0, F0 * 2.0 ** k)
    F0[:, 3:5] = np.where(inputs.uniform(9703, F0[:, 3:5].size).reshape(F0[:, 3:5].shape) < 0.5, F0[:, 3:5], 0.0)
    F0[0] = np.abs(F0[0]) + 0.5
    F0[5:] *= 0.05
    p = oracle_params(nx, ny, 2, (P, P, W, W), None, 0.05, lam=lam, s=s)
    got = gpu_post(F0, 1, dim=2, precision=lbm_sw.FP64, bc=(P, P, W, W), inflow=None, a=0.05, kernel=kernel, lam=lam, s=s)
    want = oracle_post(F0, 1, p, 2)
    assert rel_max(got, want) <= FP64_TOL


@pytest.mark.parametrize("scale", [2.0 ** -600, 2.0 ** -300, 1.0, 2.0 ** 300])
def test_depths_over_the_exponent_range(scale):
    """A lake at rest of any depth stays one (g scaled so that g h is the same)."""
    nx, ny = 40, 9
    with lbm_sw.Simulation(nx, ny, precision=lbm_sw.FP64, g=1.0 / scale) as sim:
        z = np.zeros((ny, nx))
        sim.set_state(np.full((ny, nx), 1.37 * scale), z, z)
        sim.step(20)
        h, hu, hv = sim.moments()
    assert np.abs(h / scale - 1.37).max() <= 1e-14 and np.all(hu == 0) and np.all(hv == 0)


def test_infinities_and_nan_stay_where_they_stream():
    nx, ny = 33, 8
    F0 = inputs.random_populations(13, ny, nx, seed=9710)
    F0[1, 4, 10], F0[6, 2, 20] = np.nan, np.inf
    kw = dict(dim=2, precision=lbm_sw.FP64, bc=(P, P, P, P), inflow=None, a=0.05)
    a = gpu_post(F0, 2, kernel=lbm_sw.KERNEL_SIMPLE, **kw)
    b = gpu_post(F0, 2, kernel=lbm_sw.KERNEL_VEC, **kw)
    with np.errstate(all="ignore"):
        p = oracle.params(nx, ny, a=0.05)
        want = oracle_post(F0, 2, p, 2)
    assert np.array_equal(a, b, equal_nan=True)
    assert np.array_equal(np.isfinite(a), np.isfinite(want))
