"""The FP64 collisions in 64-bit integers and its way out to fused multiply-adds: against the oracle
where the populations of a family differ much in size, and where they are zero, tiny or huge."""

import math

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


@pytest.mark.parametrize("kernel", [lbm_sw.KERNEL_SIMPLE, lbm_sw.KERNEL_VEC], ids=["simple", "vec"])
def test_mrt_sizes_apart_match_the_oracle(kernel):
    """The same inputs with every moment at its own rate, some zero."""
    ny, nx = 21, 70
    rates = [0.0, 1.1, 0.0, 1.3, 1.4, 0.0, 1.5, 0.0, 1.7, 0.0, 1.99, 1.65, 0.9]
    F0 = inputs.random_populations(13, ny, nx, seed=9730)
    k = np.floor(inputs.uniform(9731, F0.size, -70.0, 4.0)).reshape(F0.shape)
    F0 = np.where(inputs.uniform(9732, F0.size).reshape(F0.shape) < 0.5, F0, F0 * 2.0 ** k)
    F0[:, 3:5] = np.where(inputs.uniform(9733, F0[:, 3:5].size).reshape(F0[:, 3:5].shape) < 0.5, F0[:, 3:5], 0.0)
    F0[0] = np.abs(F0[0]) + 0.5
    F0[5:] *= 0.05
    p = oracle.params(nx, ny, a=0.05, bc=(P, P, W, W), s_moments=rates)
    got = gpu_post(F0, 1, dim=2, precision=lbm_sw.FP64, bc=(P, P, W, W), inflow=None, a=0.05, kernel=kernel,
                   mrt_rates=rates)
    assert rel_max(got, oracle_post(F0, 1, p, 2)) <= FP64_TOL


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


@pytest.mark.parametrize("lam", [1.0, 8.0])
@pytest.mark.parametrize("rates", [None, [1.8] * 13, [0.0, 1.1, 1.2, 1.3, 1.4, 0.0, 1.5, 1.6, 1.7, 0.0, 1.99, 1.65, 0.9]],
                         ids=["bgk", "mrt-equal", "mrt"])
@pytest.mark.parametrize("dim", [1, 2])
def test_momenta_far_above_the_depths(dim, rates, lam):
    """Momenta up to 2^5 times the depths (further up the oracle's entropy variables lose digits):
    s c q in units of the depths' leaves the integers' range in some cells, near it in others.  One
    collision (a second one would divide by depths near zero)."""
    ny, nx, q = (1, 640, 5) if dim == 1 else (10, 640, 13)
    F0 = inputs.random_populations(q, ny, nx, seed=9720)
    nf = 3 if dim == 1 else 5
    F0[:nf] = 0.245 + 0.01 * (F0[:nf] - 0.25)
    F0[nf:] *= 1e-3
    big = inputs.uniform(9721, ny * nx, -1.0, 5.0).reshape(ny, nx)  # powers of two
    F0[nf] += 2.0 ** big
    if dim == 2:
        F0[11] -= 2.0 ** inputs.uniform(9722, ny * nx, -1.0, 5.0).reshape(ny, nx)
    bc, a = ((W, W), 0.15) if dim == 1 else ((P, P, W, W), 0.05)
    if rates is not None and dim == 1:
        rates = [0.0, rates[1], rates[3], 0.0, rates[10]]
    p = oracle.params(nx, ny, a=a, lam=lam, bc=bc, inflow=None, s_moments=rates)
    got = gpu_post(F0, 0, dim=dim, precision=lbm_sw.FP64, bc=bc, inflow=None, a=a, lam=lam, mrt_rates=rates)
    assert rel_max(got, oracle_post(F0, 0, p, dim)) <= FP64_TOL


@pytest.mark.parametrize("u", [0.0, 0.2])
@pytest.mark.parametrize("s", [1.0, 1.8, 1.95, 1.99])
def test_depths_and_momenta_do_not_drift(s, u):
    """The sums of depths and momenta over 20,000 periodic steps.  Each population is rounded to nearest
    once per step; unbiased roundings of half an ulp, 2^-54 of the depth, walk by about
    2^-54 sqrt(20000 / 56^2) = 1.4e-16 of the sum.  The bar is seven times that."""
    n = 56
    y, x = np.mgrid[0:n, 0:n]
    h = np.where(np.hypot(x - n / 2, y - n / 2) < 0.2 * n, 2.0, 1.0) + 1e-3 * inputs.uniform(9740, n * n).reshape(n, n)
    with lbm_sw.Simulation(n, n, precision=lbm_sw.FP64, s=s) as sim:
        sim.set_state(h, u * h, np.zeros_like(h))
        before = sim.populations()
        sim.step(20000)
        after = sim.populations()
    total = [[math.fsum(F[a:b].ravel()) for a, b in ((0, 5), (5, 9), (9, 13))] for F in (before, after)]
    for k in range(3):
        assert abs(total[1][k] - total[0][k]) <= 1e-15 * total[0][0], (k, total)


def test_1d_lakes_at_rest_keep_their_bits():
    """A uniform depth at rest between walls whose populations add up to it (rounded once) is a
    fixed point of f + s (f^eq - f): no bit changes in 1,000 steps."""
    kept = 0
    for h in inputs.uniform(9750, 150, 0.5, 3.0):
        with lbm_sw.Simulation(8, 1, dim=1, precision=lbm_sw.FP64, bc=(W, W), a=0.15) as sim:
            sim.set_state(np.full(8, h), np.zeros(8))
            F = sim.populations()
            sim.step(1000)
            if math.fsum(F.reshape(5, 8)[:3, 0]) == h:
                kept += 1
                assert np.array_equal(sim.populations(), F), h
    assert kept >= 140
