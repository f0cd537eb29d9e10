"""Register tiles (AUTO on FP32 grids below 5 * 2^17 cells): several steps per launch give the
bits of one step per launch."""

import numpy as np
import pytest

from paper_1401_0427_gb300 import inputs, lbm_sw

from gpu_helpers import gpu_post

pytestmark = pytest.mark.gpu

P, W, O, I = lbm_sw.PERIODIC, lbm_sw.WALL, lbm_sw.OUTFLOW, lbm_sw.INFLOW
INFLOW = [(1.2, 0.1, 0.05), (0.9, -0.1, 0.02), (1.1, 0.03, 0.1), (1.0, 0.02, -0.1)]
RATES = [0.0, 1.1, 1.2, 1.3, 1.4, 0.0, 1.5, 1.6, 1.7, 0.0, 1.75, 1.65, 0.9]


@pytest.mark.parametrize("mrt", [None, RATES], ids=["bgk", "mrt"])
@pytest.mark.parametrize("bc", [(P, P, P, P), (W, W, W, W), (W, O, I, W), (I, W, P, P), (P, P, O, I)],
                         ids=lambda b: "".join("PWOI"[k] for k in b))
@pytest.mark.parametrize("nx,ny", [(1, 1), (2, 3), (7, 5), (48, 32), (53, 37), (63, 50), (64, 64), (97, 200),
                                   (300, 33), (512, 512), (809, 810)])
def test_tiles_equal_single_steps(nx, ny, bc, mrt):
    """Grids smaller than a tile, of a whole number of tiles and one cell more, odd widths (pairs
    across the seam, the last column alone in its pair), one wave of tiles and several."""
    F0 = inputs.random_populations(13, ny, nx, seed=9100 + nx + ny).astype(np.float32)
    for steps in (2, 3, 7, 8, 29):
        kw = dict(dim=2, precision=lbm_sw.FP32, bc=bc, inflow=INFLOW, a=0.05, mrt_rates=mrt)
        a = gpu_post(F0, steps, kernel=lbm_sw.KERNEL_VEC, **kw)
        b = gpu_post(F0, steps, **kw)
        assert np.array_equal(a, b, equal_nan=True), steps


def test_tile_launch_plan():
    """The launches are as even as they come and add up, and lbm_sw_step makes them."""
    with lbm_sw.Simulation(512, 512) as sim:
        sim.set_state(*inputs.circular_dam_break_2d(512, seed=1))
        for n in (1, 2, 9, 100, 1000):
            plan = sim.step_plan(n)
            assert sum(plan) == n and max(plan) <= 8 and max(plan) - min(plan) <= 1
            before = sim.info().kernel_launches
            sim.step(n)
            assert sim.info().kernel_launches - before == len(plan)


@pytest.mark.parametrize("nx,ny,bc,mrt,plan", [
    (700, 600, (P, P, P, P), None, [2]), (700, 600, (W, O, I, W), None, [2]), (701, 600, (W, O, I, W), None, [2]),
    (256, 319, (W, W, W, W), RATES, [2]), (256, 320, (W, W, W, W), RATES, [1, 1]), (256, 320, (P, P, P, P), RATES, [2]),
    (700, 600, (I, W, P, P), RATES, [1, 1]), (640, 620, (W, O, I, W), None, [2])])
def test_two_steps(nx, ny, bc, mrt, plan):
    """Two steps take what is fastest there: tiles, the wavefront (even widths from 3 * 2^17 cells on), or
    two single steps (MRT with sides from 5 * 2^14 cells on).  The same bits as one step per launch."""
    with lbm_sw.Simulation(nx, ny, bc=bc, inflow=INFLOW) as sim:
        if mrt:
            sim.set_relaxation(mrt)
        assert sim.step_plan(2) == plan
    F0 = inputs.random_populations(13, ny, nx, seed=9200 + nx + ny).astype(np.float32)
    kw = dict(dim=2, precision=lbm_sw.FP32, bc=bc, inflow=INFLOW, a=0.05, mrt_rates=mrt)
    assert np.array_equal(gpu_post(F0, 2, kernel=lbm_sw.KERNEL_VEC, **kw), gpu_post(F0, 2, **kw), equal_nan=True)


@pytest.mark.parametrize("bc", [(P, P, P, P), (W, O, I, W)], ids=["periodic", "sides"])
@pytest.mark.parametrize("nx,ny", [(640, 640), (700, 600), (701, 600), (1024, 512), (760, 740)])
def test_four_steps(nx, ny, bc):
    """Launches of four steps by tiles or by the wavefront, whichever is estimated faster: the same bits."""
    F0 = inputs.random_populations(13, ny, nx, seed=9300 + nx + ny).astype(np.float32)
    kw = dict(dim=2, precision=lbm_sw.FP32, bc=bc, inflow=INFLOW, a=0.05)
    for steps in (4, 8):
        assert np.array_equal(gpu_post(F0, steps, kernel=lbm_sw.KERNEL_VEC, **kw), gpu_post(F0, steps, **kw), equal_nan=True)
