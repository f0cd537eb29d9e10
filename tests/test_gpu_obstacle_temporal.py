"""Several steps per launch with solid cells (TEMPORAL, FP32 BGK): the bits of one step per launch."""

import numpy as np
import pytest

from paper_1401_0427_gb300 import inputs, lbm_sw

from gpu_helpers import gpu_post, torch_stream

pytestmark = pytest.mark.gpu

P, W, O, I = lbm_sw.PERIODIC, lbm_sw.WALL, lbm_sw.OUTFLOW, lbm_sw.INFLOW
INFLOW = [(1.3, 0.2, -0.1), (0.9, -0.15, 0.05), (1.1, 0.05, 0.12), (1.2, -0.08, -0.2)]


def _run(F0, steps, bc, solid, kernel, k=0):
    ny, nx = F0.shape[1:]
    with lbm_sw.Simulation(nx, ny, bc=bc, inflow=INFLOW, kernel=kernel, temporal_steps=k, stream=torch_stream()) as sim:
        sim.set_obstacle(solid)
        sim.set_populations(F0, form=lbm_sw.PRE_COLLISION)
        plan = sim.step_plan(steps)
        sim.step(steps)
        return sim.populations(), plan


@pytest.mark.parametrize("bc", [(P, P, P, P), (W, W, W, W), (O, O, O, O), (I, I, I, I), (I, O, W, W), (P, P, W, O)],
                         ids=lambda b: "".join("PWOI"[k] for k in b))
@pytest.mark.parametrize("nx,ny,fraction", [(1, 1, 0.5), (3, 2, 0.3), (7, 5, 0.3), (33, 17, 0.05), (130, 12, 0.25),
                                            (245, 9, 0.3), (257, 33, 0.02), (512, 40, 0.3), (300, 64, 1.0), (300, 64, 0.0)])
@pytest.mark.parametrize("k", [2, 4, 6, 8])
def test_fused_obstacles_equal_single_steps(nx, ny, fraction, bc, k):
    solid = inputs.random_obstacles(ny, nx, seed=960 + nx + ny, fraction=fraction)
    F0 = inputs.random_populations(13, ny, nx, seed=970 + nx + ny).astype(np.float32)
    for steps in (k, 3 * k + 1):
        a, _ = _run(F0, steps, bc, solid, lbm_sw.KERNEL_SIMPLE)
        b, plan = _run(F0, steps, bc, solid, lbm_sw.KERNEL_TEMPORAL, k)
        assert sum(plan) == steps and 1 < max(plan) <= min(k, 6)
        assert np.array_equal(a, b, equal_nan=True), steps


@pytest.mark.parametrize("nx,ny,steps", [(700, 640, 22), (1501, 1400, 20), (2900, 2900, 20)])
def test_fused_obstacles_on_the_default_shapes(nx, ny, steps):
    """AUTO: K = 4 in 128-column strips, K = 6 (and 4, 2 in the tail) in 128 and 256 columns."""
    solid = inputs.random_obstacles(ny, nx, seed=980, fraction=0.05)
    tile = inputs.random_populations(13, 96, nx, seed=985).astype(np.float32)
    F0 = np.ascontiguousarray(np.tile(tile, (1, ny // 96 + 1, 1))[:, :ny, :])
    a, _ = _run(F0, steps, (P, P, W, O), solid, lbm_sw.KERNEL_VEC)
    b, plan = _run(F0, steps, (P, P, W, O), solid, lbm_sw.KERNEL_AUTO)
    assert max(plan) > 1
    assert np.array_equal(a, b)


@pytest.mark.parametrize("mrt", [False, True], ids=["bgk", "mrt"])
@pytest.mark.parametrize("bc", [(P, P, P, P), (W, W, W, W), (I, O, W, W), (P, P, W, O)],
                         ids=lambda b: "".join("PWOI"[k] for k in b))
@pytest.mark.parametrize("nx,ny,fraction", [(1, 1, 0.5), (3, 2, 0.3), (33, 17, 0.05), (130, 12, 0.25), (97, 200, 0.3),
                                            (300, 64, 1.0), (300, 64, 0.0), (513, 500, 0.1)])
def test_tiles_with_obstacles_equal_single_steps(nx, ny, fraction, bc, mrt):
    """AUTO below 5 * 2^17 cells."""
    solid = inputs.random_obstacles(ny, nx, seed=990 + nx + ny, fraction=fraction)
    F0 = inputs.random_populations(13, ny, nx, seed=995 + nx + ny).astype(np.float32)
    rates = [0.0, 1.1, 1.2, 1.3, 1.4, 0.0, 1.5, 1.6, 1.7, 0.0, 1.75, 1.65, 0.9] if mrt else None
    for steps in (2, 8, 29):
        out = []
        for kernel in (lbm_sw.KERNEL_SIMPLE, lbm_sw.KERNEL_AUTO):
            with lbm_sw.Simulation(nx, ny, bc=bc, inflow=INFLOW, kernel=kernel, stream=torch_stream()) as sim:
                sim.set_relaxation(rates)
                sim.set_obstacle(solid)
                sim.set_populations(F0, form=lbm_sw.PRE_COLLISION)
                sim.step(steps)
                out.append(sim.populations())
        assert np.array_equal(out[0], out[1], equal_nan=True), steps


@pytest.mark.parametrize("bc", [(P, P, P, P), (W, W, W, W), (P, P, W, O), (W, O, P, P)], ids=lambda b: "".join("PWOI"[k] for k in b))
@pytest.mark.parametrize("nx,ny", [(1, 1), (2, 1), (3, 4), (4, 1), (4, 3), (5, 2), (32, 3), (63, 9), (64, 9), (66, 7), (130, 5),
                                   (516, 3), (1025, 2)])
def test_masks_from_host_and_device(nx, ny, bc):
    """The flags of the steps with obstacles come from host masks, device masks and device masks that do
    not start on a word alike: the bits of the kernel that reads the mask itself."""
    import torch

    solid = inputs.random_obstacles(ny, nx, seed=9400 + nx, fraction=0.4)
    F0 = inputs.random_populations(13, ny, nx, seed=9410 + nx)
    flat = torch.zeros(nx * ny + 1, dtype=torch.uint8, device="cuda")
    off = flat[1:]
    off.copy_(torch.from_numpy(np.ascontiguousarray(solid, dtype=np.uint8)).cuda().reshape(-1))
    masks = [solid, torch.from_numpy(np.ascontiguousarray(solid, dtype=np.uint8)).cuda(), off.reshape(ny, nx)]
    for precision in (lbm_sw.FP32, lbm_sw.FP64):
        kw = dict(dim=2, precision=precision, bc=bc, inflow=None, a=0.05)
        want = gpu_post(F0, 3, kernel=lbm_sw.KERNEL_SIMPLE, solid=solid, **kw)
        for mask in masks:
            assert np.array_equal(gpu_post(F0, 3, solid=mask, **kw), want)


@pytest.mark.parametrize("bc", [(P, P, P, P), (W, O, I, W)], ids=["periodic", "sides"])
@pytest.mark.parametrize("nx,ny", [(900, 800), (901, 760)])
def test_auto_takes_four_steps_on_middle_grids(nx, ny, bc):
    """AUTO from 5 * 2^17 cells on (three waves of register tiles and more): the wavefront of four
    steps in 128-column strips, and of two in the tail."""
    solid = inputs.random_obstacles(ny, nx, seed=990 + nx, fraction=0.03)
    F0 = np.concatenate([inputs.random_populations(13, 40, nx, seed=991)] * (ny // 40), axis=1).astype(np.float32)
    a, _ = _run(F0, 22, bc, solid, lbm_sw.KERNEL_SIMPLE)
    b, plan = _run(F0, 22, bc, solid, lbm_sw.KERNEL_AUTO)
    assert plan == [4] * 5 + [2]
    assert np.array_equal(a, b, equal_nan=True)
