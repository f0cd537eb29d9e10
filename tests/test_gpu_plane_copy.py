"""Populations and rows between a handle and CUDA tensors: one kernel for all planes gives what the
host copies give."""

import numpy as np
import pytest

from paper_1401_0427_gb300 import inputs, lbm_sw

from gpu_helpers import torch_stream

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [lbm_sw.FP32, lbm_sw.FP64])
@pytest.mark.parametrize("nx,ny", [(1, 1), (2, 3), (4, 7), (31, 5), (32, 33), (129, 4), (513, 2), (2052, 3)])
@pytest.mark.parametrize("shift", [0, 1], ids=["aligned", "one element off"])
def test_device_copies_equal_host_copies(nx, ny, precision, shift):
    import torch

    dtype = torch.float32 if precision == lbm_sw.FP32 else torch.float64
    F0 = inputs.random_populations(13, ny, nx, seed=9500 + nx)
    with lbm_sw.Simulation(nx, ny, precision=precision, stream=torch_stream()) as sim:
        sim.set_populations(F0)
        want = sim.populations()
        flat = torch.full((13 * nx * ny + 2,), -1.0, dtype=dtype, device="cuda")
        out = flat[shift:shift + 13 * nx * ny]
        sim.populations_into(out)
        assert np.array_equal(out.cpu().numpy().reshape(want.shape), want)
        assert float(flat[13 * nx * ny + 1]) == -1.0 and (not shift or float(flat[0]) == -1.0)
        part = flat[shift:shift + 13 * nx]
        sim.get_rows_into(ny - 1, 1, part)
        assert np.array_equal(part.cpu().numpy().reshape(13, nx), want[:, -1])
        half = (out.reshape(13, ny, nx) * 0.5).contiguous()
        sim.set_rows(0, ny, half)
        sim.set_rows(0, 1, part)
        now = sim.populations()
        assert np.array_equal(now[:, 0], part.cpu().numpy().reshape(13, nx))
        assert np.array_equal(now[:, 1:], half.cpu().numpy()[:, 1:])
        sim.step(1)  # the padding of the rows is still zero: same step as from host copies
        a = sim.populations()
        sim.set_populations(now)
        sim.step(1)
        assert np.array_equal(sim.populations(), a, equal_nan=True)
