"""Populations and rows between a handle and CUDA tensors: one kernel for all planes gives what the
host copies give."""

import numpy as np
import pytest

import wrapped_library
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


HOOK = r"""
#include <cuda_runtime.h>
extern "C" cudaError_t __real_cudaPointerGetAttributes(cudaPointerAttributes*, const void*);
extern "C" cudaError_t __real_cudaMemcpy2DAsync(void*, size_t, const void*, size_t, size_t, size_t, cudaMemcpyKind, cudaStream_t);
static const char *from = nullptr, *to = nullptr;
static int elsewhere_type = 0, elsewhere_device = 0, copies = 0;
// from now on memory in [p, p + n) answers as of this type on this device; returns the 2D copies so far
extern "C" __attribute__((visibility("default"))) int elsewhere(const char* p, size_t n, int type, int device) {
  from = p;
  to = p + n;
  elsewhere_type = type;
  elsewhere_device = device;
  return copies;
}
extern "C" cudaError_t __wrap_cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  const cudaError_t e = __real_cudaPointerGetAttributes(a, p);
  if (e == cudaSuccess && p >= from && p < to) {
    a->type = static_cast<cudaMemoryType>(elsewhere_type);
    a->device = elsewhere_device;
  }
  return e;
}
extern "C" cudaError_t __wrap_cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, cudaMemcpyKind k,
                                               cudaStream_t st) {
  ++copies;
  return __real_cudaMemcpy2DAsync(d, dp, s, sp, w, h, k, st);
}
"""


@pytest.fixture(scope="module")
def library(tmp_path_factory):
    return wrapped_library.link(str(tmp_path_factory.mktemp("elsewhere")), HOOK,
                                ["cudaPointerGetAttributes", "cudaMemcpy2DAsync"])


def test_memory_that_is_not_this_devices_goes_through_copies(library):
    """Only this device's memory (and managed memory) is dereferenced by a kernel; a peer's, host memory
    and unknown addresses go to the runtime's copies, which take or refuse them.  The memory here is
    this device's all the time; only the answer about it changes."""
    out = wrapped_library.run(library, r"""
lib.elsewhere.argtypes, lib.elsewhere.restype = [ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int, ctypes.c_int], ctypes.c_int
nx, ny = 36, 9
F0 = inputs.random_populations(13, ny, nx, seed=9600)
stream = torch.cuda.current_stream().cuda_stream
with lbm_sw.Simulation(nx, ny, precision=lbm_sw.FP64, stream=stream) as sim,      lbm_sw.Batch([(nx, ny)], precision=lbm_sw.FP64, stream=stream) as batch:
    z = np.zeros((ny, nx))
    batch.set_state(0, z + 1, z, z)
    sim.set_populations(F0)
    T = torch.zeros((13, ny, nx), dtype=torch.float64, device="cuda")
    n, counts, same = 8 * T.numel(), [], []
    # unregistered, host, this device's, another device's, managed
    for kind, device in ((0, 0), (1, 0), (2, 0), (2, 1), (3, 0)):
        T.zero_()
        calls = [lambda: sim.populations_into(T), lambda: sim.set_populations(T), lambda: sim.get_rows_into(0, ny, T),
                 lambda: sim.set_rows(0, ny, T),
                 lambda: lbm_sw.lbm_sw_batch_get_populations(batch.handle, 0, T.data_ptr(), True)]
        for i, call in enumerate(calls):
            before = lib.elsewhere(T.data_ptr(), n, kind, device)
            call()
            counts.append(lib.elsewhere(None, 0, 0, 0) - before)
            if i == 2:
                same.append(bool(np.array_equal(T.cpu().numpy(), F0)))
        same.append(bool(np.array_equal(sim.populations(), F0)))
print(json.dumps([counts, same]))
""")
    by_copies = [13] * 5
    assert out[0] == by_copies * 2 + [0] * 5 + by_copies + [0] * 5
    assert all(out[1])


def test_device_copies_can_be_captured():
    import torch

    nx, ny = 64, 12
    F0 = inputs.random_populations(13, ny, nx, seed=9610).astype(np.float32)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream), lbm_sw.Simulation(nx, ny, stream=torch_stream()) as sim:
        sim.set_populations(F0)
        out = torch.zeros((13, ny, nx), dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            sim.populations_into(out)
        sim.set_populations(2 * F0)
        graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), 2 * F0)
