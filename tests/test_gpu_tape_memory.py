"""Tapes and what they keep where device memory is short: a tape whose memory for the moments of every
step is not there falls back to checkpoints, and kept memory makes room for others.

cudaMalloc is wrapped: requests above a limit go to the real cudaMalloc as a request of 2^60 bytes,
which fails and leaves the runtime's last error as an exhausted device would, without using memory."""

import pytest

import wrapped_library

pytestmark = pytest.mark.gpu

HOOK = r"""
#include <cuda_runtime.h>
#include <map>
extern "C" cudaError_t __real_cudaMalloc(void**, size_t);
static cudaError_t count(cudaError_t e, void** p, size_t n);
extern "C" size_t set_budget(size_t bytes);
static bool fits(size_t n);
static size_t limit = ~size_t(0);
static int refused = 0;
extern "C" __attribute__((visibility("default"))) int refuse_above(size_t bytes) {
  limit = bytes;
  return refused;
}
extern "C" cudaError_t __wrap_cudaMalloc(void** p, size_t n) {
  if (n <= limit && fits(n)) return count(__real_cudaMalloc(p, n), p, n);
  ++refused;
  return __real_cudaMalloc(p, size_t(1) << 60);
}

// a device of `budget` bytes for blocks of 64 KB and more
extern "C" cudaError_t __real_cudaFree(void*);
static std::map<void*, size_t> blocks;
static size_t held = 0, budget = ~size_t(0);
extern "C" __attribute__((visibility("default"))) size_t set_budget(size_t bytes) {
  budget = bytes;
  return held;
}
static bool fits(size_t n) { return n < 65536 || held + n <= budget; }
static cudaError_t count(cudaError_t e, void** p, size_t n) {
  if (e == cudaSuccess && n >= 65536) {
    blocks[*p] = n;
    held += n;
  }
  return e;
}
extern "C" cudaError_t __wrap_cudaFree(void* p) {
  auto b = blocks.find(p);
  if (b != blocks.end()) {
    held -= b->second;
    blocks.erase(b);
  }
  return __real_cudaFree(p);
}
"""

LIMIT = """
lib.refuse_above.argtypes, lib.refuse_above.restype = [ctypes.c_size_t], ctypes.c_int
lib.set_budget.argtypes, lib.set_budget.restype = [ctypes.c_size_t], ctypes.c_size_t
NEVER = 2 ** 64 - 1
"""


@pytest.fixture(scope="module")
def library(tmp_path_factory):
    return wrapped_library.link(str(tmp_path_factory.mktemp("refusing")), HOOK,
                                ["cudaMalloc", "cudaFree"])


@pytest.mark.parametrize("precision", ["FP32", "FP64"])
def test_without_memory_for_the_moments_the_tape_takes_checkpoints(library, precision):
    """The record and the gradient after a refused allocation of the moments of 200 steps; the
    gradient agrees with that of a tape that keeps them as gradients of other launch splits do."""
    out = wrapped_library.run(library, LIMIT + r"""
prec = lbm_sw.%s
nx, ny, steps = 96, 64, 200
W0 = [x.reshape(ny, nx) for x in inputs.random_states(nx * ny, seed=7, h=(0.95, 1.05), speed=0.02)]
with lbm_sw.Simulation(nx, ny, precision=prec, stream=torch.cuda.current_stream().cuda_stream) as sim:
    plane = sim.info().pitch * ny
    all_steps = 3 * (steps + 1) * plane * np.dtype(sim.dtype).itemsize
    grads, kept = [], []
    for limit in (NEVER, all_steps):
        before = lib.refuse_above(limit)
        sim.set_state(*W0)
        with lbm_sw.Tape(sim, steps) as tape:
            tape.record()
            grads.append(tape.adjoint(sim.moments()[0] - 1.0))
            kept.append(tape.info().replay_bytes >= all_steps)
        refused = lib.refuse_above(NEVER) - before
        # the kept memory of the first tape would serve the second
        sim.close()
        sim.__init__(nx, ny, precision=prec, stream=torch.cuda.current_stream().cuda_stream)
print(json.dumps({"kept": kept, "refused": refused, "off": float(np.abs(grads[0] - grads[1]).max() / np.abs(grads[0]).max())}))
""" % precision)
    assert out["kept"] == [True, False] and out["refused"] >= 1
    assert out["off"] <= (1e-5 if precision == "FP32" else 1e-12)


def test_releasing_a_tape_waits_for_its_work():
    """lbm_sw_tape_destroy synchronises the owner's stream, also where it keeps the tape's memory: a
    gradient on the device may then be read on any other stream."""
    import torch

    from paper_1401_0427_gb300 import inputs, lbm_sw

    nx = ny = 512
    W0 = [x.reshape(ny, nx) for x in inputs.random_states(nx * ny, seed=8, h=(0.95, 1.05), speed=0.02)]
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream), lbm_sw.Simulation(nx, ny, stream=stream.cuda_stream) as sim:
        g = torch.full((ny, nx), 1e-3, dtype=torch.float64, device="cuda")
        for _ in range(3):
            sim.set_state(*W0)
            tape = lbm_sw.Tape(sim, 400)
            tape.record()
            tape.adjoint(g)
            assert not stream.query()  # 400 reverse steps: more than a millisecond
            tape.close()
            assert stream.query()


def test_kept_tape_memory_makes_room_for_other_allocations(library):
    """What a handle keeps for its next tape is freed when another handle, a batch, or another
    handle's tape finds no memory; what still does not fit is refused with out of memory, and the
    next calls go on."""
    out = wrapped_library.run(library, LIMIT + r"""
nx, ny, steps = 128, 128, 60
W0 = [x.reshape(ny, nx) for x in inputs.random_states(nx * ny, seed=9, h=(0.95, 1.05), speed=0.02)]
stream = torch.cuda.current_stream().cuda_stream
def new():
    return lbm_sw.Simulation(nx, ny, stream=stream)
def gradient(sim):
    sim.set_state(*W0)
    with lbm_sw.Tape(sim, steps) as tape:
        tape.record()
        return tape.adjoint(sim.moments()[0] - 1.0)
log = []
a, b = new(), new()
b.set_state(*W0)
first = gradient(a)
kept = lib.set_budget(NEVER)
def tight(call):
    gradient(a)                       # a keeps its tape's memory again
    lib.set_budget(lib.set_budget(NEVER))  # nothing more fits beside what is held
    got = call()
    held = lib.set_budget(NEVER)
    log.append(held < kept + 13 * 4 * nx * ny)
    return got
tight(lambda: new()).close()
tight(lambda: lbm_sw.Batch([(64, 64)], stream=stream)).close()
same = tight(lambda: gradient(b))
log.append(bool(np.array_equal(same, first)))
lib.set_budget(0)
try:
    new()
    log.append(False)
except lbm_sw.LbmSwError as e:
    log.append(e.status == lbm_sw.E_NOMEM and "out of memory" in str(e))
b.step(1)
lib.set_budget(NEVER)
log.append(bool(np.array_equal(gradient(a), first)))
print(json.dumps(log))
""")
    assert all(out), out
