"""A handle for which there is no host memory: an error code, not an exception through the C entry.

operator new is wrapped in a child process and fails at the n-th call inside lbm_sw_create, for each of
the allocations that a handle makes before its first CUDA call.  No GPU is needed."""

import wrapped_library

HOOK = r"""
#include <new>
extern "C" void* __real__Znwm(size_t);
static int left = -1;
extern "C" __attribute__((visibility("default"))) void fail_new_after(int calls) { left = calls; }
extern "C" void* __wrap__Znwm(size_t n) {
  if (left >= 0 && left-- == 0) throw std::bad_alloc();
  return __real__Znwm(n);
}
"""


def test_create_without_host_memory_returns_an_error(tmp_path):
    library = wrapped_library.link(str(tmp_path), HOOK, ["_Znwm"])
    out = wrapped_library.run(library, r"""
lib.fail_new_after.argtypes, lib.fail_new_after.restype = [ctypes.c_int], None
codes = []
for calls in range(3):  # the handle, its tape memory, the list that this joins
    p = lbm_sw.make_params(64, 64)
    h = ctypes.c_void_p()
    lib.fail_new_after(calls)
    codes.append(lib.lbm_sw_create(ctypes.byref(p), ctypes.byref(h)))
    lib.fail_new_after(-1)
print(json.dumps(codes))
""", on_gpu=False)
    assert out == [-6] * 3
