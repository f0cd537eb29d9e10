"""1D windows whose neighbour never publishes its borders: the wait runs out, and every cell that
depends on the missing borders is NaN; no other cell changes.

A small program compiled here launches the kernel without the CTA of one piece of the line and with a
short limit, next to the one-step kernel on the whole line.  Nothing waits without an end."""

import os
import subprocess

import pytest

from paper_1401_0427_gb300 import build as libbuild

pytestmark = pytest.mark.gpu

DRIVER = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "kernels_1d.cu"
using namespace lbm;

template <class T>
int run(int nx, int bc, int nsteps, int polls) {
  StepArgs<T> a{};
  a.nx = nx;
  a.ny = 1;
  a.pitch = a.plane = (nx + 31) / 32 * 32;
  a.bc[LBM_SW_SIDE_XM] = a.bc[LBM_SW_SIDE_XP] = bc;
  const size_t bytes = 5 * a.plane * sizeof(T);
  std::vector<T> f(5 * a.plane, T(0)), want(f), got(f);
  for (int i = 0; i < nx; ++i) {
    const double h = 1.0 + 0.3 * std::sin(0.37 * i), p = h * h / 32.0;
    const double e[5] = {0.075 * h, 0.4625 * h, 0.4625 * h, p, -p};
    for (int k = 0; k < 5; ++k) f[k * a.plane + i] = static_cast<T>(e[k]);
  }
  T *s0, *s1, *d;
  void *mail, *in;
  cudaMalloc(&s0, bytes);
  cudaMalloc(&s1, bytes);
  cudaMalloc(&d, bytes);
  cudaMalloc(&in, 20 * sizeof(T));
  cudaMemset(in, 0, 20 * sizeof(T));
  cudaMalloc(&mail, mail1d_bytes<T>(nx));
  a.inflow_feq = static_cast<T*>(in);
  const ConstsD kd{1.0, 8.0, 1.8, 0.15};
  // the whole line, one step per launch
  cudaMemcpy(s0, f.data(), bytes, cudaMemcpyHostToDevice);
  T *from = s0, *to = s1;
  for (int n = 0; n < nsteps; ++n, std::swap(from, to)) {
    a.src = from;
    a.dst = to;
    if (launch_step1d<T>(a, kd, 0) != cudaSuccess) return 2;
  }
  cudaMemcpy(want.data(), from, bytes, cudaMemcpyDeviceToHost);
  // without its last piece
  cudaMemcpy(s0, f.data(), bytes, cudaMemcpyHostToDevice);
  cudaMemset(d, 0, bytes);
  cudaMemset(mail, 0, mail1d_bytes<T>(nx));
  a.src = s0;
  a.dst = d;
  const int b = 8, out = 32 - 2 * b, pieces = (nx + out - 1) / out;
  step1d_windows<T, false><<<pieces - 1, 32>>>(a, consts1<T>(kd), nsteps, b, polls, static_cast<unsigned long long*>(mail));
  if (cudaDeviceSynchronize() != cudaSuccess) return 3;
  cudaMemcpy(got.data(), d, bytes, cudaMemcpyDeviceToHost);
  int nan = 0, wrong = 0, right = 0;
  const int end = (pieces - 1) * out;
  for (int i = 0; i < end; ++i)
    for (int k = 0; k < 5; ++k) {
      const T g = got[k * a.plane + i], w = want[k * a.plane + i];
      if (std::isnan(g))
        ++nan;
      else if (g == w)
        ++right;
      else
        ++wrong;
    }
  std::printf("%d %d %d %d\n", end * 5, nan, right, wrong);
  return 0;
}

int main(int, char** v) {
  const int nx = std::atoi(v[2]), bc = std::atoi(v[3]), n = std::atoi(v[4]);
  return v[1][0] == 'd' ? run<double>(nx, bc, n, 2000) : run<float>(nx, bc, n, 2000);
}
"""


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    folder = str(tmp_path_factory.mktemp("waits"))
    src, exe = os.path.join(folder, "waits.cu"), os.path.join(folder, "waits")
    with open(src, "w") as f:
        f.write(DRIVER)
    r = subprocess.run([libbuild.nvcc(), *libbuild.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-I", libbuild.CSRC,
                        "-I", libbuild.INCLUDE, src, "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


@pytest.mark.parametrize("bc", [0, 1], ids=["periodic", "walls"])
@pytest.mark.parametrize("nsteps", [9, 20, 61])
@pytest.mark.parametrize("kind", ["float", "double"])
def test_no_finite_value_depends_on_a_border_that_never_came(driver, kind, nsteps, bc):
    nx = 168  # ten pieces of 16 cells and one of 8, which is left out
    out = subprocess.run([driver, kind, str(nx), str(bc), str(nsteps)], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stderr
    values, nan, right, wrong = map(int, out.stdout.split())
    assert wrong == 0 and nan + right == values
    # the neighbours of the missing piece (two on a periodic line) know from the first exchange on
    assert nan >= 16 * 5 * (1 if bc else 2)
    # NaN reaches a piece further, and no more, with every exchange
    if nsteps == 9:
        assert nan == 16 * 5 * (1 if bc else 2)
