// Conserved totals and health check of a population state.
//
// h, hu, hv of every cell in the storage precision (pair-symmetric sums) are accumulated in FP64,
// with the smallest h and the number of cells with NaN/Inf or h <= 0; warp shuffles, then shared
// memory reduce a block to one partial of 5 doubles, and the partials are folded in a fixed order:
// same input, same bits.  A handle's aligned planes take one launch (diag_once); any other pitch
// takes a pass of partials with scalar loads and a final one (allocation-free diagnostics).
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <type_traits>

#include "internal.h"
#include "scheme.cuh"

namespace lbm {
namespace {

constexpr int kThreads = 256;
constexpr int kMaxBlocks = 1216;  // 8 per SM on a 152-SM GB300
constexpr unsigned kFull = 0xffffffffu;

struct Acc {
  double h, hu, hv, hmin, bad;
};

__device__ __forceinline__ Acc combine(Acc a, const Acc& b) {
  a.h += b.h;
  a.hu += b.hu;
  a.hv += b.hv;
  a.hmin = fmin(a.hmin, b.hmin);
  a.bad += b.bad;
  return a;
}

__device__ __forceinline__ Acc warp_reduce(Acc a) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    Acc o;
    o.h = __shfl_down_sync(kFull, a.h, off);
    o.hu = __shfl_down_sync(kFull, a.hu, off);
    o.hv = __shfl_down_sync(kFull, a.hv, off);
    o.hmin = __shfl_down_sync(kFull, a.hmin, off);
    o.bad = __shfl_down_sync(kFull, a.bad, off);
    a = combine(a, o);
  }
  return a;
}

// Block-wide reduction of one Acc per thread; thread 0 returns the total.
__device__ __forceinline__ Acc block_reduce(Acc a) {
  __shared__ Acc warp_part[kThreads / 32];
  a = warp_reduce(a);
  const int w = threadIdx.x / 32, lane = threadIdx.x % 32;
  if (lane == 0) warp_part[w] = a;
  __syncthreads();
  if (w == 0) {
    a = lane < kThreads / 32 ? warp_part[lane] : Acc{0.0, 0.0, 0.0, DBL_MAX, 0.0};
    a = warp_reduce(a);
  }
  return a;
}

template <class T, int Q>
__global__ void __launch_bounds__(kThreads) diag_partials(const StepArgs<T> A, double* __restrict__ part) {
  Acc a{0.0, 0.0, 0.0, DBL_MAX, 0.0};
  for (int y = blockIdx.x; y < A.ny; y += gridDim.x) {
    const T* row = A.src + static_cast<long long>(y) * A.pitch;
    for (int x = threadIdx.x; x < A.nx; x += kThreads) {
      T h, qx, qy = T(0);
      if constexpr (Q == 13) {
        T f[13];
#pragma unroll
        for (int p = 0; p < 13; ++p) f[p] = row[p * A.plane + x];
        moments13(f, h, qx, qy);
      } else {
        T f[5];
#pragma unroll
        for (int p = 0; p < 5; ++p) f[p] = row[p * A.plane + x];
        moments5(f, h, qx);
      }
      const double hd = static_cast<double>(h), ud = static_cast<double>(qx), vd = static_cast<double>(qy);
      a.h += hd;
      a.hu += ud;
      a.hv += vd;
      a.hmin = fmin(a.hmin, hd);
      if (!(hd > 0.0) || !isfinite(hd) || !isfinite(ud) || !isfinite(vd)) a.bad += 1.0;
    }
  }
  a = block_reduce(a);
  if (threadIdx.x == 0) {
    double* o = part + 5 * blockIdx.x;
    o[0] = a.h;
    o[1] = a.hu;
    o[2] = a.hv;
    o[3] = a.hmin;
    o[4] = a.bad;
  }
}

// One launch for the handle's aligned layout: the warps take pieces of 32 V cells of a row by turns
// (V = 4 FP32 values of 16 bytes, or one FP64 value), each block writes a partial, and the block
// that finishes last folds the partials in their order and writes the result where the host
// reads it (pinned memory), so a check takes no second launch and no copy.  `done` counts the
// blocks and is zero again afterwards.  FP64 additions (64 cycles of a quarter of an SM each) bound
// it: three per cell, and those of the block's reduction; the tests are integer operations.
// 701 x 401 FP64: 31 us for the call, 40 with two launches, a copy and 256-thread rows; 4096^2 FP32
// 245 against 360.
template <class T, int Q>
__global__ void __launch_bounds__(kThreads)
    diag_once(const StepArgs<T> A, double* __restrict__ part, unsigned* __restrict__ done, double* __restrict__ out) {
  constexpr int V = sizeof(T) == 4 ? 4 : 1;
  using Vec = typename std::conditional<sizeof(T) == 4, float4, double>::type;
  const int lane = threadIdx.x % 32;
  const int chunks = (A.nx + 32 * V - 1) / (32 * V);
  const long long tasks = static_cast<long long>(A.ny) * chunks;
  Acc a{0.0, 0.0, 0.0, DBL_MAX, 0.0};
  unsigned bad = 0;
  for (long long task = blockIdx.x * (kThreads / 32) + threadIdx.x / 32; task < tasks; task += gridDim.x * (kThreads / 32)) {
    const long long y = task / chunks;
    const int x0 = static_cast<int>(task - y * chunks) * (32 * V) + lane * V;
    if (x0 >= A.nx) continue;
    const T* row = A.src + y * A.pitch;
    T f[Q][V];
#pragma unroll
    for (int p = 0; p < Q; ++p) {
      const Vec t = __ldg(reinterpret_cast<const Vec*>(row + p * A.plane + x0));
      const T* tv = reinterpret_cast<const T*>(&t);
#pragma unroll
      for (int k = 0; k < V; ++k) f[p][k] = tv[k];
    }
#pragma unroll
    for (int k = 0; k < V; ++k) {
      if (x0 + k >= A.nx) break;
      T h, qx, qy = T(0);
      T g[Q];
#pragma unroll
      for (int p = 0; p < Q; ++p) g[p] = f[p][k];
      if constexpr (Q == 13)
        moments13(g, h, qx, qy);
      else
        moments5(g, h, qx);
      const double hd = static_cast<double>(h), ud = static_cast<double>(qx), vd = static_cast<double>(qy);
      a.h += hd;
      a.hu += ud;
      a.hv += vd;
      a.hmin = fmin(a.hmin, hd);
      const long long hb = __double_as_longlong(hd);  // positive and finite: between 0 and infinity as integers
      if (hb <= 0 || hb >= 0x7ff0000000000000LL || (__double2hiint(ud) & 0x7ff00000) == 0x7ff00000 ||
          (__double2hiint(vd) & 0x7ff00000) == 0x7ff00000)
        ++bad;
    }
  }
  a.bad = bad;
  a = block_reduce(a);
  __shared__ bool last;
  if (threadIdx.x == 0) {
    double* o = part + 5 * blockIdx.x;
    o[0] = a.h;
    o[1] = a.hu;
    o[2] = a.hv;
    o[3] = a.hmin;
    o[4] = a.bad;
    __threadfence();
    last = atomicInc(done, gridDim.x - 1) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  a = Acc{0.0, 0.0, 0.0, DBL_MAX, 0.0};
  for (int b = threadIdx.x; b < gridDim.x; b += kThreads) {
    const volatile double* o = part + 5 * b;
    a = combine(a, Acc{o[0], o[1], o[2], o[3], o[4]});
  }
  a = block_reduce(a);
  if (threadIdx.x == 0) {
    out[0] = a.h;
    out[1] = a.hu;
    out[2] = a.hv;
    out[3] = a.hmin;
    out[4] = a.bad;
  }
}

__global__ void __launch_bounds__(kThreads) diag_final(const double* __restrict__ part, int nblocks,
                                                      double* __restrict__ out) {
  Acc a{0.0, 0.0, 0.0, DBL_MAX, 0.0};
  for (int b = threadIdx.x; b < nblocks; b += kThreads) {
    const double* o = part + 5 * b;
    a = combine(a, Acc{o[0], o[1], o[2], o[3], o[4]});
  }
  a = block_reduce(a);
  if (threadIdx.x == 0) {
    out[0] = a.h;
    out[1] = a.hu;
    out[2] = a.hv;
    out[3] = a.hmin;
    out[4] = a.bad;
  }
}

}  // namespace

int diag_max_blocks() { return kMaxBlocks; }

template <class T>
cudaError_t launch_diagnostics(const StepArgs<T>& a, int q, double* partials, unsigned* done, double* out, int sms,
                               cudaStream_t st) {
  constexpr int V = sizeof(T) == 4 ? 4 : 1, kWarps = kThreads / 32;
  const long long tasks = static_cast<long long>(a.ny) * ((a.nx + 32 * V - 1) / (32 * V));
  // two blocks per SM: enough loads in flight, few reductions (four and eight: slower)
  const int blocks = static_cast<int>(std::min<long long>((tasks + kWarps - 1) / kWarps, std::min(2 * sms, kMaxBlocks)));
  if (q == 13)
    diag_once<T, 13><<<blocks, kThreads, 0, st>>>(a, partials, done, out);
  else
    diag_once<T, 5><<<blocks, kThreads, 0, st>>>(a, partials, done, out);
  return cudaGetLastError();
}

template <class T>
cudaError_t launch_diagnostics_blocks(const StepArgs<T>& a, int q, int nblocks, double* partials, double* out,
                                      cudaStream_t st) {
  if (q == 13)
    diag_partials<T, 13><<<nblocks, kThreads, 0, st>>>(a, partials);
  else
    diag_partials<T, 5><<<nblocks, kThreads, 0, st>>>(a, partials);
  diag_final<<<1, kThreads, 0, st>>>(partials, nblocks, out);
  return cudaGetLastError();
}

template cudaError_t launch_diagnostics<float>(const StepArgs<float>&, int, double*, unsigned*, double*, int, cudaStream_t);
template cudaError_t launch_diagnostics<double>(const StepArgs<double>&, int, double*, unsigned*, double*, int, cudaStream_t);
template cudaError_t launch_diagnostics_blocks<float>(const StepArgs<float>&, int, int, double*, double*,
                                                      cudaStream_t);
template cudaError_t launch_diagnostics_blocks<double>(const StepArgs<double>&, int, int, double*, double*,
                                                       cudaStream_t);

}  // namespace lbm
