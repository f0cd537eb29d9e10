// D1Q3Q2 kernels (section 2): populations f0, f+, f- (mass, D1Q3) and g+, g-
// (discharge, D1Q2; h_0^* does not depend on beta, so there is no g0).  One thread
// per cell; five planes of `pitch` elements, post-collision values.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "internal.h"
#include "scheme.cuh"

namespace lbm {
namespace {

// Value of population p (1: f+, 2: f-, 3: g+, 4: g-) streaming into cell i.
template <class T>
__device__ __forceinline__ T pull1(const StepArgs<T>& A, int p, int i) {
  const bool plus = (p == 1 || p == 3);  // moves +lambda: comes from i - 1
  const int is = plus ? i - 1 : i + 1;
  if (is >= 0 && is < A.nx) return A.src[p * A.plane + is];
  const int side = plus ? LBM_SW_SIDE_XM : LBM_SW_SIDE_XP;
  switch (A.bc[side]) {
    case LBM_SW_BC_PERIODIC:
      return A.src[p * A.plane + (plus ? A.nx - 1 : 0)];
    case LBM_SW_BC_WALL: {  // mirror of the boundary cell: f+ <-> f-, g+ <-> -g-
      const int m = (p == 1) ? 2 : (p == 2) ? 1 : (p == 3) ? 4 : 3;
      const T v = A.src[m * A.plane + i];
      return p >= 3 ? -v : v;
    }
    case LBM_SW_BC_OUTFLOW:
      return A.src[p * A.plane + i];
    default:
      return A.inflow_feq[side * 5 + p];
  }
}

template <class T, bool MRT>
__global__ void __launch_bounds__(256) step1d(const StepArgs<T> A, const Consts<T> K) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < A.nx; i += gridDim.x * blockDim.x) {
    T f[5];
    f[0] = A.src[i];
#pragma unroll
    for (int p = 1; p < 5; ++p) f[p] = pull1(A, p, i);
    collide5_any<T, MRT>(f, K);
#pragma unroll
    for (int p = 0; p < 5; ++p) A.dst[p * A.plane + i] = f[p];
  }
}

// ---- all n steps of a line in one launch: windows of cells in registers ----
//
// The line is cut into pieces of 32 - 2B cells.  One warp (a CTA of its own, so that the warps
// spread over the SMs) holds a piece and B cells on each side, one cell per lane, and advances
// them B steps with warp shuffles for the pulls: no shared memory and no barrier.  After s steps the window is exact but for s cells at each end that is not a
// physical boundary, which never reaches the piece within B steps.  Then the warp publishes the
// cells that its neighbours hold as halo, reads its own halo from theirs, and goes on.  Every
// cell update is the pull + collide of the per-step kernel on the same values: the same bits.
//
// What bounds it is the collision's chain of one warp: in FP64 every instruction takes 64 cycles
// of its quarter of an SM (half a lane per clock, whatever the number of active lanes), so the
// line is spread over as many quarters as it fills.  With the former collision (32 FP64 operations)
// 1000 cells took 1.23 us per step in FP64, against 1.44 with one cluster of 16 SMs (windows of
// 63 + 16 cells in shared memory, a cluster barrier per 8 steps), 16000 cells 1.66 against 9.82;
// with the one in integers 0.92 and 1.13.  FP32: 0.16 against 0.39 and 0.17 against 0.69.
//
// Exchange: a mailbox in global memory with two slots per cell, used by turns.  Each 8-byte
// word carries 4 bytes of payload and the number of the exchange, written and read as one
// access, so a reader that sees the number has the payload: one trip through L2 and no fence.  A
// slot is written again two exchanges later, when its writer has read the exchange between from
// the same neighbours, who had read the slot before they published that one.  The launch is
// cooperative, so every warp is resident; a wait gives up after `wait_polls` polls all the same.  A
// warp that gave up holds NaN from there on, and publishes it, and waits for nothing any more (a
// neighbour that misses an exchange for that gives up too): every cell that depends on what never
// came is stored as NaN, which diagnostics report, and every other cell is right.
constexpr int kWaitPolls = 1 << 22;
constexpr unsigned kAllLanes = 0xffffffffu;

template <class T>
struct MailWords;  // 8-byte words per value
template <>
struct MailWords<float> {
  static constexpr int n = 1;
};
template <>
struct MailWords<double> {
  static constexpr int n = 2;
};

__device__ __forceinline__ unsigned long long mail_word(unsigned payload, unsigned epoch) {
  return (static_cast<unsigned long long>(epoch) << 32) | payload;
}
__device__ __forceinline__ void mail_put(unsigned long long* w, float v, unsigned epoch) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(w), "l"(mail_word(__float_as_uint(v), epoch)) : "memory");
}
__device__ __forceinline__ void mail_put(unsigned long long* w, double v, unsigned epoch) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(v));
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(w),
               "l"(mail_word(static_cast<unsigned>(b), epoch)), "l"(mail_word(static_cast<unsigned>(b >> 32), epoch))
               : "memory");
}
__device__ __forceinline__ bool mail_get(const unsigned long long* w, float& v, unsigned epoch) {
  unsigned long long a;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(a) : "l"(w) : "memory");
  v = __uint_as_float(static_cast<unsigned>(a));
  return static_cast<unsigned>(a >> 32) == epoch;
}
__device__ __forceinline__ bool mail_get(const unsigned long long* w, double& v, unsigned epoch) {
  unsigned long long a, b;
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(w) : "memory");
  v = __longlong_as_double(static_cast<long long>((b << 32) | (a & 0xffffffffull)));
  return static_cast<unsigned>(a >> 32) == epoch && static_cast<unsigned>(b >> 32) == epoch;
}

template <class T, bool MRT>
__global__ void __launch_bounds__(32) step1d_windows(const StepArgs<T> A, const Consts<T> K, int nsteps, int B,
                                                     int wait_polls, unsigned long long* __restrict__ mail) {
  constexpr int MW = MailWords<T>::n;
  const int nx = A.nx;
  const int out = 32 - 2 * B;                   // cells of a piece
  const int o = blockIdx.x * out;               // this piece: cells [o, oe)
  const int oe = min(nx, o + out);
  const int g = o - B + static_cast<int>(threadIdx.x);          // this lane's cell
  const bool own = g >= o && g < oe;
  const bool per = A.bc[LBM_SW_SIDE_XM] == LBM_SW_BC_PERIODIC;  // periodic sides come in pairs
  const bool has_edge = !per && (o - B <= 0 || oe + B >= nx);   // warp-uniform: the window meets a side
  // the cell in the domain, -1: outside it, or further out than a halo (reaches no cell of the piece)
  int cell = per ? g % nx : g;
  if (per && cell < 0) cell += nx;
  if (cell < 0 || cell >= nx || g >= oe + B) cell = -1;
  T f[5];
#pragma unroll
  for (int p = 0; p < 5; ++p) f[p] = cell >= 0 ? A.src[p * A.plane + cell] : T(1);
  bool failed = false;
  unsigned epoch = 0;
  for (int done = 0; done < nsteps;) {
    const int kb = min(B, nsteps - done);
    for (int s = 0; s < kb; ++s) {
      // +lambda movers from the cell to the left, -lambda movers from the cell to the right
      T n[5] = {f[0], __shfl_up_sync(kAllLanes, f[1], 1), __shfl_down_sync(kAllLanes, f[2], 1),
                __shfl_up_sync(kAllLanes, f[3], 1), __shfl_down_sync(kAllLanes, f[4], 1)};
      if (has_edge && (cell == 0 || cell == nx - 1)) {
        if (cell == 0) {
          const int bc = A.bc[LBM_SW_SIDE_XM];
          if (bc == LBM_SW_BC_WALL) {  // mirror of the boundary cell: f+ <-> f-, g+ <-> -g-
            n[1] = f[2];
            n[3] = -f[4];
          } else if (bc == LBM_SW_BC_OUTFLOW) {
            n[1] = f[1];
            n[3] = f[3];
          } else {
            n[1] = A.inflow_feq[LBM_SW_SIDE_XM * 5 + 1];
            n[3] = A.inflow_feq[LBM_SW_SIDE_XM * 5 + 3];
          }
        }
        if (cell == nx - 1) {
          const int bc = A.bc[LBM_SW_SIDE_XP];
          if (bc == LBM_SW_BC_WALL) {
            n[2] = f[1];
            n[4] = -f[3];
          } else if (bc == LBM_SW_BC_OUTFLOW) {
            n[2] = f[2];
            n[4] = f[4];
          } else {
            n[2] = A.inflow_feq[LBM_SW_SIDE_XP * 5 + 2];
            n[4] = A.inflow_feq[LBM_SW_SIDE_XP * 5 + 4];
          }
        }
      }
      if (sizeof(T) == 4 || cell >= 0) {  // FP64 lanes outside keep their values (noise leaves the integers' path)
        collide5_any<T, MRT>(n, K);
#pragma unroll
        for (int p = 0; p < 5; ++p) f[p] = n[p];
      }
    }
    done += kb;
    if (done >= nsteps) break;
    ++epoch;
    unsigned long long* const w =
        mail + (static_cast<long long>(epoch & 1) * nx + max(cell, 0)) * static_cast<long long>(5 * MW);
    if (own && (g < o + B || g >= oe - B))  // cells that some neighbour holds as halo
#pragma unroll
      for (int p = 0; p < 5; ++p) mail_put(w + p * MW, f[p], epoch);
    __syncwarp();  // a window may wait for its own cells (a periodic line of one piece)
    if (cell >= 0 && !own) {
      for (int polls = 0;; ++polls) {
        bool ok = true;
#pragma unroll
        for (int p = 0; p < 5; ++p) ok &= mail_get(w + p * MW, f[p], epoch);
        if (ok) break;
        if (failed || polls >= wait_polls) {  // one exhausted wait ends the later ones at once
          failed = true;
          break;
        }
      }
    }
    failed = __any_sync(kAllLanes, failed);
    if (failed)
#pragma unroll
      for (int p = 0; p < 5; ++p) f[p] = T(NAN);
  }
  if (own)
#pragma unroll
    for (int p = 0; p < 5; ++p) A.dst[p * A.plane + g] = f[p];
}

template <class T>
__global__ void init1d(const StepArgs<T> A, const Consts<T> K, const double* __restrict__ h,
                       const double* __restrict__ hu) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < A.nx; i += gridDim.x * blockDim.x) {
    T e[5];
    equilibrium5(static_cast<T>(h[i]), static_cast<T>(hu[i]), K, e);
#pragma unroll
    for (int p = 0; p < 5; ++p) A.dst[p * A.plane + i] = e[p];
  }
}

template <class T, bool MRT>
__global__ void collide1d_dense(const StepArgs<T> A, const Consts<T> K, const T* __restrict__ dense) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < A.nx; i += gridDim.x * blockDim.x) {
    T f[5];
#pragma unroll
    for (int p = 0; p < 5; ++p) f[p] = dense[p * static_cast<long long>(A.nx) + i];
    collide5_any<T, MRT>(f, K);
#pragma unroll
    for (int p = 0; p < 5; ++p) A.dst[p * A.plane + i] = f[p];
  }
}

template <class T>
__global__ void moments1d(const StepArgs<T> A, double* __restrict__ h, double* __restrict__ hu) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < A.nx; i += gridDim.x * blockDim.x) {
    T f[5];
#pragma unroll
    for (int p = 0; p < 5; ++p) f[p] = A.src[p * A.plane + i];
    T d, q;
    moments5(f, d, q);
    h[i] = static_cast<double>(d);
    hu[i] = static_cast<double>(q);
  }
}

struct InflowStates1 {
  int bc[2];
  double w[2][2];
};

template <class T>
__global__ void inflow_feq1d(T* out, const InflowStates1 in, const Consts<T> K) {
  const int side = threadIdx.x;
  if (side >= 4) return;
  T e[5] = {T(0), T(0), T(0), T(0), T(0)};
  if (side < 2 && in.bc[side] == LBM_SW_BC_INFLOW)
    equilibrium5(static_cast<T>(in.w[side][0]), static_cast<T>(in.w[side][1]), K, e);
#pragma unroll
  for (int p = 0; p < 5; ++p) out[side * 5 + p] = e[p];
}

unsigned blocks_for(int n, int threads) {
  const long long b = (static_cast<long long>(n) + threads - 1) / threads;
  return static_cast<unsigned>(b < 65535 ? b : 65535);
}

}  // namespace

template <class T>
Consts<T> consts1(const ConstsD& kd) {
  return kd.mrt ? make_consts_mrt<T>(kd.g, kd.lambda, kd.s, kd.a, kd.rates, 3) : make_consts<T>(kd.g, kd.lambda, kd.s, kd.a);
}

template <class T>
cudaError_t launch_step1d(const StepArgs<T>& a, const ConstsD& kd, cudaStream_t st) {
  if (kd.mrt)
    step1d<T, true><<<blocks_for(a.nx, 128), 128, 0, st>>>(a, consts1<T>(kd));
  else
    step1d<T, false><<<blocks_for(a.nx, 128), 128, 0, st>>>(a, consts1<T>(kd));
  return cudaGetLastError();
}

template <class T>
size_t mail1d_bytes(int nx) {
  return static_cast<size_t>(2) * nx * 5 * MailWords<T>::n * sizeof(unsigned long long);
}

// Steps between exchanges (the halo's width) for a line of nx cells: an exchange takes about
// 0.5 us, so wide halos while the warps they make find free quarters of SMs (with some to spare: they
// are not dealt evenly), narrower ones (fewer warps) on longer lines.  FP64, us per step with halos
// of 4 / 6 / 8 / 10: 3000 cells 1.06 / 1.02 / 1.03 / 0.98, 8000 cells 1.08 / 1.01 / 1.00 / 1.25,
// 12000 cells 1.09 / 1.02 / 1.24 / 1.24, 16000 cells 1.34 / 1.30 / 1.26 / 1.63.  FP32 with 6 / 8 /
// 10: 3000 cells 0.20 / 0.18 / 0.16, 16000 cells 0.23 / 0.18 / 0.20.  Two or four cells per lane
// were slower at every length.
template <class T>
int window_halo(int nx, int sm_count) {
  auto pieces = [&](int b) { return (nx + 32 - 2 * b - 1) / (32 - 2 * b); };
  if constexpr (sizeof(T) == 8) {
    for (int b : {10, 8})
      if (2 * pieces(b) <= 7 * sm_count) return b;
    return pieces(6) <= 4 * sm_count ? 6 : 8;
  } else {
    return pieces(10) <= 4 * sm_count ? 10 : 8;
  }
}

// Few steps, with a halo of as many cells: nothing is exchanged, so the launch needs no cleared mailbox
// and no residency of all its warps.  Up to the halo that the line would have anyway, or 15 steps
// where every warp finds a quarter of an SM.  us per call of 1, 2, 8 and 11 steps with the exchange's launch / this way:
// 1000 cells FP64 8.2, 8.2, 12.3, 16.4 / 4.1, 4.3, 10.3, 12.3, FP32 8.2, 8.2, 8.2, 8.7 / 4.1 each.
template <class T>
int lone_halo(int nx, int nsteps, int sm_count) {
  if (nsteps <= window_halo<T>(nx, sm_count)) return nsteps;
  const int out = std::max(32 - 2 * nsteps, 1);
  return nsteps <= 15 && (nx + out - 1) / out <= 4 * sm_count ? nsteps : 0;
}

template <class T>
cudaError_t launch_step1d_windows(const StepArgs<T>& a, const ConstsD& kd, int nsteps, void* mail, int sm_count,
                                  cudaStream_t st) {
  const int lone = lone_halo<T>(a.nx, nsteps, sm_count);
  const int b = lone ? lone : window_halo<T>(a.nx, sm_count), out = 32 - 2 * b;
  const int pieces = (a.nx + out - 1) / out;
  const auto kernel = kd.mrt ? step1d_windows<T, true> : step1d_windows<T, false>;
  if (lone) {
    kernel<<<pieces, 32, 0, st>>>(a, consts1<T>(kd), nsteps, b, 0, nullptr);
    return cudaGetLastError();
  }
  if (pieces > 1 || a.bc[LBM_SW_SIDE_XM] == LBM_SW_BC_PERIODIC) {
    cudaError_t e = cudaMemsetAsync(mail, 0, mail1d_bytes<T>(a.nx), st);  // exchange numbers start at 1
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(pieces);
  cfg.blockDim = dim3(32);
  cfg.stream = st;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeCooperative;
  attr.val.cooperative = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, a, consts1<T>(kd), nsteps, b, kWaitPolls, static_cast<unsigned long long*>(mail));
}

template <class T>
cudaError_t launch_init1d(const StepArgs<T>& a, const ConstsD& kd, const double* h, const double* hu,
                          cudaStream_t st) {
  init1d<T><<<blocks_for(a.nx, 128), 128, 0, st>>>(a, make_consts<T>(kd.g, kd.lambda, kd.s, kd.a), h, hu);
  return cudaGetLastError();
}

template <class T>
cudaError_t launch_collide1d_dense(const StepArgs<T>& a, const ConstsD& kd, const T* dense, cudaStream_t st) {
  if (kd.mrt)
    collide1d_dense<T, true><<<blocks_for(a.nx, 128), 128, 0, st>>>(a, consts1<T>(kd), dense);
  else
    collide1d_dense<T, false><<<blocks_for(a.nx, 128), 128, 0, st>>>(a, consts1<T>(kd), dense);
  return cudaGetLastError();
}

template <class T>
cudaError_t launch_moments1d(const StepArgs<T>& a, double* h, double* hu, cudaStream_t st) {
  moments1d<T><<<blocks_for(a.nx, 128), 128, 0, st>>>(a, h, hu);
  return cudaGetLastError();
}

template <class T>
cudaError_t launch_inflow_feq1d(T* out, const int bc[4], const double inflow[4][3], const ConstsD& kd,
                                cudaStream_t st) {
  InflowStates1 in;
  for (int s = 0; s < 2; ++s) {
    in.bc[s] = bc[s];
    in.w[s][0] = inflow[s][0];
    in.w[s][1] = inflow[s][1];
  }
  inflow_feq1d<T><<<1, 32, 0, st>>>(out, in, make_consts<T>(kd.g, kd.lambda, kd.s, kd.a));
  return cudaGetLastError();
}

#define LBM_INSTANTIATE_1D(T)                                                                               \
  template cudaError_t launch_step1d<T>(const StepArgs<T>&, const ConstsD&, cudaStream_t);                 \
  template size_t mail1d_bytes<T>(int);                                                                     \
  template cudaError_t launch_step1d_windows<T>(const StepArgs<T>&, const ConstsD&, int, void*, int,        \
                                                cudaStream_t);                                              \
  template cudaError_t launch_init1d<T>(const StepArgs<T>&, const ConstsD&, const double*, const double*,   \
                                        cudaStream_t);                                                      \
  template cudaError_t launch_collide1d_dense<T>(const StepArgs<T>&, const ConstsD&, const T*, cudaStream_t); \
  template cudaError_t launch_moments1d<T>(const StepArgs<T>&, double*, double*, cudaStream_t);             \
  template cudaError_t launch_inflow_feq1d<T>(T*, const int[4], const double[4][3], const ConstsD&, cudaStream_t);

LBM_INSTANTIATE_1D(float)
LBM_INSTANTIATE_1D(double)

}  // namespace lbm
