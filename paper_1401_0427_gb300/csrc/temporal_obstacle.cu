// K fused D2Q5Q4Q4 steps per launch with solid cells inside the domain, FP32 BGK: the two-column
// wavefront (temporal_pair.cuh, OBST) with any sides and widths.
//
// One step per launch reads and writes 104 bytes per cell and update, and its masks' tests cost
// issue slots on top (50k MLUPS on 3000 x 2000 cells); the wavefront advances K steps per trip
// through HBM, and the faces' rule costs it some selects per cell and level.
#include <cuda_runtime.h>

#include <algorithm>

#include "internal.h"
#include "scheme.cuh"
#include "temporal.cuh"
#include "temporal_pair.cuh"

namespace lbm {
namespace {

// Four cells of a row per thread (the pitch is a multiple of 32), all of their bytes loaded at once; the
// pitch's padding gets zeros.  copy: also the mask itself ([ny][nx]), or nullptr.  us per call of lbm_sw_set_obstacle
// with one cell per thread, one neighbour after the other, and a copy of its own for the mask / this way (without any
// flags): device masks 512^2 16 / 12 (12), 3000 x 2000 43 / 22 (16), host masks 512^2 47 / 41 (36).
// W: rows of whole words that start on one (nx a multiple of 4).
template <bool W>
__global__ void __launch_bounds__(128)
    obstacle_flags_kernel(const unsigned char* __restrict__ solid, unsigned char* __restrict__ copy,
                          unsigned char* __restrict__ flags, int nx, int ny, long long pitch, bool px, bool py) {
  const int x0 = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
  if (x0 >= pitch) return;
  for (int y = blockIdx.y; y < ny; y += gridDim.y) {
    const unsigned char* const row = solid + static_cast<long long>(y) * nx;
    const unsigned char* const below = y > 0 ? row - nx : (py ? solid + static_cast<long long>(ny - 1) * nx : nullptr);
    const unsigned char* const above = y < ny - 1 ? row + nx : (py ? solid : nullptr);
    unsigned s[6], d[4], u[4];  // cells x0 - 1 .. x0 + 4, and those below and above
    auto word = [&](const unsigned char* r) { return r && x0 < nx ? *reinterpret_cast<const unsigned*>(r + x0) : 0u; };
    const unsigned w[3] = {W ? word(row) : 0, W ? word(below) : 0, W ? word(above) : 0};
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      if (W && i > 0 && i < 5) {
        s[i] = w[0] >> (8 * (i - 1)) & 255;
        continue;
      }
      int x = x0 - 1 + i;
      const bool wraps = x < 0 || x == nx;
      if (wraps) x = x < 0 ? nx - 1 : 0;
      s[i] = x < nx && (!wraps || px) ? row[x] : 0;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      d[i] = W ? w[1] >> (8 * i) & 255 : below && x0 + i < nx ? below[x0 + i] : 0;
      u[i] = W ? w[2] >> (8 * i) & 255 : above && x0 + i < nx ? above[x0 + i] : 0;
    }
    unsigned out = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const unsigned faces = (s[i] ? kSolidLeft : 0) | (s[i + 2] ? kSolidRight : 0) | (d[i] ? kSolidBelow : 0) |
                             (u[i] ? kSolidAbove : 0);
      // faces between solid cells mean nothing
      out |= (x0 + i >= nx ? 0 : s[i + 1] ? kSolidSelf : faces) << (8 * i);
    }
    *reinterpret_cast<unsigned*>(flags + static_cast<long long>(y) * pitch + x0) = out;
    if (W && copy && x0 < nx)
      *reinterpret_cast<unsigned*>(copy + static_cast<long long>(y) * nx + x0) = w[0];
    else if (copy)
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (x0 + i < nx) copy[static_cast<long long>(y) * nx + x0 + i] = static_cast<unsigned char>(s[i + 1]);
  }
}

// Every side periodic: the branch-free steady state (3000 x 2000: 35.8 us per step; the row loop
// unrolled by three 37.5).
// ODD as in temporal_mrt.cu (odd widths: 37.0).
template <int K, int COLS, int PF, bool L0R, bool PER, bool ODD>
__global__ void __launch_bounds__(COLS / 2, 2)
    step2d_temporal_obstacle(const StepArgs<float> A, const Consts<float> Kc, const Partition P,
                             const unsigned char* __restrict__ flags) {
  extern __shared__ __align__(16) float smem[];
  pdl_wait();
  run_segment(P, A.ny, [&](int strip, int ys, int ye) {
    pair_wave<K, COLS, PF, false, L0R, PER, false, ODD, false, PER, true>(A, Kc, smem, strip * P.w, P.w, ys, ye, nullptr,
                                                                           0, flags);
  });
  pdl_done();
}

template <int K, int COLS, int PF, bool L0R, bool ODD>
cudaError_t launch_obst_odd(const StepArgs<float>& a, const ConstsD& kd, const unsigned char* flags, cudaStream_t st,
                        int sm_count) {
  const size_t smem = PairShape<K, COLS, PF, L0R>::floats() * sizeof(float);
  const bool per = a.bc[LBM_SW_SIDE_XM] == LBM_SW_BC_PERIODIC && a.bc[LBM_SW_SIDE_YM] == LBM_SW_BC_PERIODIC;
  const auto fn =
      per ? step2d_temporal_obstacle<K, COLS, PF, L0R, true, ODD> : step2d_temporal_obstacle<K, COLS, PF, L0R, false, ODD>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  const int resident = cached_resident(reinterpret_cast<const void*>(fn), COLS / 2, smem);
  const Partition Q = pair_partition(a.nx, a.ny, K, COLS, resident * std::max(sm_count, 1));
  return launch_pdl(fn, dim3(Q.strips * Q.segments), dim3(COLS / 2), smem, st, a,
                    make_consts<float>(kd.g, kd.lambda, kd.s, kd.a), Q, flags);
}
template <int K, int COLS, int PF, bool L0R>
cudaError_t launch_obst(const StepArgs<float>& a, const ConstsD& kd, const unsigned char* flags, cudaStream_t st,
                        int sm_count) {
  return a.nx & 1 ? launch_obst_odd<K, COLS, PF, L0R, true>(a, kd, flags, st, sm_count)
                  : launch_obst_odd<K, COLS, PF, L0R, false>(a, kd, flags, st, sm_count);
}

}  // namespace

cudaError_t launch_obstacle_flags(const unsigned char* solid, unsigned char* copy, unsigned char* flags, int nx, int ny,
                                  long long pitch, const int bc[4], cudaStream_t st) {
  const dim3 grid(static_cast<unsigned>((pitch + 511) / 512), static_cast<unsigned>(std::min(ny, 65535)));
  const bool words = nx % 4 == 0 && reinterpret_cast<size_t>(solid) % 4 == 0 && reinterpret_cast<size_t>(copy) % 4 == 0;
  const auto kernel = words ? obstacle_flags_kernel<true> : obstacle_flags_kernel<false>;
  kernel<<<grid, 128, 0, st>>>(solid, copy, flags, nx, ny, pitch, bc[LBM_SW_SIDE_XM] == LBM_SW_BC_PERIODIC,
                                              bc[LBM_SW_SIDE_YM] == LBM_SW_BC_PERIODIC);
  return cudaGetLastError();
}

// The shapes of the walled BGK kernel (launch_k in temporal.cu).
cudaError_t launch_step2d_temporal_obstacle(const StepArgs<float>& a, const ConstsD& kd, const unsigned char* flags,
                                            int k, cudaStream_t st, int sm_count) {
  const long long cells = static_cast<long long>(a.nx) * a.ny;
  switch (k) {
    case 2: return launch_obst<2, 256, 2, true>(a, kd, flags, st, sm_count);
    case 4:
      return cells < (1LL << 21) ? launch_obst<4, 128, 2, true>(a, kd, flags, st, sm_count)
                                 : launch_obst<4, 256, 2, true>(a, kd, flags, st, sm_count);
    case 6:
      return cells < (1LL << 23) ? launch_obst<6, 128, 1, true>(a, kd, flags, st, sm_count)
                                 : launch_obst<6, 256, 1, true>(a, kd, flags, st, sm_count);
    default: return cudaErrorNotSupported;
  }
}

}  // namespace lbm
