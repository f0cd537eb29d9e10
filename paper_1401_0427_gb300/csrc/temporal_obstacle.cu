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

// The pitch's padding gets zeros.
__global__ void obstacle_flags_kernel(const unsigned char* __restrict__ solid, unsigned char* __restrict__ flags, int nx,
                                      int ny, long long pitch, bool px, bool py) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= pitch) return;
  for (int y = blockIdx.y; y < ny; y += gridDim.y) {
    unsigned b = 0;
    if (x < nx) {
      const unsigned char* row = solid + static_cast<long long>(y) * nx;
      if (row[x]) b |= kSolidSelf;
      if (x > 0 ? row[x - 1] : (px && row[nx - 1])) b |= kSolidLeft;
      if (x < nx - 1 ? row[x + 1] : (px && row[0])) b |= kSolidRight;
      if (y > 0 ? row[x - nx] : (py && solid[static_cast<long long>(ny - 1) * nx + x])) b |= kSolidBelow;
      if (y < ny - 1 ? row[x + nx] : (py && solid[x])) b |= kSolidAbove;
      if (b & kSolidSelf) b = kSolidSelf;  // faces between solid cells mean nothing
    }
    flags[static_cast<long long>(y) * pitch + x] = static_cast<unsigned char>(b);
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

cudaError_t launch_obstacle_flags(const unsigned char* solid, unsigned char* flags, int nx, int ny, long long pitch,
                                  const int bc[4], cudaStream_t st) {
  const dim3 grid(static_cast<unsigned>((pitch + 127) / 128), static_cast<unsigned>(std::min(ny, 65535)));
  obstacle_flags_kernel<<<grid, 128, 0, st>>>(solid, flags, nx, ny, pitch, bc[LBM_SW_SIDE_XM] == LBM_SW_BC_PERIODIC,
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
