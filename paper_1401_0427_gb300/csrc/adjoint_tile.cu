// Several reverse steps of the discrete adjoint per launch on tiles held in registers, FP32, for the
// grids below the wavefronts': the tiles of tile2d.cu with the populations Phi pulled in the reverse
// direction (+x movers from x + 1, and so on), the transposed side rules of adjoint_step_vec, and
// the local product (1 - s) psi + s M^T D(W)^T psi with the moments W^{n-1} of each step, which a
// thread loads a step ahead.  One step per launch is bound by the launch and the dependent reads
// from L2: 4.4, 4.6 and 6.4 us per step at 128^2, 256^2 and 512^2, here 1.7, 1.9 and 3.9 (walls the
// same within 0.1), bound by the rows' chains and the recomputed halo.
// Two rows per thread and 16 warps, 128 registers: three rows and 12 warps, 168 registers, with the
// moments loaded behind their last use, took 2.0, 2.3 and 4.4 (walls 2.7, 2.8 and 4.9).
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "internal.h"
#include "scheme.cuh"
#include "step2d_vec.cuh"
#include "temporal.cuh"
#include "tile2d.cuh"

namespace lbm {
namespace {

constexpr int kRows = 2, kWarps = 16;

template <bool PER>
__global__ void __launch_bounds__(32 * kWarps, 1)
    adjoint_tile(const StepArgs<float> A, const float* __restrict__ w0, long long wslot, const Consts<float> Kc,
                 const TilePart P) {
  constexpr int R = kRows, NW = kWarps;
  __shared__ float2 edge[2][NW][2][3][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int strip = blockIdx.x % P.strips, seg = blockIdx.x / P.strips;
  const int nx = A.nx, ny = A.ny;
  const bool px = PER || A.bc[LBM_SW_SIDE_XM] == LBM_SW_BC_PERIODIC;
  const bool py = PER || A.bc[LBM_SW_SIDE_YM] == LBM_SW_BC_PERIODIC;
  const int tx = strip * P.w - P.hl + 2 * lane;
  const int y0 = seg * P.h, y1 = min(ny, y0 + P.h);
  const int ty = y0 - P.kb + warp * R;
  pdl_wait();

  int gx = tx, gx2 = tx + 1;
  if (px) {
    gx %= nx;
    if (gx < 0) gx += nx;
    gx2 = gx + 1 == nx ? 0 : gx + 1;
  }
  const bool split = (gx & 1) || gx2 != gx + 1;  // pairs at odd columns or across the seam (odd nx)
  const bool col_live = px || (gx >= 0 && gx < nx);
  long long row[R];  // of each row in a plane, -1: outside
#pragma unroll
  for (int r = 0; r < R; ++r) {
    int gy = ty + r;
    if (py) {
      gy %= ny;
      if (gy < 0) gy += ny;
    }
    row[r] = col_live && ty + r < y1 + P.kb && gy >= 0 && gy < ny ? static_cast<long long>(gy) * A.pitch : -1;
  }
  auto load = [&](const float* plane, int r, float outside) {
    if (row[r] < 0) return dup2(outside);
    const float* g = plane + row[r];
    return split ? make_float2(__ldg(g + gx), __ldg(g + gx2)) : __ldg(reinterpret_cast<const float2*>(g + gx));
  };
  float2 F[R][13], W[R][3], N[R][3];
#pragma unroll
  for (int r = 0; r < R; ++r) {
#pragma unroll
    for (int p = 0; p < 13; ++p) F[r][p] = load(A.src + p * A.plane, r, 0.f);
#pragma unroll
    for (int c = 0; c < 3; ++c) W[r][c] = load(w0 + c * A.plane, r, 1.f);
  }

  const int tx0 = strip * P.w - P.hl;
  const bool meets_x = !px && (tx0 <= 0 || tx0 + kTileCols >= nx);
  const bool meets_y = !py && (ty <= 0 || ty + R >= ny);
  const bool at_xm = tx == 0, at_xp_x = tx == nx - 1, at_xp_y = tx + 1 == nx - 1;
  const bool wxm = A.bc[LBM_SW_SIDE_XM] == LBM_SW_BC_WALL, oxm = A.bc[LBM_SW_SIDE_XM] == LBM_SW_BC_OUTFLOW;
  const bool wxp = A.bc[LBM_SW_SIDE_XP] == LBM_SW_BC_WALL, oxp = A.bc[LBM_SW_SIDE_XP] == LBM_SW_BC_OUTFLOW;
  const bool wym = A.bc[LBM_SW_SIDE_YM] == LBM_SW_BC_WALL, oym = A.bc[LBM_SW_SIDE_YM] == LBM_SW_BC_OUTFLOW;
  const bool wyp = A.bc[LBM_SW_SIDE_YP] == LBM_SW_BC_WALL, oyp = A.bc[LBM_SW_SIDE_YP] == LBM_SW_BC_OUTFLOW;
  const float oms = 1.f - Kc.s;

  for (int s = 1; s <= P.kb; ++s) {
    float2(*const e)[2][3][32] = edge[s & 1];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      e[warp][0][c][lane] = F[R - 1][4 + 4 * c];  // pulled by the row above
      e[warp][1][c][lane] = F[0][2 + 4 * c];      // pulled by the row below
    }
    __syncthreads();
    const int rem = P.kb - s;
    if (ty + R <= y0 - rem || ty >= y1 + rem) continue;
    if (s < P.kb)
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) N[r][c] = load(w0 - s * wslot + c * A.plane, r, 1.f);
    auto step = [&](auto xs, auto ys) {
      float2 below[3], above[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        below[c] = warp > 0 ? e[warp - 1][0][c][lane] : F[0][4 + 4 * c];
        above[c] = warp < NW - 1 ? e[warp + 1][1][c][lane] : F[R - 1][2 + 4 * c];
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        float a[13], b[13];  // psi of the two cells
        a[0] = F[r][0].x;
        b[0] = F[r][0].y;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float2 xp = F[r][1 + 4 * c], xm = F[r][3 + 4 * c], yp = F[r][2 + 4 * c], ym = F[r][4 + 4 * c];
          float pa = xp.y, pb = __shfl_down_sync(kFullMask, xp.x, 1);  // +x movers, from x + 1
          float ma = __shfl_up_sync(kFullMask, xm.y, 1), mb = xm.x;    // -x movers, from x - 1
          float2 up = r < R - 1 ? F[r < R - 1 ? r + 1 : 0][2 + 4 * c] : above[c];  // +y movers, from y + 1
          float2 dn = below[c];                                                    // -y movers, from y - 1
          if constexpr (decltype(xs)::value) {
            // the front sides' rules, then the OUTFLOW ghosts' own values
            const float wx = c == 1 ? -xm.x : xm.x, wy = c == 1 ? -xm.y : xm.y, w1 = c == 1 ? -xp.x : xp.x;
            pa = at_xp_x ? (wxp ? wx : 0.f) : pa;
            pb = at_xp_y ? (wxp ? wy : 0.f) : pb;
            ma = at_xm ? (wxm ? w1 : 0.f) : ma;
            pa = at_xm && oxm ? pa + xp.x : pa;
            ma = at_xp_x && oxp ? ma + xm.x : ma;
            mb = at_xp_y && oxp ? mb + xm.y : mb;
          }
          if constexpr (decltype(ys)::value) {
            const bool first = ty + r == 0, last = ty + r == ny - 1;
            up.x = last ? (wyp ? (c == 2 ? -ym.x : ym.x) : 0.f) : up.x;
            up.y = last ? (wyp ? (c == 2 ? -ym.y : ym.y) : 0.f) : up.y;
            dn.x = first ? (wym ? (c == 2 ? -yp.x : yp.x) : 0.f) : dn.x;
            dn.y = first ? (wym ? (c == 2 ? -yp.y : yp.y) : 0.f) : dn.y;
            up.x = first && oym ? up.x + yp.x : up.x;
            up.y = first && oym ? up.y + yp.y : up.y;
            dn.x = last && oyp ? dn.x + ym.x : dn.x;
            dn.y = last && oyp ? dn.y + ym.y : dn.y;
          }
          a[1 + 4 * c] = pa;
          b[1 + 4 * c] = pb;
          a[2 + 4 * c] = up.x;
          b[2 + 4 * c] = up.y;
          a[3 + 4 * c] = ma;
          b[3 + 4 * c] = mb;
          a[4 + 4 * c] = dn.x;
          b[4 + 4 * c] = dn.y;
          below[c] = ym;  // for row r + 1
        }
        float za[3], zb[3];
        equilibrium_vjp(W[r][0].x, W[r][1].x, W[r][2].x, a, Kc, za[0], za[1], za[2]);
        equilibrium_vjp(W[r][0].y, W[r][1].y, W[r][2].y, b, Kc, zb[0], zb[1], zb[2]);
#pragma unroll
        for (int c = 0; c < 3; ++c) W[r][c] = N[r][c];
#pragma unroll
        for (int p = 0; p < 13; ++p) {
          const int f = p < 5 ? 0 : (p < 9 ? 1 : 2);
          F[r][p] = make_float2(oms * a[p] + Kc.s * za[f], oms * b[p] + Kc.s * zb[f]);
        }
      }
    };
    using std::false_type;
    using std::true_type;
    if constexpr (PER) {
      step(false_type{}, false_type{});
    } else if (meets_x) {
      if (meets_y)
        step(true_type{}, true_type{});
      else
        step(true_type{}, false_type{});
    } else {
      if (meets_y)
        step(false_type{}, true_type{});
      else
        step(false_type{}, false_type{});
    }
  }
  pdl_done();

  if (2 * lane >= P.hl && 2 * lane < P.hl + P.w && tx < nx) {
    const bool both = tx + 1 < nx;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int y = ty + r;
      if (y < y0 || y >= y1) continue;
      float* g = A.dst + static_cast<long long>(y) * A.pitch + tx;
#pragma unroll
      for (int p = 0; p < 13; ++p) {
        if (both)
          *reinterpret_cast<float2*>(g + p * A.plane) = F[r][p];
        else
          g[p * A.plane] = F[r][p].x;
      }
    }
  }
}

}  // namespace

int adjoint_tile_steps(int nx, int ny, int sms) {
  int best = 4;
  double us = 1e300;
  for (int kb = 8; kb >= 3; --kb) {
    const TilePart P = tile_part(nx, ny, kRows * kWarps, kb, sms);
    const int waves = (P.strips * P.segs + sms - 1) / sms;
    const double per_step = waves * (0.22 * (P.h + 2 * kb) + 0.5 * kb) / kb;  // a row of a tile, and a step's barrier
    if (per_step < us) {
      us = per_step;
      best = kb;
    }
  }
  return best;
}

cudaError_t launch_adjoint_tile(const StepArgs<float>& a, const float* w0, long long wslot, const ConstsD& kd, int kb,
                                cudaStream_t st, int sms) {
  if (kb < 1 || kb > 8) return cudaErrorInvalidValue;
  const TilePart P = tile_part(a.nx, a.ny, kRows * kWarps, kb, std::max(sms, 1));
  const bool per = a.bc[LBM_SW_SIDE_XM] == LBM_SW_BC_PERIODIC && a.bc[LBM_SW_SIDE_YM] == LBM_SW_BC_PERIODIC;
  return launch_pdl(per ? adjoint_tile<true> : adjoint_tile<false>, dim3(P.strips * P.segs), dim3(32 * kWarps), 0, st, a,
                    w0, wslot, make_consts<float>(kd.g, kd.lambda, kd.s, kd.a), P);
}

}  // namespace lbm
