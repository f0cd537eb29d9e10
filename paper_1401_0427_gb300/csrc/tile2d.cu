// Several D2Q5Q4Q4 steps per launch on tiles held in registers, FP32 (small and middle grids).
//
// A CTA holds a tile of 64 columns x NW R rows: warp w has R consecutive rows, lane l columns
// 2l and 2l + 1 of each.  It loads the 13
// planes of the tile, kb columns and rows of halo included, straight into registers, advances
// them kb steps, and stores the columns and rows that are still exact.  Per step a population
// moves along x by a warp shuffle, along y inside a warp by naming another register, and from
// warp to warp through shared memory (three planes of one row each way, one barrier per step).
// Halo cells are recomputed: a step makes one column and one row less exact on every side that
// is not a side of the domain.
//
// The row wavefront (temporal_pair.cuh) reads and computes less, but has 2K rows of fill per row
// segment and runs its K levels one after the other; one step per launch is bound by L2 and the
// launches.  Here a launch of 6 steps on 512^2 cells takes 11 us (150 tiles, one per SM): about
// 0.17 us per row of a tile for the loads and the collisions' chains, 0.5 us per step for the
// exchange of rows and the barrier.  us per step, one step per launch or the wavefront against
// this: 64^2 2.3 / 0.68, 256^2 2.8 / 0.92, 512^2 4.3 / 1.87, 724^2 4.2 / 3.5 (periodic), 512^2
// with inflow, outflow and walls 4.4 / 2.5; MRT 4.7 / 3.2; from about 850^2 on the wavefront wins
// (1024^2: 5.9 / 7.5).
//
// The collision is the scalar one on both cells of a lane: the paired instructions read two
// registers per operand and wait for register ports (a paired fused multiply-add with three
// register operands takes 4.6 cycles of a scheduler, two scalar ones 3.1), and the lanes of a
// pair that moves along x would have to change halves (2.22 -> 1.87 us per step at 512^2).
//
// Every cell update is the pull + collide of the single-step kernels on the same values, so kb
// steps equal kb single steps bit for bit.
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

// OBST: solid cells (kSolid* flags): a population that would come from a solid cell is the cell's
// own reflected one, the family normal to the face negated; solid cells keep their populations.
// STORE_W: the moments (h, hu, hv) of every step are also written, for the tile's output cells, to
// the three planes at wout + (step - 1) * wslot (the record of the discrete adjoint).
template <int R, int NW, bool MRT, bool PER, bool OBST, bool STORE_W>
__global__ void __launch_bounds__(32 * NW, 1)
    step2d_tile(const StepArgs<float> A, const Consts<float> Kc, const TilePart P,
                const unsigned char* __restrict__ flags, float* __restrict__ wout, long long wslot) {
  extern __shared__ __align__(16) float2 smem2[];
  float2(*const edge)[NW][2][3][32] = reinterpret_cast<float2(*)[NW][2][3][32]>(smem2);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int strip = blockIdx.x % P.strips, seg = blockIdx.x / P.strips;
  const int nx = A.nx, ny = A.ny;
  const bool px = PER || A.bc[LBM_SW_SIDE_XM] == LBM_SW_BC_PERIODIC;
  const bool py = PER || A.bc[LBM_SW_SIDE_YM] == LBM_SW_BC_PERIODIC;
  const int tx = strip * P.w - P.hl + 2 * lane;  // this lane's first column
  const int y0 = seg * P.h, y1 = min(ny, y0 + P.h);
  const int ty = y0 - P.kb + warp * R;           // this warp's first row
  pdl_wait();

  float2 F[R][13];
  unsigned solid[R];  // flags of the rows' two cells (bits 0 .. 4 and 8 .. 12)
  {
    int gx = tx, gx2 = tx + 1, gy = ty;
    if (px) {
      gx %= nx;
      if (gx < 0) gx += nx;
      gx2 = gx + 1 == nx ? 0 : gx + 1;
    }
    if (py) {
      gy %= ny;
      if (gy < 0) gy += ny;
    }
    // pairs at odd columns or across the seam (odd nx) load their lanes one by one
    const bool split = (gx & 1) || gx2 != gx + 1;
    const bool col_live = px || (gx >= 0 && gx < nx);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const bool live = col_live && ty + r < y1 + P.kb && (py || (gy >= 0 && gy < ny));
      const long long row = static_cast<long long>(gy) * A.pitch;
      if (OBST) solid[r] = live ? flags[row + gx] | (gx2 < nx ? flags[row + gx2] << 8 : 0) : 0u;
      if (live && !split) {
#pragma unroll
        for (int p = 0; p < 13; ++p)
          F[r][p] = __ldg(reinterpret_cast<const float2*>(A.src + p * A.plane + row + gx));
      } else if (live) {
#pragma unroll
        for (int p = 0; p < 13; ++p)
          F[r][p] = make_float2(__ldg(A.src + p * A.plane + row + gx), __ldg(A.src + p * A.plane + row + gx2));
      } else {
#pragma unroll
        for (int p = 0; p < 13; ++p) F[r][p] = make_float2(1.f, 1.f);  // reaches no cell of the output
      }
      ++gy;
      if (py && gy == ny) gy = 0;
    }
  }

  // Sides of the domain that this warp's cells meet (warp-uniform), the lanes that hold them, and
  // the values of INFLOW sides.  The rules are selects inside the row loop, in a copy of the
  // step's code for the warps that meet an x side, a y side or both: branches between the rows
  // would keep the code generator from overlapping them.
  const int tx0 = strip * P.w - P.hl;
  const bool meets_x = !px && (tx0 <= 0 || tx0 + kTileCols >= nx);
  const bool meets_y = !py && (ty <= 0 || ty + R >= ny);
  const bool at_xm = tx == 0, at_xp_x = tx == nx - 1, at_xp_y = tx + 1 == nx - 1;
  const bool wxm = A.bc[LBM_SW_SIDE_XM] == LBM_SW_BC_WALL, oxm = A.bc[LBM_SW_SIDE_XM] == LBM_SW_BC_OUTFLOW;
  const bool wxp = A.bc[LBM_SW_SIDE_XP] == LBM_SW_BC_WALL, oxp = A.bc[LBM_SW_SIDE_XP] == LBM_SW_BC_OUTFLOW;
  const bool wym = A.bc[LBM_SW_SIDE_YM] == LBM_SW_BC_WALL, oym = A.bc[LBM_SW_SIDE_YM] == LBM_SW_BC_OUTFLOW;
  const bool wyp = A.bc[LBM_SW_SIDE_YP] == LBM_SW_BC_WALL, oyp = A.bc[LBM_SW_SIDE_YP] == LBM_SW_BC_OUTFLOW;
  const float* const in = A.inflow_feq;

  for (int s = 1; s <= P.kb; ++s) {
    float2(*const e)[2][3][32] = edge[s & 1];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      e[warp][0][c][lane] = F[R - 1][2 + 4 * c];
      e[warp][1][c][lane] = F[0][4 + 4 * c];
    }
    __syncthreads();
    // rows that the remaining steps need: a warp with none of them waits
    const int rem = P.kb - s;
    if (ty + R <= y0 - rem || ty >= y1 + rem) continue;
    auto step = [&](auto xs, auto ys) {
      float2 below[3], above[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        below[c] = warp > 0 ? e[warp - 1][0][c][lane] : F[0][2 + 4 * c];
        above[c] = warp < NW - 1 ? e[warp + 1][1][c][lane] : F[R - 1][4 + 4 * c];
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        float a[13], b[13];  // the two cells' pulled populations
        a[0] = F[r][0].x;
        b[0] = F[r][0].y;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float2 xp = F[r][1 + 4 * c], xm = F[r][3 + 4 * c], yp = F[r][2 + 4 * c], ym = F[r][4 + 4 * c];
          float l = __shfl_up_sync(kFullMask, xp.y, 1), rr = __shfl_down_sync(kFullMask, xm.x, 1), mid = xm.y;
          float2 dn = below[c], up = r < R - 1 ? F[r < R - 1 ? r + 1 : 0][4 + 4 * c] : above[c];
          if constexpr (decltype(xs)::value) {
            const float vm = wxm ? (c == 1 ? -xm.x : xm.x) : oxm ? xp.x : in[LBM_SW_SIDE_XM * 13 + 1 + 4 * c];
            const float ip = in[LBM_SW_SIDE_XP * 13 + 3 + 4 * c];
            const float vx = wxp ? (c == 1 ? -xp.x : xp.x) : oxp ? xm.x : ip;
            const float vy = wxp ? (c == 1 ? -xp.y : xp.y) : oxp ? xm.y : ip;
            l = at_xm ? vm : l;
            mid = at_xp_x ? vx : mid;
            rr = at_xp_y ? vy : rr;
          }
          if constexpr (decltype(ys)::value) {
            const float im = in[LBM_SW_SIDE_YM * 13 + 2 + 4 * c], ip = in[LBM_SW_SIDE_YP * 13 + 4 + 4 * c];
            const bool first = ty + r == 0, last = ty + r == ny - 1;
            dn.x = first ? (wym ? (c == 2 ? -ym.x : ym.x) : oym ? yp.x : im) : dn.x;
            dn.y = first ? (wym ? (c == 2 ? -ym.y : ym.y) : oym ? yp.y : im) : dn.y;
            up.x = last ? (wyp ? (c == 2 ? -yp.x : yp.x) : oyp ? ym.x : ip) : up.x;
            up.y = last ? (wyp ? (c == 2 ? -yp.y : yp.y) : oyp ? ym.y : ip) : up.y;
          }
          float lb = xp.x;
          if constexpr (OBST) {
            const unsigned q = solid[r];
            l = q & kSolidLeft ? (c == 1 ? -xm.x : xm.x) : l;
            lb = q & kSolidLeft << 8 ? (c == 1 ? -xm.y : xm.y) : lb;
            mid = q & kSolidRight ? (c == 1 ? -xp.x : xp.x) : mid;
            rr = q & kSolidRight << 8 ? (c == 1 ? -xp.y : xp.y) : rr;
            dn.x = q & kSolidBelow ? (c == 2 ? -ym.x : ym.x) : dn.x;
            dn.y = q & kSolidBelow << 8 ? (c == 2 ? -ym.y : ym.y) : dn.y;
            up.x = q & kSolidAbove ? (c == 2 ? -yp.x : yp.x) : up.x;
            up.y = q & kSolidAbove << 8 ? (c == 2 ? -yp.y : yp.y) : up.y;
          }
          a[1 + 4 * c] = l;
          b[1 + 4 * c] = lb;
          a[3 + 4 * c] = mid;
          b[3 + 4 * c] = rr;
          a[2 + 4 * c] = dn.x;
          b[2 + 4 * c] = dn.y;
          a[4 + 4 * c] = up.x;
          b[4 + 4 * c] = up.y;
          below[c] = yp;  // for row r + 1
        }
        float2 h, qx, qy;
        collide13_any<float, MRT>(a, Kc, h.x, qx.x, qy.x);
        collide13_any<float, MRT>(b, Kc, h.y, qx.y, qy.y);
        if constexpr (STORE_W) {
          if (2 * lane >= P.hl && 2 * lane < P.hl + P.w && tx < nx && ty + r >= y0 && ty + r < y1) {
            float* const g = wout + (s - 1) * wslot + static_cast<long long>(ty + r) * A.pitch + tx;
            if (tx + 1 < nx) {
              *reinterpret_cast<float2*>(g) = h;
              *reinterpret_cast<float2*>(g + A.plane) = qx;
              *reinterpret_cast<float2*>(g + 2 * A.plane) = qy;
            } else {
              g[0] = h.x;
              g[A.plane] = qx.x;
              g[2 * A.plane] = qy.x;
            }
          }
        }
#pragma unroll
        for (int p = 0; p < 13; ++p) {
          F[r][p].x = OBST && (solid[r] & kSolidSelf) ? F[r][p].x : a[p];
          F[r][p].y = OBST && (solid[r] & kSolidSelf << 8) ? F[r][p].y : b[p];
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

  const int col = 2 * lane;
  if (col >= P.hl && col < P.hl + P.w && tx < nx) {
    const bool both = tx + 1 < nx;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int y = ty + r;
      if (y < y0 || y >= y1) continue;
      float* g = A.dst + static_cast<long long>(y) * A.pitch + tx;
      if (both) {
#pragma unroll
        for (int p = 0; p < 13; ++p) *reinterpret_cast<float2*>(g + p * A.plane) = F[r][p];
      } else {
#pragma unroll
        for (int p = 0; p < 13; ++p) g[p * A.plane] = F[r][p].x;
      }
    }
  }
}

// The tile of 48 rows (BGK 12 warps of 4 rows, MRT 16 warps of 3, whose transforms want the
// registers) or of 32 (16 warps of 2: less latency per step where a wave of them covers the
// grid), by the time in us per launch fitted to grids of 64^2 to 800^2: a wave of tiles takes
// 0.165 per loaded row and 0.5 per step (48 rows), 0.22 and 0.14 (32 rows).
struct TileChoice {
  TilePart P;
  bool tall;
  double us;
};
TileChoice tile_choose(int nx, int ny, int kb, int sms) {
  TileChoice best{};
  for (const bool tall : {true, false}) {
    const TilePart P = tile_part(nx, ny, tall ? 48 : 32, kb, sms);
    const int waves = (P.strips * P.segs + sms - 1) / sms, rows = P.h + 2 * kb;
    const double us = waves * (tall ? 0.165 * rows + 0.5 * kb : 0.22 * rows + 0.14 * kb);
    if (tall || us < best.us) best = {P, tall, us};
  }
  return best;
}

struct TileExtra {
  const unsigned char* flags;
  float* wout;
  long long wslot;
};

template <int R, int NW, bool MRT, bool OBST, bool STORE_W>
cudaError_t launch_tile(const StepArgs<float>& a, const ConstsD& kd, const TilePart& P, const TileExtra& x,
                        cudaStream_t st) {
  constexpr size_t smem = sizeof(float2) * 2 * NW * 2 * 3 * 32;
  static_assert(smem <= 48 * 1024, "dynamic shared memory without an attribute");
  const bool per = a.bc[LBM_SW_SIDE_XM] == LBM_SW_BC_PERIODIC && a.bc[LBM_SW_SIDE_YM] == LBM_SW_BC_PERIODIC;
  return launch_pdl(per ? step2d_tile<R, NW, MRT, true, OBST, STORE_W> : step2d_tile<R, NW, MRT, false, OBST, STORE_W>,
                    dim3(P.strips * P.segs), dim3(32 * NW), smem, st, a, to_consts<float>(kd), P, x.flags, x.wout, x.wslot);
}

template <bool OBST>
cudaError_t launch_tile_choice(const StepArgs<float>& a, const ConstsD& kd, const TileChoice& c, const TileExtra& x,
                               cudaStream_t st) {
  if (c.tall)
    return kd.mrt ? launch_tile<3, 16, true, OBST, false>(a, kd, c.P, x, st)
                  : launch_tile<4, 12, false, OBST, false>(a, kd, c.P, x, st);
  return kd.mrt ? launch_tile<2, 16, true, OBST, false>(a, kd, c.P, x, st)
                : launch_tile<2, 16, false, OBST, false>(a, kd, c.P, x, st);
}

}  // namespace

int tile_steps(int nx, int ny, int sms, int* waves) {
  int best = 8;
  double us = 1e300;
  for (int kb = 8; kb >= 4; --kb) {
    const TileChoice c = tile_choose(nx, ny, kb, sms);
    if (c.us / kb < us) {
      us = c.us / kb;
      best = kb;
      if (waves) *waves = (c.P.strips * c.P.segs + sms - 1) / sms;
    }
  }
  return best;
}

// Launches of four steps on grids of 3 to 5 * 2^17 cells took 0.82 to 0.98 of tile_choose's fit periodic, 0.93 to 1.2 with
// sides.
double tile4_us(int nx, int ny, bool periodic, int sms) {
  return tile_choose(nx, ny, 4, std::max(sms, 1)).us * (periodic ? 0.91 : 1.07);
}

cudaError_t launch_step2d_tile(const StepArgs<float>& a, const ConstsD& kd, int kb, const unsigned char* flags,
                               cudaStream_t st, int sms) {
  if (kb < 1 || kb > 8) return cudaErrorInvalidValue;
  const TileChoice c = tile_choose(a.nx, a.ny, kb, std::max(sms, 1));
  const TileExtra x{flags, nullptr, 0};
  return flags ? launch_tile_choice<true>(a, kd, c, x, st) : launch_tile_choice<false>(a, kd, c, x, st);
}

cudaError_t launch_step2d_tile_store_w(const StepArgs<float>& a, const ConstsD& kd, int kb, float* wout, long long wslot,
                                       cudaStream_t st, int sms) {
  if (kb < 1 || kb > 8 || kd.mrt) return cudaErrorInvalidValue;
  const TileChoice c = tile_choose(a.nx, a.ny, kb, std::max(sms, 1));
  const TileExtra x{nullptr, wout, wslot};
  return c.tall ? launch_tile<4, 12, false, false, true>(a, kd, c.P, x, st)
                : launch_tile<2, 16, false, false, true>(a, kd, c.P, x, st);
}

}  // namespace lbm
