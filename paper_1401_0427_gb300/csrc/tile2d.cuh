// The cut of a grid into register tiles, shared by the steps (tile2d.cu) and the reverse steps of the
// adjoint (adjoint_tile.cu).
#pragma once

#include <algorithm>

namespace lbm {
namespace {

constexpr int kTileCols = 64;

// Output columns and rows per tile (w even), tiles per row of tiles, steps, left halo (kb
// rounded up to even, so that pairs start at even columns).
struct TilePart {
  int w, h, strips, segs, kb, hl;
};

// Tiles of a launch of kb steps: strips of equal even width, row segments for whole waves of
// one CTA per SM.
TilePart tile_part(int nx, int ny, int rows, int kb, int sms) {
  TilePart P;
  P.kb = kb;
  P.hl = kb + (kb & 1);
  const int wmax = (kTileCols - P.hl - kb) & ~1, hmax = rows - 2 * kb;
  P.strips = (nx + wmax - 1) / wmax;
  P.w = (nx + P.strips - 1) / P.strips;
  P.w += P.w & 1;
  P.strips = (nx + P.w - 1) / P.w;
  const int need = (ny + hmax - 1) / hmax;
  const int waves = (P.strips * need + sms - 1) / sms;
  const int segs = std::max(need, std::min(waves * sms / P.strips, (ny + 3) / 4));
  P.h = (ny + segs - 1) / segs;
  P.segs = (ny + P.h - 1) / P.h;
  return P;
}

}  // namespace
}  // namespace lbm
