// Shared pieces of the half-shell pair kernels (pair_f32.cu, pair_f64.cu).
//
// A CTA works on one pair cell and meets every unordered pair of neighbouring cells from exactly one
// side: its own cell and the 13 neighbour cells of a half shell, offsets (dx, dy, dz) with dz = +1, or
// dz = 0 and dy = +1, or dz = dy = 0 and dx = +1 (m_i >= 3 keeps them distinct modulo m_i). Cells
// adjacent in x are contiguous in the cell-sorted arrays, so the 14 cells are at most ten index ranges.
#pragma once

#include "fcm_internal.cuh"

namespace fcm {

constexpr int kPieces = 10;   // x ranges of a half shell: 5 rows, each split in two where it wraps in x

// Called by the 32 lanes of one warp: meta[2 q] = first cell-sorted index of piece q, meta[2 q + 1] = staged
// slots before it, meta[2 kPieces + 1] = all staged slots; shift[q] = the piece's periodic image. Lane l
// describes piece l: row l / 2, part l % 2 of a row that wraps in x. Row 0 is the own cell and its +x
// neighbour (the own cell first); rows 1 .. 4 are dy = +1 at dz = 0 and dy = -1, 0, +1 at dz = +1, cells
// cx - 1 .. cx + 1. A piece that a row does not need stays empty.
template <typename R>
__device__ inline void half_shell_pieces(const Geometry<R>& g, int cell, const int* __restrict__ cstart, int* meta,
                                         float4* shift) {
  const int lane = threadIdx.x & 31;
  const int mx = g.mcell[0], my = g.mcell[1], mz = g.mcell[2];
  const int cs = g.nsys > 1 ? cell / g.cells_per : 0;   // system of this cell (batched launches)
  const int cbase = cs * g.cells_per;
  const int lc = cell - cbase;
  const int cx = lc % mx, cy = (lc / mx) % my, cz = lc / (mx * my);
  const int r = lane >> 1, part = lane & 1;
  int xa = 0, xb = -1;   // cells xa .. xb of the row; empty when xb < xa
  float sx = 0.f;
  if (r == 0) {
    if (part == 0) { xa = cx; xb = (cx + 1 < mx) ? cx + 1 : cx; }
    else if (cx + 1 >= mx) { xa = 0; xb = 0; sx = (float)g.L[0]; }
  } else if (r < 5) {
    if (cx - 1 >= 0 && cx + 1 < mx) { if (part == 0) { xa = cx - 1; xb = cx + 1; } }
    else if (cx - 1 < 0) {
      if (part == 0) { xa = mx - 1; xb = mx - 1; sx = -(float)g.L[0]; } else { xa = 0; xb = 1; }
    } else {
      if (part == 0) { xa = mx - 2; xb = mx - 1; } else { xa = 0; xb = 0; sx = (float)g.L[0]; }
    }
  }
  const int yu = r == 1 ? cy + 1 : cy + r - 3, zu = r <= 1 ? cz : cz + 1;   // row 0: (cy, cz)
  const int yr = r == 0 ? cy : yu;
  int a = 0, cnt = 0;
  if (lane < kPieces && xb >= xa) {
    const int rowbase = cbase + mx * (pmod(yr, my) + my * pmod(zu, mz));
    a = cstart[rowbase + xa];
    cnt = cstart[rowbase + xb + 1] - a;
  }
  int pre = cnt;   // inclusive prefix over the pieces
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, pre, o);
    if (lane >= o) pre += v;
  }
  if (lane < kPieces) {
    meta[2 * lane] = a;
    meta[2 * lane + 1] = pre - cnt;
    const float sy = yr < 0 ? -(float)g.L[1] : (yr >= my ? (float)g.L[1] : 0.f);
    const float sz = zu < 0 ? -(float)g.L[2] : (zu >= mz ? (float)g.L[2] : 0.f);
    shift[lane] = make_float4(sx, sy, sz, 0.f);
  }
  if (lane == kPieces - 1) meta[2 * kPieces + 1] = pre;   // prefix sentinel
}

}  // namespace fcm
