// Launch shapes that must fit a fixed buffer (plain C++, no CUDA needed).
#pragma once

namespace topo {

constexpr int MAXB = 16;        // PARM / CARM columns
constexpr int RED_BLOCKS = 608; // blocks of a deterministic reduction, at most (4 x 152 SMs)
// float64 values in a context's buffer of per-block partial sums
constexpr long long PARTIALS = (long long)RED_BLOCKS * MAXB * MAXB;

// The mixed 3D sensitivity: a block owns SN_X x SN_Y element columns of zc
// layers and writes one partial sum.
constexpr int SN_X = 32, SN_Y = 4;

inline long long sensitivity_columns(int nx, int ny) {
  return (long long)((nx + SN_X - 1) / SN_X) * ((ny + SN_Y - 1) / SN_Y);
}
inline long long sensitivity_blocks(int nx, int ny, int nz, int zc) {
  return sensitivity_columns(nx, ny) * ((nz + zc - 1) / zc);
}
// Layers per block.  A chunk's first face is loaded and transformed again, so
// 16 as long as the blocks still fill the SMs (six resident on each), fewer on
// small grids; more only where the blocks would outnumber the partial sums
// (from 318 million elements on).
inline int sensitivity_chunk(int nx, int ny, int nz) {
  int zc = 16;
  while (zc > 1 && sensitivity_blocks(nx, ny, nz, zc) < 6 * 152) zc /= 2;
  while (zc < nz && sensitivity_blocks(nx, ny, nz, zc) > PARTIALS) zc *= 2;
  return zc;
}

}  // namespace topo
