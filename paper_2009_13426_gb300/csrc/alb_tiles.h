// Shape of a block's tile of nodes: 2^lg along x by block >> lg rows.
#pragma once

namespace alb {

// log2 of the tile's width, at least lg: doubled while half the rows would still
// hold a grid of ny rows, so that a flat grid's tiles keep their threads busy
// (a step of 16 tubes of 4000 x 1 nodes in one batch: 315 us with tiles of 32 x 8,
// seven threads of eight idle, 112 us with 256 x 1; 2000 x 2: 192 and 107 us).
inline int tile_lg(int lg, int block, int ny) {
  while ((1 << lg) < block && (block >> lg) >= 2 * (long long)ny) ++lg;
  return lg;
}

}  // namespace alb
