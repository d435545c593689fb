// mask_look.cuh -- which columns of a mask row the pipelined update looks at for a
// lane's node.  Apart from the kernel, so that the rule can be checked on the host
// for every row length: the mask is exactly nx * ny * nz bytes, and in the last row a
// column beyond nx would lie behind it.
#pragma once

namespace lbm {

// The column of node x itself.  Nodes beyond the row's end (lanes of a ragged tile
// that have no node) look at the last column.
__host__ __device__ constexpr int mask_column(int x, int nx) { return x < nx ? x : nx - 1; }

// The column beside the warp's 32 consecutive nodes: lane 0 (the first) looks to
// the left of its own, lane 31 to the right, with the wrap of a periodic row; other
// lanes have none and repeat their own.  A lane 31 at or beyond the row's last node looks
// at column 0, so that the wrapped neighbour of a last node in mid-warp is seen.
__host__ __device__ constexpr int mask_column_beside(int x, int nx, int lane) {
  const int c = mask_column(x, nx);
  return lane == 0    ? (c == 0 ? nx - 1 : c - 1)
         : lane == 31 ? (c == nx - 1 ? 0 : c + 1)
                      : c;
}

}  // namespace lbm
