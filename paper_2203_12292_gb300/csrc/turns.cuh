// Additions of a warp's lanes into the DoF buffer of a tile, in a fixed order.
// No CUDA header is needed, so the order can be checked on the host as well.
#pragma once

namespace gcmg {

// x[i] += v[i] for the C nodes of one slot: lanes whose slot starts at the same
// DoF take turns in lane order (rank and turns come with the tile: finding the
// lanes that meet with a match over the warp's addresses at every node was the
// largest part of a hanging tile: Q4 sphere postsmoothing 311 -> 261 us with the
// turns and the hanging lines dealt evenly to the warps).
//   Lanes also meet across slots: node k of one cell is node 0 of its neighbour.
// Every call therefore ends with the warp together, so the additions of one slot
// are complete before those of the next, and their order is the program's
// whatever the lanes ran apart on before (a hanging line interpolated by some of
// them).  turns is uniform over the warp, and all its lanes call.
template <int C, typename T>
__device__ __forceinline__ void add_turns(T* x, const T* v, int rank, int turns) {
  if (turns <= 1) {
#pragma unroll
    for (int i = 0; i < C; ++i) x[i] += v[i];
    __syncwarp();
    return;
  }
#pragma unroll 1
  for (int q = 0; q < turns; ++q) {
    if (rank == q) {
#pragma unroll
      for (int i = 0; i < C; ++i) x[i] += v[i];
    }
    __syncwarp();
  }
}

}  // namespace gcmg
