// Where the packets of a fused CG loop lie (cgloop.cu).
//
// A packet is recognised by the number of its exchange, and exchanges are numbered per mesh.  So the
// packets of a mesh must lie where no other mesh of the batch ever writes, whatever the solve: with a
// range that moved with the number of components, a mesh could find a neighbour's old packet under the
// number that it waits for.  Each mesh has three values per row, piece and aggregate, at the same place
// for block (three components) and scalar rows (one to three right-hand sides).
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define GSPM_HD __host__ __device__
#else
#define GSPM_HD
#endif

namespace gspm {

// p of block rows: component c of row j
GSPM_HD inline int64_t p_packet3(int64_t j, int c) { return 3 * j + c; }
// p of scalar rows: right-hand side c of row j, of a mesh of `rows` rows (whole slices) from row0
GSPM_HD inline int64_t p_packet1(int64_t row0, int64_t rows, int64_t j, int c) {
  return 2 * row0 + c * rows + j;
}
// nc values of item i (an aggregate, or a piece of one) of a mesh whose items start at first
GSPM_HD inline int64_t coarse_packet(int64_t first, int64_t i, int nc, int c) {
  return 3 * first + (i - first) * nc + c;
}

}  // namespace gspm
