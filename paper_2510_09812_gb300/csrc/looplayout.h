// Where the packets of a fused CG loop lie (cgloop.cu).
//
// A packet is recognised by the number of its exchange, and exchanges are numbered per mesh.  So the
// packets of a mesh must lie where no other mesh of the batch ever writes, whatever the solve: with a
// range that moved with the number of components, a mesh could find a neighbour's old packet under the
// number that it waits for.  Each mesh has three values per row, piece and aggregate, at the same place
// for block (three components) and scalar rows (several right-hand sides), and one per row for one.
#pragma once

#include <cstdint>

#ifndef GSPM_HD
#ifdef __CUDACC__
#define GSPM_HD __host__ __device__
#else
#define GSPM_HD
#endif
#endif

namespace gspm {

// p of block rows: component c of row j
GSPM_HD inline int64_t p_packet3(int64_t j, int c) { return 3 * j + c; }
// p of scalar rows, right-hand side c of row j.  Nothing of the mesh is in the address, so that it costs
// the gather no registers (with the mesh's first row and row count in it, spills made steps 3 % slower):
// one right-hand side has an array of its own, several lie by slices, [slice][right-hand side][32 rows]
// (a mesh has whole slices), beside the block rows' packets.
GSPM_HD inline int p_packet1(int j) { return j; }
GSPM_HD inline int p_packet1(int j, int c) { return j + 64 * (j >> 5) + 32 * c; }
// nc values of item i (an aggregate, or a piece of one) of a mesh whose items start at first
GSPM_HD inline int coarse_packet(int first, int i, int nc, int c) {
  return 3 * first + (i - first) * nc + c;
}

}  // namespace gspm
