// How the s-rows of a cell go over the lanes of a warp and, for the streaming
// kernels, over the chunks of its ring (host only).
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>

namespace mmh {

// Rows a warp takes at once: packed, ceil(ns / 8) lanes of eight nodes each, or
// V nodes to a lane over a power of two of lanes.
inline int packed_rpp(int ns) { return 32 / ((ns + 7) / 8); }
inline int lane_rpp(int ns, int V) {
  int seg = 1;
  while (seg < ns / V) seg <<= 1;
  return 32 / seg;
}

struct RowPlan {
  bool packed;
  int rows, chunks;  // rows per chunk (the last may be shorter), chunks
  int passes;        // passes of rows over all chunks
};

// `total` rows of row_bytes each in chunks of at most chunk_bytes, each of them
// whole passes of rpp rows but the last (a pass is at most 2 KB): equal chunks that
// divide the rows left most lanes idle where they hold less than a pass (a row each
// for 31 or 37 orientations: up to 3.9 times the substep). Chunks of a whole
// number of 16-byte vectors, which bulk copies need, take up to four passes more.
inline RowPlan chunk_plan(bool packed, int total, size_t row_bytes, int rpp, int chunk_bytes) {
  int unit = rpp;
  while (unit * row_bytes % 16 != 0) unit += rpp;
  if ((size_t)unit * row_bytes > (size_t)chunk_bytes) unit = rpp;
  const int most = std::max<int>(1, (int)(chunk_bytes / (unit * row_bytes))) * unit;
  const int n = (total + most - 1) / most;
  RowPlan p;
  p.packed = packed;
  p.rows = std::min(total, ((total + n - 1) / n + unit - 1) / unit * unit);
  p.chunks = (total + p.rows - 1) / p.rows;
  const int last = total - (p.chunks - 1) * p.rows;
  p.passes = (p.chunks - 1) * ((p.rows + rpp - 1) / rpp) + (last + rpp - 1) / rpp;
  // equal chunks after all where they take no more passes
  const int even = total / n;
  if (even * n == total && n * ((even + rpp - 1) / rpp) <= p.passes &&
      (total * row_bytes % 16 != 0 || even * row_bytes % 16 == 0)) {
    p.rows = even;
    p.chunks = n;
  }
  return p;
}

// What a pass costs: the nodes of a lane times what one costs, whether the lane
// has a row or not. float64, bound by its pipe: 12.3 operations a node with eight
// nodes to a lane, 18 with two, 23 with one (the differences and fluxes at a lane's
// edges are formed once a lane). float32, bound by issue: alike.
inline double pass_cost(bool packed, int V, int tsz) {
  if (tsz == 4) return packed ? 8.0 : V;
  return packed ? 8 * 12.3 : V == 2 ? 2 * 18.0 : 23.0;
}

// Packed rows or V nodes to a lane, whichever costs less for `total` rows of ns
// nodes: packed wastes lanes on few rows (float64 8 x 8 a cell: 733 against 507 us),
// V nodes to a lane on rows that are no power of two of lanes (float32 48 x 36: 63
// against 49). float32 rows of a multiple of eight nodes have eight to a lane
// already (packing them leaves fewer idle lanes where their lanes are no power of
// two, but its remainders cost more: 400^2 x 24 x 24 343 against 266 us), and of no
// multiple of four are always packed (one node to a lane: 200 x 150 x 24 x 30 228
// against 69).
inline RowPlan row_plan(int total, int ns, int V, int tsz, int chunk_bytes) {
  const size_t row_bytes = (size_t)ns * tsz;
  const RowPlan p = chunk_plan(true, total, row_bytes, packed_rpp(ns), chunk_bytes);
  const RowPlan q = chunk_plan(false, total, row_bytes, lane_rpp(ns, V), chunk_bytes);
  if (tsz == 4 && V != 4) return V == 8 ? q : p;
  return p.passes * pass_cost(true, V, tsz) <= q.passes * pass_cost(false, V, tsz) ? p : q;
}

// Most bytes of Mb for which one resident launch (mm_resident.cu) of n substeps is
// taken rather than the streaming kernel. Up to 32 orientations, a lane each in the
// psi phase, it is the faster one up to 250 MB, twice the L2, where HBM comes to
// bound both (256^2 x 32^2 in us: 124 against 134; 256^2 x 64^2 498 against 390);
// beyond, a lane takes several and the streaming kernel wins earlier, the sooner
// the fuller its lanes: rows of a power of two of full lanes from 100 MB on (64
// orientations x 16: 80 MB 0.94 of its time, 140 MB 1.13, 245 MB 1.20; x 32 1.12 at
// 245 MB), of three quarters of one from 140 MB (x 24). Rows of no multiple of four
// nodes leave the streaming kernel the slower one up to what the resident plan
// holds at all (400^2 x 24 x 30, 460 MB: 244 against 331 us; beyond 32 orientations
// they part at 200 MB: 48 x 31 1.06 at 450 MB). A call of two substeps pays for
// loading and storing what is kept: half of the bytes (192^2 x 32^2, 151 MB, 85
// against 79 us a substep).
inline size_t resident_limit(int nth, int ns, int n) {
  size_t mb = 250;
  if (ns % 4 != 0) {
    if (nth <= 32) return SIZE_MAX;
    mb = 200;
  } else if (nth > 32 && ns % 8 == 0) {
    int seg = 1;
    while (seg < ns / 8) seg <<= 1;
    mb = ns / 8 == seg ? 100 : 4 * (ns / 8) >= 3 * seg ? 140 : 250;
  }
  return (mb << 20) / (n == 2 ? 2 : 1);
}

}  // namespace mmh
