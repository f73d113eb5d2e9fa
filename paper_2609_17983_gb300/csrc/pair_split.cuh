// pair_split.cuh -- which cluster of the paired GEMM computes what, and which of them
// waits for which.  Needs no CUDA header, so that a test can compile it alone.
#pragma once

#ifdef __CUDACC__
#define KVR_HD __host__ __device__
#else
#define KVR_HD
#endif

namespace kvr {

struct PairSplit {
  int KU;           // units of K of a tile
  int m_tiles;      // token tiles (tile = feature tile * m_tiles + token tile)
  int clusters;     // clusters of the grid
  int left, parts;  // tiles 0 .. left - 1 go to `parts` clusters each
  int rounds;       // whole tiles per cluster after them
};

// One accumulator's worth of work of a cluster: units [ku0, ku1) of a tile.
struct Segment {
  int tile, ntile, mtile, ku0, ku1;
};

// The cluster that computes part k of left-over tile t, and the one that sums the
// tile: the last part's.  It waits for the others' parts, so they are clusters of
// lower numbers, which are dispatched before it and wait for nothing before they
// publish: the wait ends whatever share of the chip other work holds.
KVR_HD inline int part_cluster(const PairSplit &p, int t, int k) { return t + k * p.left; }
KVR_HD inline bool sums_parts(const PairSplit &p, int cluster) {
  return cluster >= (p.parts - 1) * p.left;
}

// Segments of cluster c in order: its part of a left-over tile (part c / left of
// tile c % left), then its whole tiles.
struct Walk {
  int k, c;
  KVR_HD Walk(const PairSplit &p, int cluster)
      : k(cluster < p.left * p.parts ? -1 : 0), c(cluster) {}
  KVR_HD bool next(const PairSplit &p, Segment &s) {
    if (k >= p.rounds) return false;
    s.ku0 = 0;
    s.ku1 = p.KU;
    if (k < 0) {
      const int j = c / p.left;
      s.tile = c - j * p.left;
      s.ku0 = (int)((long long)j * p.KU / p.parts);
      s.ku1 = (int)((long long)(j + 1) * p.KU / p.parts);
    } else {
      s.tile = p.left + c + k * p.clusters;
    }
    ++k;
    s.ntile = s.tile / p.m_tiles;
    s.mtile = s.tile - s.ntile * p.m_tiles;
    return true;
  }
};

}  // namespace kvr
