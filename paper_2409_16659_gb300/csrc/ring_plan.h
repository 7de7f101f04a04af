// ring_plan.h -- how the ring sums of a lattice are shared out over blocks of
// 256 threads. Host code.
#pragma once

namespace mlsw {

// A block's turn is `tr` rows of one of `segs` segments of `seg` columns, 2^lgx
// threads beside one another in a row: item = row group * segs + segment, and
// block b takes the items b, b + blocks, ...
struct RingPlan {
  int lgx, tr;        // threads in a row (log2), rows at once: 2^lgx * tr = 256
  int segs, seg;      // segments of a row, columns of a segment (whole turns)
  int groups;         // row groups
  int blocks;
};

constexpr int kRingBlocks = 608;  // four blocks an SM

// Lattices of fewer than 256 columns put several rows side by side, those of
// fewer rows than blocks cut their rows: with a block per row, whatever their
// length, 1000000 x 1 cells took 2470 us a call (267 now), 100000 x 8 493 (277),
// 8 x 100000 562 (271); 1024^2, the same turns as before, 327 (321).
inline RingPlan ring_plan(int nx, int ny) {
  RingPlan p;
  p.lgx = 3;
  while (p.lgx < 8 && (1 << p.lgx) < nx) ++p.lgx;
  const int tx = 1 << p.lgx;
  p.tr = 256 >> p.lgx;
  p.groups = (int)(((long)ny + p.tr - 1) / p.tr);
  const int turns = (int)(((long)nx + tx - 1) / tx);  // of a row
  int want = p.groups < kRingBlocks ? (kRingBlocks + p.groups - 1) / p.groups : 1;
  if (want > turns) want = turns;
  const int per = (turns + want - 1) / want;
  p.seg = per * tx;
  p.segs = (turns + per - 1) / per;
  const long items = (long)p.groups * p.segs;
  p.blocks = (int)(items < kRingBlocks ? items : kRingBlocks);
  return p;
}

}  // namespace mlsw
