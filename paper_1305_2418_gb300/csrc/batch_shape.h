// batch_shape.h -- launch shape of a batched solve from the amount of work, and the shapes
// that the tuner times.  `vecs`: the work items of a half-sweep of the finest grids (four
// cells each).  Plain C++.
//
// Beyond 2^20 items the device is full either way and 512 threads x 2 per SM are the
// fastest (96 solves of 32^3..128^3, ms, all on one build: 45.0; 256 x 2 54.5, 256 x 3
// 47.1, 128 x 8 50.3; 40 to 42 for 512 x 2 now), below it smaller blocks spread the items
// better (one 64^3 1.68 for 1.82, one 128^3 3.46 for 3.64).  A batch of few items is little
// but barriers, whose time grows with the blocks that arrive at them: no more blocks than
// there are items for (and one per solve, for the 4^3 grids).  Up to 16384 items (one 32^3:
// 4096) blocks of 128 threads, 32 items each up to 128 blocks: what a block does between
// two barriers is then short (two blocks of 256 made one 16^3 to 1e-11 15% slower than a
// full grid), ms to 1e-8 (1e-11):
//   one 8^3   0.365 (0.529), 256 threads with all items 0.369 (0.549), a full grid 0.375 (0.526)
//   one 16^3  0.669 (0.936), 256 threads x 2 blocks 0.729 (1.095), a full grid 0.702 (0.954)
//   one 32^3  0.962 (1.456), 64 blocks 0.967 (1.488), a full grid 1.027 (1.512)
// (the full grid: 304 blocks of 256, one cell per thread, an earlier build).
#pragma once
#include <algorithm>

struct BatchShape {
  int threads, per_sm;  // of a block; blocks per SM
};

// Most blocks of a launch with `threads` per block.  Blocks of 128 take 32 items each up to
// 128 blocks (four blocks at least), so that a small batch is on many SMs.
inline long long batch_blocks(int threads, long long vecs, int nsolves) {
  long long b = (vecs + threads - 1) / threads;
  if (threads == 128) b = std::max(b, std::min(128LL, std::max(4LL, vecs / 32)));
  return std::max(b, (long long)nsolves);
}

inline long long batch_grid(BatchShape s, long long vecs, int nsolves, int nsm) {
  return std::min((long long)nsm * s.per_sm, batch_blocks(s.threads, vecs, nsolves));
}

// the shape of a batch that was not tuned; no more blocks per SM than its blocks need
inline BatchShape batch_rule(long long vecs, int nsolves, int nsm) {
  const int threads = vecs > (1 << 20) ? 512 : (vecs > 16384 ? 256 : 128);
  const long long need = (batch_blocks(threads, vecs, nsolves) + nsm - 1) / nsm;
  return BatchShape{threads, (int)std::min(threads == 512 ? 2LL : 3LL, std::max(1LL, need))};
}

// the launches worth timing, the untuned one first (so that a tuned batch is not slower),
// each once; at most 10 into out, their number returned
inline int batch_candidates(long long vecs, int nsolves, int nsm, BatchShape* out) {
  int n = 0;
  auto add = [&](BatchShape s) {
    for (int i = 0; i < n; ++i)
      if (out[i].threads == s.threads && batch_grid(out[i], vecs, nsolves, nsm) ==
                                             batch_grid(s, vecs, nsolves, nsm))
        return;
    out[n++] = s;
  };
  add(batch_rule(vecs, nsolves, nsm));
  for (int t : {128, 256, 512})
    for (int b : {1, 2, 4}) add(BatchShape{t, b});
  return n;
}
