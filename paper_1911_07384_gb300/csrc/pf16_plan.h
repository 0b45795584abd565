// Launch plans as host arithmetic without CUDA, so that they can be checked on a
// machine that has no GPU.
#pragma once

#ifdef __CUDACC__
#define PF16_PLAN_FN __host__ __device__ inline
#else
#define PF16_PLAN_FN inline
#endif

namespace pf16 {

enum LoadMode : int {
  LD_TILED_K = 0,
  LD_TILED_MN = 1,
  LD_IM2COL_K = 2,
  LD_IM2COL_MN = 3,
  LD_TAP3D_MN = 4
};

// Whether k_gemm's producer is compiled for A in mode a and B in mode b: forward
// (1x1, others), data gradient (1x1, stride phases), weight gradient (1x1 and
// patches, others); with an operand transform only the 1x1 forward and weight
// gradient.  Any other pair is refused before a launch.
inline bool gemm_modes_ok(int a, int b, bool transform) {
  if (a == LD_TILED_K) return b == LD_TILED_K || (b == LD_TILED_MN && !transform);
  if (a == LD_TILED_MN) return b == LD_TILED_MN || (b == LD_IM2COL_MN && !transform);
  return a == LD_IM2COL_K && (b == LD_TILED_K || b == LD_TAP3D_MN) && !transform;
}

// Split-K reduction of `total` 8-column chunks over `splits` partial planes.
//
// The tree over the splits, padded with zeros to a power of two, is part of the
// result (FP16 sums round): the splits are cut into 2^tree_groups_log2 aligned
// runs, a run is summed pairwise, neighbours first, and the runs' sums at a
// stride, run i with run i + half, half halving down to 1.  As many runs as it
// takes to give the GPU's 152 SMs 512 threads each with one thread per chunk and
// run, at most 256: a function of the two sizes and of nothing that a launch
// may choose.
//
// The launch: groups of 2^leaves_log2 splits, at most 16, one thread each per
// chunk.  A group lies inside a run; only where a run is a single split does
// a thread take two of them, half of the splits apart (leaf_step), which is the
// first level of the stride.
struct SplitkPlan {
  int tree_groups_log2;
  int leaves_log2;  // splits a thread sums itself, loads all in flight
  int groups_log2;  // groups of splits
  int leaf_step;    // planes between a thread's splits
};

inline SplitkPlan splitk_plan(int splits, long long total) {
  int sp_log2 = 0;
  while ((1 << sp_log2) < splits) ++sp_log2;
  SplitkPlan p;
  p.tree_groups_log2 = 0;
  while (p.tree_groups_log2 < sp_log2 && p.tree_groups_log2 < 8 && (total << p.tree_groups_log2) < 152ll * 512)
    ++p.tree_groups_log2;
  // as many groups as leave a thread at most 16 splits, and more while the GPU
  // has fewer than 512 threads per SM and a thread more than two loads (against
  // 16 loads a thread throughout: 819 against 829 us over 24 weight gradients);
  // at most 256, a CTA's threads (splits <= 4,096 keeps the first condition
  // below that: a small result with more than 512 splits meets the second)
  p.groups_log2 = 0;
  while (sp_log2 - p.groups_log2 > 4 ||
         (p.groups_log2 < 8 && sp_log2 - p.groups_log2 > 1 && (total << p.groups_log2) < 152ll * 512))
    ++p.groups_log2;
  p.leaves_log2 = sp_log2 - p.groups_log2;
  p.leaf_step = p.groups_log2 < p.tree_groups_log2 ? 1 << p.groups_log2 : 1;
  return p;
}

// A ring of `stages` buffers that a producer fills and `groups` consumer groups
// empty, group g taking tiles g, g + groups, ...: a position in it, one per role,
// the producer's advanced tile by tile, a group's by `groups` (at most `stages`).
struct RingPos {
  int stage, bar;
  unsigned phase;  // parity of the tile's use of its full barrier
  PF16_PLAN_FN void advance(int by, int stages, int bars) {
    if ((stage += by) >= stages) stage -= stages;
    if ((bar += by) >= bars) {
      bar -= bars;
      phase ^= 1u;
    }
  }
};
// Full barriers.  A wait by parity is only sound for who saw the barrier's phase
// before: until that is over, the other parity lets it pass at once.  With a
// barrier per stage a group would meet the uses that other groups waited for
// (three stages and two groups: every second one), and pass while the copy of
// such a use, or its own, is in flight.  (Waiting for that use first is no way
// out: the copy after it may already have landed, and its phase come round.)
// With the least common multiple of both numbers each barrier serves one group,
// which sees all of its phases.
PF16_PLAN_FN int ring_bars(int stages, int groups) {
  int bars = stages;
  while (bars % groups != 0) bars += stages;
  return bars;
}
PF16_PLAN_FN RingPos ring_start(int tile) { return RingPos{tile, tile, 0u}; }

}  // namespace pf16
