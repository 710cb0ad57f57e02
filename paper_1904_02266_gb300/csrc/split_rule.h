// The weight of an active source group in the rebalanced work split of a reused plan
// (pair_kernels.cuh: split_work), apart from the kernels so that the host can check it.
#pragma once

#ifdef __CUDACC__
#define CVO_HD __host__ __device__
#else
#define CVO_HD
#endif

namespace cvo {

// work model: the pair bodies of a source group that kept a pair, in pair-test units
constexpr int kCostActive = 12;
// and for shares that are large enough for the bodies to count and small enough to fit the
// cache when they are weighed that much
constexpr int kCostActiveShort = 24;

// The weight, from the plan's first split (no group weighed): `total` units of work on
// `warps` warps, ncl clusters of `points` source points, the caller's cost model, and the
// cache: cap floats a warp, of which a point takes point_floats. Told in chunks and floats,
// not in units: a unit is the caller's to choose, and what fits hangs on the features.
// kCostActiveShort from 1.75 chunks a warp on (fewer: within 1% either way) as long as the
// mean share takes seven tenths of the cache. The largest is 1.5 times the mean and more, and
// a plan of which one does not fit goes back to kCostActive (check_fits): one warp of
// 2280 that streams its rest in every pass holds up the team. Whole room solves, means of
// six pairs, with 12, with 24, and with 24 and the way back: five features, 20k points 5.33,
// 5.16, 5.18 ms, 28k 7.43, 7.33, 7.29, 30k 8.12, 8.48, 8.09; eight features, 20k 5.87, 5.89, 5.76,
// 22k 6.60, 7.00, 6.61, 24k 7.69, 7.96, 7.73.
CVO_HD inline int active_weight(long long total, long long warps, int ncl, int points,
                                int cost_chunk, int cost_cluster, int point_floats, int cap) {
  // over all warps, and times `unit`, so that nothing is divided (a division's subroutine
  // would cost the callers registers): the work without the clusters' staging; clusters times
  // the units of a chunk, a cluster's points rounded up to fours on average; and the chunks
  const float work = (float)total - (float)ncl * (float)cost_cluster;
  const float size = (float)points + 1.5f * (float)ncl;
  const float unit = size + (float)ncl * (float)cost_chunk;
  const float chunks = work * (float)ncl, w = (float)warps * unit;
  const float need = (32.0f * chunks + size * unit) * (float)point_floats;
  return chunks >= 1.75f * w && need <= 0.7f * (float)cap * w ? kCostActiveShort
                                                                  : kCostActive;
}

}  // namespace cvo
