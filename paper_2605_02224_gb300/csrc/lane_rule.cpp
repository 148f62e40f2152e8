// The rule that picks a launch's lanes per query.
#include "batch.h"
#include "knn_kernels.h"

namespace mknn {

namespace {

// Untuned default on a cloud whose long lists have no trees (a dynamic
// cloud): with a successor list of 2^12 entries or more, a whole warp per
// query, which scans the long rows 32 entries at a time.
constexpr int kHubBucketWide = 12;

// Queries of one launch from which one lane per query is faster than one
// warp per query. One lane per query takes about the time of its longest
// query whatever the number of queries, until they fill the GPU; one warp
// per query takes time in proportion to it, so the line grows with the number
// of SMs; the figures are of 152. On a 300k-site torus (queries
// half in the box, half near the surface; us for one lane / one warp per
// query at 40,000 and 80,000 queries, the locality sort included):
//   k = 1: 102 / 102, 103 / 163     k = 8: 184 / 159, 198 / 277
//   k = 16: 273 / 214, 297 / 379    k = 32: 503 / 323, 555 / 576
// above k = 32, where the one-lane list moves keys, at 100,000 and 400,000:
//   k = 40: 1204 / 874, 2949 / 3249   k = 47: 1473 / 987, 4116 / 3689
// and on a 200k-site patch cloud with trees, at 100,000 and 150,000:
//   k = 1: 278 / 256, 311 / 359     k = 8: 492 / 418, 527 / 599
//   k = 16: 706 / 629, 789 / 909    k = 32: 1145 / 1012, 1547 / 1471
// A lane that scans a list of hundreds of entries takes as long as one that
// gives up at a tree (12k-site patch cloud, longest list 757, no trees, 60,000
// queries at k = 4: 340 / 157), so such clouds take that line too.
// Register groups of 4, 8 and 16 lanes are slower than both at every size
// (100,000 queries, k = 16: 1,638 / 994 / 837 us against 320), so the rule
// never takes them.
// On a cloud with trees and no scratch for the hand-over, a lane reads lists of
// up to 2^(hub + 1) entries through while one warp per query walks the trees.
// Queries from which one lane is the faster all the same (patch clouds of 20k
// to 90k sites, k = 1, 4, 16, 32, 40):
//   longest list 1,100: 135k 155k 175k 180k 205k   1,625: 120k 180k 195k 245k 310k
//   2,404: 195k 300k 340k 390k 430k   2,695: 275k 340k 280k 270k 280k
//   3,579: 310k 480k 425k 470k 490k   9,682: 600k 850k 650k 550k 550k
// (longest 2,695, k = 16, us for one lane / one warp: 150,000 queries 1223 /
// 704, 300,000 1264 / 1338, 1,000,000 1956 / 4247).
constexpr int kHubBucketLong = 9;  // a list of 2^9 - 1 entries or more
int64_t one_lane_min_queries(int k, int hub, bool trees, bool handover) {
  int64_t q = 40960 + 1100 * (int64_t)k;
  if (trees && !handover) {
    q += 61440 + ((int64_t)90 << hub);
  } else {
    if (k > 32) q += 32768 * (int64_t)(k - 32);
    if (trees || hub >= kHubBucketLong) q += 81920;
  }
  return q * num_sms() / 152;
}

}  // namespace

Mode choose_mode(int k, int64_t n, int hub, int64_t nq, bool trees, bool handover) {
  const Mode t = tuned_mode(k, n, hub);
  const int wide = (hub >= kHubBucketWide && !trees) ? 32 : default_lanes(k);
  int lanes = t.lanes ? t.lanes : wide;
  // a table made by an earlier tuner may hold register groups: slower than
  // one warp per query in a small launch (100k-site torus, k = 8, 4 / 8 / 16
  // lanes: 64 queries 205 / 90 / 51 us against 21, 10,000 259 / 132 / 79
  // against 57)
  if (lanes < 32 && nq < one_lane_min_queries(k, hub, trees, handover)) lanes = 32;
  const int placement = (t.lanes && lanes == t.lanes) ? t.placement : default_placement(k, lanes);
  return Mode{lanes, placement};
}

}  // namespace mknn
