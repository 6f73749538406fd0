// How a launch of the cluster kernel (lqer_decode_cluster.cu: the layer for 3 to 16 tokens, paper Section 2.1) is cut: cluster size, clusters,
// shared memory.  Plain C++ over the shapes and over how many clusters the device holds: the host's tests run it too.
#pragma once
#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <cstring>

#include "lqer_ring.h"

namespace lqer {
namespace dcl {

constexpr int kColumnWarps = 4, kPhases = 3;                       // consumer warps: 32 columns of a tile each, and every third stage
constexpr int kConsumers = kColumnWarps * kPhases, kEpilogue = 4;  // warps; one more is the producer, and one looks after T
constexpr int kWorkerWarps = kConsumers + kEpilogue, kWorkers = kWorkerWarps * 32, kThreads = kWorkers + 64;
constexpr int kMaxLayers = 4;                // layers of a launch, at most
constexpr int kUnit = 16;                    // columns of a unit, one side of an MMA
constexpr int kTileColumns = 128, kUnits = kTileColumns / kUnit;   // columns and units of a tile
constexpr int kRows = 16;
constexpr int kMaxSlots = 20;                // ring slots, at most (RingCursor: each phase has its own of them, a third if the ring is filled again)
constexpr int kRed = 3;                      // tiles whose sums may be under way
constexpr int kSmemMax = 222 * 1024;
constexpr int kLocalStages = 10, kLocalBlocks = 8;   // stages of a cluster that forms all of T itself, and blocks of T (of eight rows) to a warp, at most

// Bytes of the mantissas of a packed tile's slab, with 4- or 2-bit weights, and of the whole slab; a stage is two of them.
constexpr int slab_mantissa_bytes(int w_bits) { return w_bits == 4 ? 4096 : 2048; }
constexpr int slab_bytes(int w_bits) { return slab_mantissa_bytes(w_bits) + kTileColumns * 4; }
// Words from column to column of a unit on its way to Y: tokens, two more against bank conflicts.
LQER_RING_FN constexpr int token_stride(int mt) { return 8 * mt + 2; }

// The planes lie 16, 64 and 80 bytes beyond multiples of 128 from the first, so that the lanes that store neighbouring blocks meet four to a bank
// (with none of that sixteen: 16 rows, K = 2048 in clusters of four, 2 us of 8).
LQER_RING_FN constexpr uint32_t plane_bytes(int steps, int mt) { return (uint32_t)steps * (512u * mt) + 16u; }
LQER_RING_FN constexpr uint32_t plane_offset(uint32_t m, uint32_t plane) { return m * plane + (m >> 1) * 32u; }

struct Shape {
  int dev, n, M, w_bits, k_slabs[kMaxLayers], tiles[kMaxLayers], r_blocks[kMaxLayers];
};
// The cluster size, the clusters of each layer and the shared memory of a launch over these layers: functions of the shapes (and of
// what the device holds) alone.
struct Plan {
  int CS, steps_max, slots;
  int off_red, red_bytes, off_xq, off_xe, off_tpart, off_trecv, off_tq, off_ring;
  size_t smem;
  int resident, clusters[kMaxLayers], total;
  int t_blocks[kMaxLayers], t_clusters[kMaxLayers], t_tiles[kMaxLayers];
  bool local;                               // every cluster forms all of T for itself
  double cost;
};
// `resident`: clusters of CS CTAs that the device holds at a time, or -1 where it could not be asked.  false: no such launch.
inline bool plan_with(const Shape& sh, int CS, int resident, Plan& q) {
  const int MT = sh.M > 8 ? 2 : 1, n = sh.n;
  int k_slabs_max = 0, r_blocks_max = 0, tiles_max = 0, steps[kMaxLayers];
  for (int i = 0; i < n; ++i) {
    k_slabs_max = std::max(k_slabs_max, sh.k_slabs[i]);
    r_blocks_max = std::max(r_blocks_max, sh.r_blocks[i]);
    tiles_max = std::max(tiles_max, sh.tiles[i]);
    steps[i] = ((sh.k_slabs[i] + CS - 1) / CS + 1) / 2;
  }
  q.CS = CS;
  auto al = [](int v) { return (v + 127) / 128 * 128; };
  const int red = al(kUnits * kPhases * kUnit * token_stride(MT) * 4), stage = 2 * slab_bytes(sh.w_bits);
  q.steps_max = ((k_slabs_max + CS - 1) / CS + 1) / 2;
  if ((long long)q.steps_max * 2048 * MT > kSmemMax) return false;
  const int off = al((int)plane_offset(4, plane_bytes(q.steps_max, MT)));
  // X_q for the projection and the partial sums of T share their room with the sums of the tiles
  q.off_red = off;
  q.red_bytes = red;
  q.off_xq = off;
  q.off_xe = q.off_xq + al(8 * MT * (q.steps_max * 128 + 16));
  q.off_tpart = q.off_xe + al(8 * MT * q.steps_max * 8);
  const int t_width = std::max(8 * kWorkerWarps, 16 * r_blocks_max);
  q.off_trecv = q.off_tpart + 64 * MT * t_width;
  q.off_tq = r_blocks_max > 0 ? std::max(off + kRed * red, q.off_trecv + 64 * MT * 16 * r_blocks_max) : off + kRed * red;
  q.off_ring = q.off_tq + 2048 * MT;
  // a slot for each phase at least, unless a CTA has fewer stages than that
  if (kSmemMax - q.off_ring < kPhases * stage) return false;
  q.slots = (int)std::min<long long>(std::min((kSmemMax - q.off_ring) / stage, kMaxSlots), (long long)tiles_max * q.steps_max);
  q.smem = (size_t)q.off_ring + (size_t)q.slots * stage;
  q.resident = resident;
  if (q.resident < n) return false;
  // each layer has a cluster, the others go one by one where the time is longest, as long as every cluster keeps a tile
  double length[kMaxLayers];                // 0: each of its clusters has one tile
  auto count = [&](int i, int clusters) {
    q.clusters[i] = clusters;
    length[i] = clusters < sh.tiles[i] ? (double)sh.tiles[i] / clusters * steps[i] : 0.0;
  };
  // (to begin with, nearly what each one's part of the work comes to: one by one no layer gets more than that and one, so none gets
  // less than n - 1 below it)
  double work = 0.0;
  for (int i = 0; i < n; ++i) work += (double)sh.tiles[i] * steps[i];
  q.total = 0;
  for (int i = 0; i < n; ++i) {
    count(i, std::max(1, std::min(sh.tiles[i], (int)(q.resident * (sh.tiles[i] * (double)steps[i] / work)) - n)));
    q.total += q.clusters[i];
  }
  while (q.total < q.resident) {
    int best = 0;
    for (int i = 1; i < n; ++i)
      if (length[i] > length[best]) best = i;
    if (length[best] == 0.0) break;
    count(best, q.clusters[best] + 1);
    ++q.total;
  }
  // In the time of a stage: the stages, what a tile costs beyond them (many CTAs hand over more sums in less time), the rounds in which
  // X is quantised, and what T costs the clusters that form it, which get fewer tiles for that.  Fitted to calls of 3, 8, 9 and 16 rows with
  // clusters of 2, 4 and 8.  us for the groups (qkv, o, gate and up, down) of a 4096 / 11008 and of a 5120 / 13824 layer, 2 | 4 | 8:
  //    3 rows: 18.0 10.9 25.5 28.2 | 15.0 10.6 26.0 13.9 | 17.8 10.7 30.5 18.6;  21.9 12.9 31.6 36.0 | 21.9 12.5 35.8 28.2 | 24.7 11.9 41.4 22.6
  //   16 rows: 23.5 17.4 31.6 -    | 20.5 13.3 30.7 22.2 | 27.5 14.6 45.9 23.2;  29.4 21.7 41.7 -    | 27.5 16.9 42.4 39.3 | 34.7 16.3 56.9 29.2
  // (At hidden sizes of 1024 to 2048 the model is at times off: 1536 / 4096, rank 32, 16 rows, gate and up 13.9 with 4, 11.6 with 2.)
  const double tile_cost = CS == 8 ? (MT == 1 ? 2.0 : 3.5) : CS == 4 ? (MT == 1 ? 0.7 : 1.2) : (MT == 1 ? 0.3 : 0.6);
  const int most = std::max(q.resident / 4 / n, 1);  // clusters that form a layer's T: a quarter of the places, whatever the rank
  auto share = [&](int i) { return (sh.tiles[i] + q.clusters[i] - 1) / q.clusters[i]; };
  // few stages: T's way through global memory would take longer than they do
  q.local = r_blocks_max > 0 && r_blocks_max <= 8;
  for (int i = 0; i < n; ++i)
    q.local = q.local && steps[i] * 8 * 2 * sh.r_blocks[i] * MT <= kLocalBlocks * kWorkerWarps && share(i) * steps[i] <= kLocalStages;
  q.cost = 0.0;
  for (int i = 0; i < n; ++i) {
    const int tiles = sh.tiles[i], formers = q.local ? 1 : std::min(q.clusters[i], most);
    q.t_blocks[i] = (sh.r_blocks[i] + formers - 1) / formers;
    int f = !q.local && q.t_blocks[i] > 0 ? (sh.r_blocks[i] + q.t_blocks[i] - 1) / q.t_blocks[i] : 0, tf = 0;
    const double per_tile = steps[i] + tile_cost;
    const double t_cost = sh.r_blocks[i] > 0 ? 2.0 + 0.15 * MT * steps[i] * 16 * q.t_blocks[i] / kWorkerWarps : 0.0;
    if (f > 0 && f < q.clusters[i]) {
      // equal times: f * tf + (clusters - f) * (tf + t_cost / per_tile) = tiles
      const double level = (tiles - (q.clusters[i] - f) * t_cost / per_tile) / q.clusters[i];
      tf = std::max(1, (int)(level + 0.5));
      if (tiles - f * tf < q.clusters[i] - f) tf = 0;
    }
    if (tf == 0) f = 0;                              // equal shares for all
    q.t_clusters[i] = f;
    q.t_tiles[i] = tf;
    const int longest = (tiles - f * tf + q.clusters[i] - f - 1) / (q.clusters[i] - f);
    q.cost = std::max(q.cost, std::max(longest * per_tile + (f > 0 ? 0.0 : t_cost), f > 0 ? tf * per_tile + t_cost : 0.0) +
                                  (MT == 1 ? 3.0 : 3.5) * ((sh.M * steps[i] * 8 + kWorkers - 1) / kWorkers));
  }
  return true;
}
// The plan that costs least.  resident(CS): see plan_with; sure: no cluster size was left out because the device could not be asked.
template <class Resident>
bool make_plan(const Shape& sh, Resident&& resident, Plan& best, bool& sure) {
  int k_slabs_min = sh.k_slabs[0];
  for (int i = 1; i < sh.n; ++i) k_slabs_min = std::min(k_slabs_min, sh.k_slabs[i]);
  bool found = false;
  sure = true;
  for (int CS = 8; CS >= 1; CS >>= 1) {
    if (CS > 1 && k_slabs_min < 2 * CS) continue;                    // at least one step of two slabs to a CTA
    const int places = resident(CS);
    if (places < 0) sure = false;
    Plan q;
    if (!plan_with(sh, CS, places, q)) continue;
    if (!found || q.cost < best.cost) { best = q; found = true; }
  }
  return found;
}
// The plans of the shapes that a thread has asked for, as long as no other shape takes their place (a call asks twice, and working one out takes
// 0.2 to 0.8 us).  What was
// worked out while the device could not be asked is not kept.
class PlanCache {
 public:
  template <class Resident>
  bool find(const Shape& sh, Resident&& resident, Plan& q) {
    uint32_t h = 2166136261u;
    const int* words = reinterpret_cast<const int*>(&sh);
    for (size_t i = 0; i < sizeof(sh) / sizeof(int); ++i) h = (h ^ (uint32_t)words[i]) * 16777619u;
    Known& k = known_[(h ^ (h >> 16)) % kKnown];
    if (std::memcmp(&k.shape, &sh, sizeof(sh)) == 0) { q = k.plan; return k.found; }
    bool sure;
    const bool found = make_plan(sh, resident, q, sure);
    if (sure) { k.shape = sh; k.plan = q; k.found = found; }
    return found;
  }

 private:
  static constexpr int kKnown = 128;
  struct Known {
    Shape shape;                            // n == 0: none
    Plan plan;
    bool found;
  };
  Known known_[kKnown] = {};
};

}  // namespace dcl
}  // namespace lqer
