// How a launch of the collision kernel runs its work items: shape and chunks (host code only).
#pragma once

#include <cmath>

#include "dgfs_internal.h"

namespace dgfs {

// entries of a plan's dearest task, and the mean over its tasks as a fraction of that
struct TaskLoad {
  double most = 1.0, mean = 1.0;
};
inline TaskLoad task_load(const Plan& pl) {
  TaskLoad l;
  double sum = 0.0;
  l.most = 0.0;
  for (const TaskDesc& t : pl.tasks) {
    sum += t.n_ent;
    l.most = t.n_ent > l.most ? t.n_ent : l.most;
  }
  l.mean = sum / (pl.tasks.size() * l.most);
  return l;
}

// How a launch of `items` work items (task, node) runs: the shape W and the number of chunks each
// item's radial nodes are split into, by a cost model in units of one radial node of the dearest
// task on a full device.  A chunk of `len` nodes costs len + 1/2 (its own f_hat), or len + 4 / entries
// where the dearest task has so few entries that a radial node is cheap beside that (400 nodes of N = 4,
// three entries: 23 us whole, 30 in two chunks).  Chunks go out one by one, so a launch takes its share of
// the device, sum of costs / clusters, and about 0.38 of the last chunk; a chunk on a nearly idle device
// runs at 0.6 of its cost.  Fitted to N = 24, 45 nodes
// (W = 0: 1.42, 1.21, 1.11, 0.98, 1.10 ms with 1, 2, 4, 6, 12 chunks) and N = 32, 5 nodes, 3 species
// (W = 0: 2.30, 1.22, 0.99, 1.11 ms with 1, 4, 8, 16; W = 1: 0.97, 0.74, 0.75, 0.84 with 1, 2, 4, 16).
// The wide shape takes `slow` times longer per node and cluster-share of the device.  All products
// of all items must fit the parts buffer.
struct LaunchPlan {
  int wide = 0, chunks = 1;
};
inline LaunchPlan plan_launch(int items, int n_rho, int clusters0, int clusters1, double slow, const TaskLoad& load,
                              int part_slots) {
  LaunchPlan best;
  double best_t = 1e300;
  for (int w = 0; w < 2; ++w) {
    const int C = w == 0 ? clusters0 : clusters1;
    if (C <= 0) continue;
    const double unit = w == 0 ? 1.0 : slow * double(clusters1) / double(clusters0);
    for (int s = 1; s <= n_rho; ++s) {
      if (s > 1 && double(items) * n_rho > double(part_slots)) break;
      const int len = (n_rho + s - 1) / s;
      if (s > 1 && (n_rho + s - 2) / (s - 1) == len) continue;  // no shorter than with s - 1 chunks
      const double own = 4.0 / load.most, one = (own > 0.5 ? own : 0.5) + len;
      const double share = double(items) * s * load.mean * one / C + 0.38 * one;
      const double t = (share > 0.6 * one ? share : 0.6 * one) * unit;
      if (t < best_t * (1.0 - 1e-9)) {
        best_t = t;
        best.wide = w;
        best.chunks = s;
      }
    }
  }
  return best;
}

// VSS: chunks of whole parts, in the same units.  An item's own cost (f_hat, its share of the finish) is about
// 4 / entries radial nodes, a split one's sum of its parts half an entry each; a launch takes its share of the
// device and about 0.8 of its last chunk.  With up to two clusters per SM (N >= 16) a chunk's speed hardly
// depends on its neighbours, so whole waves count: half share and last chunk, half the number of waves.
// Fitted to 521 launches (N = 4 to 48, 1 to 5000 nodes, tasks of 3 to 32 entries, 2 to 24 radial nodes, split
// into 1, 2, 4 and 8 parts): the split taken costs 0.9 % more than the best of them on average and 27 % at most.
// One three-species node of N = 48, 24 radial nodes, M = 32: 31.3 -> 6.6 ms with 8 parts (4: 10.2).
constexpr int kFewClusters = 304;
inline int vss_chunks(int items, int n_rho, int clusters, const TaskLoad& load, int part_slots) {
  const int parts = vss_parts(n_rho);
  if (double(items) * parts > double(part_slots)) return 1;
  int best = 1;
  double best_t = 1e300;
  for (int s = 1;; s = 2 * s < parts ? 2 * s : parts) {
    const double own = 4.0 / load.most, len = double((parts + s - 1) / s) * n_rho / parts;
    const double one = (own > 0.25 ? own : 0.25) + len + (s > 1 ? 0.5 * parts / load.most : 0.0);
    const double share = double(items) * s * load.mean / clusters;
    const double waves = std::ceil(double(items) * s / clusters) * load.mean;
    const double t = one * std::fmax(1.0, clusters > kFewClusters ? share + 0.8 : 0.5 * (share + 1.0) + 0.5 * waves);
    if (t < best_t * (1.0 - 1e-9)) {
      best_t = t;
      best = s;
    }
    if (s == parts) return best;
  }
}

}  // namespace dgfs
