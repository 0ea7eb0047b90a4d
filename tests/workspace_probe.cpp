// Host-side probe of the workspace's allocation (test infrastructure, no GPU needed): a plan whose launch
// shapes are given, an allocator that refuses what passes a limit, and the sizes that result.
//
// stdin: N s precision flags max_batch clusters0 clusters1 slot part_slots part_size tasks n_rho vss
//        limit batch
#include <cstdio>

#include "dgfs_internal.h"

namespace {
size_t limit_bytes = 0, used = 0;
char memory[1];
int refuse_above_limit(dgfs::Plan&, void** p, size_t bytes) {
  if (used + bytes > limit_bytes) {
    *p = nullptr;
    return DGFS_ERR_OOM;
  }
  used += bytes;
  *p = memory;
  return DGFS_OK;
}
}  // namespace

int main() {
  dgfs::Plan p;
  int batch, tasks, vss;
  if (std::scanf("%d %d %d %u %d %d %d %zu %d %zu %d %d %d %zu %d", &p.N, &p.s, &p.precision, &p.flags, &p.max_batch,
                 &p.shapes[0].clusters, &p.shapes[1].clusters, &p.shape.slot, &p.part_slots, &p.part_size, &tasks,
                 &p.N_rho, &vss, &limit_bytes, &batch) != 15)
    return 2;
  p.tasks.resize(size_t(tasks));
  p.vss = vss != 0;
  dgfs::size_workspace(p);
  const size_t wanted = p.scratch_bytes;
  const int rc = dgfs::alloc_workspace(p, refuse_above_limit);
  if ((p.flags & DGFS_SUM_SPECIES) && (p.flags & DGFS_CONSERVE)) {
    p.cons.resize(size_t(p.s) * (p.s + 1) / 2);
    p.d_Qfull = p.d_lam = reinterpret_cast<double*>(memory);
  }
  std::printf("{\"rc\": %d, \"wanted\": %zu, \"scratch\": %zu, \"used\": %zu, \"clusters\": [%d, %d], \"part_slots\": %d, "
              "\"part_off\": %zu, \"counters\": %zu, \"reported\": %zu, \"second\": %zu, \"part_slots2\": %d}\n",
              rc, wanted, p.scratch_bytes, used, p.shapes[0].clusters, p.shapes[1].clusters, p.part_slots, p.part_off,
              p.counter_bytes(), dgfs::workspace_bytes(p, batch), p.scratch_bytes_of(1), p.part_slots_of(1));
  return 0;
}
