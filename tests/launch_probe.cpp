// Host-side probe of the launch rules (test infrastructure, no GPU needed): one launch per input line,
// the chunks that each rule takes on standard output.
//
// stdin: vhs items n_rho clusters0 clusters1 slow most mean part_slots   -> "wide chunks"
//        vss items n_rho clusters most mean part_slots                   -> "0 chunks"
#include <cstdio>
#include <cstring>

#include "launch_plan.h"

int main() {
  char kind[8];
  while (std::scanf("%7s", kind) == 1) {
    int items, n_rho, c0, c1 = 0, slots;
    double slow = 1.0;
    dgfs::TaskLoad load;
    const bool vss = std::strcmp(kind, "vss") == 0;
    if (std::scanf("%d %d %d", &items, &n_rho, &c0) != 3) return 2;
    if (!vss && std::scanf("%d %lf", &c1, &slow) != 2) return 2;
    if (std::scanf("%lf %lf %d", &load.most, &load.mean, &slots) != 3) return 2;
    dgfs::LaunchPlan run;
    if (vss)
      run.chunks = dgfs::vss_chunks(items, n_rho, c0, load, slots);
    else
      run = dgfs::plan_launch(items, n_rho, c0, c1, slow, load, slots);
    std::printf("%d %d\n", run.wide, run.chunks);
  }
  return 0;
}
