// Host-side check of the general kernel's block geometry (gen_geom in
// paper_1302_0120_gb300/csrc/gs_internal.h). Built with nvcc as host code by
// tests/test_gen_geom_host.py. With no argument: every valid pair of sides,
// several batches and devices against the limits of a block; prints "ok N" or
// the first violation. With "nx ny masks": prints "teams warps" on 152 SMs.
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "gs_internal.h"

int main(int argc, char** argv) {
  using namespace gsk;
  if (argc == 4) {
    const GenGeom g = gen_geom(std::atoi(argv[1]), std::atoi(argv[2]), std::atoi(argv[3]), 152);
    std::printf("%d %d\n", g.teams, 1 << (g.team_log - 5));
    return 0;
  }
  std::vector<int> sides;
  for (int n = 8; n <= 4096; ++n) {
    int left = n;
    for (int f : {2, 3, 5})
      while (left % f == 0) left /= f;
    if (left == 1 && (n <= kMaxGeneralSide || (n & (n - 1)) == 0)) sides.push_back(n);
  }
  long checked = 0;
  for (int nx : sides)
    for (int ny : sides) {
      if (!uses_general(nx, ny) || uses_rg(nx, ny)) continue;
      if (gen_smem_bytes(nx, ny, kGenMinTeams) > static_cast<size_t>(kGenSmemLimit)) continue;  // no context
      for (int masks : {1, 3, 64})
        for (int sms : {152, 7}) {
          const GenGeom g = gen_geom(nx, ny, masks, sms);
          if (g.teams < kGenMinTeams || g.teams > kGenMaxTeams || g.team_log < 6 || g.team_log > 7 ||
              (g.teams << g.team_log) > kGenMaxThreads ||
              gen_smem_bytes(nx, ny, g.teams) > static_cast<size_t>(kGenSmemLimit)) {
            std::printf("%d x %d, %d masks, %d SMs: %d teams of 2^%d threads\n", nx, ny, masks, sms, g.teams, g.team_log);
            return 0;
          }
          ++checked;
        }
    }
  std::printf("ok %ld\n", checked);
  return 0;
}
