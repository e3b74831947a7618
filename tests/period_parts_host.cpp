// Host driver for the placement of the check period's partial sums
// (paper_2311_12180_gb300/csrc/pdlp_period.cuh), used by
// tests/test_period_parts_host.py: reads "cluster grid primal dual
// check_primal check_dual infeas restart" and prints the room that a solver
// reserves, then "place length" (in doubles) of the primal sums of trials 0 to
// 3, the dual sums, the check's, the infeasibility's and the restart's.
#include <cstdio>

#include "pdlp_period.cuh"

using namespace pdlp;

template <bool CLUSTER>
void print(const PeriodGrids &g, int grid) {
  const PeriodParts p = period_parts<CLUSTER>(g, grid);
  std::printf("%zu\n", period_part_doubles());
  for (int t = 0; t < 4; ++t) std::printf("%zu %zu\n", p.primal_of(t), partials<CLUSTER>(NV_A, g.primal, grid));
  std::printf("%zu %zu\n", p.dual, partials<CLUSTER>(NV_B, g.dual, grid));
  std::printf("%zu %zu\n", p.check_primal, partials<CLUSTER>(NV_R1, g.check_primal, grid));
  std::printf("%zu %zu\n", p.check_dual, partials<CLUSTER>(NV_R2, g.check_dual, grid));
  std::printf("%zu %zu\n", p.infeas, partials<CLUSTER>(NV_I, g.infeas, grid));
  std::printf("%zu %zu\n", p.restart, partials<CLUSTER>(NV_R3, g.restart, grid));
}

int main() {
  int cluster, grid;
  PeriodGrids g;
  while (std::scanf("%d %d %d %d %d %d %d %d", &cluster, &grid, &g.primal, &g.dual, &g.check_primal, &g.check_dual,
                    &g.infeas, &g.restart) == 8)
    cluster ? print<true>(g, grid) : print<false>(g, grid);
  return 0;
}
