// Where the one-launch check period (pdlp_period.cu) deals the kernels' groups
// and where it keeps the partial sums: host and device code, so that the
// placement can be checked without a GPU.
#pragma once

#include "pdlp_internal.cuh"

namespace pdlp {

// ---- the kernels' grids, dealt out over this launch's CTAs ----
//
// A multiple of G groups is dealt out whole: a group's eight virtual warps run
// on one CTA (a snake over the CTAs, as the groups' costs fall), which adds
// them, and part[a][group] is what the other CTAs read.  The rest, the first
// and most expensive groups (in a small LP: all of them), is spread by virtual
// warps, so that every CTA gets the same number of them and the longest rows
// meet on no scheduler; their sums go to part[a][v], and the totals add a
// group's eight.

constexpr int MAX_SLOTS = 8;  // whole groups of one CTA

template <bool CLUSTER>
__host__ __device__ __forceinline__ int spread_groups(int groups, int grid) {
  return CLUSTER ? groups : groups % grid;
}
// round r of a snake over the CTAs: this CTA's turn in it
__host__ __device__ __forceinline__ int snake(int round, int block, int grid) {
  return round * grid + ((round & 1) ? grid - 1 - block : block);
}
// doubles of nv values' partials
template <bool CLUSTER>
__host__ __device__ __forceinline__ size_t partials(int nv, int groups, int grid) {
  const int sg = spread_groups<CLUSTER>(groups, grid);
  return (size_t)nv * (8 * sg + groups - sg);
}

// The places (in doubles) of a launch's partial sums.  Each sum has one of its
// own, since a slower CTA may still read one phase's while the next phase
// writes; and ||dx||^2 has two, taken in turn.  Trial t's totals are read
// behind its second barrier, and the next trial's primal phase writes before
// the next barrier has let anyone through: into the other copy.  A copy is
// written again two trials later, behind the first barrier of trial t + 1,
// which every CTA reaches only after its totals of trial t.  (The dual step's
// sums are written behind that barrier as it is, and the check's once a
// launch.)
struct PeriodParts {
  size_t primal, primal_copy, dual, check_primal, check_dual, infeas, restart, end;
  __host__ __device__ __forceinline__ size_t primal_of(int trial) const { return primal + (trial & 1) * primal_copy; }
};
template <bool CLUSTER>
__host__ __device__ __forceinline__ PeriodParts period_parts(const PeriodGrids &g, int grid) {
  PeriodParts p;
  p.primal = 0;
  p.primal_copy = partials<CLUSTER>(NV_A, g.primal, grid);
  p.dual = p.primal + 2 * p.primal_copy;
  p.check_primal = p.dual + partials<CLUSTER>(NV_B, g.dual, grid);
  p.check_dual = p.check_primal + partials<CLUSTER>(NV_R1, g.check_primal, grid);
  p.infeas = p.check_dual + partials<CLUSTER>(NV_R2, g.check_dual, grid);
  p.restart = p.infeas + partials<CLUSTER>(NV_I, g.infeas, grid);
  p.end = p.restart + partials<CLUSTER>(NV_R3, g.restart, grid);
  return p;
}
// room for any plan's
inline size_t period_part_doubles() {
  return (size_t)(2 * NV_A + NV_B + NV_R1 + NV_R2 + NV_I + NV_R3) * PERIOD_PART_GROUPS;
}

}  // namespace pdlp
