// One check period of restarted PDHG in one launch, for LPs whose iteration is
// bound by latency rather than by its gathers: up to `max_trials` Algorithm 2
// trials, then (when due) the restart / termination check and the restart,
// with the phases separated by a barrier over the CTAs instead of by kernel
// boundaries.
//
// What bounds it.  A small LP's iteration is a serial chain: gather latency,
// the row sums' FMAs, the sums over rows, the step test, and one barrier per
// half-step.  On GB300 a scheduler issues one FP64 warp instruction every 64
// cycles whatever the number of active lanes (measured: 64 cycles per
// dependent add, and no more with four independent chains), a division takes
// 575, a 64-bit shuffle 25, a load from the L2 300-500, a barrier over 152
// CTAs through an L2 counter 2400, the cluster barrier over 16 CTAs 470.
// Hence:
//   * Every CTA evaluates the step test for itself from the block partials:
//     two barriers a trial.  Several sums over rows go through one transposed
//     butterfly (14 values: 15 additions instead of 70), the step test divides
//     once (eta / omega and ||dy||^2 / omega come from 1 / omega by one
//     correction step, div_rn).
//   * A warp keeps the same rows for the whole period, so its indices and
//     values are copied into shared memory once and its inner loop waits for
//     the gathers only.
//   * LPs with little work run as one cluster (the rule is at period_plan).
//   * The check's phases are out of line, and little that the steps use lives
//     in local memory: each barrier's acquire empties the L1, so a spilled
//     register costs an L2 round trip.
// Measured per iteration of a long run, step and check kernels against this
// one: 16.9 / 8.2 us on a 200 x 500 LP, 18.5 / 15.5 on the 200 x 300
// transportation LP, 21.5 / 14.8 at 1e5 nonzeros of the power-law recipe, 35.5 /
// 29.9 at 1e6, 42.5 / 40.2 at 2e6.  From 1e6 on the FP64 pipe bounds it (each row's epilogue and
// each virtual warp's sums take whole warp instructions), and the gathers in
// flight: half of the step kernels' warps are gone.
//
// Results are those of the step and check kernels, bit for bit.  Every row is
// summed in the same order, and the sums over rows follow the kernels' trees:
// the phase is dealt out as the kernel's grid of 256-thread CTAs ("groups" of
// eight virtual warps, each with the kernel's items or elements), a virtual
// warp's lanes, a group's eight warps and the groups are added in the kernel's
// order, whichever SM they ran on.  So which path an LP takes never shows in
// its results, and pdlp_time_kernels may run the kernels one by one.
// Vectors that a phase reads and an earlier one wrote on another SM are
// loaded with plain coherent loads behind the barrier's acquire, never
// through the read-only path.

#include <algorithm>
#include <vector>

#include "pdlp_internal.cuh"
#include "pdlp_period.cuh"
#include "pdlp_step.cuh"

namespace pdlp {

namespace {

// Threads per CTA and gathers in flight per lane with the matrix resident in
// shared memory: a cluster has few rows for many registers, the whole GPU more
// rows (16 gathers would spill at 512 threads; 256 threads take 34.0 us an
// iteration at 1e6 nonzeros where 512 take 29.9, 13.5 against 14.9 at 1e5).
template <bool CLUSTER>
constexpr int PT = CLUSTER ? 256 : 512;
template <bool CLUSTER>
constexpr int PW = PT<CLUSTER> / 32;
template <bool CLUSTER>
constexpr int RU = CLUSTER ? 16 : 6;
constexpr int MAX_PW = 16;
constexpr int PU = 8;         // strides of 32 entries in flight per warp, matrix read from the L2
constexpr int PU2 = 4;        // the same for two gathered vectors
constexpr unsigned long long BAR_WAIT_NS = 2000000000ull;

__device__ __forceinline__ unsigned long long timer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// 0 for a negative index, else p[c] by a plain coherent load
__device__ __forceinline__ double ld_at(const double *p, int c) {
  double v;
  asm volatile("{\n .reg .pred q;\n setp.ge.s32 q, %2, 0;\n mov.f64 %0, 0d0000000000000000;\n @q ld.global.f64 %0, [%1];\n}\n"
               : "=d"(v)
               : "l"(p + (c >= 0 ? c : 0)), "r"(c));
  return v;
}

// Barrier over the grid: a cluster's hardware barrier, or a counter in global
// memory that only grows (`target`: its value once every CTA has arrived; the
// next launch starts from the value this one leaves in sync->base, a new state
// from 0).  All threads of a CTA call both halves; the barrier orders the CTA's
// writes before arrive() before every CTA's reads after wait().  The counter's
// wait() returns false in every thread after BAR_WAIT_NS.  The hardware barrier
// has no limit and needs none: a cluster is scheduled as a whole, and its CTAs
// total the same partials behind the same barriers (see period_parts for what
// keeps them the same), so they take the same decisions and pass the same
// number of barriers.
template <bool CLUSTER>
struct Barrier {
  PeriodSync *s;
  unsigned target;
  int *s_ok;
  __device__ __forceinline__ void arrive() {
    if constexpr (CLUSTER) {
      asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    } else {
      target += gridDim.x;
      __syncthreads();
      if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&s->count) : "memory");
    }
  }
  __device__ __forceinline__ bool wait() {
    if constexpr (CLUSTER) {
      asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
      return true;
    } else {
      if (threadIdx.x == 0) {
        int ok = 1, spins = 0;
        unsigned v;
        const unsigned long long t0 = timer_ns();
        for (;;) {
          asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&s->count) : "memory");
          if ((int)(v - target) >= 0) break;
          if ((++spins & 1023) == 0 && timer_ns() - t0 > BAR_WAIT_NS) {
            ok = 0;
            break;
          }
        }
        *s_ok = ok;
      }
      __syncthreads();
      return *s_ok != 0;
    }
  }
  __device__ __forceinline__ bool both() {
    arrive();
    return wait();
  }
};

// f(v, slot) for each of the warp's virtual warps; slot < 0: spread.
template <bool CLUSTER, class F>
__device__ __forceinline__ void for_virtual_warps(int groups, F &&f) {
  const int G = (int)gridDim.x, blk = (int)blockIdx.x, wid = threadIdx.x >> 5;
  const int sg = spread_groups<CLUSTER>(groups, G), slots = (groups - sg) / G;
  // whole groups: warps 0-7 take even slots, 8-15 odd ones; spread warps start
  // with those that have a slot less
  int round = (wid + ((slots & 1) && !CLUSTER ? PW<CLUSTER> - 8 : 0)) % PW<CLUSTER>, slot = wid >> 3;
  for (;;) {  // one call of f: it is inlined
    int v, s = -1;
    if (slot < slots) {
      s = slot;
      v = 8 * (sg + snake(slot, blk, G)) + (wid & 7);
      slot += PW<CLUSTER> / 8;
    } else {
      if (round * G >= 8 * sg) break;
      v = snake(round, blk, G);
      round += PW<CLUSTER>;
      if (v >= 8 * sg) continue;
    }
    f(v, s);
  }
}

// items v, 2 nv - 1 - v, 2 nv + v, ... of the cost-sorted list, as spmv_sell
template <class F>
__device__ __forceinline__ void for_items(int v, int nv, int nitems, F &&f) {
  for (int b = 0;; ++b) {
    const long long first = (long long)b * nv, it = first + ((b & 1) ? nv - 1 - v : v);
    if (first >= nitems || it >= nitems) break;
    f((int)it);
  }
}

// A virtual warp's lane sums x[0..NV) -> its warp sums, to the partials
// (spread) or to the CTA's table.
template <bool CLUSTER, int NV, int STRIDE = 16>
__device__ __forceinline__ void put_sums(double (&x)[NV], int v, int slot, int groups, double *part,
                                         double (*tab)[8][STRIDE], int at) {
  constexpr int NP = pow2_at_least(NV), SPAN = 32 / NP;
  const int lane = threadIdx.x & 31;
  bool any = false;
#pragma unroll
  for (int a = 0; a < NV; ++a) any |= __double_as_longlong(x[a]) != 0;
  const unsigned mask = __ballot_sync(0xffffffffu, any);
  auto put = [&](int a, double s) {
    if (slot < 0)
      part[(size_t)a * 8 * spread_groups<CLUSTER>(groups, (int)gridDim.x) + v] = s;
    else
      tab[slot][v & 7][at + a] = s;
  };
  if (mask & (mask - 1)) {
    butterfly<NV, NP, 16>(x, lane);
    if (lane % SPAN == 0 && lane / SPAN < NV) put(lane / SPAN, x[0]);
  } else if (lane == (mask ? __ffs(mask) - 1 : 0)) {  // one lane holds all (a long row) or none does: nothing to add
#pragma unroll
    for (int a = 0; a < NV; ++a) put(a, x[a]);
  }
}

// The CTA's table -> part[a][group] for the values [at, at + NV): eight lanes
// add a group's eight warps.  Call with the table complete (a CTA barrier).
template <bool CLUSTER, int NV, int STRIDE = 16>
__device__ __forceinline__ void put_groups(int groups, double *part, const double (*tab)[8][STRIDE], int at) {
  const int G = (int)gridDim.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int sg = spread_groups<CLUSTER>(groups, G), slots = (groups - sg) / G;
  for (int t0 = 4 * wid; t0 < NV * slots; t0 += 4 * PW<CLUSTER>) {
    const int t = t0 + (lane >> 3), a = t % NV, slot = t / NV;
    const int c = snake(slot, (int)blockIdx.x, G);
    const bool on = t < NV * slots;
    double s = on ? tab[slot][lane & 7][at + a] : 0.0;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((lane & 7) == 0 && on) part[(size_t)NV * 8 * sg + (size_t)a * (groups - sg) + c] = s;
  }
}

// Partials of value a of nv; group c's sum is its partial or (spread) its
// eight warps' in the order of the xor tree over eight lanes.
struct Source {
  const double *part;
  int groups, a, nv;
};
// What lane `lane` of warp r of the kernel's last CTA adds up: its thread's
// groups t, t + 256, ...
template <bool CLUSTER>
__device__ __forceinline__ double last_cta_lane(const Source &p, int r, int lane) {
  const int sg = spread_groups<CLUSTER>(p.groups, (int)gridDim.x);
  const double *const rest = p.part + (size_t)p.nv * 8 * sg + (size_t)p.a * (p.groups - sg) - sg;
  double s = 0.0;
  bool have = false;
#pragma unroll 1
  for (int c0 = 32 * r; c0 < p.groups; c0 += 256) {
    const int c = c0 + lane;
    double g;
    g = __ldcg(c < sg ? p.part : rest + min(c, p.groups - 1));
    if (c0 < sg) {  // some of the warp's groups are spread
      const double *q = p.part + ((size_t)p.a * sg + min(c, sg - 1)) * 8;
      double w[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) w[k] = __ldcg(q + k);
      const double t = ((w[0] + w[4]) + (w[2] + w[6])) + ((w[1] + w[5]) + (w[3] + w[7]));
      if (c < sg) g = t;
    }
    if (c < p.groups) s = have ? s + g : g;
    have = true;
  }
  return s;
}

// Totals over the groups (behind a grid barrier) into tot[0..NV), value a's
// partials given by src(a), in the order of the kernel's last CTA: its
// threads, the tree over a warp's lanes, the tree over its eight warps.  A
// warp takes one value of one of those warps while there are few, all values
// of one otherwise (a transposed butterfly).  Ends with a CTA barrier.
template <bool CLUSTER, int NV, class F>
__device__ __forceinline__ void grid_totals(F &&src, double *tot, double (*tw)[8]) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int most = 0;
#pragma unroll
  for (int a = 0; a < NV; ++a) most = max(most, src(a).groups);
  const int rows = (min(most, 256) + 31) / 32;
  if (NV * rows <= PW<CLUSTER>) {
    if (wid < NV * rows) {
      const int a = wid % NV, r = wid / NV;
      double s = last_cta_lane<CLUSTER>(src(a), r, lane);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) (rows == 1 ? tot[a] : tw[a][r]) = s;
    }
  } else if (wid < rows) {
    constexpr int NP = pow2_at_least(NV), SPAN = 32 / NP;
    double x[NV];
#pragma unroll
    for (int a = 0; a < NV; ++a) x[a] = last_cta_lane<CLUSTER>(src(a), wid, lane);
    butterfly<NV, NP, 16>(x, lane);
    if (lane % SPAN == 0 && lane / SPAN < NV) (rows == 1 ? tot[lane / SPAN] : tw[lane / SPAN][wid]) = x[0];
  }
  __syncthreads();
  if (rows == 1) return;
  for (int a = wid; a < NV; a += PW<CLUSTER>) {
    double s = (lane & 7) < rows ? tw[a][lane & 7] : 0.0;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) tot[a] = s;
  }
  __syncthreads();
}

// ---- SpMV of a virtual warp ----

// As strided_dot for a matrix that stays in the L2: the last, partial batch
// is loaded in one go as well (its latency would otherwise be paid once per
// leftover stride).
template <int U, typename VT, int NV, bool SCALED>
__device__ __forceinline__ void batch_dot(const int32_t *__restrict__ ip, const VT *__restrict__ vp, int cnt,
                                          const double *const (&xs)[NV], const double (&sc)[NV], double (&acc)[NV]) {
  for (int k = 0; k < cnt; k += U) {
    int c[U];
    VT v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {  // past the end: the last stride again, not used
      const int e = 32 * min(k + u, cnt - 1);
      c[u] = __ldg(ip + e);
      v[u] = __ldg(vp + e);
    }
    double g[NV][U];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int a = 0; a < NV; ++a) g[a][u] = ld_at(xs[a], c[u]);
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (u == 0 || k + u < cnt) {
#pragma unroll
        for (int a = 0; a < NV; ++a) acc[a] = fma(widen(v[u]), SCALED && (NV == 1 || a > 0) ? sc[a] * g[a][u] : g[a][u], acc[a]);
      }
  }
}

// A warp's items of one matrix, copied into shared memory for the length of
// a period: descriptors, then column indices and values in the order the warp
// walks them, 32 per stride.  The pointers move on as a phase walks.
struct WarpShare {
  const int4 *desc;
  const int32_t *idx;
  const void *val;
  int bits;  // of a value: 64 or 32; 0: not resident
};

__device__ __forceinline__ int item_strides(const int4 &d) { return d.y > 0 ? d.z : (d.z + 31) >> 5; }

// Sum over `cnt` resident strides.
template <int U, typename VT>
__device__ __forceinline__ double resident_dot(const int32_t *ip, const VT *vp, int cnt, const double *x) {
  double acc = 0.0;
  for (int k = 0; k < cnt; k += U) {
    double g[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      int c = ip[32 * min(k + u, cnt - 1)];
      if (k + u >= cnt) c = -1;
      g[u] = ld_at(x, c);
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (u == 0 || k + u < cnt) acc = fma(widen(vp[32 * (k + u)]), g[u], acc);
  }
  return acc;
}

// The rows of virtual warp v of nv, each finished through ep.  w != null: the
// warp's resident share, which moves on.
template <int U, int UR, typename VT, int NV, bool SCALED, class Epi>
__device__ __forceinline__ void vwarp_spmv(const SellMat &A, const VT *__restrict__ val, WarpShare *w, int v, int nv,
                                           const double *const (&xs)[NV], const double (&sc)[NV], Epi &ep, int *rows,
                                           double *tot) {
  const int lane = threadIdx.x & 31;
  LongRows<NV> lr;
  lr.t = 0;
  lr.rows = rows;
  lr.tot = tot;
  for_items(v, nv, A.nitems, [&](int it) {
    const int4 d = w ? *w->desc : __ldg(A.items + it);
    const int cnt = item_strides(d);
    const bool slice = d.y > 0, has = slice && lane < d.y;
    if (has) ep.prefetch(d.x + lane);
    double acc[NV];
#pragma unroll
    for (int a = 0; a < NV; ++a) acc[a] = 0.0;
    if (w) {
      if constexpr (NV == 1) acc[0] = resident_dot<UR, VT>(w->idx + lane, static_cast<const VT *>(w->val) + lane, cnt, xs[0]);
      w->desc += 1;
      w->idx += 32 * cnt;
      w->val = static_cast<const VT *>(w->val) + 32 * cnt;
    } else {
      batch_dot<U, VT, NV, SCALED>(A.idx + d.w + lane, val + d.w + lane, cnt, xs, sc, acc);
    }
    if (slice) {
      if (has) ep.finish(d.x + lane, acc);
    } else {
      long_push(lr, acc, d.x, ep);
    }
  });
  if (lr.t > 0) long_flush(lr, ep);
}

// A step's product.  VT: the values a resident share holds; in the FP32-values
// mode (VT float) the steps may have moved to the FP64 values (f32 = 0), which
// are then read from the L2.
template <bool CLUSTER, typename VT, class Epi>
__device__ __forceinline__ void step_spmv(const SellMat &A, WarpShare &w, int f32, int v, int nv, const double *x,
                                          Epi &ep, int *rows, double *tot) {
  const double *const xs[1] = {x};
  const double sc[1] = {1.0};
  if constexpr (sizeof(VT) == 4) {
    if (!f32)
      vwarp_spmv<PU2, RU<CLUSTER>, double, 1, false>(A, A.val, nullptr, v, nv, xs, sc, ep, rows, tot);
    else if (w.bits)
      vwarp_spmv<PU, RU<CLUSTER>, float, 1, false>(A, A.val32, &w, v, nv, xs, sc, ep, rows, tot);
    else
      vwarp_spmv<PU, RU<CLUSTER>, float, 1, false>(A, A.val32, nullptr, v, nv, xs, sc, ep, rows, tot);
  } else {
    if (w.bits)
      vwarp_spmv<PU, RU<CLUSTER>, double, 1, false>(A, A.val, &w, v, nv, xs, sc, ep, rows, tot);
    else
      vwarp_spmv<PU, RU<CLUSTER>, double, 1, false>(A, A.val, nullptr, v, nv, xs, sc, ep, rows, tot);
  }
}

// Copies the warp's items of one matrix into the CTA's dynamic shared memory
// (`limit` bytes, `used` so far): the warps count their items and strides,
// take consecutive blocks, and copy.  A CTA whose share does not fit reads
// this matrix from the L2 instead (the same sums in the same order).
template <bool CLUSTER, typename VT>
__device__ __forceinline__ void take_share(const SellMat &A, const VT *__restrict__ val, int groups, unsigned char *dyn,
                                           int limit, int &used, int (*s_cnt)[2], WarpShare &w) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int items = 0, strides = 0;
  for_virtual_warps<CLUSTER>(groups, [&](int v, int) {
    for_items(v, 8 * groups, A.nitems, [&](int it) {
      ++items;
      strides += item_strides(__ldg(A.items + it));
    });
  });
  __syncthreads();  // s_cnt of the matrix before has been read
  if (lane == 0) {
    s_cnt[wid][0] = items;
    s_cnt[wid][1] = strides;
  }
  __syncthreads();
  int i0 = 0, e0 = 0, it = 0, et = 0;
  for (int v = 0; v < PW<CLUSTER>; ++v) {
    if (v == wid) {
      i0 = it;
      e0 = et;
    }
    it += s_cnt[v][0];
    et += s_cnt[v][1];
  }
  const int bytes = 16 * it + 32 * et * (4 + (int)sizeof(VT));
  w.bits = 0;
  if (used + bytes > limit) return;
  int4 *desc = reinterpret_cast<int4 *>(dyn + used) + i0;
  VT *sv = reinterpret_cast<VT *>(dyn + used + 16 * it) + 32 * e0;
  int32_t *si = reinterpret_cast<int32_t *>(dyn + used + 16 * it + 32 * et * (int)sizeof(VT)) + 32 * e0;
  w = WarpShare{desc, si, sv, 8 * (int)sizeof(VT)};
  for_virtual_warps<CLUSTER>(groups, [&](int v, int) {
    for_items(v, 8 * groups, A.nitems, [&](int i) {
      const int4 d = __ldg(A.items + i);
      if (lane == 0) *desc = d;
      ++desc;
      const int n = item_strides(d);
#pragma unroll 4
      for (int k = 0; k < n; ++k) {
        si[32 * k + lane] = __ldg(A.idx + d.w + 32 * k + lane);
        sv[32 * k + lane] = __ldg(val + d.w + 32 * k + lane);
      }
      si += 32 * n;
      sv += 32 * n;
    });
  });
  __syncwarp();
  used += (bytes + 15) & ~15;
}

// ---- phases ----

// The solver state a CTA keeps while it steps: every CTA computes the same
// values, CTA 0 writes them back.
struct StepState {
  double eta, omega, romega, tau, sigma, W;
  long long k, t, attempts;
  long long left;  // accepted steps until the next check
  int cur, need_g, pending, status;
};

struct Scratch {
  double tab[MAX_SLOTS][8][16];
  double tw[NV_I][8];
  double tot[16], tot2[NV_R2], tot3[NV_I];
  double ltot[MAX_PW][64];
  int rows[MAX_PW][32];
  StepState S;
  int cnt[MAX_PW][2];
  int ok;
};

// Algorithm 2's acceptance test (one thread): step_test's operations, with
// the divisions by omega taken from 1 / omega (div_rn) and what does not need
// the sums (e1f = 1 - (k + 2)^-0.3, e2 = (1 + (k + 2)^-0.6) eta, W + eta) ready
// before they are.
__device__ __forceinline__ void step_rule(StepState &S, const double *tot, double e1f, double e2, double Wn) {
  const double dx2 = tot[0], dy2 = tot[1], cross = tot[2], eta = S.eta, omega = S.omega, ia = fabs(cross);
  const double eta_bar = ia > 0.0 ? fma(omega, dx2, div_rn(dy2, omega, S.romega)) / (2.0 * ia) : CUDART_INF;
  const double e1 = e1f * eta_bar;
  const double eta_next = e1 < e2 ? e1 : e2;
  S.attempts += 1;
  if (!finite_bits(dx2) || !finite_bits(dy2) || !finite_bits(cross) || isnan(eta_bar) || !(eta_next > 0.0)) {
    S.status = ST_NUMERICAL;
    return;
  }
  S.eta = eta_next;
  S.tau = div_rn(eta_next, omega, S.romega);
  S.sigma = eta_next * omega;
  if (eta <= eta_bar) {
    S.cur ^= 1;
    S.k += 1;
    S.t += 1;
    S.W = Wn;
    S.need_g = 1;
    if (--S.left == 0) S.pending = 1;
  } else {
    S.need_g = 0;
  }
}

// The primal half-step.  The lane sums of the warp's last virtual warp stay in
// `pend` (pv, ps: where they go): they are added while the barrier fills.
template <bool CLUSTER, bool QP, typename VT>
__device__ __forceinline__ void primal_phase(const SellMat &KT, WarpShare w, const Vecs &V, const PeriodGrids &g,
                                             int f32, Scratch &sm, double *part, double &pend, int &pv, int &ps) {
  const StepState &S = sm.S;
  const int cur = S.cur, nxt = cur ^ 1, wid = threadIdx.x >> 5, lane = threadIdx.x & 31, nv = 8 * g.primal;
  PrimalEpi<QP> ep;
  ep.c = V.c;
  ep.l = V.l;
  ep.u = V.u;
  ep.qd = V.qd;
  ep.x = V.x[cur];
  ep.sx = V.sx[cur];
  ep.g = V.g;
  ep.xn = V.x[nxt];
  ep.sxn = V.sx[nxt];
  ep.tau = S.tau;
  ep.eta = S.eta;
  const bool need_g = S.need_g != 0;
  pv = -1;
  for_virtual_warps<CLUSTER>(g.primal, [&](int v, int slot) {
    if (pv >= 0) {
      double s[1] = {pend};
      put_sums<CLUSTER, 1>(s, pv, ps, g.primal, part, sm.tab, 0);
    }
    ep.dx2 = 0.0;
    if (need_g) {
      step_spmv<CLUSTER, VT>(KT, w, f32, v, nv, V.y[cur], ep, sm.rows[wid], sm.ltot[wid]);
    } else {  // rejected trial: g = K'y is unchanged, only the projection reruns
      for (int j = 32 * v + lane; j < V.n; j += 32 * nv) {
        ep.prefetch(j);
        ep.apply(j, V.g[j], false);
      }
    }
    pend = ep.dx2;
    pv = v;
    ps = slot;
  });
}

template <bool CLUSTER, typename VT>
__device__ __forceinline__ void dual_phase(const SellMat &K, WarpShare w, const Vecs &V, const PeriodGrids &g, int f32,
                                           Scratch &sm, double *part) {
  const StepState &S = sm.S;
  const int cur = S.cur, nxt = cur ^ 1, wid = threadIdx.x >> 5;
  DualEpi ep;
  ep.q = V.q;
  ep.y = V.y[cur];
  ep.kx = V.Kx[cur];
  ep.sy = V.sy[cur];
  ep.yn = V.y[nxt];
  ep.kxn = V.Kx[nxt];
  ep.syn = V.sy[nxt];
  ep.sigma = S.sigma;
  ep.eta = S.eta;
  ep.n_eq = V.n_eq;
  for_virtual_warps<CLUSTER>(g.dual, [&](int v, int slot) {
    ep.dy2 = 0.0;
    ep.cross = 0.0;
    step_spmv<CLUSTER, VT>(K, w, f32, v, 8 * g.dual, V.x[nxt], ep, sm.rows[wid], sm.ltot[wid]);
    double s[2] = {ep.dy2, ep.cross};
    put_sums<CLUSTER, 2>(s, v, slot, g.dual, part, sm.tab, 1);
  });
}

// ---- the check's passes (K' and K), as k_check_primal and k_check_dual, its
// infeasibility sums and the restart: once a period, from the L2, and out of
// line (their registers would spill the steps' into local memory, which the
// barriers' acquire empties from the L1) ----

template <bool CLUSTER>
__device__ __noinline__ void check_primal_phase(const SellMat &KT, const Vecs &V, int groups, bool check, double invW,
                                                bool keep, Scratch &sm, double *part) {
  const int cur = sm.S.cur, wid = threadIdx.x >> 5;
  CheckPrimalEpi ep;
  ep.c = V.c;
  ep.l = V.l;
  ep.u = V.u;
  ep.rd2 = V.rD2;
  ep.x = V.x[cur];
  ep.sx = V.sx[cur];
  ep.g = V.g;
  ep.gbar = V.gbar;
  ep.g0 = V.g0;
  ep.gprev = V.gprev;
  ep.qd = V.qd;
  ep.invW = invW;
  ep.kind = !check ? 0 : (sm.S.need_g ? 1 : 2);
  ep.keep = keep;
  for_virtual_warps<CLUSTER>(groups, [&](int v, int slot) {
#pragma unroll
    for (int a = 0; a < NV_R1; ++a) ep.acc[a] = 0.0;
    if (ep.kind == 1) {
      const double *const xs[2] = {V.y[cur], V.sy[cur]};
      const double sc[2] = {1.0, invW};
      vwarp_spmv<PU2, RU<CLUSTER>, double, 2, true>(KT, KT.val, nullptr, v, 8 * groups, xs, sc, ep, sm.rows[wid], sm.ltot[wid]);
    } else if (ep.kind == 0) {
      const double *const xs[1] = {V.y[cur]};
      const double sc[1] = {1.0};
      vwarp_spmv<PU2, RU<CLUSTER>, double, 1, false>(KT, KT.val, nullptr, v, 8 * groups, xs, sc, ep, sm.rows[wid], sm.ltot[wid]);
    } else {
      const double *const xs[1] = {V.sy[cur]};
      const double sc[1] = {invW};
      vwarp_spmv<PU2, RU<CLUSTER>, double, 1, true>(KT, KT.val, nullptr, v, 8 * groups, xs, sc, ep, sm.rows[wid], sm.ltot[wid]);
    }
    put_sums<CLUSTER, NV_R1>(ep.acc, v, slot, groups, part, sm.tab, 0);
  });
}

template <bool CLUSTER>
__device__ __noinline__ void check_dual_phase(const SellMat &K, const Vecs &V, int groups, bool check, double invW,
                                              bool keep, Scratch &sm, double *part) {
  const int cur = sm.S.cur, wid = threadIdx.x >> 5;
  CheckDualEpi ep;
  ep.q = V.q;
  ep.rd1 = V.rD1;
  ep.y = V.y[cur];
  ep.sy = V.sy[cur];
  ep.kx = V.Kx[cur];
  ep.kxbar = V.Kxbar;
  ep.kx0 = V.kx0;
  ep.invW = invW;
  ep.check = check ? 1 : 0;
  ep.n_eq = V.n_eq;
  ep.keep = keep;
  for_virtual_warps<CLUSTER>(groups, [&](int v, int slot) {
#pragma unroll
    for (int a = 0; a < NV_R2; ++a) ep.acc[a] = 0.0;
    if (!check) {
      const double *const xs[1] = {V.x[cur]};
      const double sc[1] = {1.0};
      vwarp_spmv<PU2, RU<CLUSTER>, double, 1, false>(K, K.val, nullptr, v, 8 * groups, xs, sc, ep, sm.rows[wid], sm.ltot[wid]);
    } else {
      const double *const xs[1] = {V.sx[cur]};
      const double sc[1] = {invW};
      vwarp_spmv<PU2, RU<CLUSTER>, double, 1, true>(K, K.val, nullptr, v, 8 * groups, xs, sc, ep, sm.rows[wid], sm.ltot[wid]);
    }
    put_sums<CLUSTER, NV_R2>(ep.acc, v, slot, groups, part, sm.tab, 0);
  });
}

template <bool CLUSTER>
__device__ __noinline__ void infeas_phase(const Vecs &V, int groups, Scratch &sm, double *part) {
  for_virtual_warps<CLUSTER>(groups, [&](int v, int slot) {
    double a[NV_I];
    infeas_sums(V, sm.S.cur, sm.S.need_g ? 0 : 1, 32 * v + (int)(threadIdx.x & 31), 256 * groups, a);
    put_sums<CLUSTER, NV_I>(a, v, slot, groups, part, sm.tab, 0);
  });
}

template <bool CLUSTER>
__device__ __noinline__ void restart_phase(const Vecs &V, int groups, bool avg, bool keep, double invW, Scratch &sm,
                                           double *part) {
  for_virtual_warps<CLUSTER>(groups, [&](int v, int slot) {
    double a[2];
    restart_sums(V, sm.S.cur, avg, keep, invW, 32 * v + (int)(threadIdx.x & 31), 256 * groups, a);
    put_sums<CLUSTER, 2>(a, v, slot, groups, part, sm.tab, 0);
  });
}

template <bool CLUSTER, int NV>
__device__ __noinline__ void check_totals(const double *part, int groups, double *tot, double (*tw)[8]) {
  grid_totals<CLUSTER, NV>([&](int a) { return Source{part, groups, a, NV}; }, tot, tw);
}
__device__ __noinline__ void decide(DevState *st, TraceRec *trace, const double *p, const double *d, const double *inf) {
  check_decide(st, trace, p, d, inf);
}
__device__ __noinline__ void finish_restart(DevState *st, TraceRec *trace, double dx2, double dy2) {
  restart_finish(st, trace, dx2, dy2);
}

// Trials until a check is due (at most max_trials), the check, the restart.
template <bool CLUSTER, bool QP, typename VT>
__global__ void __launch_bounds__(PT<CLUSTER>, 1) k_period(const __grid_constant__ SellMat K, const __grid_constant__ SellMat KT,
                                                  const __grid_constant__ Vecs V, const __grid_constant__ PeriodGrids g,
                                                  DevState *st, PeriodSync *ps, double *part, int max_trials,
                                                  int share_bytes, int stall) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ Scratch sm;
  StepState &S = sm.S;
  if (st->status != ST_RUNNING) return;
  if (!CLUSTER && stall && blockIdx.x == 1) return;
  const int f32 = st->use_f32, tid = threadIdx.x;
  const bool keep = st->eps_infeas > 0.0, check = st->mode == MODE_CHECK;
  Barrier<CLUSTER> bar{ps, CLUSTER ? 0u : ps->base, &sm.ok};
  if (tid == 0) {
    const int P = st->P;
    const long long max_iter = st->max_iter;
    S.eta = st->eta;
    S.omega = st->omega;
    S.romega = 1.0 / S.omega;
    S.tau = S.eta / S.omega;
    S.sigma = S.eta * S.omega;
    S.W = st->W;
    S.k = st->k;
    S.t = st->t;
    S.attempts = st->attempts;
    S.cur = st->cur;
    S.need_g = st->need_g;
    S.pending = st->check_pending;
    S.status = ST_RUNNING;
    S.left = P - S.k % P;
    if (S.left > max_iter - S.k) S.left = max_iter - S.k;
    if (S.left < 1) S.left = 1;
  }
  const PeriodParts pp = period_parts<CLUSTER>(g, (int)gridDim.x);
  double *const pB = part + pp.dual, *const pR1 = part + pp.check_primal, *const pR2 = part + pp.check_dual,
               *const pI = part + pp.infeas, *const pR3 = part + pp.restart;
  WarpShare wk, wt;
  wk.bits = wt.bits = 0;
  if (share_bytes && max_trials > 0 && (sizeof(VT) == 8 || f32)) {
    int used = 0;
    const VT *kv, *tv;
    if constexpr (sizeof(VT) == 4) {
      kv = K.val32;
      tv = KT.val32;
    } else {
      kv = K.val;
      tv = KT.val;
    }
    take_share<CLUSTER>(KT, tv, g.primal, dyn, share_bytes, used, sm.cnt, wt);
    take_share<CLUSTER>(K, kv, g.dual, dyn, share_bytes, used, sm.cnt, wk);
  }
  __syncthreads();
  bool ok = true, stepped = false;
  // CTA 0 writes the state only behind a barrier that every CTA reaches after
  // reading it
  for (int trial = 0; trial < max_trials && !S.pending && S.status == ST_RUNNING; ++trial) {
    double e1f = 0.0, e2 = 0.0, Wn = 0.0, pend = 0.0;
    int pv, psl = 0;
    double *const pA = part + pp.primal_of(trial);  // a slower CTA may still read the last trial's
    if (tid == PT<CLUSTER> - 32) {  // the step test's factors, by a warp with little else to do
      const long long k = S.k;
      const double p3 = k < V.npw ? __ldg(V.pw + k) : pow((double)(k + 2), -0.3);
      const double p6 = k < V.npw ? __ldg(V.pw + V.npw + k) : pow((double)(k + 2), -0.6);
      e1f = 1.0 - p3;
      e2 = (1.0 + p6) * S.eta;
      Wn = S.W + S.eta;
    }
    primal_phase<CLUSTER, QP, VT>(KT, wt, V, g, f32, sm, pA, pend, pv, psl);
    bar.arrive();
    if (pv >= 0) {
      double s[1] = {pend};
      put_sums<CLUSTER, 1>(s, pv, psl, g.primal, pA, sm.tab, 0);
    }
    ok = bar.wait();
    if (!ok) break;
    dual_phase<CLUSTER, VT>(K, wk, V, g, f32, sm, pB);
    if constexpr (!CLUSTER) {
      __syncthreads();
      put_groups<CLUSTER, 1>(g.primal, pA, sm.tab, 0);
      put_groups<CLUSTER, 2>(g.dual, pB, sm.tab, 1);
    }
    ok = bar.both();
    if (!ok) break;
    grid_totals<CLUSTER, 3>([&](int a) { return a ? Source{pB, g.dual, a - 1, 2} : Source{pA, g.primal, 0, 1}; }, sm.tot,
                            sm.tw);
    if (tid == PT<CLUSTER> - 32) step_rule(S, sm.tot, e1f, e2, Wn);
    __syncthreads();
    stepped = true;
  }
  const bool first = blockIdx.x == 0 && tid == 0;
  if (stepped && ok && first) {
    st->eta = S.eta;
    st->W = S.W;
    st->k = S.k;
    st->t = S.t;
    st->attempts = S.attempts;
    st->cur = S.cur;
    st->need_g = S.need_g;
    st->check_pending = S.pending;
    st->status = S.status;
  }
  if (ok && S.pending && S.status == ST_RUNNING) {
    const double invW = check ? 1.0 / S.W : 0.0;
    const bool inf = check && keep;
    check_primal_phase<CLUSTER>(KT, V, g.check_primal, check, invW, keep, sm, pR1);
    __syncthreads();
    put_groups<CLUSTER, NV_R1>(g.check_primal, pR1, sm.tab, 0);
    __syncthreads();
    check_dual_phase<CLUSTER>(K, V, g.check_dual, check, invW, keep, sm, pR2);
    __syncthreads();
    put_groups<CLUSTER, NV_R2>(g.check_dual, pR2, sm.tab, 0);
    if (inf) {  // by elements: behind a barrier, it reads this check's K'y
      ok = bar.both();
      if (ok) {
        infeas_phase<CLUSTER>(V, g.infeas, sm, pI);
        __syncthreads();
        put_groups<CLUSTER, NV_I>(g.infeas, pI, sm.tab, 0);
      }
    }
    if (ok) ok = bar.both();
    if (ok && blockIdx.x == 0) {
      check_totals<CLUSTER, NV_R1>(pR1, g.check_primal, sm.tot, sm.tw);
      check_totals<CLUSTER, NV_R2>(pR2, g.check_dual, sm.tot2, sm.tw);
      if (inf) check_totals<CLUSTER, NV_I>(pI, g.infeas, sm.tot3, sm.tw);
      if (tid == 0) decide(st, V.trace, sm.tot, sm.tot2, inf ? sm.tot3 : nullptr);
    }
    if (ok) ok = bar.both();
    if (ok && __ldcg(&st->status) == ST_RUNNING && __ldcg(&st->restart_to)) {
      restart_phase<CLUSTER>(V, g.restart, __ldcg(&st->restart_to) == 2, keep, invW, sm, pR3);
      __syncthreads();
      put_groups<CLUSTER, 2>(g.restart, pR3, sm.tab, 0);
      ok = bar.both();
      if (ok && blockIdx.x == 0) {
        check_totals<CLUSTER, 2>(pR3, g.restart, sm.tot, sm.tw);
        if (tid == 0) finish_restart(st, V.trace, sm.tot[0], sm.tot[1]);
      }
    }
  }
  if (first) {
    if (!CLUSTER) ps->base = bar.target;
    if (!ok) {
      ps->error = 1;
      st->status = ST_NUMERICAL;
    }
  }
}

}  // namespace

namespace {
// grid, block, shared memory and attribute of a plan's launch
void launch_config(const PeriodPlan &p, cudaStream_t s, cudaLaunchConfig_t &cfg, cudaLaunchAttribute (&at)[1]) {
  cfg = cudaLaunchConfig_t{};
  at[0] = cudaLaunchAttribute{};
  cfg.gridDim = dim3(p.ctas);
  cfg.blockDim = dim3(p.cluster ? PT<true> : PT<false>);
  cfg.dynamicSmemBytes = p.share_bytes;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (p.cluster) {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = p.ctas;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  } else {  // its CTAs wait on one another: all resident or none
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
  }
}
}  // namespace

// Which LPs run as one cluster of PERIOD_CLUSTER CTAs and which on the whole
// GPU: the FP64 instructions of an iteration (one per 32 stored entries, 6 and
// 9 per 32 rows for the epilogues) take 19 cycles each on an SM; the cluster's
// two barriers save 2 x 1900 cycles over the grid's, so it wins while its
// extra share of the work, (1/16 - 1/152) of them, costs less.
//
// `share_bytes`: the shared memory that holds the largest CTA's items of K and
// K', or 0 when that is more than PERIOD_SHARE_MAX: the rest of the SM's 256
// KB is the L1 that holds a line for every gather in flight.
//
// Where a cluster does not fit the SMs that the stream has (a cluster's CTAs
// share a GPC), the step and check kernels run the LP; too few SMs for the
// whole-GPU kernel show at its cooperative launch.
//
// Larger LPs keep the step and check kernels, whose grids have twice the warps:
// with many items, this path's warps walk them one after another.  Where the
// lines lie, in us an iteration, step kernels / this path:
//   stored entries  power-law recipe, 1e6 nonzeros 36 / 30 (2.0e6 stored), 2e6
//                   42.5 / 40.2 (4.07e6), 2.2e6 42.3 / 42.1 (4.47e6), 2.3e6
//                   43.8 / 45.0 (4.68e6), 3e6 48.5 / 67
//   long rows       rows of 60 entries in K and K': 7000 of each 29.7 / 27.8,
//                   10000 of each 31.8 / 36.4, 30000 of each 47 / 66
//   slices          transportation, 600 x 900 (16900, resident) 37.0 / 31.5,
//                   600 x 1000 (18800, not resident) 38.0 / 40.3; not resident:
//                   power law 1.8e5 x 1.8e5 (11100) 46.9 / 44.5, 3e5 x 1e5 of 4
//                   a row (12500) 34.7 / 38.7
//   long rows on one cluster, whose few warps pay each row's own sums: 300 in all
//                   (150 x 150 of 80) 15.9 / 13.6, 400 15.0 (whole GPU 13.5),
//                   600 19.5 (11.5)
//   FP32 values     the whole-GPU kernel of this mode also holds the FP64 product
//                   and spills: 2e5 nonzeros 21.6 / 19.3, 5e5 24.0 / 24.1, 1e6
//                   34.2 / 36.0; 60000 x 60000 of 4 a row (3750 slices) 18.9 /
//                   18.3, 1e5 x 1e5 of 3 (6250) 21.8 / 23.0
void period_plan(PeriodPlan &p, int32_t m, int32_t n, const int4 *k_items, int nk, const int4 *t_items, int nt,
                 int64_t stored, int value_bytes, int num_sms, cudaStream_t s) {
  int slices = 0;
  for (int i = 0; i < nk; ++i) slices += k_items[i].y > 0;
  for (int i = 0; i < nt; ++i) slices += t_items[i].y > 0;
  const int longs = nk + nt - slices;
  if (stored > PERIOD_STORED_MAX || longs > PERIOD_LONG_MAX || slices > PERIOD_SLICES_MAX) return;
  const PeriodGrids &g = p.grids;
  const double f64 = (double)stored / 32 + 6.0 * n / 32 + 9.0 * m / 32;
  const double extra = 19.0 * f64 * (1.0 / PERIOD_CLUSTER - 1.0 / num_sms);
  p.cluster = extra < 2.0 * 1900.0 && longs <= PERIOD_LONG_CLUSTER_MAX;
  if (!p.cluster && value_bytes == 4 && (stored > PERIOD_STORED_F32_MAX || slices > PERIOD_SLICES_F32_MAX)) return;
  p.ctas = p.cluster ? PERIOD_CLUSTER : num_sms;
  const int most_groups = std::max({g.primal, g.dual, g.check_primal, g.check_dual, g.infeas, g.restart});
  if (most_groups > (p.cluster ? PERIOD_PART_GROUPS / 8 : MAX_SLOTS * num_sms)) {
    p.ctas = 0;
    return;
  }
  std::vector<int64_t> bytes(p.ctas, 64);
  auto deal = [&](const int4 *items, int count, int groups) {
    const int nv = 8 * groups;
    for (int i = 0; i < count; ++i) {
      const int b = i / nv, r = i % nv, v = (b & 1) ? nv - 1 - r : r;
      const int strides = items[i].y > 0 ? items[i].z : (items[i].z + 31) >> 5;
      const int sg = p.cluster ? groups : groups % p.ctas;
      const int u = v < 8 * sg ? v : v / 8 - sg, round = u / p.ctas;
      bytes[snake(round, u % p.ctas, p.ctas) - round * p.ctas] += 16 + 32LL * strides * (4 + value_bytes);
    }
  };
  deal(k_items, nk, g.dual);
  deal(t_items, nt, g.primal);
  const int64_t most = *std::max_element(bytes.begin(), bytes.end());
  p.share_bytes = most <= PERIOD_SHARE_MAX ? (int)((most + 1023) / 1024 * 1024) : 0;
  if (!p.share_bytes && slices > PERIOD_SLICES_L2_MAX) {
    p.ctas = 0;
    return;
  }
  if (p.cluster) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[1];
    launch_config(p, s, cfg, at);
    int fit = 0;
    const cudaError_t e = value_bytes == 4 ? cudaOccupancyMaxActiveClusters(&fit, k_period<true, true, float>, &cfg)
                                           : cudaOccupancyMaxActiveClusters(&fit, k_period<true, true, double>, &cfg);
    if (e != cudaSuccess || fit < 1) {
      cudaGetLastError();
      p.ctas = 0;
    }
  }
}

cudaError_t period_init() {
  cudaError_t e = cudaSuccess;
  auto set = [&](const void *f, bool cluster) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, PERIOD_SHARE_MAX);
    if (e == cudaSuccess && cluster) e = cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  };
  set((const void *)k_period<true, false, double>, true);
  set((const void *)k_period<true, true, double>, true);
  set((const void *)k_period<true, false, float>, true);
  set((const void *)k_period<true, true, float>, true);
  set((const void *)k_period<false, false, double>, false);
  set((const void *)k_period<false, true, double>, false);
  set((const void *)k_period<false, false, float>, false);
  set((const void *)k_period<false, true, float>, false);
  return e;
}

cudaError_t launch_period(const PeriodPlan &p, const SellMat &K, const SellMat &KT, const Vecs &V, DevState *st,
                          int max_trials, cudaStream_t s) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[1];
  launch_config(p, s, cfg, at);
  auto go = [&](auto kernel) {
    return cudaLaunchKernelEx(&cfg, kernel, K, KT, V, p.grids, st, p.sync, p.part, max_trials, p.share_bytes, p.stall);
  };
  if (p.cluster) {
    if (K.val32) return V.qd ? go(k_period<true, true, float>) : go(k_period<true, false, float>);
    return V.qd ? go(k_period<true, true, double>) : go(k_period<true, false, double>);
  }
  if (K.val32) return V.qd ? go(k_period<false, true, float>) : go(k_period<false, false, float>);
  return V.qd ? go(k_period<false, true, double>) : go(k_period<false, false, double>);
}

}  // namespace pdlp
