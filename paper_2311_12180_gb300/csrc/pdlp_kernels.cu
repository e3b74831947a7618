// Hot-path kernels of restarted PDHG (cuPDLP.jl paper, Algorithms 1 and 2,
// eq. (pdhg), eq. (step-size), eq. (kkt), Sec. 3.4 and Sec. 4.1).
//
// One accepted PDHG iteration is two kernels:
//   k_primal  (rows of K'):  g = K'y (only when y changed), then
//             x' = proj_X(x - (eta/omega)(c - g)),  sx' = sx + eta x',
//             block partial of ||x' - x||^2.
//   k_dual    (rows of K):   Kx', then
//             y' = proj_Y(y + eta*omega (q - (2 Kx' - Kx))),  sy' = sy + eta y',
//             partials of ||y'-y||^2 and (y'-y)'(Kx' - Kx) = (y'-y)'K(x'-x);
//             its last CTA finishes all partials in a fixed order and runs the
//             Algorithm 2 test (accept: flip the buffer parity; reject: retry
//             with eta').
// Every P accepted steps the check kernels run:
//   k_check_primal (rows of K'):  K'y (if stale) and K'ybar in one pass over
//             K', dual residual / objective pieces for the current and the
//             average iterate, scaled (restart) and original (termination).
//   k_check_dual   (rows of K):   K xbar, primal residual pieces; its last CTA
//             applies Sec. 4.1 termination, GetRestartCandidate and the three
//             restart criteria of Sec. 3.4.
//   k_infeas (elementwise, between the two):  pieces of the infeasibility
//             certificates (Sec. 2.2, last bullet) for the difference of the
//             last two accepted iterates and for the normalised iterate,
//             from stored products (no SpMV).
//   k_restart (elementwise):      moves the candidate into the iterate, resets
//             the epoch average, and (last CTA) PrimalWeightUpdate.
// Every kernel reads the device state at entry and returns at once when it
// has nothing to do, so a fixed CUDA graph of P + E trial slots followed by the
// check kernels advances the solve by exactly one check period.
//
// SpMV (sliced ELL, see SellMat): rows are renumbered by length within
// their group at create, so that 32 consecutive internal rows have nearly
// equal lengths; such a slice is stored column-major (entry k of lane l at
// off + 32 k + l) and one warp computes it with one row per lane: coalesced
// 4-byte index loads, 8-byte value loads, random gathers of x / y straight
// into registers, FMAs in the row's own order, and the row's epilogue in the
// same lane -- no shared memory, no barriers, no cross-lane reduction.  The
// random gathers bind on GB300 (about 0.85 per clock per SM whatever the
// cache qualifier; 2e7 of them take ~74 us), then the narrow FP64 pipe
// (~1.6 DFMA per clock per SM), so the layout spends one FMA per stored
// entry and one epilogue per 32 rows.  Rows longer than SELL_LONG are stored
// contiguously and taken by a whole warp (lane-strided partial sums); their
// totals come out of a butterfly over 32 such rows at a time, followed by
// one vectorised epilogue.  Warps walk a cost-sorted item list in a snake
// order, independently: every warp keeps its own loads and gathers in
// flight.  Reductions are deterministic: fixed per-lane order, fixed
// butterfly and shuffle trees, fixed block order in the last CTA.  No
// atomics touch floating point.

#include "pdlp_internal.cuh"
#include "pdlp_step.cuh"

namespace pdlp {

// ---------------------------------------------------------------- reductions

// CTA-wide sums of NV values in a fixed order; totals land in every lane of
// warp 0.  s_red holds NV * NW doubles.  Every warp of the SM comes through
// here at the end of its launch, on an FP64 pipe that takes one warp
// instruction per 64 cycles and scheduler, so the sums are transposed (6
// additions for 3 values instead of 15, the same trees).  With this, the
// quotients below taken by one thread, and one pass over the partials in
// k_dual, an iteration at 2e7 nonzeros takes 216 us instead of 220, 207
// instead of 214 with FP32 values and 238 instead of 244 for a QP.
template <int NV>
__device__ __forceinline__ void block_sum(double (&v)[NV], double *s_red) {
  constexpr int NP = pow2_at_least(NV), SPAN = 32 / NP;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  butterfly<NV, NP, 16>(v, lane);
  if (lane % SPAN == 0 && lane / SPAN < NV) s_red[(lane / SPAN) * NW + wid] = v[0];
  __syncthreads();
  if (wid == 0) {
#pragma unroll
    for (int a = 0; a < NV; ++a) v[a] = lane < NW ? s_red[a * NW + lane] : 0.0;
    butterfly<NV, NP, 16>(v, lane);
    const double s = v[0];
#pragma unroll
    for (int a = 0; a < NV; ++a) v[a] = __shfl_sync(0xffffffffu, s, SPAN * a);
  }
  __syncthreads();
}

// a / b, computed by one thread for the CTA: a division is about nine FP64
// instructions, and every warp's copy of one would hold each scheduler for
// thousands of cycles (one FP64 warp instruction per 64).  `slot`: shared, of
// no other use in the kernel.
__device__ __forceinline__ double cta_quotient(double a, double b, double *slot) {
  if (threadIdx.x == 0) *slot = a / b;
  __syncthreads();
  return *slot;
}

// Writes this CTA's NV partial sums, and returns true in every thread of the
// CTA that finishes last; there `tot` holds the grid totals summed in block
// order (deterministic for a fixed grid).  The counter is reset for the next
// launch by that CTA.
// The NX values of each of `xcount` blocks in `xpart`, written by an earlier
// kernel, are summed with them into tot[NV..]: one pass over the L2 and one
// pair of barriers for both.
template <int NV, int NX = 0>
__device__ __forceinline__ bool grid_finish(double (&v)[NV], double *part, unsigned int *counter, double *s_red,
                                            int *s_flag, double (&tot)[NV + NX], const double *xpart = nullptr,
                                            int xcount = 0) {
  block_sum<NV>(v, s_red);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int a = 0; a < NV; ++a) part[(size_t)blockIdx.x * NV + a] = v[a];
    __threadfence();
    const unsigned int prev = atomicAdd(counter, 1u);
    *s_flag = (prev == gridDim.x - 1);
  }
  __syncthreads();
  if (!*s_flag) return false;
  __threadfence();
  double acc[NV + NX];
#pragma unroll
  for (int a = 0; a < NV + NX; ++a) acc[a] = 0.0;
  for (int b = threadIdx.x; b < (int)gridDim.x; b += NT) {
#pragma unroll
    for (int a = 0; a < NV; ++a) acc[a] += __ldcg(part + (size_t)b * NV + a);
  }
  if constexpr (NX > 0) {
    for (int b = threadIdx.x; b < xcount; b += NT) {
#pragma unroll
      for (int a = 0; a < NX; ++a) acc[NV + a] += __ldcg(xpart + (size_t)b * NX + a);
    }
  }
  block_sum<NV + NX>(acc, s_red);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int a = 0; a < NV + NX; ++a) s_red[a] = acc[a];
    *counter = 0u;
  }
  __syncthreads();
#pragma unroll
  for (int a = 0; a < NV + NX; ++a) tot[a] = s_red[a];
  __syncthreads();
  return true;
}

// Sums a partial array of `count` blocks x NV values written by an earlier
// kernel, in block order.  Totals valid in every lane of warp 0.
template <int NV>
__device__ __forceinline__ void sum_partials(const double *part, int count, double *s_red, double (&tot)[NV]) {
#pragma unroll
  for (int a = 0; a < NV; ++a) tot[a] = 0.0;
  for (int b = threadIdx.x; b < count; b += NT) {
#pragma unroll
    for (int a = 0; a < NV; ++a) tot[a] += __ldcg(part + (size_t)b * NV + a);
  }
  block_sum<NV>(tot, s_red);
}

template <bool QP>
__device__ __forceinline__ void primal_step(const SellMat &KT, const Vecs &V, const DevState *st, double *s_red,
                                            int (*s_rows)[32], double (*s_tot)[64]) {
  const int cur = st->cur, nxt = cur ^ 1, need_g = st->need_g, f32 = st->use_f32;
  const double eta = st->eta, omega = st->omega;
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
  ep.tau = cta_quotient(eta, omega, s_red + 16 * NW - 1);
  ep.eta = eta;
  ep.dx2 = 0.0;
  if (need_g) {
    const double *const xs[1] = {V.y[cur]};
    const double sc[1] = {1.0};
    if (f32)
      spmv_sell<SELL_U_P, float, 1, false>(KT, KT.val32, xs, sc, ep, s_rows[threadIdx.x >> 5], s_tot[threadIdx.x >> 5]);
    else
      spmv_sell<SELL_U_P, double, 1, false>(KT, KT.val, xs, sc, ep, s_rows[threadIdx.x >> 5], s_tot[threadIdx.x >> 5]);
  } else {
    // rejected trial: g = K'y is unchanged, only the projection reruns
    for (int j = blockIdx.x * NT + threadIdx.x; j < V.n; j += gridDim.x * NT) {
      ep.prefetch(j);
      ep.apply(j, V.g[j], false);
    }
  }
  double acc[1] = {ep.dx2};
  block_sum<1>(acc, s_red);
  if (threadIdx.x == 0) V.partA[blockIdx.x] = acc[0];
}

// STEP_MINB CTAs per SM: as many warps (gathers in flight) as the registers allow
__global__ void __launch_bounds__(NT, STEP_MINB) k_primal(SellMat KT, Vecs V, DevState *__restrict__ st) {
  __shared__ double s_red[16 * NW];
  __shared__ int s_rows[NW][32];
  __shared__ double s_tot[NW][64];
  if (st->status != ST_RUNNING || st->check_pending) return;
  primal_step<false>(KT, V, st, s_red, s_rows, s_tot);
}

// The QP's primal step (V.qd set), a kernel of its own so that the LP's
// keeps its register budget.
__global__ void __launch_bounds__(NT, STEP_MINB) k_primal_qp(SellMat KT, Vecs V, DevState *__restrict__ st) {
  __shared__ double s_red[16 * NW];
  __shared__ int s_rows[NW][32];
  __shared__ double s_tot[NW][64];
  if (st->status != ST_RUNNING || st->check_pending) return;
  primal_step<true>(KT, V, st, s_red, s_rows, s_tot);
}

// ---------------------------------------------------------------- dual step + Algorithm 2 test

// Algorithm 2 acceptance test (one thread).  eq. (step-size) with the
// interaction taken in absolute value; the exponent base counts the step
// being taken from 1 (k + 2 for k accepted steps so far).
__device__ void step_test(DevState *st, const Vecs &V, double dx2, double dy2, double cross) {
  const double eta = st->eta, omega = st->omega;
  const long long k = st->k;
  const double ia = fabs(cross);
  const double eta_bar = ia > 0.0 ? (omega * dx2 + dy2 / omega) / (2.0 * ia) : CUDART_INF;
  const double kk = (double)(k + 2);
  // the exponent factors come from a table built at create by the same pow()
  // (two FP64 powers are microseconds of serial latency on GB300's FP64 pipe,
  // on the critical path of every step)
  const double p3 = k < V.npw ? V.pw[k] : pow(kk, -0.3), p6 = k < V.npw ? V.pw[V.npw + k] : pow(kk, -0.6);
  const double e1 = (1.0 - p3) * eta_bar;
  const double e2 = (1.0 + p6) * eta;
  const double eta_next = e1 < e2 ? e1 : e2;
  st->attempts += 1;
  if (!isfinite(dx2) || !isfinite(dy2) || !isfinite(cross) || isnan(eta_bar) || !(eta_next > 0.0)) {
    st->status = ST_NUMERICAL;
    return;
  }
  st->eta = eta_next;
  if (eta <= eta_bar) {
    st->cur ^= 1;
    st->k = k + 1;
    st->t += 1;
    st->W += eta;
    st->need_g = 1;
    if ((k + 1) % st->P == 0 || k + 1 >= st->max_iter) st->check_pending = 1;
  } else {
    st->need_g = 0;  // g = K'y was refreshed by this trial's primal kernel
  }
}

__global__ void __launch_bounds__(NT, STEP_MINB) k_dual(SellMat K, Vecs V, DevState *__restrict__ st) {
  __shared__ double s_red[16 * NW];
  __shared__ int s_flag;
  __shared__ int s_rows[NW][32];
  __shared__ double s_tot[NW][64];
  if (st->status != ST_RUNNING || st->check_pending) return;
  const int cur = st->cur, nxt = cur ^ 1, f32 = st->use_f32;
  const double eta = st->eta, omega = st->omega;
  DualEpi ep;
  ep.q = V.q;
  ep.y = V.y[cur];
  ep.kx = V.Kx[cur];
  ep.sy = V.sy[cur];
  ep.yn = V.y[nxt];
  ep.kxn = V.Kx[nxt];
  ep.syn = V.sy[nxt];
  ep.sigma = eta * omega;
  ep.eta = eta;
  ep.dy2 = 0.0;
  ep.cross = 0.0;
  ep.n_eq = V.n_eq;
  const double *const xs[1] = {V.x[nxt]};
  const double sc[1] = {1.0};
  if (f32)
    spmv_sell<SELL_U_D, float, 1, false, DualEpi>(K, K.val32, xs, sc, ep, s_rows[threadIdx.x >> 5], s_tot[threadIdx.x >> 5]);
  else
    spmv_sell<SELL_U_D, double, 1, false, DualEpi>(K, K.val, xs, sc, ep, s_rows[threadIdx.x >> 5], s_tot[threadIdx.x >> 5]);
  double acc[2] = {ep.dy2, ep.cross};
  double tot[3];
  if (!grid_finish<2, 1>(acc, V.partB, &st->cnt[CNT_DUAL], s_red, &s_flag, tot, V.partA, V.gridA)) return;
  if (threadIdx.x == 0) step_test(st, V, tot[2], tot[0], tot[1]);
}

// ---------------------------------------------------------------- restart / termination check

__global__ void __launch_bounds__(NT, CHECK_MINB) k_check_primal(SellMat KT, Vecs V, DevState *__restrict__ st) {
  __shared__ double s_red[16 * NW];
  __shared__ int s_rows[NW][32];
  __shared__ double s_tot[NW][64];
  if (st->status != ST_RUNNING || !st->check_pending) return;
  const int mode = st->mode, cur = st->cur, need_g = st->need_g;
  const bool check = mode == MODE_CHECK;
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
  ep.invW = check ? cta_quotient(1.0, st->W, s_red + 16 * NW - 1) : 0.0;
  ep.kind = !check ? 0 : (need_g ? 1 : 2);
  ep.keep = st->eps_infeas > 0.0;
#pragma unroll
  for (int a = 0; a < NV_R1; ++a) ep.acc[a] = 0.0;
  if (ep.kind == 0) {
    const double *const xs[1] = {V.y[cur]};
    const double sc[1] = {1.0};
    spmv_sell<SELL_U_C, double, 1, false>(KT, KT.val, xs, sc, ep, s_rows[threadIdx.x >> 5], s_tot[threadIdx.x >> 5]);
  } else if (ep.kind == 1) {
    const double *const xs[2] = {V.y[cur], V.sy[cur]};
    const double sc[2] = {1.0, ep.invW};
    spmv_sell<SELL_U_C, double, 2, true>(KT, KT.val, xs, sc, ep, s_rows[threadIdx.x >> 5], s_tot[threadIdx.x >> 5]);
  } else {
    const double *const xs[1] = {V.sy[cur]};
    const double sc[1] = {ep.invW};
    spmv_sell<SELL_U_C, double, 1, true>(KT, KT.val, xs, sc, ep, s_rows[threadIdx.x >> 5], s_tot[threadIdx.x >> 5]);
  }
  block_sum<NV_R1>(ep.acc, s_red);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int a = 0; a < NV_R1; ++a) V.partR1[(size_t)blockIdx.x * NV_R1 + a] = ep.acc[a];
  }
}

__global__ void __launch_bounds__(NT) k_check_dual(SellMat K, Vecs V, DevState *__restrict__ st) {
  __shared__ double s_red[16 * NW];
  __shared__ int s_flag;
  __shared__ int s_rows[NW][32];
  __shared__ double s_tot[NW][64];
  if (st->status != ST_RUNNING || !st->check_pending) return;
  const int mode = st->mode, cur = st->cur;
  const bool check = mode == MODE_CHECK;
  CheckDualEpi ep;
  ep.q = V.q;
  ep.rd1 = V.rD1;
  ep.y = V.y[cur];
  ep.sy = V.sy[cur];
  ep.kx = V.Kx[cur];
  ep.kxbar = V.Kxbar;
  ep.kx0 = V.kx0;
  ep.invW = check ? cta_quotient(1.0, st->W, s_red + 16 * NW - 1) : 0.0;
  ep.check = check ? 1 : 0;
  ep.n_eq = V.n_eq;
  ep.keep = st->eps_infeas > 0.0;
#pragma unroll
  for (int a = 0; a < NV_R2; ++a) ep.acc[a] = 0.0;
  if (!check) {
    const double *const xs[1] = {V.x[cur]};
    const double sc[1] = {1.0};
    spmv_sell<SELL_U_C, double, 1, false>(K, K.val, xs, sc, ep, s_rows[threadIdx.x >> 5], s_tot[threadIdx.x >> 5]);
  } else {
    const double *const xs[1] = {V.sx[cur]};
    const double sc[1] = {ep.invW};
    spmv_sell<SELL_U_C, double, 1, true>(K, K.val, xs, sc, ep, s_rows[threadIdx.x >> 5], s_tot[threadIdx.x >> 5]);
  }
  double tot[NV_R2];
  if (!grid_finish<NV_R2>(ep.acc, V.partR2, &st->cnt[CNT_R2], s_red, &s_flag, tot)) return;
  double p[NV_R1];
  sum_partials<NV_R1>(V.partR1, V.gridR1, s_red, p);
  double inf[NV_I];
  const bool infeas = check && st->eps_infeas > 0.0;
  if (infeas) sum_partials<NV_I>(V.partI, V.gridI, s_red, inf);
  if (threadIdx.x == 0) check_decide(st, V.trace, p, tot, infeas ? inf : nullptr);
}

// ---------------------------------------------------------------- infeasibility detection

// Runs between k_check_primal (which refreshed g = K'y) and k_check_dual,
// whose last CTA sums the block partials and decides.
__global__ void __launch_bounds__(NT) k_infeas(Vecs V, DevState *__restrict__ st) {
  __shared__ double s_red[16 * NW];
  if (st->status != ST_RUNNING || !st->check_pending || st->mode != MODE_CHECK || !(st->eps_infeas > 0.0)) return;
  double a[NV_I];
  // the difference ray needs this check's stored K'y_prev
  infeas_sums(V, st->cur, st->need_g ? 0 : 1, blockIdx.x * NT + threadIdx.x, gridDim.x * NT, a);
  block_sum<NV_I>(a, s_red);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < NV_I; ++k) V.partI[(size_t)blockIdx.x * NV_I + k] = a[k];
  }
}

// ---------------------------------------------------------------- restart

__global__ void __launch_bounds__(NT) k_restart(Vecs V, DevState *__restrict__ st) {
  __shared__ double s_red[16 * NW];
  __shared__ int s_flag;
  if (st->status != ST_RUNNING || !st->check_pending || st->restart_to == 0) return;
  double acc[2];
  restart_sums(V, st->cur, st->restart_to == 2, st->eps_infeas > 0.0,
               cta_quotient(1.0, st->W, s_red + 16 * NW - 1), blockIdx.x * NT + threadIdx.x,
               gridDim.x * NT, acc);
  double tot[2];
  if (!grid_finish<2>(acc, V.partR3, &st->cnt[CNT_R3], s_red, &s_flag, tot)) return;
  if (threadIdx.x == 0) restart_finish(st, V.trace, tot[0], tot[1]);
}

// ---------------------------------------------------------------- output

// Original-space output, written in the original order of rows and
// columns: the current iterate or the average (projected onto X), or, for an
// infeasibility status, the certificate ray in place of the
// iterate it concerns (y for primal infeasibility, x for dual
// infeasibility; unprojected).
__global__ void __launch_bounds__(NT) k_output(Vecs V, DevState *__restrict__ st) {
  const int which = st->which, cur = st->cur, prv = cur ^ 1, status = st->status;
  const bool avg = which == 1;
  const bool xray = status == ST_DUAL_INFEASIBLE, yray = status == ST_PRIMAL_INFEASIBLE;
  const double invW = avg ? 1.0 / st->W : 0.0;
  const int stride = gridDim.x * NT;
  for (int j = blockIdx.x * NT + threadIdx.x; j < V.n; j += stride) {
    if (xray) {
      V.xout[V.perm_c[j]] = V.D2[j] * (V.x[cur][j] - (which == 2 ? V.x[prv][j] : V.xlast[j]));
      continue;
    }
    const double xs = avg ? invW * V.sx[cur][j] : V.x[cur][j];
    double v = V.D2[j] * xs;
    if (v < V.l0[j]) v = V.l0[j];
    if (v > V.u0[j]) v = V.u0[j];
    V.xout[V.perm_c[j]] = v;
  }
  for (int i = blockIdx.x * NT + threadIdx.x; i < V.m; i += stride) {
    if (yray) {
      V.yout[V.perm_r[i]] = V.D1[i] * (V.y[cur][i] - (which == 2 ? V.y[prv][i] : V.ylast[i]));
      continue;
    }
    const double ys = avg ? invW * V.sy[cur][i] : V.y[cur][i];
    V.yout[V.perm_r[i]] = V.D1[i] * ys;
  }
}

__global__ void k_time_limit(DevState *st) {
  if (st->status == ST_RUNNING) st->status = ST_TIME_LIMIT;
}

// ---------------------------------------------------------------- launchers

const char *kernel_class_name(int kc) {
  static const char *names[KC_NUM] = {"k_primal", "k_dual", "k_check_primal", "k_check_dual", "k_restart",
                                      "k_output", "k_primal_reuse_g", "k_infeas"};
  return (kc >= 0 && kc < KC_NUM) ? names[kc] : "";
}

int occupancy_grid(int kc, int num_sms) {
  int nb = 1;
  switch (kc) {
    case KC_PRIMAL: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_primal, NT, 0); break;
    case KC_DUAL: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_dual, NT, 0); break;
    case KC_R1: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_check_primal, NT, 0); break;
    case KC_R2: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_check_dual, NT, 0); break;
    case KC_R3: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_restart, NT, 0); break;
    case KC_INFEAS: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_infeas, NT, 0); break;
    default: nb = 4;
  }
  if (nb < 1) nb = 1;
  return nb * num_sms;
}

// Preferred shared-memory carveout of the step kernels, in percent of the
// largest configuration: 8 % is the smallest that holds four CTAs' static
// shared memory, so the L1 keeps the rest.  Every in-flight gather of x or y
// holds an L1 line until it returns, so the L1's size bounds the gathers in
// flight (measured on the 1e6 x 2e6 LP: 8 % 83.5 / 117.9 us per k_primal /
// k_dual launch, the driver's default 86.2 / 119.0, 28 % 92.1 / 120.4,
// 58 % 112.5 / 132.9).
#ifndef PDLP_STEP_CARVEOUT
#define PDLP_STEP_CARVEOUT 8
#endif
cudaError_t kernels_init() {
  if (PDLP_STEP_CARVEOUT < 0) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(k_primal, cudaFuncAttributePreferredSharedMemoryCarveout, PDLP_STEP_CARVEOUT);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_primal_qp, cudaFuncAttributePreferredSharedMemoryCarveout, PDLP_STEP_CARVEOUT);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_dual, cudaFuncAttributePreferredSharedMemoryCarveout, PDLP_STEP_CARVEOUT);
  return e;
}
cudaError_t launch_primal(const SellMat &KT, const Vecs &V, DevState *st, int grid, cudaStream_t s) {
  if (V.qd)
    k_primal_qp<<<grid, NT, 0, s>>>(KT, V, st);
  else
    k_primal<<<grid, NT, 0, s>>>(KT, V, st);
  return cudaGetLastError();
}
cudaError_t launch_dual(const SellMat &K, const Vecs &V, DevState *st, int grid, cudaStream_t s) {
  k_dual<<<grid, NT, 0, s>>>(K, V, st);
  return cudaGetLastError();
}
cudaError_t launch_check_primal(const SellMat &KT, const Vecs &V, DevState *st, int grid, cudaStream_t s) {
  k_check_primal<<<grid, NT, 0, s>>>(KT, V, st);
  return cudaGetLastError();
}
cudaError_t launch_check_dual(const SellMat &K, const Vecs &V, DevState *st, int grid, cudaStream_t s) {
  k_check_dual<<<grid, NT, 0, s>>>(K, V, st);
  return cudaGetLastError();
}
cudaError_t launch_restart(const Vecs &V, DevState *st, int grid, cudaStream_t s) {
  k_restart<<<grid, NT, 0, s>>>(V, st);
  return cudaGetLastError();
}
cudaError_t launch_infeas(const Vecs &V, DevState *st, int grid, cudaStream_t s) {
  k_infeas<<<grid, NT, 0, s>>>(V, st);
  return cudaGetLastError();
}
cudaError_t launch_output(const Vecs &V, DevState *st, cudaStream_t s) {
  const int n = V.n > V.m ? V.n : V.m;
  int grid = (n + NT - 1) / NT;
  if (grid > 4096) grid = 4096;
  if (grid < 1) grid = 1;
  k_output<<<grid, NT, 0, s>>>(V, st);
  return cudaGetLastError();
}
cudaError_t launch_time_limit(DevState *st, cudaStream_t s) {
  k_time_limit<<<1, 1, 0, s>>>(st);
  return cudaGetLastError();
}

}  // namespace pdlp
