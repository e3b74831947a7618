// Device code shared by the step and check kernels of pdlp_kernels.cu and the
// one-launch check period of pdlp_period.cu: the sliced-ELL SpMV, the row
// epilogues of the half-steps and of the check passes, and the scalar rules of
// Sec. 3.4, Sec. 4.1 and Sec. 2.2.
#pragma once

#include <math.h>
#include <math_constants.h>

#include "pdlp_internal.cuh"

namespace pdlp {

// ---------------------------------------------------------------- sliced-ELL SpMV

// float -> double from the IEEE bits with integer operations, exact for
// every normal float and for zero: with t the magnitude bits, the high word
// is the sign | ((t >> 3) + (896 << 20)) (exponent re-biased by 1023 - 127,
// top 20 mantissa bits), the low word the last 3 mantissa bits << 29, and
// t = 0 gives the signed zero.  The FP32 copies the step kernels read hold
// only normal floats and zeros (setup_f32 flushes the subnormals, and the
// scaled matrix is finite), so no hardware conversion and no branch: the
// widening stays off GB300's narrow FP64 pipe.
__device__ __forceinline__ double f2d(float f) {
  const unsigned int b = __float_as_uint(f);
  const unsigned int t = b & 0x7fffffffu;
  const unsigned int hi = (b ^ t) | (t ? (t >> 3) + 0x38000000u : 0u);
  return __hiloint2double((int)hi, (int)(b << 29));
}
__device__ __forceinline__ double widen(double v) { return v; }
__device__ __forceinline__ double widen(float v) { return f2d(v); }

// Sum over `cnt` strides of 32 stored entries, this lane's entry of each
// stride: acc[a] += val * xs[a][col] in stride order (FMA), padding (column
// -1) skipped.  U strides are loaded (streaming, coalesced across the
// warp) before their gathers are issued, and all gathers before the FMAs.
template <int U, typename VT, int NV, bool SCALED>
__device__ __forceinline__ void strided_dot(const int32_t *__restrict__ ip, const VT *__restrict__ vp, int cnt,
                                            const double *const (&xs)[NV], const double (&sc)[NV],
                                            double (&acc)[NV]) {
  int k = 0;
  for (; k + U <= cnt; k += U) {
    int c[U];
    VT v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      c[u] = __ldcs(ip + 32 * (k + u));
      v[u] = __ldcs(vp + 32 * (k + u));
    }
    double g[NV][U];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int a = 0; a < NV; ++a) {
        const double xv = c[u] >= 0 ? __ldg(xs[a] + c[u]) : 0.0;
        g[a][u] = SCALED && (NV == 1 || a > 0) ? sc[a] * xv : xv;
      }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int a = 0; a < NV; ++a) acc[a] = fma(widen(v[u]), g[a][u], acc[a]);
  }
  for (; k < cnt; ++k) {
    const int c = __ldcs(ip + 32 * k);
    const VT v = __ldcs(vp + 32 * k);
#pragma unroll
    for (int a = 0; a < NV; ++a) {
      const double xv = c >= 0 ? __ldg(xs[a] + c) : 0.0;
      acc[a] = fma(widen(v), SCALED && (NV == 1 || a > 0) ? sc[a] * xv : xv, acc[a]);
    }
  }
}

// One butterfly level: lanes with the `off` bit clear keep row a's pair sum,
// lanes with it set keep row b's.
__device__ __forceinline__ double bfly(double a, double b, int off, int lane) {
  const bool hi = (lane & off) != 0;
  const double recv = __shfl_xor_sync(0xffffffffu, hi ? a : b, off);
  return (hi ? b : a) + recv;
}

// Long rows (whole warp per row) are reduced 32 at a time: the per-lane
// partial sums of the batch's rows go through a five-level butterfly
// (31 additions per lane for 32 rows instead of 5 per row), after which
// lane l holds the total of the batch's row rev5(l), and one vectorised
// epilogue finishes all 32 rows.  The tree is fixed, so the sums are too.
template <int NV>
struct LongRows {
  double buf[5][NV];
  int t;        // rows in the current batch (warp-uniform)
  int *rows;    // this warp's 32 row slots in shared memory
  double *tot;  // this warp's 32 x NV totals in shared memory (partial batch)
};

template <int NV, class Epi>
__device__ __forceinline__ void long_push(LongRows<NV> &lr, const double (&p)[NV], int row, Epi &ep) {
  const int lane = threadIdx.x & 31;
  if (lane == 0) lr.rows[lr.t] = row;
  const int t = lr.t;
  double v[NV];
#pragma unroll
  for (int a = 0; a < NV; ++a) v[a] = p[a];
  bool done = false;
  if (!(t & 1)) {
#pragma unroll
    for (int a = 0; a < NV; ++a) lr.buf[0][a] = v[a];
  } else {
#pragma unroll
    for (int a = 0; a < NV; ++a) v[a] = bfly(lr.buf[0][a], v[a], 16, lane);
    if (!(t & 2)) {
#pragma unroll
      for (int a = 0; a < NV; ++a) lr.buf[1][a] = v[a];
    } else {
#pragma unroll
      for (int a = 0; a < NV; ++a) v[a] = bfly(lr.buf[1][a], v[a], 8, lane);
      if (!(t & 4)) {
#pragma unroll
        for (int a = 0; a < NV; ++a) lr.buf[2][a] = v[a];
      } else {
#pragma unroll
        for (int a = 0; a < NV; ++a) v[a] = bfly(lr.buf[2][a], v[a], 4, lane);
        if (!(t & 8)) {
#pragma unroll
          for (int a = 0; a < NV; ++a) lr.buf[3][a] = v[a];
        } else {
#pragma unroll
          for (int a = 0; a < NV; ++a) v[a] = bfly(lr.buf[3][a], v[a], 2, lane);
          if (!(t & 16)) {
#pragma unroll
            for (int a = 0; a < NV; ++a) lr.buf[4][a] = v[a];
          } else {
#pragma unroll
            for (int a = 0; a < NV; ++a) v[a] = bfly(lr.buf[4][a], v[a], 1, lane);
            done = true;
          }
        }
      }
    }
  }
  lr.t = t + 1;
  if (done) {
    __syncwarp();
    const int r = lr.rows[__brev(lane) >> 27];
    __syncwarp();
    if (r >= 0) {
      ep.prefetch(r);
      ep.finish(r, v);
    }
    lr.t = 0;
  }
}

// Finishes a partial batch of t < 32 long rows without padding it: buf[k]
// (present when bit k of t is set) holds slots [t & ~(2^(k+1) - 1), +2^k)
// after k butterfly levels, lane l carrying a partial of the block's slot
// rev_k(l >> (5 - k)); the remaining 5 - k levels are a plain xor reduction,
// after which the first lane of every group of 32 >> k holds its row's
// total.  The totals go through shared memory so that lane s finishes slot
// s: one epilogue (one round of operand loads) for the whole batch.
template <int NV, class Epi>
__device__ __forceinline__ void long_flush(LongRows<NV> &lr, Epi &ep) {
  const int lane = threadIdx.x & 31, t = lr.t;
  __syncwarp();
  const int r = lane < t ? lr.rows[lane] : -1;
  if (r >= 0) ep.prefetch(r);  // the epilogue's operands arrive during the reductions
#pragma unroll
  for (int k = 4; k >= 0; --k) {
    if (!(t & (1 << k))) continue;
    const int start = t & ~((2 << k) - 1);
    double v[NV];
#pragma unroll
    for (int a = 0; a < NV; ++a) v[a] = lr.buf[k][a];
#pragma unroll
    for (int off = 16 >> k; off >= 1; off >>= 1)
#pragma unroll
      for (int a = 0; a < NV; ++a) v[a] += __shfl_xor_sync(0xffffffffu, v[a], off);
    if ((lane & ((32 >> k) - 1)) == 0) {
      const int slot = start + (k ? (int)(__brev((unsigned)(lane >> (5 - k))) >> (32 - k)) : 0);
#pragma unroll
      for (int a = 0; a < NV; ++a) lr.tot[slot * NV + a] = v[a];
    }
  }
  __syncwarp();
  if (r >= 0) {
    double v[NV];
#pragma unroll
    for (int a = 0; a < NV; ++a) v[a] = lr.tot[lane * NV + a];
    ep.finish(r, v);
  }
  __syncwarp();
  lr.t = 0;
}

// y = A x for NV (1 or 2) gathered vectors, each finished row r passed to
// ep.finish(r, sums) after ep.prefetch(r).  With SCALED, gathered entries of
// vector a are multiplied by sc[a] (the epoch average (1/W) sum); sc[0] of two
// is 1 and costs no multiply.  Warp w of
// the grid takes items w, 2G - 1 - w, 2G + w, ... of the schedule (G warps):
// a snake over the cost-sorted items, so every warp gets about the same work.
template <int U, typename VT, int NV, bool SCALED, class Epi>
__device__ __forceinline__ void spmv_sell(const SellMat &A, const VT *__restrict__ val,
                                          const double *const (&xs)[NV], const double (&sc)[NV], Epi &ep,
                                          int *warp_rows, double *warp_tot) {
  const int lane = threadIdx.x & 31;
  const int nw = (int)((gridDim.x * (unsigned)NT) >> 5);
  const int gw = (int)((blockIdx.x * (unsigned)NT + threadIdx.x) >> 5);
  LongRows<NV> lr;
  lr.t = 0;
  lr.rows = warp_rows;
  lr.tot = warp_tot;
  // the warp's b-th item of the snake order (-1: none)
  auto item_of = [&](int b) -> long long {
    const long long first = (long long)b * nw;
    if (first >= A.nitems) return -1;
    const long long it = first + ((b & 1) ? nw - 1 - gw : gw);
    return it < A.nitems ? it : -1;
  };
  long long it = item_of(0);
  int4 d = it >= 0 ? __ldg(A.items + it) : make_int4(0, 0, 0, 0);
  for (int b = 0; it >= 0; ++b) {
    const long long itn = item_of(b + 1);
    int4 dn = make_int4(0, 0, 0, 0);
    double acc[NV];
#pragma unroll
    for (int a = 0; a < NV; ++a) acc[a] = 0.0;
    if (d.y > 0) {  // slice: one row per lane
      const bool has = lane < d.y;
      const int row = d.x + lane;
      if (has) ep.prefetch(row);
      strided_dot<U, VT, NV, SCALED>(A.idx + d.w + lane, val + d.w + lane, d.z, xs, sc, acc);
      if (has) ep.finish(row, acc);
    } else {  // long row: the whole warp
      strided_dot<U, VT, NV, SCALED>(A.idx + d.w + lane, val + d.w + lane, (d.z + 31) >> 5, xs, sc, acc);
      long_push(lr, acc, d.x, ep);
    }
    if (itn >= 0) dn = __ldg(A.items + itn);  // the next item's descriptor
    it = itn;
    d = dn;
  }
  if (lr.t > 0) long_flush(lr, ep);
}

// ---------------------------------------------------------------- primal step

// QP: qd (the scaled diagonal of Q) non-null, and the primal step is the
// exact proximal step of x'Qx/2 + (c - K'y)'x over X, coordinate by
// coordinate: x' = proj_X((x - tau (c - g)) / (1 + tau Q_jj)).
template <bool QP>
struct PrimalEpi {
  const double *c, *l, *u, *x, *sx;
  const double *qd;
  double *g, *xn, *sxn;
  double tau, eta, dx2;
  double pc, pl, pu, px, psx, pq;
  __device__ __forceinline__ void prefetch(int j) {
    pc = c[j];
    pl = l[j];
    pu = u[j];
    px = x[j];
    psx = sx[j];
    if (QP) pq = qd[j];
  }
  __device__ __forceinline__ void finish(int j, const double (&gs)[1]) { apply(j, gs[0], true); }
  __device__ __forceinline__ void apply(int j, double gj, bool store_g) {
    if (store_g) g[j] = gj;
    const double v = QP ? clamp_bits(fma(-tau, pc - gj, px) / fma(tau, pq, 1.0), pl, pu)
                        : clamp_bits(fma(-tau, pc - gj, px), pl, pu);
    xn[j] = v;
    sxn[j] = fma(eta, v, psx);
    const double d = v - px;
    dx2 = fma(d, d, dx2);
  }
};

struct DualEpi {
  const double *q, *y, *kx, *sy;
  double *yn, *kxn, *syn;
  double sigma, eta, dy2, cross;
  int n_eq;
  double pq, py, pkx, psy;
  __device__ __forceinline__ void prefetch(int i) {
    pq = q[i];
    py = y[i];
    pkx = kx[i];
    psy = sy[i];
  }
  __device__ __forceinline__ void finish(int i, const double (&ks)[1]) {
    const double kn = ks[0];
    double v = fma(sigma, pq - fma(2.0, kn, -pkx), py);
    if (i >= n_eq && __double_as_longlong(v) < 0) v = 0.0;  // proj_Y: sign bit test
    yn[i] = v;
    kxn[i] = kn;
    syn[i] = fma(eta, v, psy);
    const double d = v - py;
    dy2 = fma(d, d, dy2);
    cross = fma(d, kn - pkx, cross);
  }
};

// IEEE-bit tests (integer pipe): sign of a nonzero, finiteness
__device__ __forceinline__ bool neg_bits(double v) { return __double_as_longlong(v) < 0; }
__device__ __forceinline__ bool pos_bits(double v) { return __double_as_longlong(v) > 0; }
__device__ __forceinline__ bool finite_bits(double v) {
  return ((unsigned long long)__double_as_longlong(v) & 0x7ff0000000000000ull) != 0x7ff0000000000000ull;
}

// proj_Lambda (reading 5 of the paper's lambda): every test on the IEEE
// bits, so GB300's narrow FP64 pipe does none of it.  -0.0 maps to -0.0 or
// +0.0, which no sum below can tell from 0.
__device__ __forceinline__ double proj_lambda(double d, double l, double u) {
  const bool lf = finite_bits(l), uf = finite_bits(u);
  if (lf && uf) return d;
  if (lf) return pos_bits(d) ? d : 0.0;
  if (uf) return neg_bits(d) ? d : 0.0;
  return 0.0;
}

// Dual-side pieces of eq. (kkt) / Sec. 4.1 for one variable.
// With qp (Q_jj = qdj), the objective's gradient c + Qx replaces c in the
// reduced cost, and x'Qx/2 is added to the primal objective c'x and taken
// from the dual one (the QP's objectives).
// The original-space residual is r / D2, taken as r times the stored 1/D2
// (rd2): no FP64 division on the hot check path.
__device__ __forceinline__ void dual_piece(double c, double g, double l, double u, double rd2, double x,
                                           double *acc, bool qp = false, double qdj = 0.0) {
  const double d = qp ? fma(qdj, x, c) - g : c - g;
  const double lam = proj_lambda(d, l, u);
  const double r = d - lam;
  acc[0] = fma(r, r, acc[0]);
  const double ro = r * rd2;
  acc[1] = fma(ro, ro, acc[1]);
  acc[2] = fma(c, x, acc[2]);
  if (pos_bits(lam)) acc[3] = fma(l, lam, acc[3]);
  if (neg_bits(lam) && (__double_as_longlong(lam) << 1) != 0) acc[3] = acc[3] - u * (-lam);
  if (qp) {
    const double h = 0.5 * qdj * x * x;
    acc[2] += h;
    acc[3] -= h;
  }
}

// Epilogue of the dual-side check pass.  kind 0: start point (sums = {K'y});
// kind 1: check with stale g (sums = {K'y, K'ybar}); kind 2: check with g
// current (sums = {K'ybar}, g loaded).
struct CheckPrimalEpi {
  const double *c, *l, *u, *rd2, *x,
      *sx;
  double *g, *gbar;
  double *g0, *gprev;  // kept for infeasibility detection when keep
  const double *qd;                 // QP: the scaled diagonal of Q (else null)
  double invW;
  int kind, keep;
  double acc[NV_R1];
  double pc, pl, pu, pd2, px, psx, pg, pq;
  __device__ __forceinline__ void prefetch(int j) {
    pc = c[j];
    pl = l[j];
    pu = u[j];
    pd2 = rd2[j];
    px = x[j];
    psx = kind ? sx[j] : 0.0;
    pg = (kind == 2 || (kind == 1 && keep)) ? g[j] : 0.0;
    pq = qd ? qd[j] : 0.0;
  }
  template <int NV>
  __device__ __forceinline__ void finish(int j, const double (&s)[NV]) {
    double gj = pg, gb = 0.0;
    if (kind == 0) {
      gj = s[0];
      g[j] = gj;
      if (keep) g0[j] = gj;  // K'y at the epoch start
    } else if (kind == 1) {
      gj = s[0];
      gb = s[NV - 1];
      if (keep) gprev[j] = pg;  // K'y of the previous accepted iterate
      g[j] = gj;
    } else {
      gb = s[0];
    }
    const bool qp = qd != nullptr;
    dual_piece(pc, gj, pl, pu, pd2, px, acc, qp, pq);
    if (kind) {
      gbar[j] = gb;
      dual_piece(pc, gb, pl, pu, pd2, invW * psx, acc + 4, qp, pq);
    }
  }
};

// The original-space residual is r / D1, taken as r times the stored 1/D1.
__device__ __forceinline__ void primal_piece(double q, double kx, bool ineq, double rd1, double y, double *acc) {
  double r = q - kx;
  if (ineq && neg_bits(r)) r = 0.0;
  acc[0] = fma(r, r, acc[0]);
  const double ro = r * rd1;
  acc[1] = fma(ro, ro, acc[1]);
  acc[2] = fma(q, y, acc[2]);
}

__device__ __forceinline__ double kkt_omega(double rp2, double rd2, double pobj, double dobj, double omega) {
  const double gap = dobj - pobj;
  return sqrt(omega * omega * rp2 + rd2 / (omega * omega) + gap * gap);
}

__device__ __forceinline__ bool sec41_pass(double pobj, double dobj, double rp, double rd, double tol, double qn,
                                           double cn) {
  if (!(fabs(dobj - pobj) <= tol * (1.0 + fabs(dobj) + fabs(pobj)))) return false;
  if (!(rp <= tol * (1.0 + qn))) return false;
  if (!(rd <= tol * (1.0 + cn))) return false;
  return true;
}

__device__ __forceinline__ double sec41_rel(double pobj, double dobj, double rp, double rd, double qn, double cn) {
  const double a = fabs(dobj - pobj) / (1.0 + fabs(dobj) + fabs(pobj));
  const double b = rp / (1.0 + qn);
  const double c = rd / (1.0 + cn);
  return fmax(a, fmax(b, c));
}

// p: the 8 dual-side sums (current 0..3, average 4..7); d: the 6 primal-side
// sums (current 0..2, average 3..5).
// Sec. 2.2 infeasibility detection on k_infeas' sums for one ray (original
// LP): the dual ray certifies primal infeasibility when its objective
// q'yr + l'lam+ - u'lam- is positive and ||(-K'yr - lam, min(yr_G, 0))||
// is at most eps times it; the primal ray certifies dual infeasibility when
// -c'xr is positive and ||(K_E xr, min(K_G xr, 0), cone violation)|| is at
// most eps times it.  Returns the status, or ST_RUNNING.
__device__ inline int infeas_status(const double *a, double eps, double *ray) {
  const double obj_d = a[5] + a[1], res_d = sqrt(a[0] + a[6]);
  if (obj_d > 0.0 && res_d <= eps * obj_d) {
    ray[0] = obj_d;
    ray[1] = res_d;
    return ST_PRIMAL_INFEASIBLE;
  }
  const double obj_p = -a[2], res_p = sqrt(a[4] + a[3]);
  if (obj_p > 0.0 && res_p <= eps * obj_p) {
    ray[0] = obj_p;
    ray[1] = res_p;
    return ST_DUAL_INFEASIBLE;
  }
  return ST_RUNNING;
}

__device__ inline void check_decide(DevState *st, TraceRec *trace, const double *p, const double *d, const double *inf) {
  const double omega = st->omega;
  if (st->mode == MODE_INIT) {
    const double k0 = kkt_omega(d[0], p[0], p[2], d[2] + p[3], omega);
    st->kkt_start = k0;
    st->kkt_prev = k0;
    st->mode = MODE_CHECK;
    st->need_g = 0;
    st->check_pending = 0;
    return;
  }
  st->checks += 1;
  st->need_g = 0;
  const double pc = p[2], dc = d[2] + p[3], rpc = sqrt(d[1]), rdc = sqrt(p[1]);
  const double pa = p[6], da = d[5] + p[7], rpa = sqrt(d[4]), rda = sqrt(p[5]);
  const double tol = st->tol, qn = st->q_norm, cn = st->c_norm;
  st->term[0] = pc;
  st->term[1] = dc;
  st->term[2] = rpc;
  st->term[3] = rdc;
  if (sec41_pass(pc, dc, rpc, rdc, tol, qn, cn)) {
    st->status = ST_OPTIMAL;
    st->which = 0;
    return;
  }
  if (sec41_pass(pa, da, rpa, rda, tol, qn, cn)) {
    st->term[0] = pa;
    st->term[1] = da;
    st->term[2] = rpa;
    st->term[3] = rda;
    st->status = ST_OPTIMAL;
    st->which = 1;
    return;
  }
  if (inf) {  // difference ray, then normalised-iterate ray
    for (int r = 0; r < 2; ++r) {
      const int stt = infeas_status(inf + r * NV_I1, st->eps_infeas, st->ray);
      if (stt != ST_RUNNING) {
        st->status = stt;
        st->which = 2 + r;
        return;
      }
    }
  }
  if (st->k >= st->max_iter) {
    st->status = ST_ITER_LIMIT;
    st->which = 0;
    return;
  }
  const double kc = kkt_omega(d[0], p[0], pc, dc, omega);
  const double ka = kkt_omega(d[3], p[4], pa, da, omega);
  const int cand_avg = !(kc < ka);
  const double kcand = cand_avg ? ka : kc;
  const double ks = st->kkt_start;
  int mask = 0;
  if (kcand <= st->beta_suff * ks) mask |= 1;
  if (kcand <= st->beta_nec * ks && kcand > st->kkt_prev) mask |= 2;
  if ((double)st->t >= st->beta_art * (double)st->k) mask |= 4;
  if (mask) {
    st->restart_to = cand_avg ? 2 : 1;
    if (cand_avg) {
      st->cand[0] = d[3];
      st->cand[1] = p[4];
      st->cand[2] = pa;
      st->cand[3] = da;
    } else {
      st->cand[0] = d[0];
      st->cand[1] = p[0];
      st->cand[2] = pc;
      st->cand[3] = dc;
    }
    if (st->use_f32 && st->polish) {
      // FP32-values mode: move the steps to the FP64 K once the original-space
      // relative KKT of the restart point stops improving for two restarts.
      const double rel = cand_avg ? sec41_rel(pa, da, rpa, rda, qn, cn) : sec41_rel(pc, dc, rpc, rdc, qn, cn);
      if (rel < st->rel_kkt_best) {
        st->rel_kkt_best = rel;
        st->stall = 0;
      } else if (++st->stall >= 2) {
        st->use_f32 = 0;
        st->f64_switch_k = st->k;
      }
    }
  } else {
    st->kkt_prev = kcand;
    st->check_pending = 0;
  }
  {  // the check's record, into the ring
    TraceRec &r = trace[st->ntrace % st->trace_cap];
    r.k = st->k;
    r.attempts = st->attempts;
    r.restarts = st->restarts + (mask ? 1 : 0);
    r.restart = mask;
    r.cand_avg = cand_avg;
    r.kkt_cur = kc;
    r.kkt_avg = ka;
    r.kkt_start = st->kkt_start;
    r.omega = omega;
    r.eta_hat = st->eta;
    r.rel_gap = fabs(pc - dc) / (1.0 + fabs(pc) + fabs(dc));
    r.rel_primal = rpc / (1.0 + qn);
    r.rel_dual = rdc / (1.0 + cn);
    st->ntrace += 1;
  }
}

// Epilogue of the primal-side check pass.  check = 0: start point (sums =
// {Kx}, stored as Kx); check = 1: sums = {K xbar}.
struct CheckDualEpi {
  const double *q, *rd1, *y, *sy;
  double *kx, *kxbar, *kx0;
  double invW;
  int check, n_eq, keep;
  double acc[NV_R2];
  double pq, pd1, py, psy, pkx;
  __device__ __forceinline__ void prefetch(int i) {
    pq = q[i];
    pd1 = rd1[i];
    py = y[i];
    psy = check ? sy[i] : 0.0;
    pkx = check ? kx[i] : 0.0;
  }
  __device__ __forceinline__ void finish(int i, const double (&s)[1]) {
    const bool ineq = i >= n_eq;
    double kxi = pkx;
    if (!check) {
      kxi = s[0];
      kx[i] = kxi;
      if (keep) kx0[i] = kxi;  // K x at the epoch start
    }
    primal_piece(pq, kxi, ineq, pd1, py, acc);
    if (check) {
      kxbar[i] = s[0];
      primal_piece(pq, s[0], ineq, pd1, invW * psy, acc + 3);
    }
  }
};

// Pieces of the two certificates (NV_I1 each, layout of NV_I1) for the rays
// z - z_prev (difference of the last two accepted iterates; only when this
// check's K'y pass stored K'y_prev) and z - z^{n,0} (the normalised iterate
// times t: the tests are invariant to positive scaling), unscaled to the
// original LP: xr = D2 dx^, yr = D1 dy^, K xr = (K~ dx^) / D1 and
// K'yr = (K~' dy^) / D2 from the stored products, c'xr = c~'dx^ and
// q'yr = q~'dy^.  Since D2 > 0, lambda = proj_Lambda(-K'yr) = p / D2 with
// p = proj_Lambda(-K~' dy^), so l'lambda+ - u'lambda- = sum of l~ p (p > 0)
// and u~ p (p < 0) in scaled terms.  Sign and finiteness tests read the IEEE
// bits (integer pipe); GB300's FP64 pipe does only the arithmetic.  The
// caller takes elements first, first + stride, ...; r0 = 1 leaves out the
// difference ray.
__device__ __forceinline__ void infeas_sums(const Vecs &V, int cur, int r0, int first, int stride, double (&a)[NV_I]) {
  const int prv = cur ^ 1;
#pragma unroll
  for (int k = 0; k < NV_I; ++k) a[k] = 0.0;
  for (int j = first; j < V.n; j += stride) {
    const double d2 = V.D2[j], rd2 = V.rD2[j], lt = V.l[j], ut = V.u[j], cj = V.c[j], gj = V.g[j];
    const double xj = V.x[cur][j];
    const bool lf = finite_bits(lt), uf = finite_bits(ut);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      if (r < r0) continue;
      double *b = a + r * NV_I1;
      const double mg = (r == 0 ? V.gprev[j] : V.g0[j]) - gj;  // -(K~' dy^)_j
      double p = mg;                                             // proj onto the cone of the bounds
      if (!lf && !uf) p = 0.0;
      else if (!uf && neg_bits(p)) p = 0.0;
      else if (!lf && pos_bits(p)) p = 0.0;
      const double res = (mg - p) * rd2;
      b[0] = fma(res, res, b[0]);
      if (pos_bits(p)) b[1] = fma(lt, p, b[1]);
      else if (neg_bits(p)) b[1] = fma(ut, p, b[1]);
      const double dx = xj - (r == 0 ? V.x[prv][j] : V.xlast[j]);
      b[2] = fma(cj, dx, b[2]);
      if ((lf && neg_bits(dx)) || (uf && pos_bits(dx))) {
        const double xo = d2 * dx;
        b[3] = fma(xo, xo, b[3]);
      }
    }
  }
  for (int i = first; i < V.m; i += stride) {
    const double d1 = V.D1[i], rd1 = V.rD1[i], qi = V.q[i], yi = V.y[cur][i], kxi = V.Kx[cur][i];
    const bool ineq = i >= V.n_eq;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      if (r < r0) continue;
      double *b = a + r * NV_I1;
      double kr = (kxi - (r == 0 ? V.Kx[prv][i] : V.kx0[i])) * rd1;
      if (ineq && pos_bits(kr)) kr = 0.0;
      b[4] = fma(kr, kr, b[4]);
      const double dy = yi - (r == 0 ? V.y[prv][i] : V.ylast[i]);
      b[5] = fma(qi, dy, b[5]);
      if (ineq && neg_bits(dy)) {
        const double yo = d1 * dy;
        b[6] = fma(yo, yo, b[6]);
      }
    }
  }
}

// Restart: moves the candidate (with avg, the average) into the iterate and
// resets the epoch, elements first, first + stride, ...; acc = this thread's
// shares of ||x_new - x_last||^2 and ||y_new - y_last||^2.
__device__ __forceinline__ void restart_sums(const Vecs &V, int cur, bool avg, bool keep, double invW, int first,
                                             int stride, double (&acc)[2]) {
  acc[0] = acc[1] = 0.0;
  double *x = V.x[cur];
  double *sx = V.sx[cur];
  for (int j = first; j < V.n; j += stride) {
    double xn;
    if (avg) {
      xn = invW * sx[j];
      x[j] = xn;
      V.g[j] = V.gbar[j];
    } else {
      xn = x[j];
    }
    if (keep) V.g0[j] = V.g[j];  // K'y at the new epoch start
    const double d = xn - V.xlast[j];
    acc[0] = fma(d, d, acc[0]);
    V.xlast[j] = xn;
    sx[j] = 0.0;
  }
  double *y = V.y[cur];
  double *sy = V.sy[cur];
  double *kx = V.Kx[cur];
  for (int i = first; i < V.m; i += stride) {
    double yn;
    if (avg) {
      yn = invW * sy[i];
      y[i] = yn;
      kx[i] = V.Kxbar[i];
    } else {
      yn = y[i];
    }
    if (keep) V.kx0[i] = kx[i];  // K x at the new epoch start
    const double d = yn - V.ylast[i];
    acc[1] = fma(d, d, acc[1]);
    V.ylast[i] = yn;
    sy[i] = 0.0;
  }
}

// The restart's scalars (one thread).
__device__ __forceinline__ void restart_finish(DevState *st, TraceRec *trace, double dx2, double dy2) {
  // Sec. 2.2 PrimalWeightUpdate, read in log space
  const double dx = sqrt(dx2), dy = sqrt(dy2);
  double omega = st->omega;
  if (dx > st->eps_zero && dy > st->eps_zero)
    omega = exp(st->theta * log(dy / dx) + (1.0 - st->theta) * log(omega));
  st->omega = omega;
  st->W = 0.0;
  st->t = 0;
  st->restarts += 1;
  const double k0 = kkt_omega(st->cand[0], st->cand[1], st->cand[2], st->cand[3], omega);
  st->kkt_start = k0;
  st->kkt_prev = k0;
  st->restart_to = 0;
  st->check_pending = 0;
  if (st->ntrace > 0 && trace[(st->ntrace - 1) % st->trace_cap].k == st->k) {
    trace[(st->ntrace - 1) % st->trace_cap].omega = omega;
    trace[(st->ntrace - 1) % st->trace_cap].kkt_start = k0;
  }
}

}  // namespace pdlp
