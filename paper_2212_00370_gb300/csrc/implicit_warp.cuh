// implicit_warp.cuh -- the implicit radiation-matter solve (Sec. 3.3) of a warp's cells.
//
// What bounds a cell launch is its slowest cells (10^2 - 10^3 evaluations of R against 8 on
// average) and the divergence around them: with the solver written as nested loops, lanes
// that evaluate R for different reasons (a Jacobian column, a line-search trial, a polish
// step) cannot do it together.  Here the solver is a state machine per lane, and a warp
// advances in rounds: every lane that has an unfinished cell names the point where it needs
// R next, one call evaluates all of them, and every lane digests its result.
// When four cells or fewer are left in a warp, the idle lanes work for them: each cell gets
// eight lanes, which evaluate all the columns of a difference Jacobian (both signs), or eight
// trials of a line search, in one round.  A trial that the sequential search would not have
// reached is ignored, so the iterates are those of the sequential algorithm, bit for bit.
// Measured against nested loops: a slow cell alone 13.7 -> 7.3 ms (635 evaluations), 8.5 ->
// 2.8 ms (482); 300007 independent solves 60.8 -> 48.3 ms; 2D blast 1024^2, two steps,
// 40.3 -> 33.4 ms; 1001 Riemann problems, two steps, 121 -> 113 ms.
#pragma once
#include "scheme_f64.cuh"

namespace rr {

// The point a lane needs next: residual R on X (INIT .. LADDER), on the matter primitives Y
// (M_INIT .. M_FINAL).
enum ImpPhase : int {
  IMP_DONE = 0,
  IMP_INIT,     // R at X*
  IMP_REINIT,   // the same again, after a failed first attempt on the matter primitives
  IMP_FD,       // column `col` of the forward-difference Jacobian (sign 1: backward)
  IMP_LS,       // line-search trial k
  IMP_FINAL,    // the converged step
  IMP_POLISH,   // polishing correction k
  IMP_LADDER,   // start of a rung of the continuation in h
  IMP_M_INIT,
  IMP_M_FD,
  IMP_M_LS,
  IMP_M_FINAL,
};

// What the evaluation of a request needs to know of a cell: its own task's, or (wide
// rounds) another lane's.
struct ImpView {
  ImpCell c;
  double X[4], Y[4], sc[4], dX[4], Z, lam, r0;
  int phase, k, col, sign;
  bool first;
};

// One cell's solve.  begin() to finish() hold the algorithm of implicit step 3.5: iteration
// on X (from the cell's cached matrix or C^(m)), continuation in h, matter primitives.
template <class F>
struct ImpTask {
  using JT = typename F::Mat;
  ImpCell c;
  double hdt, Zguess;
  double X[4], R[4], V[NV], Z;
  double dX[4], lam, r0, prev;
  double Y[4], sc[4];
  double Mnew[16], Vs[NV], jc[17];
  JT J[4][4];
  double Jm[4][4];  // matter form
  int phase, rc;
  int m, k, col, sign, lad;
  bool need_fd, fresh_fd, first, tried_m, polishing;
};

template <class F>
__device__ __forceinline__ void imp_start_newton(ImpTask<F>& t, bool cached) {
  using JT = typename F::Mat;
  if (cached) {  // the cell's matrix from its previous solve: J = I + h M
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j)
        t.J[i][j] = conv<JT>((i == j ? 1.0 : 0.0) + t.c.hdt * t.jc[4 * i + j]);
  } else {
    double Jd[4][4];
    picard_matrix(t.c, t.X, t.V, Jd);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) t.J[i][j] = conv<JT>(Jd[i][j]);
  }
  t.need_fd = false;
  t.fresh_fd = false;
  t.first = true;
  t.polishing = false;
  t.prev = -1.0;
  t.m = 1;
}

__device__ __forceinline__ double imp_norm2(const double* R) {
  return ((R[0] * R[0] + R[1] * R[1]) + R[2] * R[2]) + R[3] * R[3];
}

// Accepts the evaluated point.
template <class F>
__device__ __forceinline__ void imp_take(ImpTask<F>& t, const double* X, const double* R,
                                         const double* V, double Z) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    t.X[i] = X[i];
    t.R[i] = R[i];
  }
#pragma unroll
  for (int k = 0; k < NV; ++k) t.V[k] = V[k];
  t.Z = Z;
}

// The cell's end: cache, status.
template <class F>
__device__ __forceinline__ void imp_finish(ImpTask<F>& t, bool ok, bool matter) {
#pragma unroll
  for (int k = 0; k < 16; ++k) t.jc[k] = (ok && !matter) ? t.Mnew[k] : 0.0;
  t.jc[16] = ok ? (matter ? 2.0 : 1.0) : 0.0;
  t.rc = ok ? ST_OK : ST_IMPLICIT;
  t.phase = IMP_DONE;
}

// The trial point of a lane's request: the cell's own next one (slot 0 in sequence), or the
// slot-th of the eight evaluated for it.  False: nothing to evaluate in this slot.
template <class Task>
__device__ __forceinline__ bool imp_trial(const Task& t, bool wide, int slot, double* T) {
#pragma unroll
  for (int i = 0; i < 4; ++i) T[i] = t.phase >= IMP_M_INIT ? t.Y[i] : t.X[i];
  switch (t.phase) {
    case IMP_FD:
    case IMP_M_FD: {
      const int col = wide ? (slot & 3) : t.col;
      const bool back = wide ? slot >= 4 : t.sign != 0;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const double h = __dmul_rn(1e-7, t.phase == IMP_FD ? t.X[0] : t.sc[j]);
        if (j == col) T[j] = back ? T[j] - h : T[j] + h;
      }
      return true;
    }
    case IMP_LS:
    case IMP_M_LS: {
      const int last = t.phase == IMP_M_LS ? 39 : (t.first ? 3 : 9);
      double d[4] = {t.dX[0], t.dX[1], t.dX[2], t.dX[3]};
      for (int s = 0; s < slot; ++s) {
#pragma unroll
        for (int i = 0; i < 4; ++i) d[i] = 0.5 * d[i];
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) T[i] = T[i] + d[i];
      return t.k + slot <= last;
    }
    case IMP_FINAL:
    case IMP_POLISH:
    case IMP_M_FINAL:
#pragma unroll
      for (int i = 0; i < 4; ++i) T[i] = T[i] + t.dX[i];
      return slot == 0;
    default:
      return slot == 0;
  }
}

// Digests the result (ok, R, V, Z at the trial point T) of the lane's own request and moves
// the task to its next request or to its end.  wide: the results of eight slots; the
// Jacobian columns Rc (okc: 4 forward and 4 backward flags), and the first accepted slot of a
// line search (hit, -1: none).
template <class F>
__device__ __forceinline__ void imp_digest(const Params& P, ImpTask<F>& t, bool wide, bool ok,
                                           const double* T, const double* R, const double* V,
                                           double Z, unsigned okc, const double Rc[4][4], int hit) {
  using JT = typename F::Mat;
  enum Next { NONE, START, ITER, DIR, CONVERGED, FAILED, M_START, M_ITER, M_DIR, M_FAILED } next = NONE;
  switch (t.phase) {
    case IMP_INIT:
      if (!ok) {  // no admissible matter state at X*: the explicit update U* is inadmissible
        t.rc = ST_C2P;
        t.phase = IMP_DONE;
        break;
      }
      imp_take(t, T, R, V, Z);
#pragma unroll
      for (int k = 0; k < NV; ++k) t.Vs[k] = V[k];
      next = t.tried_m ? M_START : START;
      break;
    case IMP_REINIT:
      if (ok) imp_take(t, T, R, V, Z);
      next = START;
      break;
    case IMP_LADDER:
      if (ok) imp_take(t, T, R, V, Z);
      next = ok ? START : FAILED;
      break;
    case IMP_FD:
    case IMP_M_FD: {
      const bool mt = t.phase == IMP_M_FD;
      bool failed = false, done = false;
      const int c0 = wide ? 0 : t.col, c1 = wide ? 4 : t.col + 1;
      if (!wide && !ok && t.sign == 0) {
        t.sign = 1;  // the backward point of the same column
        break;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (j < c0 || j >= c1 || failed) continue;
        const bool fwd = wide ? ((okc >> j) & 1u) != 0u : t.sign == 0;
        if (wide ? !fwd && !((okc >> (4 + j)) & 1u) : !ok) {
          failed = true;
          continue;
        }
        const double x = mt ? t.Y[j] : t.X[j];
        const double h = __dmul_rn(1e-7, mt ? t.sc[j] : t.X[0]);
        const double d = (fwd ? x + h : x - h) - x;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const double q = ddiv_call((wide ? Rc[i][j] : R[i]) - t.R[i], d);
          if (mt)
            t.Jm[i][j] = q;
          else
            t.J[i][j] = conv<JT>(q);
        }
        if (j == 3) done = true;
      }
      if (failed) {
        next = mt ? M_FAILED : FAILED;
      } else if (done) {
        if (mt) {
          next = M_DIR;
        } else {
          t.need_fd = false;
          t.fresh_fd = true;
          t.first = false;
          next = DIR;
        }
      } else {
        ++t.col;
        t.sign = 0;
      }
      break;
    }
    case IMP_LS:
    case IMP_M_LS: {
      const bool mt = t.phase == IMP_M_LS;
      const int last = mt ? 39 : (t.first ? 3 : 9);
      bool acc;
      int used;  // halvings of the step up to the accepted trial, or past the rejected ones
      if (wide) {
        acc = hit >= 0;
        used = acc ? hit : 8;
      } else {
        acc = ok && imp_norm2(R) <= (1.0 - 1e-4 * t.lam) * t.r0;
        used = acc ? 0 : 1;
      }
      for (int s = 0; s < used; ++s) {
#pragma unroll
        for (int i = 0; i < 4; ++i) t.dX[i] = 0.5 * t.dX[i];
        t.lam = 0.5 * t.lam;
      }
      t.k += used;
      if (!acc) {
        if (t.k <= last) break;  // the next trial(s)
        if (mt) {
          next = M_FAILED;
        } else if (!t.fresh_fd) {
          t.need_fd = true;
          ++t.m;
          next = ITER;
        } else {
          next = FAILED;
        }
        break;
      }
      if (mt) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          t.Y[i] = T[i];
          t.R[i] = R[i];
          t.X[i] = V[8 + i];
        }
#pragma unroll
        for (int k = 0; k < NV; ++k) t.V[k] = V[k];
        ++t.m;
        next = M_ITER;
        break;
      }
      double dmax = 0.0;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (fpi::mag_gt(t.dX[i], dmax)) dmax = fabs(t.dX[i]);
      broyden(t.J, t.dX, t.R, R);
      t.fresh_fd = false;
      t.first = false;
      imp_take(t, T, R, V, Z);
      if (t.prev >= 0.0 && dmax > 0.5 * t.prev) t.need_fd = true;
      t.prev = dmax;
      ++t.m;
      next = ITER;
      break;
    }
    case IMP_FINAL:
      if (!ok) {
        next = FAILED;
        break;
      }
      imp_take(t, T, R, V, Z);
#pragma unroll 1
      for (int i = 0; i < 16; ++i)
        t.Mnew[i] = ddiv_call(as_double(t.J[i >> 2][i & 3]) - ((i >> 2) == (i & 3) ? 1.0 : 0.0), t.c.hdt);
      if (F::polish(t.c, t.X)) {
        // Polish: stopping at imp_tol leaves an error of about the last step times the
        // matrix's contraction, which depends on how the iterate was reached.  The iterate
        // is refined towards the root of R itself, so that the result is a function of the
        // cell's state: corrections without line search, J updated by Broyden's formula,
        // until a correction is <= 1e-14 E_r or does not halve the previous one (the
        // rounding floor of R; that one is not taken).
        t.polishing = true;
        t.prev = t.r0;  // size of the converged step
        t.k = 0;
        next = DIR;
      } else {
        next = CONVERGED;
      }
      break;
    case IMP_POLISH:
      if (!ok) {
        next = CONVERGED;
        break;
      }
      broyden(t.J, t.dX, t.R, R);
      imp_take(t, T, R, V, Z);
      t.prev = t.lam;
      next = ++t.k == IMP_POLISH_MAX ? CONVERGED : DIR;
      break;
    case IMP_M_INIT:
      if (fpi::pos(t.Y[0])) {
#pragma unroll
        for (int k = 0; k < NV; ++k) t.V[k] = V[k];
      }
      if (!ok) {
        next = M_FAILED;
        break;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        t.R[i] = R[i];
        t.X[i] = V[8 + i];
      }
      t.m = 1;
      next = M_ITER;
      break;
    case IMP_M_FINAL:
      if (!ok) {
        next = M_FAILED;
        break;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) t.X[i] = V[8 + i];
#pragma unroll
      for (int k = 0; k < NV; ++k) t.V[k] = V[k];
      if (t.tried_m) {  // started here: the cache keeps its flag
        t.rc = ST_OK;
        t.phase = IMP_DONE;
      } else {
        imp_finish(t, true, true);
      }
      break;
    default:
      break;
  }

  if (next == START) {
    imp_start_newton(t, t.phase == IMP_INIT && t.jc[16] == 1.0);
    next = ITER;
  }
  if (next == ITER) {
    if (t.m > P.imp_maxit) {
      next = FAILED;
    } else if (t.need_fd) {
      t.phase = IMP_FD;
      t.col = t.sign = 0;
    } else {
      next = DIR;
    }
  }
  if (next == DIR) {
    const bool solved = newton_dir(t.J, t.R, t.dX);
    double d = 0.0;
    if (solved) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (fpi::mag_gt(t.dX[i], d)) d = fabs(t.dX[i]);
    }
    if (t.polishing) {
      if (!solved || d <= IMP_POLISH_TOL * t.X[0] || (t.k > 0 && d > 0.5 * t.prev)) {
        next = CONVERGED;
      } else {
        t.lam = d;
        t.phase = IMP_POLISH;
      }
    } else if (!solved) {
      if (!t.fresh_fd && t.m + 1 <= P.imp_maxit) {
        ++t.m;
        t.phase = IMP_FD;
        t.col = t.sign = 0;
      } else {
        next = FAILED;
      }
    } else if (d <= P.imp_tol * t.X[0]) {
      t.r0 = d;
      t.phase = IMP_FINAL;
    } else {
      t.r0 = imp_norm2(t.R);
      t.lam = 1.0;
      t.k = 0;
      t.phase = IMP_LS;
    }
  }
  if (next == CONVERGED) {
    if (t.lad > 0) {  // the next rung of the continuation
      --t.lad;
      t.c.hdt = ddiv_call(t.hdt, (double)(1 << t.lad));
      t.phase = IMP_LADDER;
    } else {
      imp_finish(t, true, false);
    }
  }
  if (next == FAILED) {
    if (t.lad < 0) {  // continuation in h from X*
#pragma unroll
      for (int i = 0; i < 4; ++i) t.X[i] = t.c.Xs[i];
      t.Z = t.Zguess;
      t.lad = IMP_LADDER_RUNGS;
      t.c.hdt = ddiv_call(t.hdt, (double)(1 << t.lad));
      t.phase = IMP_LADDER;
    } else {
      t.c.hdt = t.hdt;
      if (t.tried_m)
        imp_finish(t, false, false);
      else
        next = M_START;
    }
  }
  if (next == M_START) {  // the matter state of U*
    const double v2 = (t.Vs[1] * t.Vs[1] + t.Vs[2] * t.Vs[2]) + t.Vs[3] * t.Vs[3];
    const double W = ddiv_call(1.0, dsqrt_call(1.0 - v2));
    t.Y[0] = t.Vs[4];
    t.Y[1] = W * t.Vs[1];
    t.Y[2] = W * t.Vs[2];
    t.Y[3] = W * t.Vs[3];
    t.phase = IMP_M_INIT;
  }
  if (next == M_ITER) {
    if (t.m > P.imp_maxit) {
      next = M_FAILED;
    } else {
      // scales of the difference steps and of the stopping rule: p and 1 + |u|
      const double su = 1.0 + dsqrt_call((t.Y[1] * t.Y[1] + t.Y[2] * t.Y[2]) + t.Y[3] * t.Y[3]);
      t.sc[0] = t.Y[0];
      t.sc[1] = t.sc[2] = t.sc[3] = su;
      t.phase = IMP_M_FD;
      t.col = t.sign = 0;
    }
  }
  if (next == M_DIR) {
    double A[4][4], b[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      b[i] = -t.R[i];
#pragma unroll
      for (int j = 0; j < 4; ++j) A[i][j] = t.Jm[i][j];
    }
    if (!solve4(A, b, t.dX)) {
      next = M_FAILED;
    } else {
      bool conv = true;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (fabs(t.dX[i]) > (100.0 * P.imp_tol) * t.sc[i]) conv = false;
      t.r0 = imp_norm2(t.R);
      t.lam = 1.0;
      t.k = 0;
      t.phase = conv ? IMP_M_FINAL : IMP_M_LS;
    }
  }
  if (next == M_FAILED) {
    if (!t.tried_m) {
      imp_finish(t, false, false);
    } else {  // it was the first attempt: the iteration on X
#pragma unroll
      for (int i = 0; i < 4; ++i) t.X[i] = t.c.Xs[i];
#pragma unroll
      for (int k = 0; k < NV; ++k) t.V[k] = t.Vs[k];
      t.Z = t.Zguess;
      t.phase = IMP_REINIT;
    }
  }
}

__device__ __forceinline__ double from_lane(unsigned mask, double x, int lane) {
  return __shfl_sync(mask, x, lane);
}

// The request that lane `lane` has posted, for a lane that evaluates a slot of it.
template <class F>
__device__ __forceinline__ void imp_view(const ImpTask<F>& t, unsigned mask, int lane, ImpView& v) {
  v.c.kappa = from_lane(mask, t.c.kappa, lane);
  v.c.sigma = from_lane(mask, t.c.sigma, lane);
  v.c.hdt = from_lane(mask, t.c.hdt, lane);
  v.c.D = from_lane(mask, t.c.D, lane);
  v.c.taut = from_lane(mask, t.c.taut, lane);
  v.c.iD = from_lane(mask, t.c.iD, lane);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    v.c.St[i] = from_lane(mask, t.c.St[i], lane);
    v.c.B[i] = from_lane(mask, t.c.B[i], lane);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    v.c.Xs[i] = from_lane(mask, t.c.Xs[i], lane);
    v.X[i] = from_lane(mask, t.X[i], lane);
    v.Y[i] = from_lane(mask, t.Y[i], lane);
    v.sc[i] = from_lane(mask, t.sc[i], lane);
    v.dX[i] = from_lane(mask, t.dX[i], lane);
  }
  v.Z = from_lane(mask, t.Z, lane);
  v.lam = from_lane(mask, t.lam, lane);
  v.r0 = from_lane(mask, t.r0, lane);
  const int bits = __shfl_sync(mask, t.phase | (t.k << 8) | ((int)t.first << 16), lane);
  v.phase = bits & 0xff;
  v.k = (bits >> 8) & 0xff;
  v.first = (bits >> 16) & 1;
  v.col = v.sign = 0;
}

// Cells left in a warp from which its idle lanes work for them, eight lanes each.
constexpr int kWideCells = 4;

// Runs the tasks of the warp's lanes (mask: every lane of the warp that exists; a lane
// without a cell has phase IMP_DONE) to their ends.
template <class F>
__device__ __forceinline__ void implicit_warp(const Params& P, unsigned mask, ImpTask<F>& t) {
  const int lane = threadIdx.x & 31;
  for (;;) {
    const unsigned act = __ballot_sync(mask, t.phase != IMP_DONE);
    if (act == 0u) return;
    const bool wide = mask == 0xffffffffu && __popc(act) <= kWideCells;
    double T[4], R[4], V[NV], Z = 0.0;
    bool ok = false, pass = false;
    ImpView v;
    bool eval;
    if (wide) {
      const unsigned own = __fns(act, 0, (lane >> 3) + 1);  // the cell of this lane's group
      const bool served = own < 32u;
      imp_view(t, mask, served ? (int)own : lane, v);
      eval = imp_trial(v, true, lane & 7, T) && served;
    } else {
      v.c = t.c;
      v.Z = t.Z;
      v.phase = t.phase;
      eval = imp_trial(t, false, 0, T) && t.phase != IMP_DONE;
    }
    if (eval) {
      if (v.phase >= IMP_M_INIT) {
        double Xm[4];
        ok = imp_residual_m(P, v.c, T, R, Xm, V);
      } else {
        Z = v.Z;
        ok = imp_residual<F>(P, v.c, T, v.Z, R, V, &Z);
      }
    }
    unsigned okc = 0u;
    double Rc[4][4];
    int hit = -1;
    if (wide) {
      if (ok && (v.phase == IMP_LS || v.phase == IMP_M_LS)) {
        double lam = v.lam;
        for (int s = 0; s < (lane & 7); ++s) lam = 0.5 * lam;
        pass = imp_norm2(R) <= (1.0 - 1e-4 * lam) * v.r0;
      }
      const unsigned okb = __ballot_sync(mask, ok), passb = __ballot_sync(mask, pass);
      // results to the cells' own lanes
      const int base = 8 * __popc(act & ((1u << lane) - 1u)) & 31;
      okc = (okb >> base) & 0xffu;
      const unsigned hits = (passb >> base) & 0xffu;
      hit = hits ? __ffs(hits) - 1 : -1;
      if (__any_sync(mask, (t.phase == IMP_FD || t.phase == IMP_M_FD))) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int i = 0; i < 4; ++i)
            Rc[i][j] = from_lane(mask, R[i], base + (((okc >> j) & 1u) ? j : 4 + j));
      }
      const int src = base + (hit > 0 ? hit : 0);
      ok = (okc & 1u) != 0u;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        R[i] = from_lane(mask, R[i], src);
        T[i] = from_lane(mask, T[i], src);
      }
#pragma unroll
      for (int k = 0; k < NV; ++k) V[k] = from_lane(mask, V[k], src);
      Z = from_lane(mask, Z, src);
    }
    if (t.phase != IMP_DONE) imp_digest(P, t, wide, ok, T, R, V, Z, okc, Rc, hit);
    __syncwarp(mask);
  }
}

// Sets a lane's task up for the implicit step of one cell (Sec. 3.3) from the explicit state
// Us; jc: the cell's Jacobian cache (17 words: M = (J - I)/h of its last converged solve and
// a flag; flag 1: M replaces C^(m) as the first matrix; flag 2: the last solve needed the
// matter primitives, and this one starts there).  Order: [flag 2: matter solve]; iteration on
// X; continuation in h on X; matter solve (unless it was the first attempt).  A cell without
// opacity needs no solve: its primitives are recovered here.
template <class F>
__device__ __forceinline__ void imp_begin(const Params& P, ImpTask<F>& t, double kappa, double sigma,
                                          double hdt, const double* Us, double Zguess,
                                          const double* jc) {
  t.rc = ST_OK;
  t.phase = IMP_DONE;
  t.k = 0;
  t.first = true;
#pragma unroll
  for (int k = 0; k < 17; ++k) t.jc[k] = jc ? jc[k] : 0.0;
  if ((kappa == 0.0 && sigma == 0.0) || hdt == 0.0) {
    t.rc = con2prim(P, Us, Zguess, t.V, nullptr);
    t.m = 0;  // U is Us itself
    return;
  }
  t.m = 1;
  t.c.kappa = kappa;
  t.c.sigma = sigma;
  t.c.hdt = t.hdt = hdt;
  t.c.D = Us[0];
  t.c.taut = Us[4] + Us[8];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    t.c.St[j] = Us[1 + j] + Us[9 + j];
    t.c.B[j] = Us[5 + j];
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) t.X[i] = t.c.Xs[i] = Us[8 + i];
  if constexpr (F::kReuseW) t.c.iD = ddiv_call(1.0, t.c.D);
  t.Z = t.Zguess = Zguess;
  t.tried_m = t.jc[16] == 2.0;
  t.lad = -1;
  t.phase = IMP_INIT;
}

// U of a converged task.
template <class F>
__device__ __forceinline__ void imp_result(const ImpTask<F>& t, const double* Us, double* U) {
  if (t.m == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) U[k] = Us[k];
  } else {
    matter_state(t.c, t.X, U);
  }
}

}  // namespace rr
