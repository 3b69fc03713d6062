// physics_f64.cuh -- FP64 device functions of the gray-M1 relativistic radiation
// MHD update (Lopez-Miralles, Marti & Perucho 2022, arXiv:2212.00370).
//
// Arithmetic contract of the FP64 path: every value is produced by IEEE
// +, -, *, /, sqrt in the association order written here, and the translation
// unit is compiled with --fmad=false, so the results are a pure function of the
// inputs.  The nested flux differences of the PVM viscosity divide rounding
// noise by eps = 1e-8, so a one-ulp change anywhere upstream shows up at the
// 1e-8 level; this order is therefore part of the specification of the path.
//
// Variable order (Sec. 2.1, Eq. eqU):
//   U = (D, S^x, S^y, S^z, tau_e, B^x, B^y, B^z, E_r, F^x, F^y, F^z)
//   V = (rho, v^x, v^y, v^z, p,   B^x, B^y, B^z, E_r, F^x, F^y, F^z)
#pragma once
#include <cstdint>

#include "fp64_int.cuh"

namespace rr {

constexpr int NV = 12;

// Correctly rounded a / b and sqrt(x) of the FP64 path (fp64_int.cuh).  The _call forms are
// one shared copy of the code, for places off the innermost loops: an inline quotient is
// ~60 instructions (1 KB), and the solvers' instruction footprint matters.
static __device__ __noinline__ double ddiv_call(double a, double b) { return fpi::div(a, b); }
static __device__ __noinline__ double dsqrt_call(double x) { return fpi::sqrt(x); }
__device__ __forceinline__ float ddiv_call(float a, float b) { return a / b; }
#ifdef RR_DIV_CALLS
__device__ __forceinline__ double ddiv(double a, double b) { return ddiv_call(a, b); }
__device__ __forceinline__ double dsqrt(double x) { return dsqrt_call(x); }
#else
__device__ __forceinline__ double ddiv(double a, double b) { return fpi::div(a, b); }
__device__ __forceinline__ double dsqrt(double x) { return fpi::sqrt(x); }
#endif

enum Status : int {
  ST_OK = 0,
  ST_C2P = 1,       // con2prim found no admissible root
  ST_IMPLICIT = 2,  // implicit radiation-matter solve failed
  ST_UNPHYS = 3,    // inadmissible conserved state (D <= 0 or E_r <= 0)
};

// A cell update the admissibility fallback retries with first-order faces: no
// admissible explicit state, or no converged implicit solve from it.
__host__ __device__ inline bool fallback_retry(int rc) {
  return rc == ST_C2P || rc == ST_IMPLICIT || rc == ST_UNPHYS;
}

enum Recon : int { RECON_GODUNOV = 0, RECON_MINMOD = 1, RECON_MC = 2, RECON_VANLEER = 3 };

// Scheme constants shared by every kernel of a context (passed by value).
struct Params {
  double gamma, a_rad, cfl, pvm_eps;
  int recon, beta_mode, c2p_maxit, imp_maxit;
  int pvm_k;  // PVM-int-2^k: 3 (PVM-int-8) or 4 (PVM-int-16)
  int pvm_products;  // FP64 A w products: 0 nested flux differences (Eq. utilde), 1 tangent
  int solver;        // 0 PVM-int (Sec. 3.2.2), 1 radiative HLL (Sec. 3.2.1)
  double imp_tol;
  double gfac;  // gamma/(gamma-1)
  double gm1g;  // (gamma-1)/gamma
};

// Products of prim2con.  SOFT (the pointwise kernel): on the integer pipes (fpi::mul_fast, ~30
// integer instructions, 14 clocks per warp and SM against 18.7 on the FP64 pipe, and both pipes
// run side by side); the factors must be zeros or normal, and the products normal, which the
// caller's window test (soft_matter) ensures.  Same roundings either way.  8 M prim2con: 857 us
// with FP64 products, 482 with these.  The flux keeps FP64 products: 47 more inline ones (24 KB)
// take a third of its FP64 instructions away and slow the faces of a Riemann batch by
// 15-25 % (instruction fetches).
template <bool SOFT>
__device__ __forceinline__ double mul(double a, double b) {
  if constexpr (SOFT)
    return fpi::mul_fast<true>(a, b);
  else
    return a * b;
}
// b + p a for p a power of two: one rounding either way where p a is exact.  (It is not where
// it is subnormal: the multiply-add then keeps the bit that the product would round off, and
// the last bit of a sum next to 2^-1022 may differ from the plain form's.)
__device__ __forceinline__ double scale_add(double p, double a, double b) {
#ifdef RR_DIV_CALLS
  return b + p * a;
#else
  return __fma_rn(p, a, b);
#endif
}

// Window in which the SOFT products of prim2con are valid: |v_k| from 2^-200 to 1 and
// |B_k| within 2^+-100, or zeros; rho and p within 2^+-150; v^2 < 1, so that W is a
// number in [1, 2^27); gamma/(gamma-1), which is in [1, 2^52] for a finite gamma and NaN for an
// infinite one.  Every product there has at most six factors and every difference keeps at
// least the last bit of its terms: all of them stay far inside 2^+-1022 or are exact zeros.  v^2
// is the sum aux_of forms.  8 M prim2con: 503 us without the test of v^2 (and finite numbers
// where W is not one), 510 with it, 482 with that of gamma as well (another schedule of the
// same products); with the test of v^2, 527 with v^2, 1/W and W formed once ahead of the branch,
// 529 with the test after the products, 509 with a bound of v^2 in FP32 first.
__device__ __forceinline__ bool soft_matter(const Params& P, const double* V) {
  using namespace fpi;
  bool ok = in_window(P.gfac, 1023, 60) && in_window(V[0], 1023 - 150, 300) &&
            in_window(V[4], 1023 - 150, 300);
#pragma unroll
  for (int k = 1; k < 4; ++k)
    ok = ok && in_window_or_zero(V[k], 1023 - 200, 200) && in_window_or_zero(V[4 + k], 1023 - 100, 200);
  return ok && below_one((V[1] * V[1] + V[2] * V[2]) + V[3] * V[3]);
}

// ---------------------------------------------------------------- aux state
// W = 1/sqrt(1-v^2), b^0 = W v.B, b^i = B^i/W + v^i b^0, |b|^2 = B^2/W^2 + (v.B)^2,
// rho h = rho + gamma/(gamma-1) p, p* = p + |b|^2/2   (Sec. 2.1).
struct Aux {
  double v2, iW, W, vB, B2, b0, b[3], bsq, rhoh, ptot;
};

// B2 (may be null): |B|^2 of the state, where the caller has it.
// The squares of v and B stay on the FP64 pipe in either form: with all 34 products of
// prim2con on the integer pipes these hold a warp for ~615 clocks and the FP64 pipe, with the
// sums alone, for ~410; six products moved back even the two out (8 M prim2con, products
// moved back: none 537 us, three 529, six 503, nine 503).
template <bool SOFT = false>
__device__ __forceinline__ void aux_of(const Params& P, const double* V, Aux& a,
                                       const double* B2 = nullptr) {
  const double vx = V[1], vy = V[2], vz = V[3];
  const double Bx = V[5], By = V[6], Bz = V[7];
  a.v2 = (vx * vx + vy * vy) + vz * vz;
  a.iW = dsqrt(1.0 - a.v2);
  a.W = ddiv(1.0, a.iW);
  a.vB = (mul<SOFT>(vx, Bx) + mul<SOFT>(vy, By)) + mul<SOFT>(vz, Bz);
  a.B2 = B2 ? *B2 : (Bx * Bx + By * By) + Bz * Bz;
  a.b0 = mul<SOFT>(a.W, a.vB);
  a.b[0] = mul<SOFT>(Bx, a.iW) + mul<SOFT>(vx, a.b0);
  a.b[1] = mul<SOFT>(By, a.iW) + mul<SOFT>(vy, a.b0);
  a.b[2] = mul<SOFT>(Bz, a.iW) + mul<SOFT>(vz, a.b0);
  a.bsq = mul<SOFT>(a.B2, mul<SOFT>(a.iW, a.iW)) + mul<SOFT>(a.vB, a.vB);
  a.rhoh = V[0] + mul<SOFT>(P.gfac, V[4]);
  a.ptot = scale_add(0.5, a.bsq, V[4]);
}

// rho h W^2: the con2prim unknown Z of a primitive state (warm starts).
__device__ __forceinline__ double prim_Z(const Params& P, const double* V) {
  Aux a;
  aux_of(P, V, a);
  return a.rhoh * (a.W * a.W);
}

// Eq. eqU, with rho W^2 - rho W = D u^2/(W+1) (u^2 = W^2 v^2).
template <bool SOFT>
__device__ __forceinline__ void prim2con_t(const Params& P, const double* V, double* U) {
  Aux a;
  aux_of<SOFT>(P, V, a);
  const double W2 = mul<SOFT>(a.W, a.W);
  const double D = mul<SOFT>(V[0], a.W);
  const double hw = mul<SOFT>(a.rhoh + a.bsq, W2);
  U[0] = D;
  U[1] = mul<SOFT>(hw, V[1]) - mul<SOFT>(a.b0, a.b[0]);
  U[2] = mul<SOFT>(hw, V[2]) - mul<SOFT>(a.b0, a.b[1]);
  U[3] = mul<SOFT>(hw, V[3]) - mul<SOFT>(a.b0, a.b[2]);
  const double u2 = mul<SOFT>(W2, a.v2);
  const double e1 = mul<SOFT>(D, ddiv(u2, a.W + 1.0));
  const double e2 = mul<SOFT>(mul<SOFT>(P.gfac, V[4]) + a.bsq, W2);
  U[4] = (e1 + e2) - (a.ptot + mul<SOFT>(a.b0, a.b0));
#pragma unroll
  for (int k = 5; k < NV; ++k) U[k] = V[k];
}
__device__ __forceinline__ void prim2con(const Params& P, const double* V, double* U) {
  prim2con_t<false>(P, V, U);
}

// a / b inline, or the shared copy
template <bool INL>
__device__ __forceinline__ double cdiv(double a, double b) {
  return INL ? ddiv(a, b) : ddiv_call(a, b);
}

// ------------------------------------------------------------- M1 closure
// xi(f) = (3 + 4f^2)/(5 + 2 sqrt(4 - 3f^2)), P = [(1-xi)/2 delta + (3xi-1)/2 n n] E
// (Sec. 2.2, Eq. xi); f clamped to 1; no n n term when F_r = 0.
struct M1 {
  double a, c;  // P_ij = c F_i F_j (+ a on the diagonal)
};

// INL: quotients and root inline (the faces), else the shared ones (the cell solver).
template <bool INL = true>
__device__ __forceinline__ M1 m1_coef(double E, double Fx, double Fy, double Fz) {
#ifndef RR_DIV_CALLS
  // factors 2, 4 and 1/2 folded into multiply-adds (their products are exact)
  const double F2 = (Fx * Fx + Fy * Fy) + Fz * Fz;
  double f2 = cdiv<INL>(F2, E * E);
  if (fpi::gt_nonneg(f2, 1.0)) f2 = 1.0;
  const double r = 4.0 - 3.0 * f2;
  const double xi = cdiv<INL>(__fma_rn(4.0, f2, 3.0), __fma_rn(2.0, (INL ? dsqrt(r) : dsqrt_call(r)), 5.0));
  M1 m;
  m.a = __fma_rn(-0.5, xi, 0.5) * E;
  const bool z = !fpi::pos(F2);
  const double mc = cdiv<INL>(__fma_rn(0.5, 3.0 * xi, -0.5) * E, z ? 1.0 : F2);
  m.c = z ? 0.0 : mc;
  return m;
#else
  // uncontracted in every unit: the FP32-bulk unit's results must not depend on how the
  // compiler fuses this sum with what is inlined around it
  const double F2 = __dadd_rn(__dadd_rn(__dmul_rn(Fx, Fx), __dmul_rn(Fy, Fy)), __dmul_rn(Fz, Fz));
  double f2 = ddiv(F2, E * E);
  if (f2 > 1.0) f2 = 1.0;
  const double xi = ddiv(3.0 + 4.0 * f2, 5.0 + 2.0 * dsqrt(4.0 - 3.0 * f2));
  M1 m;
  m.a = (0.5 * (1.0 - xi)) * E;
  m.c = 0.0;
  const double mc = ddiv((0.5 * (3.0 * xi - 1.0)) * E, F2 > 0.0 ? F2 : 1.0);
  if (F2 > 0.0) m.c = mc;
  return m;
#endif
}

__device__ __forceinline__ double m1_P(const M1& m, const double* F, int i, int j) {
  const double t = m.c * (F[i] * F[j]);
  return (i == j) ? t + m.a : t;
}

// Eddington tensor D_r = P_r/E_r (coefficients without the E_r factor).
__device__ __forceinline__ void eddington(double E, const double* F, double Dr[3][3]) {
  const double F2 = (F[0] * F[0] + F[1] * F[1]) + F[2] * F[2];
  double f2 = ddiv(F2, E * E);
  if (f2 > 1.0) f2 = 1.0;
  const double xi = ddiv(3.0 + 4.0 * f2, 5.0 + 2.0 * dsqrt(4.0 - 3.0 * f2));
  const double a = 0.5 * (1.0 - xi);
  const double c = (F2 > 0.0) ? ddiv(0.5 * (3.0 * xi - 1.0), F2) : 0.0;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) Dr[i][j] = c * (F[i] * F[j]) + (i == j ? a : 0.0);
}

// ------------------------------------------------------------- fluxes
// Eq. eqF along direction d, using the conserved variables of the same state:
//   momentum  S^j v^d - b^j B^d/W + p* delta^{dj}
//   energy    (tau_e + p*) v^d - b^0 B^d/W
//   induction v^d B^j - B^d v^j;  radiation F^d, P^{dj}.
// B2 as in aux_of.
__device__ __forceinline__ void flux(const Params& P, int d, const double* V, const double* U,
                                     double* F, const double* B2 = nullptr) {
  Aux a;
  aux_of(P, V, a, B2);
  const double vd = V[1 + d];
  const double Bd = V[5 + d];
  const double BdW = Bd * a.iW;
  F[0] = U[0] * vd;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const double t = U[1 + j] * vd - a.b[j] * BdW;
    F[1 + j] = (j == d) ? t + a.ptot : t;
  }
  F[4] = (U[4] + a.ptot) * vd - a.b0 * BdW;
#pragma unroll
  for (int j = 0; j < 3; ++j) F[5 + j] = (j == d) ? 0.0 : vd * V[5 + j] - Bd * V[1 + j];
  F[8] = V[9 + d];
  const double* Fr = V + 9;
  const M1 m = m1_coef(V[8], V[9], V[10], V[11]);
#pragma unroll
  for (int j = 0; j < 3; ++j) F[9 + j] = m1_P(m, Fr, d, j);
}

// ------------------------------------------------------------- con2prim
// One-dimensional Newton-Raphson in W' = Z - D, Z = rho h W^2, for the
// ideal-gas law (Mignone & McKinney 2007); it ends with the step |dW'| <= 1e-10 W';
// steps leaving W' > 0, v^2 < 1 are halved.
struct C2PIn {
  double D, S[3], tau, B[3], S2, B2, SB, SB2, gm1g;
};
struct C2PPt {  // the root
  double Z, iZ, iZB, v2, W, p;
};

// Newton's iteration from x > 0: the point of the last step, or false.  One loop holds the
// one copy of the evaluation, whatever it is for (the first point, doubled until
// admissible; Newton points, the step halved until admissible), and f and df are formed
// only where another Newton step follows.
// A point is admissible when x > 0 and v^2(x) < 1.  v^2 falls with x (Z = x + D > 0,
// B^2 >= 0), so every point at or below one whose v^2 came out >= 1 + 1e-9, and every point
// with Z + B^2 <= |S| (1 - 1e-12), where v^2 >= S^2/(Z + B^2)^2, is inadmissible and is
// passed over unevaluated: the margins are 10^4 times the rounding of the evaluation.
// Nearly all halvings are such points (C1, three steps: 35 of 37.7 million, 60 % of all
// the evaluations of the cell solves).
// FAST (the FP32-bulk form's cells): 1/Z and 1/(Z+B^2) from one division, W from rsqrt
// (the same values to a few ulps) and an inexact Newton step with an FP32 reciprocal of
// df (~6e-8 relative).
// Whether the products of the evaluation may be formed by mul_fast: D and S^2 within
// 2^+-80, B^2 and (S.B)^2 as well or zero, (gamma-1)/gamma in [2^-60, 2) (NaN for an infinite
// gamma).  With x in [2^-400, 2^80) every factor and every
// product of the evaluation is then normal (|h| <= 3/Z, the sums that can cancel to zero
// are tested where they are used).
__device__ __forceinline__ bool lo_hi_zero(double x) { return fpi::bits(x) == 0; }
__device__ __forceinline__ bool exp_zero(double x) { return (fpi::hi_word(x) & 0x7ff00000u) == 0; }
// 0 where z, else x
__device__ __forceinline__ double zsel(bool z, double x) { return z ? 0.0 : x; }
__device__ __forceinline__ bool c2p_window(const C2PIn& c) {
  using namespace fpi;
  constexpr uint32_t lo = 1023 - 80, n = 160;
  return in_window(c.gm1g, 1023 - 60, 61) && in_window(c.D, lo, n) && in_window(c.S2, lo, n) &&
         (in_window(c.B2, lo, n) || lo_hi_zero(c.B2)) &&
         (in_window(c.SB2, lo, n) || lo_hi_zero(c.SB2));
}

// pm: a product of the evaluation inside the window; z: one of its factors is zero.
template <bool SOFT>
__device__ __forceinline__ double pm(bool z, double a, double b) {
  if constexpr (SOFT)
    return zsel(z, fpi::mul_fast(a, b));
  else
    return a * b;
}

template <bool FAST, bool SOFT>
__device__ __forceinline__ bool c2p_root(const C2PIn& c, double x, int maxit, C2PPt& e) {
  using namespace fpi;
  double xt = x, dx = 0.0, bad = 0.0;
  int it = 0, k = 0;
  bool bound = false;
  const bool window = SOFT && c2p_window(c);
  const bool zB = lo_hi_zero(c.B2), zSB = lo_hi_zero(c.SB2);
  for (;;) {
    bool ok = gt_nonneg(xt, bad);
    double Z, iZ, iZB, iZ2, iZB2, v2;
    const bool in = window && in_window(xt, 1023 - 400, 480);
    if (ok) {
      Z = xt + c.D;
      const double ZB = Z + c.B2;
      if constexpr (FAST) {
        const double q = ddiv(1.0, Z * ZB);
        iZ = ZB * q;
        iZB = Z * q;
        iZ2 = iZ * iZ;
        v2 = (c.S2 + c.SB2 * ((2.0 * Z + c.B2) * iZ2)) * (iZB * iZB);
      } else {
        iZ = cdiv<SOFT>(1.0, Z);
        iZB = cdiv<SOFT>(1.0, ZB);
        if (in) {
          const double u = __fma_rn(2.0, Z, c.B2);
          iZ2 = pm<SOFT>(false, iZ, iZ);
          iZB2 = pm<SOFT>(false, iZB, iZB);
          v2 = pm<SOFT>(false, c.S2 + pm<SOFT>(zSB, c.SB2, pm<SOFT>(false, u, iZ2)), iZB2);
        } else {
          iZ2 = iZ * iZ;
          iZB2 = iZB * iZB;
          v2 = (c.S2 + c.SB2 * ((2.0 * Z + c.B2) * iZ2)) * iZB2;
        }
      }
      ok = below_one(v2);
      if (!ok && c.S2 < 1e200) {
        if (v2 >= 1.0 + 1e-9) bad = xt;
        if (!bound) {
          const double xs = dsqrt_call(c.S2) * (1.0 - 1e-12) - (c.B2 + c.D);
          if (xs > bad) bad = xs;
          bound = true;
        }
      }
    }
    if (!ok) {
      if (k == (it == 0 ? 200 : 60)) return false;
      ++k;
      if (it == 0) {
        xt = 2.0 * xt;
      } else {
        dx = 0.5 * dx;
        // halvings that cannot suffice, at once: while |dx| >= 2^(g+2), g the exponent of
        // x - bad, x + dx lies below bad
        const uint32_t ed = hi_word(dx) >> 20, eg = hi_word(x - bad) >> 20;
        if (ed - 0x801u < 0x7feu && eg - 1u < 0x7feu) {  // dx negative, both normal
          int n = (int)(ed - 0x800u) - (int)eg - 1;
          if (n > 60 - k) n = 60 - k;
          if (n > 0) {
            dx = make(hi_word(dx) - ((uint32_t)n << 20), lo_word(dx));
            k += n;
          }
        }
        xt = x + dx;
      }
      continue;
    }
    x = xt;
    const double omv2 = 1.0 - v2;
    double W, p;
    bool conv;
    if constexpr (FAST) {
      W = rsqrt(omv2);
      p = c.gm1g * (x * omv2 - c.D * ddiv(v2, W + 1.0));
      conv = mag_le(dx, 1e-10 * x);
    } else {
      W = cdiv<SOFT>(1.0, SOFT ? dsqrt(omv2) : dsqrt_call(omv2));
      const double q = cdiv<SOFT>(v2, W + 1.0);
      double tol;
      if (in) {
        const double t = pm<SOFT>(false, x, omv2) - pm<SOFT>(false, c.D, q);
        p = pm<SOFT>(exp_zero(t), c.gm1g, t);
        tol = pm<SOFT>(false, 1e-10, x);
      } else {
        p = c.gm1g * (x * omv2 - c.D * q);
        tol = 1e-10 * x;
      }
      conv = mag_le(dx, tol);
    }
    if (it > 0 && conv) {
      e.Z = Z;
      e.iZ = iZ;
      e.iZB = iZB;
      e.v2 = v2;
      e.W = W;
      e.p = p;
      return true;
    }
    if (it == maxit) return false;
    if constexpr (FAST) {
      const double f = ((x - p) + (0.5 * c.B2) * (1.0 + v2)) - ((0.5 * c.SB2) * iZ2 + c.tau);
      const double dv2 = (-2.0 * ((iZB * iZB) * iZB)) *
                         (c.S2 + c.SB2 * (((3.0 * Z + 3.0 * c.B2) * Z + c.B2 * c.B2) * (iZ2 * iZ)));
      const double dp = c.gm1g * (omv2 + dv2 * ((0.5 * c.D) * W - Z));
      const double df = ((1.0 - dp) + (0.5 * c.B2) * dv2) + c.SB2 * (iZ2 * iZ);
      const float d32 = to_float(df);
      dx = (fabsf(d32) > 1e-30f && fabsf(d32) < 1e30f) ? -f * to_double(__frcp_rn(d32)) : ddiv(-f, df);
    } else {
      double f, df;
      const double opv2 = 1.0 + v2;
      if (in) {
        // h = -dv^2/dx / 2.  Factors 2 and 1/2 are folded into multiply-adds (products with
        // them are exact): the same roundings as with the factor multiplied first.
        const double fb = __fma_rn(0.5, pm<SOFT>(zB, c.B2, opv2), x - p);
        f = fb - __fma_rn(0.5, pm<SOFT>(zSB, c.SB2, iZ2), c.tau);
        const double iZ3 = pm<SOFT>(false, iZ2, iZ), iZB3 = pm<SOFT>(false, iZB2, iZB);
        const double g = pm<SOFT>(false, pm<SOFT>(false, 3.0, Z) + 3.0 * c.B2, Z) + c.B2 * c.B2;
        const double h = pm<SOFT>(false, iZB3, c.S2 + pm<SOFT>(zSB, c.SB2, pm<SOFT>(false, g, iZ3)));
        const double y = __fma_rn(0.5, pm<SOFT>(false, c.D, W), -Z);
        const double w = __fma_rn(-2.0, pm<SOFT>(exp_zero(y), h, y), omv2);
        const double dp = pm<SOFT>(exp_zero(w), c.gm1g, w);
        df = ((1.0 - dp) - pm<SOFT>(zB, c.B2, h)) + pm<SOFT>(zSB, c.SB2, iZ3);
      } else {
        f = ((x - p) + (0.5 * c.B2) * opv2) - ((0.5 * c.SB2) * iZ2 + c.tau);
        const double iZ3 = iZ2 * iZ;
        const double g = (3.0 * Z + 3.0 * c.B2) * Z + c.B2 * c.B2;
        const double dv2 = (-2.0 * (iZB2 * iZB)) * (c.S2 + c.SB2 * (g * iZ3));
        const double dp = c.gm1g * (omv2 + dv2 * ((0.5 * c.D) * W - Z));
        df = ((1.0 - dp) + (0.5 * c.B2) * dv2) + c.SB2 * iZ3;
      }
      dx = cdiv<SOFT>(-f, df);
    }
    xt = x + dx;
    ++it;
    k = 0;
  }
}

// Returns a Status; V, *Zout, *Wout (the Lorentz factor) and *B2out (|B|^2; all may be null)
// are written only on success.
// Stopping rule: the iteration stops at the Newton step with |dx| <= 1e-10 x (the
// step is taken).  In Newton's quadratic regime the error left is of order
// (1e-10 x)^2 / x, below rounding, so the PVM's finite-difference products, which
// differentiate con2prim at the 1e-8 level, see a recovery exact to rounding.
// SOFT: the products of the evaluation on the integer pipes where the state allows it.  Half
// of the FP64 instructions less per recovery (1 M C1 states: 825 -> 447 us), but a longer
// chain (a product is ~100 clocks instead of 64) and 20 KB of code: the faces, whose warps
// run in step, and the recovery itself take it; the cell solver, paced by its slowest cells
// and its instruction fetches, does not, and calls the shared quotient and root (inline ones
// cost 3-5 % there: 3D box 89.3 -> 84.8 ms per step with calls here and in the residual).
template <bool FAST = false, bool SOFT = false>
static __device__ __noinline__ int con2prim(const Params& P, const double* U, double Zguess,
                                            double* V, double* Zout, double* Wout = nullptr,
                                            double* B2out = nullptr) {
  C2PIn c;
  c.D = U[0];
  c.S[0] = U[1];
  c.S[1] = U[2];
  c.S[2] = U[3];
  c.tau = U[4];
  c.B[0] = U[5];
  c.B[1] = U[6];
  c.B[2] = U[7];
  c.S2 = (c.S[0] * c.S[0] + c.S[1] * c.S[1]) + c.S[2] * c.S[2];
  c.B2 = (c.B[0] * c.B[0] + c.B[1] * c.B[1]) + c.B[2] * c.B[2];
  c.SB = (c.S[0] * c.B[0] + c.S[1] * c.B[1]) + c.S[2] * c.B[2];
  c.SB2 = c.SB * c.SB;
  c.gm1g = P.gm1g;
  if (!fpi::pos(c.D) || !fpi::pos(U[8])) return ST_UNPHYS;

  double x = Zguess - c.D;
  if (!fpi::pos(x)) x = fpi::pos(c.tau) ? c.tau : c.D;
  C2PPt e;
  if (!c2p_root<FAST, SOFT>(c, x, P.c2p_maxit, e) || !fpi::pos(e.p)) return ST_C2P;
  const double rho = FAST ? c.D * ((1.0 - e.v2) * e.W) : ddiv(c.D, e.W);  // D/W = D (1 - v^2) W
  const double SBiZ = c.SB * e.iZ;
  V[0] = rho;
  V[1] = (c.S[0] + SBiZ * c.B[0]) * e.iZB;
  V[2] = (c.S[1] + SBiZ * c.B[1]) * e.iZB;
  V[3] = (c.S[2] + SBiZ * c.B[2]) * e.iZB;
  V[4] = e.p;
#pragma unroll
  for (int k = 5; k < NV; ++k) V[k] = U[k];
  if (Zout) *Zout = e.Z;
  if (Wout) *Wout = e.W;
  if (B2out) *B2out = c.B2;
  return ST_OK;
}

// ------------------------------------------------------------- signal speed
// max |lambda| along d, capped at 1: fast-magnetosonic estimate (Del Zanna et
// al. 2007) and the radiation eigenvalues lambda_r1, lambda_r3 (Eqs. lam1-lam3).
// Signed fast-magnetosonic speed estimates lm <= lp along d (Del Zanna et al. 2007).
__device__ __forceinline__ void mhd_speeds(const Params& P, int d, const double* V, double& lm,
                                           double& lp) {
  Aux a;
  aux_of(P, V, a);
  const double cs2 = ddiv_call(P.gamma * V[4], a.rhoh);
  const double ca2 = ddiv_call(a.bsq, a.rhoh + a.bsq);
  const double a2 = (cs2 + ca2) - cs2 * ca2;
  const double vd = V[1 + d];
  const double den = 1.0 - a.v2 * a2;
  double disc = (a2 * (1.0 - a.v2)) * (den - (vd * vd) * (1.0 - a2));
  if (disc < 0.0) disc = 0.0;
  const double sq = dsqrt(disc);
  lp = ddiv_call(vd * (1.0 - a2) + sq, den);
  lm = ddiv_call(vd * (1.0 - a2) - sq, den);
}

// Outer radiation eigenvalues l1 <= l3 (Eqs. lam1-lam3), theta between F_r and d.
__device__ __forceinline__ void rad_speeds(int d, const double* V, double& l1, double& l3) {
  const double E = V[8];
  const double F2 = (V[9] * V[9] + V[10] * V[10]) + V[11] * V[11];
  const double Fn = dsqrt(F2);
  double f = ddiv_call(Fn, E);
  if (f > 1.0) f = 1.0;
  const double cq = ddiv_call(V[9 + d], Fn > 0.0 ? Fn : 1.0);
  const double cth = (Fn > 0.0) ? cq : 0.0;
  const double f2 = f * f;
  const double s = dsqrt(4.0 - 3.0 * f2);
  double arg = (2.0 / 3.0) * ((4.0 - 3.0 * f2) - s) + (2.0 * (cth * cth)) * ((2.0 - f2) - s);
  if (arg < 0.0) arg = 0.0;
  const double zeta = dsqrt(arg);
  l1 = ddiv_call(f * cth - zeta, s);
  l3 = ddiv_call(f * cth + zeta, s);
}

__device__ __forceinline__ double signal_speed(const Params& P, int d, const double* V) {
  double lm, lp, l1, l3;
  mhd_speeds(P, d, V, lm, lp);
  const double lf = fabs(lp) > fabs(lm) ? fabs(lp) : fabs(lm);
  rad_speeds(d, V, l1, l3);
  const double lr = fabs(l1) > fabs(l3) ? fabs(l1) : fabs(l3);
  double lam = lf > lr ? lf : lr;
  if (lam > 1.0) lam = 1.0;
  return lam;
}

// ------------------------------------------------------------- four-force
// Eqs. g0, gi with u^i = W v^i, W^2 - 1 = u^2, 2W^2 - 1 = 2u^2 + 1, BP = a_R T^4.
__device__ __forceinline__ void four_force(double kappa, double sigma, double rho,
                                           const double* u, double W, double BP, double E,
                                           const double* F, const double Pr[3][3],
                                           double* G) {
  const double u2 = (u[0] * u[0] + u[1] * u[1]) + u[2] * u[2];
  const double uF = (u[0] * F[0] + u[1] * F[1]) + u[2] * F[2];
  double Pu[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) Pu[i] = (Pr[i][0] * u[0] + Pr[i][1] * u[1]) + Pr[i][2] * u[2];
  const double uPu = (u[0] * Pu[0] + u[1] * Pu[1]) + u[2] * Pu[2];
  const double rk = rho * kappa;
  const double rs = rho * sigma;
  G[0] = -(rk * (W * (BP - E) + uF)) - rs * (((W * u2) * E + W * uPu) - (2.0 * u2 + 1.0) * uF);
  const double q = ((W * W) * E - (2.0 * W) * uF) + uPu;
#pragma unroll
  for (int i = 0; i < 3; ++i)
    G[1 + i] = ((-(BP * rk)) * u[i] + (rk + rs) * (W * F[i] - Pu[i])) - (rs * u[i]) * q;
}

}  // namespace rr
