// Exact Riemann solver for the ideal gas, device side (Sec. 3.3: exact
// solver with a treatment of vacuum; the mathematics is that of the 1D Euler
// Riemann problem).
//
// The star pressure p* is the root of
//   f(p) = f_L(p) + f_R(p) + (u_R - u_L),
//   f_K(p) = (p - p_K) sqrt(A_K / (p + B_K))                      p > p_K (shock)
//          = 2 c_K / (gamma-1) ((p/p_K)^z - 1),  z=(gamma-1)/(2gamma)  p <= p_K (rarefaction)
//   A_K = 2 / ((gamma+1) rho_K), B_K = (gamma-1)/(gamma+1) p_K,
// found by Newton's method to the relative change 2|dp|/(p_new+p_old) < tol
// from a starting value, then sampled at x/t = 0.  The rarefaction derivative
// uses (p/p_K)^(z-1) = (p/p_K)^z / (p/p_K) so one power serves f and f'.
// Vacuum generated between two rarefactions (2(c_L+c_R)/(gamma-1) <= u_R-u_L)
// is handled in closed form; the extrapolated states reaching this solver are
// always positive (non-positive ones fall back to first order before).
//
// FP32 form: the iteration runs in float.  Near vacuum and in strong
// rarefactions float cannot resolve the relative tolerance (f is a
// difference of terms ~2c/(gamma-1) that cancel), so once an iterate falls
// below GUARD * min(p_L, p_R), or the float loop has not converged after
// FLOAT_ITERS iterations, the solve continues in FP64 (pressure functions,
// step and convergence test), and the face is counted.
#pragma once

#include <cuda_runtime.h>
#include <float.h>

#include "amm_internal.cuh"
#include "fixed64.cuh"

namespace amm {


__device__ __forceinline__ double xpow(double a, double b) { return pow64(a, b); }
__device__ __forceinline__ float xpow(float a, float b) { return __powf(a, b); }
__device__ __forceinline__ double xsqrt(double a) { return sqrt64(a); }
__device__ __forceinline__ float xsqrt(float a) { return sqrtf(a); }
__device__ __forceinline__ double xrsqrt(double a) { return rsqrt64(a); }
__device__ __forceinline__ float xrsqrt(float a) { return rsqrtf(a); }
__device__ __forceinline__ double xdiv(double a, double b) { return div64(a, b); }
__device__ __forceinline__ float xdiv(float a, float b) { return a / b; }
__device__ __forceinline__ double xrecip(double a) { return recip64(a); }
__device__ __forceinline__ float xrecip(float a) { return 1.0f / a; }

// an FP64 value in the bulk precision
template <typename real>
__device__ __forceinline__ real bulk(double x) {
  if constexpr (sizeof(real) == 4)
    return to_float(x);
  else
    return x;
}

__device__ __forceinline__ double widen(float x) { return to_double(x); }
__device__ __forceinline__ double widen(double x) { return x; }

// Comparisons; FP64 ones in integers (an FP64 comparison takes the FP64 pipe): x > 0;
// a < b and a <= b for a >= 0 (or its magnitude) and b >= 0, false where b is a NaN.
__device__ __forceinline__ bool positive(float x) { return x > 0.0f; }
__device__ __forceinline__ bool positive(double x) {
  return (u64)__double_as_longlong(x) - 1ull < 0x7ff0000000000000ull;
}
__device__ __forceinline__ bool mag_less(double a, double b) {
  const i64 i = __double_as_longlong(a) & 0x7fffffffffffffffll, j = __double_as_longlong(b);
  return i < j && j <= 0x7ff0000000000000ll;
}
__device__ __forceinline__ bool mag_leq(double a, double b) {
  const i64 i = __double_as_longlong(a) & 0x7fffffffffffffffll, j = __double_as_longlong(b);
  return i <= j && j <= 0x7ff0000000000000ll;
}

// Explicitly rounded products, sums and fused multiply-adds: the compiler
// neither fuses nor splits them, so a formula written with them rounds the
// same in every kernel it is inlined into.  Whether a plain a * b + c is
// fused depends on where the compiler places the product relative to the
// branches of an inlined FP64 division or square root, which differs
// between kernels.  The per-phase kernels and the persistent step kernel
// must agree bit for bit.
__device__ __forceinline__ double rn_mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float rn_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double rn_add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float rn_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double rn_fma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float rn_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
// a . b of two 3-vectors, x first
template <typename real>
__device__ __forceinline__ real rn_dot3(real ax, real ay, real az, real bx, real by, real bz) {
  return rn_fma(az, bz, rn_fma(ay, by, rn_mul(ax, bx)));
}

// f_K(p) and f_K'(p), FP32
__device__ __forceinline__ void wave_curve(float p, float rhoK, float pK, float cK, const GasC<float>& G, float& f,
                                           float& df) {
  using real = float;
  {
    // both branches, selected.  The sides of a warp's faces split
    // between shocks and rarefactions, so a branch would run both anyway;
    // unconditional, the per-side constants leave the Newton loop.
    const real A = G.two_gp1 / rhoK;
    const real id = (real)1 / (p + G.gm1_gp1 * pK);
    const real q = xsqrt(A * id);
    const real fs = (p - pK) * q;
    const real dfs = q * ((real)1 - (real)0.5 * (p - pK) * id);
    const real pr = p / pK;
    const real prz = xpow(pr, G.z);
    const real fr = G.two_gm1 * cK * (prz - (real)1);
    const real dfr = prz / (pr * rhoK * cK);
    const bool shock = p > pK;
    f = shock ? fs : fr;
    df = shock ? dfs : dfr;
  }
}

// FP64: f_K(p) and f_K'(p).  The shock takes one reciprocal square root, with h =
// rho (gamma+1)/2: q = (h (p + B))^(-1/2), whose roundings (h, p + B, their product,
// halved, and the root's) are no more than those of sqrt(A / (p + B)), and 1/(p + B) =
// h q^2 for the slope; the rarefaction f' = (p/p_K)^z c_K / (gamma p) (rho_K c_K =
// gamma p_K / c_K), with 1/p given (both sides need it).  The slopes only steer Newton's
// iteration; the values are rounded as the formulas' own quotients and powers.
// (explicitly rounded: the persistent step kernel must round alike)
struct WaveSide {
  double h, p, B, two_c, c_g;   // (gamma+1)/2 rho, p, B, 2c/(gamma-1), c/gamma
};
__device__ __forceinline__ WaveSide wave_side(double rho, double p, double c, const GasC<double>& G) {
  WaveSide s;
  s.h = rn_mul(G.half_gp1, rho);
  s.p = p;
  s.B = rn_mul(G.gm1_gp1, p);
  s.two_c = rn_mul(G.two_gm1, c);
  s.c_g = rn_mul(c, G.inv_g);
  return s;
}
__device__ __forceinline__ void wave_curve(double p, double ip, const WaveSide& K, const GasC<double>& G, double& f,
                                           double& df) {
  const double d = rn_add(p, -K.p);
  if (positive(d)) {
    const double q = rsqrt64(rn_mul(K.h, rn_add(p, K.B)));
    const double dh = rn_mul(d, rn_mul(rn_mul(q, q), K.h));
    f = rn_mul(d, q);
    df = rn_mul(q, rn_fma(-0.5, dh, 1.0));
  } else {
    const double prz = pow64(div64(p, K.p), G.z);
    f = rn_mul(K.two_c, rn_add(prz, -1.0));
    df = rn_mul(rn_mul(prz, K.c_g), ip);
  }
}

// Linearised (primitive-variable) star pressure, clipped at 0, and the
// two-shock estimate evaluated at it.
template <typename real>
__device__ __forceinline__ real linearised_pstar(real rhoL, real uL, real pL, real cL, real rhoR, real uR, real pR,
                                                 real cR) {
  const real ppv = (real)0.5 * (pL + pR) - (real)0.125 * (uR - uL) * (rhoL + rhoR) * (cL + cR);
  return ppv > (real)0 ? ppv : (real)0;
}

template <typename real>
__device__ __forceinline__ real two_shock_pstar(real rhoL, real uL, real pL, real rhoR, real uR, real pR, real ppv,
                                                const GasC<real>& G) {
  if constexpr (sizeof(real) == 8) {
    // one reciprocal square root per side (in units of sqrt(2/(gamma+1)))
    const double gL = rsqrt64(rn_mul(rhoL, rn_fma(G.gm1_gp1, pL, ppv)));
    const double gR = rsqrt64(rn_mul(rhoR, rn_fma(G.gm1_gp1, pR, ppv)));
    const double du = rn_mul(rn_add(uR, -uL), G.isqrt_two_gp1);
    return div64(rn_add(rn_fma(gL, pL, rn_mul(gR, pR)), -du), rn_add(gL, gR));
  } else {
    const real gL = xsqrt((G.two_gp1 / rhoL) / (ppv + G.gm1_gp1 * pL));
    const real gR = xsqrt((G.two_gp1 / rhoR) / (ppv + G.gm1_gp1 * pR));
    return (gL * pL + gR * pR - (uR - uL)) / (gL + gR);
  }
}

// Standard starting value: the linearised (primitive-variable) estimate when
// the pressure ratio is small and it lies between p_L and p_R, else the
// two-rarefaction estimate when it lies below both, else the two-shock
// estimate evaluated at the linearised pressure; floored positive.  With a
// proposal (`have`), the proposal replaces the two-shock estimate -- the one
// approximate branch: the two-rarefaction estimate is the exact star pressure
// when both waves are rarefactions, and the linearised one is kept where it
// passes its own test.
template <typename real>
__device__ __forceinline__ real standard_guess_ppv(real rhoL, real uL, real pL, real cL, real rhoR, real uR, real pR,
                                                   real cR, real ppv, const GasC<real>& G, bool have = false,
                                                   real proposal = (real)0) {
  const real du = uR - uL;
  const bool lowL = sizeof(real) == 8 ? mag_less(pL, pR) : pL < pR;
  const real pmin = lowL ? pL : pR, pmax = lowL ? pR : pL;
  real p0;
  if constexpr (sizeof(real) == 4) {
    // FP32: every estimate, selected (a warp's faces take all three, so
    // branches would run them all anyway)
    const bool pv = pmax <= (real)2 * pmin && ppv >= pmin && ppv <= pmax;
    const real num = cL + cR - (real)0.5 * G.gm1 * du;
    const real den = cL / xpow(pL, G.z) + cR / xpow(pR, G.z);
    const real ptr = xpow(num / den, G.inv_z);
    const real pts = have ? proposal : two_shock_pstar(rhoL, uL, pL, rhoR, uR, pR, ppv, G);
    p0 = pv ? ppv : (ppv < pmin ? ptr : pts);
  } else if (mag_leq(pmax, rn_mul(2.0, pmin)) && mag_leq(pmin, ppv) && mag_leq(ppv, pmax)) {
    p0 = ppv;
  } else if (mag_less(ppv, pmin)) {
    const real num = rn_add(rn_add(cL, cR), -rn_mul(rn_mul((real)0.5, G.gm1), du));
    const real den = rn_fma(cL, xpow(pL, -G.z), rn_mul(cR, xpow(pR, -G.z)));
    p0 = xpow(div64(num, den), G.inv_z);
  } else if (have) {
    p0 = proposal;
  } else {
    p0 = two_shock_pstar(rhoL, uL, pL, rhoR, uR, pR, ppv, G);
  }
  const real pfloor = (real)1e-10 * (real)0.5 * (pL + pR);
  if constexpr (sizeof(real) == 8) return positive(p0) && mag_less(pfloor, p0) ? p0 : pfloor;
  return (p0 > pfloor) ? p0 : pfloor;
}

template <typename real>
__device__ __forceinline__ real standard_guess(real rhoL, real uL, real pL, real cL, real rhoR, real uR, real pR,
                                               real cR, const GasC<real>& G, bool have = false,
                                               real proposal = (real)0) {
  return standard_guess_ppv(rhoL, uL, pL, cL, rhoR, uR, pR, cR, linearised_pstar(rhoL, uL, pL, cL, rhoR, uR, pR, cR),
                            G, have, proposal);
}

struct RiemannInfo {
  int iters;
  int guard;      // finished in FP64
  int vacuum;
  int fail;       // hit the iteration cap
};

// State of the last Newton step: f_L, f_R and their derivatives at the
// previous iterate p_prev; u* at the final p follows to first order,
// u* = (u_L+u_R)/2 + (f_R - f_L + (f_R' - f_L')(p - p_prev))/2, with an error
// of order (p - p_prev)^2, far below the tolerance.
template <typename real>
struct NewtonTail {
  real fL, dL, fR, dR, dp;
};

// The FP64 Newton loops also stop when f(p) vanishes to rounding (|f| within
// RESIDUAL_ULPS ulps of the size of its terms): p is then the root in working
// precision.  Near vacuum f is a small difference of large terms and the
// relative change of p cannot fall below a 1e-12 tolerance.
constexpr double RESIDUAL_ULPS = 64.0;

// One step from p, whose f_K and f_K' are in t; true when p (or the new p) is converged
__device__ __forceinline__ bool newton_step64(double& p, double du, double tol, int& it, NewtonTail<double>& t) {
  t.dp = 0.0;
  const double f = rn_add(rn_add(t.fL, t.fR), du);
  const double small = rn_mul(RESIDUAL_ULPS * DBL_EPSILON, rn_add(rn_add(fabs(t.fL), fabs(t.fR)), fabs(du)));
  if (mag_leq(f, small)) return true;
  const double D = rn_add(t.dL, t.dR);
  double pn = rn_add(p, -div64(f, D));
  if (!positive(pn)) pn = rn_mul(1e-3, p);
  it++;
  t.dp = rn_add(pn, -p);
  // 2 |dp| / (p_new + p_old) < tol, without the division
  const bool done = mag_less(t.dp, rn_mul(0.5 * tol, rn_add(pn, p)));
  p = pn;
  return done;
}

// The FP64 Newton iteration: p* from the iterate p; it and conv as in newton_pstar.
__device__ __forceinline__ double newton_pstar64(double p, const WaveSide& KL, const WaveSide& KR, double du,
                                                 const GasC<double>& G, double tol, int maxit, int& it, bool& conv,
                                                 NewtonTail<double>& t) {
  t.fL = t.dL = t.fR = t.dR = t.dp = 0.0;
  while (it < maxit) {
    const double ip = recip64(p);
    wave_curve(p, ip, KL, G, t.fL, t.dL);
    wave_curve(p, ip, KR, G, t.fR, t.dR);
    if (newton_step64(p, du, tol, it, t)) {
      conv = true;
      break;
    }
  }
  return p;
}

// The same iteration by two lanes, l and l ^ 16, that hold the same problem: each
// evaluates the wave curve of its own side (side: 1 right) and passes it to the
// other, which halves the chain of FP64 instructions of a warp with few problems.
// All lanes of `in` call it; the values and their order are newton_pstar64's.
__device__ __forceinline__ double newton_pstar64_pair(double p, const WaveSide& K, int side, double du,
                                                      const GasC<double>& G, double tol, int maxit, unsigned in,
                                                      int& it, bool& conv, NewtonTail<double>& t) {
  t.fL = t.dL = t.fR = t.dR = t.dp = 0.0;
  while (__any_sync(in, !conv && it < maxit)) {
    const double ip = recip64(p);
    double f1, d1;
    wave_curve(p, ip, K, G, f1, d1);
    const double f2 = __shfl_xor_sync(in, f1, 16), d2 = __shfl_xor_sync(in, d1, 16);
    if (conv || it >= maxit) continue;
    t.fL = side ? f2 : f1;
    t.fR = side ? f1 : f2;
    t.dL = side ? d2 : d1;
    t.dR = side ? d1 : d2;
    conv = newton_step64(p, du, tol, it, t);
  }
  return p;
}

// The FP32 forms' rare continuation in FP64: in place, or left to the caller
// (info.guard set, the returned state unfinished), whose kernel then holds no
// FP64 solve.
// SOLVE_PAIRED: FP64 problems held by lanes l and l ^ 16 alike (all lanes call).
enum GuardKind { GUARD_INLINE, GUARD_DEFER, SOLVE_PAIRED };
struct GuardOut {
  float p, us;
  int iters, conv;
};
__device__ __forceinline__ GuardOut guard_solve(float p, float rhoL, float uL, float pL, float rhoR, float uR,
                                                    float pR, float g, double tol, int maxit, int it) {
  const GasC<double> G((double)g);
  const double rL = rhoL, pLd = pL, rR = rhoR, pRd = pR;
  NewtonTail<double> t;
  bool done = false;
  const double ps = newton_pstar64((double)p, wave_side(rL, pLd, sqrt64(div64(G.g * pLd, rL)), G),
                                   wave_side(rR, pRd, sqrt64(div64(G.g * pRd, rR)), G), (double)uR - (double)uL, G, tol, maxit,
                                   it, done, t);
  GuardOut o;
  o.p = (float)ps;
  o.us = 0.5f * (uL + uR) + 0.5f * (((float)t.fR - (float)t.fL) + ((float)t.dR - (float)t.dL) * (float)t.dp);
  o.iters = it;
  o.conv = done;
  return o;
}
// Newton iteration for p*; returns p* in `real`, with the FP64 guard in the
// FP32 form, and the star velocity us.  iterations counted in info.
template <GuardKind GUARD = GUARD_INLINE, typename real>
__device__ __forceinline__ real newton_pstar(real p, real rhoL, real uL, real pL, real cL, real rhoR, real uR,
                                             real pR, real cR, const GasC<real>& G, double tol, real tol_r, int maxit,
                                             RiemannInfo& info, real& us, unsigned in = 0u) {
  const real du = uR - uL;
  NewtonTail<real> tail;
  int it = 0;
  bool conv = false;
  if constexpr (sizeof(real) == 8 && GUARD == SOLVE_PAIRED) {
    const int side = ((int)threadIdx.x >> 4) & 1;
    p = newton_pstar64_pair(p, wave_side(side ? rhoR : rhoL, side ? pR : pL, side ? cR : cL, G), side, du, G, tol,
                            maxit, in, it, conv, tail);
  } else if constexpr (sizeof(real) == 8) {
    p = newton_pstar64(p, wave_side(rhoL, pL, cL, G), wave_side(rhoR, pR, cR, G), du, G, tol, maxit, it, conv, tail);
  } else {
    constexpr int FLOAT_ITERS = 12;
    const float tol_f = (float)tol_r;   // the tolerance in FP32, converted once on the host
    const float guard_p = 1e-3f * (pL < pR ? (float)pL : (float)pR);
    bool to64 = false;
    while (it < maxit) {
      if (it >= FLOAT_ITERS || (float)p < guard_p) {
        to64 = true;
        break;
      }
      real fL, dL, fR, dR;
      wave_curve(p, rhoL, pL, cL, G, fL, dL);
      wave_curve(p, rhoR, pR, cR, G, fR, dR);
      real pn = p - (fL + fR + du) / (dL + dR);
      if (!(pn > (real)0)) pn = (real)1e-3 * p;
      it++;
      // 2 |dp| / (p_new + p_old) < tol, without the division
      const bool done = (real)2 * fabsf((float)(pn - p)) < tol_f * (pn + p);
      tail.fL = fL; tail.dL = dL; tail.fR = fR; tail.dR = dR; tail.dp = pn - p;
      p = pn;
      if (done) {
        conv = true;
        break;
      }
    }
    if (to64) {
      info.guard = 1;
      if constexpr (GUARD == GUARD_DEFER) {
        info.iters = it;
        info.fail = 0;
        us = (real)0;
        return p;
      }
      const GuardOut o = guard_solve(p, rhoL, uL, pL, rhoR, uR, pR, G.g, tol, maxit, it);
      info.iters = o.iters;
      info.fail = o.conv ? 0 : 1;
      us = o.us;
      return o.p;
    }
  }
  if constexpr (sizeof(real) == 8)
    us = rn_mul(0.5, rn_add(rn_add(uL, uR),
                            rn_fma(rn_add(tail.dR, -tail.dL), tail.dp, rn_add(tail.fR, -tail.fL))));
  else
    us = (real)0.5 * (uL + uR) + (real)0.5 * ((tail.fR - tail.fL) + (tail.dR - tail.dL) * tail.dp);
  info.iters = it;
  info.fail = conv ? 0 : 1;
  return p;
}

// Sampled state at x/t = 0 of the Riemann problem (rho, u, p per side).
// Returns side of the contact (0: left, 1: right) for the transverse
// velocity; rho = P = 0 inside generated vacuum.  pstar: the star pressure
// (0 when vacuum is generated).
// cL, cR: the sides' sound speeds; ppv: the linearised star pressure (the
// caller may have formed them already, for the proposal's gate).
template <GuardKind GUARD = GUARD_INLINE, typename real>
__device__ __forceinline__ int riemann_sample_c(real rhoL, real uL, real pL, real rhoR, real uR, real pR, real cL,
                                                real cR, real ppv, const GasC<real>& G, double tol, real tol_r,
                                                int maxit, bool have_guess, real guess, real& rhoF, real& uF, real& pF,
                                                RiemannInfo& info, real& pstar) {
  pstar = (real)0;
  info.iters = 0;
  info.guard = 0;
  info.vacuum = 0;
  info.fail = 0;
  const bool vacuum = G.two_gm1 * (cL + cR) <= uR - uL;
  unsigned in = 0u;
  if constexpr (GUARD == SOLVE_PAIRED) in = __ballot_sync(0xffffffffu, !vacuum);
  if (vacuum) {
    // two rarefactions with vacuum between them
    info.vacuum = 1;
    const real frontL = uL + G.two_gm1 * cL;
    const real frontR = uR - G.two_gm1 * cR;
    if ((real)0 <= frontL) {
      if ((real)0 <= uL - cL) {
        rhoF = rhoL; uF = uL; pF = pL;
      } else {
        const real c = G.two_gp1 * cL + G.gm1_gp1 * uL;
        const real r = xdiv(c, cL);
        uF = c;
        rhoF = rhoL * xpow(r, G.fan_rho);
        pF = pL * xpow(r, G.fan_p);
      }
      return 0;
    }
    if ((real)0 >= frontR) {
      if ((real)0 >= uR + cR) {
        rhoF = rhoR; uF = uR; pF = pR;
      } else {
        const real c = G.two_gp1 * cR - G.gm1_gp1 * uR;
        const real r = xdiv(c, cR);
        uF = -c;
        rhoF = rhoR * xpow(r, G.fan_rho);
        pF = pR * xpow(r, G.fan_p);
      }
      return 1;
    }
    rhoF = (real)0; uF = (real)0.5 * (frontL + frontR); pF = (real)0;
    return 0;
  }
  const real p0 = standard_guess_ppv(rhoL, uL, pL, cL, rhoR, uR, pR, cR, ppv, G, have_guess, guess);
  real us;
  const real ps = newton_pstar<GUARD>(p0, rhoL, uL, pL, cL, rhoR, uR, pR, cR, G, tol, tol_r, maxit, info, us, in);
  pstar = ps;
  // the side the face sees (the contact's upwind side): s = +1 left, -1
  // right; the right side's formulas are the left side's with the velocity
  // signs flipped (products with s are exact), so one path serves both
  const int side = ((real)0 <= us) ? 0 : 1;
  const real s = side ? (real)-1 : (real)1;
  const real rhoK = side ? rhoR : rhoL, uK = side ? uR : uL, pK = side ? pR : pL, cK = side ? cR : cL;
  const real r = xdiv(ps, pK);
  if constexpr (sizeof(real) == 4) {
    // FP32: the shock and rarefaction cases evaluated and selected; only the
    // sonic rarefaction (the face inside the fan, rare) branches
    const bool shock = ps > pK;
    const real sq = xsqrt(G.shock_a * r + G.shock_b);
    const real lr = __log2f(r);
    const real rz = exp2f(G.z * lr), rig = exp2f(G.inv_g * lr);
    const bool orig = shock ? ((real)0 <= s * (uK - s * cK * sq)) : ((real)0 <= s * (uK - s * cK));
    const bool fan = !shock && !orig && !((real)0 > s * (us - s * cK * rz));
    const real rho_star = shock ? rhoK * (r + G.gm1_gp1) / (G.gm1_gp1 * r + (real)1) : rhoK * rig;
    rhoF = orig ? rhoK : rho_star;
    uF = orig ? uK : us;
    pF = orig ? pK : ps;
    if (fan) {
      const real c = G.two_gp1 * cK + s * G.gm1_gp1 * uK;
      const real q = xdiv(c, cK);
      uF = s * c;
      rhoF = rhoK * xpow(q, G.fan_rho);
      pF = pK * xpow(q, G.fan_p);
    }
  } else if (mag_less(pK, ps)) {
    const real SK = uK - s * cK * xsqrt(G.shock_a * r + G.shock_b);
    if ((real)0 <= s * SK) {
      rhoF = rhoK; uF = uK; pF = pK;
    } else {
      rhoF = xdiv(rhoK * (r + G.gm1_gp1), G.gm1_gp1 * r + (real)1); uF = us; pF = ps;
    }
  } else {
    if ((real)0 <= s * (uK - s * cK)) {
      rhoF = rhoK; uF = uK; pF = pK;
    } else {
      const real tail = us - s * cK * xpow(r, G.z);
      if ((real)0 > s * tail) {
        rhoF = rhoK * xpow(r, G.inv_g); uF = us; pF = ps;
      } else {
        const real c = G.two_gp1 * cK + s * G.gm1_gp1 * uK;
        const real q = xdiv(c, cK);
        uF = s * c;
        rhoF = rhoK * xpow(q, G.fan_rho);
        pF = pK * xpow(q, G.fan_p);
      }
    }
  }
  return side;
}

// x truncated to FP32 (zero or infinite beyond its range), in integers: a conversion
// takes the FP64 pipe
__device__ __forceinline__ float coarse_float(double x) {
  const unsigned h = (unsigned)__double2hiint(x);
  const int e = (int)exponent_bits((int)h) - 896;
  const unsigned m = (h & 0xfffffu) << 3 | (unsigned)__double2loint(x) >> 29;
  const unsigned b = e <= 0 ? 0u : (e >= 255 ? 0x7f800000u : (unsigned)e << 23 | m);
  return __uint_as_float((h & 0x80000000u) | b);
}

// Which way the FP64 solve of these states will go, judged in FP32: 0 for two
// rarefactions (the standard guess is then the root itself), else one plus the
// waves' kinds and whether the guess is far off (more iterations).  Only the
// grouping of faces into warps uses it.
constexpr int SOLVE_KINDS = 8;
__device__ __forceinline__ int solve_kind(double rL, double uL, double pL, double cL, double rR, double uR, double pR,
                                          double cR, double ppv, const GasC<float>& G) {
  const float rl = coarse_float(rL), pl = coarse_float(pL), cl = coarse_float(cL), rr = coarse_float(rR),
              pr = coarse_float(pR), cr = coarse_float(cR);
  const float du = coarse_float(uR - uL);
  const float p0 = standard_guess_ppv<float>(rl, 0.0f, pl, cl, rr, du, pr, cr, coarse_float(ppv), G);
  float fL, dL, fR, dR;
  wave_curve(p0, rl, pl, cl, G, fL, dL);
  wave_curve(p0, rr, pr, cr, G, fR, dR);
  const float dp = -(fL + fR + du) / (dL + dR);
  const float p = p0 + dp;
  if (p <= pl && p <= pr) return 0;
  const int far = fabsf(dp) > 3e-4f * p0 ? 1 : 0;
  // left shock, both, right shock: neighbours in this order share a branch
  return p <= pr ? 1 + far : (p <= pl ? 6 + far : 3 + far);
}

template <GuardKind GUARD = GUARD_INLINE, typename real>
__device__ __forceinline__ int riemann_sample(real rhoL, real uL, real pL, real rhoR, real uR, real pR,
                                              const GasC<real>& G, double tol, real tol_r, int maxit, bool have_guess,
                                              real guess, real& rhoF, real& uF, real& pF, RiemannInfo& info,
                                              real& pstar) {
  const real cL = xsqrt(xdiv(G.g * pL, rhoL)), cR = xsqrt(xdiv(G.g * pR, rhoR));
  return riemann_sample_c<GUARD>(rhoL, uL, pL, rhoR, uR, pR, cL, cR, linearised_pstar(rhoL, uL, pL, cL, rhoR, uR, pR, cR), G,
                          tol, tol_r, maxit, have_guess, guess, rhoF, uF, pF, info, pstar);
}

}  // namespace amm
