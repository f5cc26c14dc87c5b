// physics.cuh -- per-cell and per-face device arithmetic of the FVCW scheme
// (Guo, Xiong & Shi): the Zhang-Shu limiter and the HLLC flux with Batten's
// wave speeds (Sec. 2.4), and the arithmetic helpers the line code shares.
//
// Line variables are ordered (rho, m_n, [m_t,] E): m_n is the momentum
// normal to the faces of the line, m_t (2-D only) the tangential one.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

namespace ppk {

template <typename real>
__device__ __forceinline__ real sqr(real x) { return x * x; }

// Reciprocal and square root in the arithmetic of the line.  FP32 compiles to
// the approximate instructions (fast math).  FP64: every FP64 instruction
// occupies the SM's FP64 pipe for 16 cycles (2 lanes), so both are written
// with as few as the result needs: the hardware's approximation (about 20
// bits) and one third-order step, y (1 + e + e^2) with e = 1 - x y for 1/x and
// y (1 + e/2 + 3 e^2/8) with e = 1 - x y^2 for x^(-1/2) (the truncated
// binomial series), whose error e^3 is below FP64's: at most one unit in the last
// place from the rounded value.  3 FP64 instructions for 1/x and 6 for a square
// root; the operators take 5.3 and 9 instruction times (measured).
// root() leaves what the approximation flushes (zeros, subnormals) to the
// operator.  rcp() wants a normal, finite argument: zeros, subnormals and
// infinities give NaN where 1/x is infinite or zero, and so does root() of an
// infinity.  Its arguments are densities of limited face states and of cells (a
// cell of any other density is outside G, which a NaN energy says too), sums of
// weights (z_terms keeps them normal), pivots 1 - c b > 0, and differences of
// wave speeds, zero only where no sound speed is left and the flux has no value.
__device__ __forceinline__ float rcp(float x) { return 1.0f / x; }
__device__ __forceinline__ double rcp(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ float root(float x) { return sqrtf(x); }
__device__ __forceinline__ double root(double x) {
  if (__double2hiint(x) < 0x00200000) return sqrt(x);   // zero, subnormal, negative
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double t = x * y;
  const double e = fma(-t, y, 1.0);
  return fma(t * e, fma(0.375, e, 0.5), t);
}

// Tests on FP64 values by integer instructions (an FP64 comparison would take
// a slot of the FP64 pipe).  positive(): x > 0 and not NaN.  less(): a < b
// for arguments that are not NaN.
__device__ __forceinline__ bool positive(float x) { return x > 0.0f; }
__device__ __forceinline__ bool positive(double x) {
  const long long b = __double_as_longlong(x);
  return b > 0 && b <= 0x7ff0000000000000ll;
}
__device__ __forceinline__ bool less(float a, float b) { return a < b; }
__device__ __forceinline__ bool less(double a, double b) {
  // bit patterns ordered as signed magnitudes
  long long p = __double_as_longlong(a), q = __double_as_longlong(b);
  p ^= (p >> 63) & 0x7fffffffffffffffll;
  q ^= (q >> 63) & 0x7fffffffffffffffll;
  return p < q;
}
// a NaN an FP64 operation returned (quiet)
__device__ __forceinline__ bool is_nan(double x) {
  return (__double2hiint(x) & 0x7ff80000) == 0x7ff80000;
}
__device__ __forceinline__ bool is_nan(float x) { return x != x; }
__device__ __forceinline__ bool is_finite(float x) { return isfinite(x); }
__device__ __forceinline__ bool is_finite(double x) {
  return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000;
}

// FP64 to FP32, round to nearest (ties away), by integer instructions: the
// conversion instruction takes a slot of the FP64 pipe.  Values beyond FP32's
// range, infinities and NaN become infinite, below its normal range zero.
__device__ __forceinline__ float to_f32(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x) + 0x10000000ull;
  const unsigned int hi = (unsigned int)(b >> 32), e = hi & 0x7fffffffu, sign = hi & 0x80000000u;
  unsigned int r = ((e - 0x38000000u) << 3) | ((unsigned int)b >> 29);
  r = e < 0x38100000u ? 0u : (e >= 0x47f00000u ? 0x7f800000u : r);
  return __uint_as_float(sign | r);
}
__device__ __forceinline__ float to_f32(float x) { return x; }

// FP32: eps of eq. (weight) is lifted to the FP32 noise floor of the
// indicators.  The FP32 averages the indicators are computed from carry,
// besides their own rounding (up to u max|ubar|, u = 2^-24), the rounding noise the FP32
// fluxes leave in the state step after step: a random walk of about
// cfl u |F| per step, tens to hundreds of u max|ubar| after 10^4 steps.
// The eps, meant to sit above the indicators' zero level and
// below every real one, becomes eps + 2^20 (u max|ubar|)^2 over the stencil:
// above 33 (150 u max|ubar|)^2, the indicators of a flat stencil carrying
// that noise, and still about 4e-9 max|ubar|^2, below the indicators of
// any feature the FP32 form resolves.  With the FP64 value alone, or a
// floor that the accumulated noise overtakes, the weights follow rounding
// noise where the solution is flat to FP32 precision and a grid-scale mode
// that the nonlinear weights otherwise damp grows from it (isentropic
// vortex on 1024^2 to t = 10: density L1 1.9e-4 with the floor at
// 4096 (u max|ubar|)^2, 1.7e-6 at 2^20 (u max|ubar|)^2).
constexpr float FP32_BETA_FLOOR = 1048576.0f * 5.9604645e-08f * 5.9604645e-08f;

// ---------------------------------------------------------------- Euler
template <typename real, int NV>
__device__ __forceinline__ real kin2(const real *U) {  // |m|^2
  real m2 = U[1] * U[1];
  if (NV == 4) m2 += U[2] * U[2];
  return m2;
}

// physical flux from the normal velocity un = m_n / rho and the pressure
template <typename real, int NV>
__device__ __forceinline__ void phys_flux_u(const real *U, real un, real p, real *F) {
  F[0] = U[1];
  F[1] = U[1] * un + p;
  if (NV == 4) F[2] = U[2] * un;
  F[NV - 1] = un * (U[NV - 1] + p);
}

// HLLC flux (Sec. 2.4, eqs. (HLLC), (contact-v), (star-l), (acoustic ws)).
// S_M's denominator uses rho_r on the right-state term, S_R is the max of
// the two estimates and the right star flux uses S_R.  In 2-D the
// tangential velocity is carried by the contact.  smax receives the larger
// |u| + a of the two face states (the speed eq. (CFL-CD) bounds) if want.
// With X_K = rho_K (S_K - u_K) and q = X_K / (S_K - S_M) the star density,
// the star state moves at S_M with pressure p* = p_K + X_K (S_M - u_K), and
// F_K + S_K (U*_K - U_K) is its physical flux (the jump conditions across
// S_K): q S_M (1, S_M, v_K) + p* (0, 1, 0) and (E* + p*) S_M.  Evaluated so
// the star flux takes 9 operations instead of 19.
template <typename real, int NV>
__device__ __forceinline__ void hllc(const real *Ul, const real *Ur, real gamma, real *F,
                                     real &smax, bool want = true) {
  const real rl = Ul[0], rr = Ur[0];
  const real irl = rcp(rl), irr = rcp(rr);
  const real ml = Ul[1], mr = Ur[1];
  const real ul = ml * irl, ur = mr * irr;
  const real vl = NV == 4 ? Ul[2] * irl : real(0), vr = NV == 4 ? Ur[2] * irr : real(0);
  const real El = Ul[NV - 1], Er = Ur[NV - 1];
  const real g1 = gamma - real(1);
  // p = (gamma - 1)(E - |m|^2 / (2 rho)) with |m|^2 / rho = m . u
  real pl = g1 * (El - real(0.5) * (ml * ul + (NV == 4 ? Ul[2] * vl : real(0))));
  real pr = g1 * (Er - real(0.5) * (mr * ur + (NV == 4 ? Ur[2] * vr : real(0))));
  if constexpr (sizeof(real) == 4) {   // FP32 form: never a NaN sound speed from rounding
    pl = fmaxf(pl, 0.0f);
    pr = fmaxf(pr, 0.0f);
  }
  const real al = root(gamma * pl * irl), ar = root(gamma * pr * irr);
  if (want) {
    const real sl = fabs(ul) + al, sr = fabs(ur) + ar;
    smax = fmax(sl, sr);
  }
  const real Hl = (El + pl) * irl, Hr = (Er + pr) * irr;
  const real R = root(rr * irl);
  const real iR = rcp(real(1) + R);
  const real ut = (ul + ur * R) * iR;
  const real vt = (vl + vr * R) * iR;
  const real Ht = (Hl + Hr * R) * iR;
  const real a2 = g1 * (Ht - real(0.5) * (ut * ut + vt * vt));
  const real at = root(a2);
  real SL = ul - al, SR = ur + ar;
  // The smaller and the larger of two speeds, of which either may be NaN:
  // rounding may leave no real Roe sound speed, and a face state of negative
  // pressure (limiter off) has none of its own.
  if (a2 >= real(0)) {
    const real tl = ut - at, tr = ut + at;
    SL = less(tl, SL) || is_nan(SL) ? tl : SL;
    SR = less(SR, tr) || is_nan(SR) ? tr : SR;
  }
  if (positive(SL)) {
    phys_flux_u<real, NV>(Ul, ul, pl, F);
    return;
  }
  const real dl = SL - ul, dr = SR - ur;
  const real Xl = rl * dl, Xr = rr * dr;
  const real SM = (Xr * ur - Xl * ul + pl - pr) * rcp(Xr - Xl);
  const bool left = positive(SM);
  if (!left && !(SR >= real(0))) {
    phys_flux_u<real, NV>(Ur, ur, pr, F);
    return;
  }
  // side K (K = l if S_M > 0, else r)
  const real X = left ? Xl : Xr, uK = left ? ul : ur, pK = left ? pl : pr, d = left ? dl : dr;
  const real SK = left ? SL : SR, EK = left ? El : Er, vK = left ? vl : vr;
  const real ps = X * (SM - uK) + pK;
  const real inv = rcp(SK - SM);
  const real Es = (d * EK - pK * uK + ps * SM) * inv;
  F[0] = X * inv * SM;
  F[1] = F[0] * SM + ps;
  if (NV == 4) F[2] = F[0] * vK;
  F[NV - 1] = (Es + ps) * SM;
}

// The HLLC flux of the same two face states relative to a reference state
// R (FP32, the mixed form): returns F_HLLC(U_l, U_r) - F(R) from the full
// states U_K (wave speeds, signal speed smax) and their differences
// d_K = U_K - R, arranged so that every term that reaches the result is a
// product of a difference with an O(1) factor: its rounding is relative to
// |U - R|, not to |F|.  With u_K - u_R = (dm_K - u_R drho_K) / rho_K and
// p_K - p_R from (gamma-1)(dE - d(m.u)/2), the physical flux difference is
//   d(rho u) = dm, d(rho u^2 + p) = dm u + m_R du + dp,
//   d(rho u v) = dt u + t_R du, d((E+p) u) = (dE + dp) u + (E_R + p_R) du,
// and the star-state jump of eq. (star-l) is proportional to S_M - u_K,
//   S_M - u_l = (p_r - p_l - rho_r (S_R - u_r)(u_r - u_l)) / den,
//   S_M - u_r = (p_r - p_l - rho_l (S_L - u_l)(u_r - u_l)) / den,
// with den the denominator of S_M, p_r - p_l and u_r - u_l again from the
// differences.  R carries (rho, m_n, [m_t,] E) and rp = (u_R, v_R, p_R,
// E_R + p_R).  The branches and wave speeds are those of hllc().
template <int NV>
__device__ __forceinline__ void hllc_delta(const float *Ul, const float *Ur, const float *dl,
                                           const float *dr, const float *R, const float *rp,
                                           float gamma, float *dF, float &smax) {
  const float rl = Ul[0], rr = Ur[0];
  const float ipair = 1.0f / (rl * rr);
  const float irl = rr * ipair, irr = rl * ipair;
  const float ul = Ul[1] * irl, ur = Ur[1] * irr;
  const float vl = NV == 4 ? Ul[2] * irl : 0.0f, vr = NV == 4 ? Ur[2] * irr : 0.0f;
  const float El = Ul[NV - 1], Er = Ur[NV - 1];
  const float g1 = gamma - 1.0f;
  const float uR = rp[0], vR = rp[1], pR = rp[2], HR = rp[3];
  // differences of the primitive quantities from the reference
  const float dul = (dl[1] - uR * dl[0]) * irl, dur = (dr[1] - uR * dr[0]) * irr;
  const float dvl = NV == 4 ? (dl[2] - vR * dl[0]) * irl : 0.0f;
  const float dvr = NV == 4 ? (dr[2] - vR * dr[0]) * irr : 0.0f;
  const float dmul = dl[1] * ul + R[1] * dul + (NV == 4 ? dl[2] * vl + R[2] * dvl : 0.0f);
  const float dmur = dr[1] * ur + R[1] * dur + (NV == 4 ? dr[2] * vr + R[2] * dvr : 0.0f);
  const float dpl = g1 * (dl[NV - 1] - 0.5f * dmul), dpr = g1 * (dr[NV - 1] - 0.5f * dmur);
  const float pl = fmaxf(pR + dpl, 0.0f), pr = fmaxf(pR + dpr, 0.0f);
  const float al = sqrtf(gamma * pl * irl), ar = sqrtf(gamma * pr * irr);
  smax = fmaxf(fabsf(ul) + al, fabsf(ur) + ar);
  const float Hl = (El + pl) * irl, Hr = (Er + pr) * irr;
  const float Rq = sqrtf(rr * irl);
  const float iR = 1.0f / (1.0f + Rq);
  const float ut = (ul + ur * Rq) * iR, vt = (vl + vr * Rq) * iR, Ht = (Hl + Hr * Rq) * iR;
  const float at = sqrtf(g1 * (Ht - 0.5f * (ut * ut + vt * vt)));
  const float SL = fminf(ul - al, ut - at);
  const float SR = fmaxf(ur + ar, ut + at);
  // the physical flux difference of side K
  auto dphys = [&](const float *d, float u, float du, float dp, float *o) {
    o[0] = d[1];
    o[1] = d[1] * u + R[1] * du + dp;
    if (NV == 4) o[2] = d[2] * u + R[2] * du;
    o[NV - 1] = (d[NV - 1] + dp) * u + HR * du;
  };
  if (SL > 0.0f) {
    dphys(dl, ul, dul, dpl, dF);
    return;
  }
  const float Xl = rl * (SL - ul), Xr = rr * (SR - ur);
  const float iden = rcp(Xl - Xr);
  const float dpn = dpr - dpl, dun = dur - dul;
  const float sml = (dpn - Xr * dun) * iden;   // S_M - u_l
  const float SM = ul + sml;
  const bool left = SM > 0.0f;
  if (!left && !(SR >= 0.0f)) {
    dphys(dr, ur, dur, dpr, dF);
    return;
  }
  const float d = left ? sml : (dpn - Xl * dun) * iden;   // S_M - u_K
  const float rK = left ? rl : rr, uK = left ? ul : ur, pK = left ? pl : pr, SK = left ? SL : SR;
  const float vK = left ? vl : vr, EKr = left ? El * irl : Er * irr;
  float dK[NV];   // element-wise selects: no run-time indexing of the arrays
#pragma unroll
  for (int k = 0; k < NV; ++k) dK[k] = left ? dl[k] : dr[k];
  const float iss = 1.0f / (SK - SM);
  const float Jr = rK * d * iss;                 // rho*_K - rho_K
  const float chi = (SK - uK) * iss;
  float J[NV];
  J[0] = Jr;
  J[1] = Jr * SM + rK * d;
  if (NV == 4) J[2] = Jr * vK;
  J[NV - 1] = EKr * Jr + chi * d * (rK * SM + pK / (SK - uK));
  dphys(dK, uK, left ? dul : dur, left ? dpl : dpr, dF);
#pragma unroll
  for (int k = 0; k < NV; ++k) dF[k] += SK * J[k];
}

// Local Lax-Friedrichs flux, the alternative Sec. 3 names for the
// near-vacuum double rarefaction: the mean of the two physical fluxes minus
// alpha/2 times the jump, alpha the larger signal speed |u| + a of the two
// face states (also returned in smax, the speed eq. (CFL-CD) bounds)
template <typename real, int NV>
__device__ __forceinline__ void llf(const real *Ul, const real *Ur, real gamma, real *F,
                                    real &smax) {
  const real irl = rcp(Ul[0]), irr = rcp(Ur[0]);
  const real ul = Ul[1] * irl, ur = Ur[1] * irr;
  const real vl = NV == 4 ? Ul[2] * irl : real(0), vr = NV == 4 ? Ur[2] * irr : real(0);
  const real g1 = gamma - real(1);
  real pl = g1 * (Ul[NV - 1] - real(0.5) * (Ul[1] * ul + (NV == 4 ? Ul[2] * vl : real(0))));
  real pr = g1 * (Ur[NV - 1] - real(0.5) * (Ur[1] * ur + (NV == 4 ? Ur[2] * vr : real(0))));
  if constexpr (sizeof(real) == 4) {
    pl = fmaxf(pl, 0.0f);
    pr = fmaxf(pr, 0.0f);
  }
  smax = fmax(fabs(ul) + root(gamma * pl * irl), fabs(ur) + root(gamma * pr * irr));
  real ha = real(0.5) * smax;
  real Fl[NV], Fr[NV];
  phys_flux_u<real, NV>(Ul, ul, pl, Fl);
  phys_flux_u<real, NV>(Ur, ur, pr, Fr);
#pragma unroll
  for (int k = 0; k < NV; ++k) F[k] = real(0.5) * (Fl[k] + Fr[k]) - ha * (Ur[k] - Ul[k]);
}

template <typename real>
__device__ __forceinline__ constexpr real unit_roundoff() {
  return sizeof(real) == 8 ? real(1.1102230246251565e-16) : real(5.9604645e-08);
}

// g(W) = rho E - |m|^2 / 2 - eps rho^2: for rho > 0, e(W) >= eps iff g >= 0
template <typename real, int NV>
__device__ __forceinline__ real energy_form(const real *w, real eps) {
  return w[0] * w[NV - 1] - real(0.5) * kin2<real, NV>(w) - eps * w[0] * w[0];
}

// round-off allowance of g along the segment from Ubar to W: forming
// (1-t) Ubar + t W costs a few ulps of |Ubar| + |W| per component, which
// moves the bilinear form g by at most a small multiple of
// u [(|E|+|E_w|)(|rho|+|rho_w|) + (|m|+|m_w|)^2]; the limiter asks g >= eta
// so that the rounded limited states stay inside G
template <typename real, int NV>
__device__ __forceinline__ real energy_allowance(const real *ub, const real *w, real uu) {
  real sm = real(0);
#pragma unroll
  for (int k = 1; k < NV - 1; ++k) sm += sqr(fabs(ub[k]) + fabs(w[k]));
  return real(16) * uu *
         ((fabs(ub[NV - 1]) + fabs(w[NV - 1])) * (fabs(ub[0]) + fabs(w[0])) + sm);
}

// root t in (0, 1] of g((1 - t) Ubar + t W) = eta: the quadratic
// A t^2 + B t + (C - eta) = 0 with C - eta > 0; the cancellation-free form
// 2C' / (-B + sqrt(B^2 - 4AC')) picks the root in (0, 1)
template <typename real, int NV>
__device__ __forceinline__ real energy_root(const real *ub, const real *w, real eps, real eta) {
  real dr = w[0] - ub[0], dE = w[NV - 1] - ub[NV - 1];
  real dm1 = w[1] - ub[1], dm2 = NV == 4 ? w[2] - ub[2] : real(0);
  real m1 = ub[1], m2 = NV == 4 ? ub[2] : real(0);
  real A = dE * dr - real(0.5) * (dm1 * dm1 + dm2 * dm2) - eps * dr * dr;
  real B = ub[NV - 1] * dr + dE * ub[0] - (m1 * dm1 + m2 * dm2) - real(2) * eps * ub[0] * dr;
  real C = ub[NV - 1] * ub[0] - real(0.5) * (m1 * m1 + m2 * m2) - eps * ub[0] * ub[0] - eta;
  if (!(C > real(0))) return real(0);
  real D = fmax(B * B - real(4) * A * C, real(0));
  real den = -B + sqrt(D);
  real t = den > real(0) ? real(2) * C / den : real(0);
  if (!(t >= real(0))) t = real(0);
  return fmin(t, real(1));
}

// Zhang-Shu limiter of one cell (Sec. 2.4, steps 1-4).  um = U^-_{i+1/2},
// up = U^+_{i-1/2} are limited in place.  Returns bit 0 if theta_1 < 1 and
// bit 1 if theta_2 < 1.  theta = 1 leaves the values untouched.  Both
// thresholds carry the round-off allowance that keeps the rounded limited
// states in G.
// uu is the unit round-off of the arithmetic in which the limited faces are
// stored and used (FP64 for the plain form, FP32 for the mixed form)
template <typename real, int NV>
__device__ __forceinline__ int limit_cell(const real *ub, real *um, real *up, real wgl, real eps,
                                          real uu) {
  int flags = 0;
  real inv12 = real(1) / (real(1) - real(2) * wgl);
  real rho_star = (ub[0] - wgl * up[0] - wgl * um[0]) * inv12;
  real rho_min = fmin(fmin(um[0], up[0]), rho_star);
  real eps_r = eps + real(8) * uu * (fabs(ub[0]) + fabs(rho_min));
  if (rho_min < eps_r) {
    real th1 = fmin(fmax((ub[0] - eps_r) / (ub[0] - rho_min), real(0)), real(1));
    um[0] = th1 * (um[0] - ub[0]) + ub[0];
    up[0] = th1 * (up[0] - ub[0]) + ub[0];
    flags |= 1;
  }
  real th2 = real(1);
  real w3[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) w3[k] = (ub[k] - wgl * up[k] - wgl * um[k]) * inv12;
  {
    real eta = energy_allowance<real, NV>(ub, um, uu);
    if (energy_form<real, NV>(um, eps) < eta) th2 = fmin(th2, energy_root<real, NV>(ub, um, eps, eta));
  }
  {
    real eta = energy_allowance<real, NV>(ub, up, uu);
    if (energy_form<real, NV>(up, eps) < eta) th2 = fmin(th2, energy_root<real, NV>(ub, up, eps, eta));
  }
  {
    real eta = energy_allowance<real, NV>(ub, w3, uu);
    if (energy_form<real, NV>(w3, eps) < eta) th2 = fmin(th2, energy_root<real, NV>(ub, w3, eps, eta));
  }
  if (th2 < real(1)) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      um[k] = th2 * (um[k] - ub[k]) + ub[k];
      up[k] = th2 * (up[k] - ub[k]) + ub[k];
    }
    flags |= 2;
  }
  return flags;
}

// A cell the limiter cannot touch, from the deviations of its two face values
// from the average alone (FP32, both forms): with dk = max |face - average|
// of component k, all three quadrature points of the limiter lie in the box
// ub +- d (the interior one is ub - wgl/(1 - 2 wgl) (dm + dp), inside it for
// wgl <= 1/4), so rho >= r = ub_0 - d_0 and g >= r (E - d_E) - |m|^2/2 at the
// box's worst corner.  The thresholds are twice the FP32 allowances of
// limiter_cell at the box's largest magnitudes, which leaves the evaluation's
// own rounding (about a tenth of them) ample room.  NaN fails every comparison,
// and a threshold within reach of the products' underflow fails.  Smooth cells
// pass, and skip the pretest below (a third of its instructions).
template <int NV>
__device__ __forceinline__ bool limit_box_free(const float *ub, const float *dm, const float *dp,
                                               float wgl, float eps) {
  const float uf = 5.9604645e-08f;
  const float d0 = fmaxf(fabsf(dm[0]), fabsf(dp[0]));
  const float dE = fmaxf(fabsf(dm[NV - 1]), fabsf(dp[NV - 1]));
  float S = 0.0f;
#pragma unroll
  for (int k = 1; k < NV - 1; ++k) {
    const float m = fabsf(ub[k]) + fmaxf(fabsf(dm[k]), fabsf(dp[k]));
    S = fmaf(m, m, S);
  }
  const float r = ub[0] - d0, R = ub[0] + d0, E = ub[NV - 1] + dE;
  const float g = fmaf(r, ub[NV - 1] - dE, -0.5f * S);
  const float need = fmaf(eps * R, R, 128.0f * uf * fmaf(E, R, S));
  return r > fmaf(32.0f * uf, R, 2.0f * eps) && g > need && need < 3.0e38f && need > 1.0e-36f &&
         wgl <= 0.25f;
}

// Mixed form: an FP32 test of the limiter's conditions with doubled
// allowances; only cells that may need limiting compute the scaling factors
// theta_1, theta_2 in FP64 (with the FP32 allowance, since the limited faces
// are stored in FP32).  Returns the limiter flags.
// FP32 pretest of a cell: true when the exact (FP64) limiter might change
// its face values; the caller then runs the exact limiter on it.  Used by
// both forms (the FP64 form passes its values rounded to FP32).
template <int NV>
__device__ __forceinline__ bool limit_need_mixed(const float *ub, const float *um, const float *up,
                                                 float wgl, float inv12, float eps) {
  const float uf = 5.9604645e-08f;
  float w3[NV];   // the interior quadrature point implied by the cell average
#pragma unroll
  for (int k = 0; k < NV; ++k) w3[k] = (ub[k] - wgl * up[k] - wgl * um[k]) * inv12;
  const float rho_min = fminf(fminf(um[0], up[0]), w3[0]);
  bool need = rho_min < 2.0f * (eps + 8.0f * uf * (fabsf(ub[0]) + fabsf(rho_min)));
  // one allowance for the three points, with each magnitude replaced by the
  // largest over them: it bounds the three allowances, so the test (doubled
  // for FP32) flags every cell the exact test would (a superset; the FP64
  // pass decides)
  const float rmx = fmaxf(fmaxf(fabsf(um[0]), fabsf(up[0])), fabsf(w3[0]));
  const float emx = fmaxf(fmaxf(fabsf(um[NV - 1]), fabsf(up[NV - 1])), fabsf(w3[NV - 1]));
  float sm = 0.0f;
#pragma unroll
  for (int k = 1; k < NV - 1; ++k) {
    const float mk = fmaxf(fmaxf(fabsf(um[k]), fabsf(up[k])), fabsf(w3[k]));
    sm += sqr(fabsf(ub[k]) + mk);
  }
  const float eta2 =
      32.0f * uf * ((fabsf(ub[NV - 1]) + emx) * (fabsf(ub[0]) + rmx) + sm);
  need = need | (energy_form<float, NV>(um, eps) < eta2) |
         (energy_form<float, NV>(up, eps) < eta2) | (energy_form<float, NV>(w3, eps) < eta2);
  // magnitudes beyond FP32's range (or NaN) make the allowance non-finite, and
  // below 1e-36 the products' underflow (1e-38) is no longer small against it:
  // such a cell always goes to the exact test
  return need | !(eta2 <= 3.0e38f && eta2 >= 1.0e-36f);
}

// The FP64 limiter of a flagged cell of the mixed form, on FP32 face values
// limited in place (with the FP32 round-off allowance: the limited faces are
// stored in FP32).  Returns the limiter flags.
template <int NV>
__device__ __forceinline__ int limit_cell_mixed_fp64(const float *ub, float *um, float *up,
                                                     float wgl, float eps) {
  const double uf = 5.9604645e-08;
  double b[NV], m[NV], p[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    b[k] = ub[k];
    m[k] = um[k];
    p[k] = up[k];
  }
  const int f = limit_cell<double, NV>(b, m, p, (double)wgl, (double)eps, uf);
  if (f) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      um[k] = (float)m[k];
      up[k] = (float)p[k];
    }
  }
  return f;
}

}  // namespace ppk
