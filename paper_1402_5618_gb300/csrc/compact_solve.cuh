// compact_solve.cuh -- the compact-WENO reconstruction of one line (Sec. 2.2)
// in partitioned form: weights, rows, chunk elimination, and the composition
// of runs of rows into the solution at their ends.
//
// Unknowns.  Both systems of a variable (minus: U^- at the right face of
// every cell, plus: U^+ at the left face) are solved for y_i = U_i - ubar_i,
// the deviation of the face value from the cell average.  With ubar_{i-1},
// ubar_i, ubar_{i+1} subtracted the right-hand side of eq. (CWENO-FV) is a
// combination of the two neighbouring differences alone,
//   s_i = dm (2 + w0 - 2 w2)/6 + dp (1 - w0 + 2 w2)/6,
// dm = ubar_i - ubar_{i-1}, dp = ubar_{i+1} - ubar_i, so every operation
// between the cell differences and the final ubar + y rounds relative to the
// differences.  The plus system is the mirror image.
//
// Rows.  A row may carry any factor, so the weights of eq. (weight) are never
// normalised: with S_k proportional to 1 + (tau/(beta_k + eps))^2 and
// alpha = (2 S0, 5 S1, 3 S2), the row times 3/2 sum(alpha) is
//   a = 2 S0 + 5/2 S1, b = S0 + 5 S1 + 3 S2, c = 3/2 S2,
//   s = dm (3/2 S0 + 5/2 S1) + dp (5/4 S1 + 9/4 S2).
//
// Walk order.  "Previous" and "next" follow the elimination: left to right
// for the minus system, right to left for the plus system; in walk order
// both have the same rows.
//
// A run of consecutive rows is reduced to its two end unknowns as functions
// of the unknowns just outside it (X_in before, X_out after):
//   first = A - B X_in - G X_out,   last = D - F X_in - C X_out.
// The order of elimination is free: b_i 2^i >= a_i 2^(i-1) + c_i 2^(i+1) in
// every row (b - a/2 - 2c = 15/4 S1 >= 0), so the matrix scaled by 2^i is
// diagonally dominant and every pivot and every 1 - C B of a composition stays
// positive, as in the serial elimination.
#pragma once

#include <cuda_runtime.h>

#include "physics.cuh"

namespace ppk {

// halves of a cluster barrier; the relaxed arrival publishes no data
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release;\n" ::: "memory");
}
__device__ __forceinline__ void cluster_arrive_relaxed() {
  asm volatile("barrier.cluster.arrive.relaxed;\n" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire;\n" ::: "memory");
}

// ---------------------------------------------------------------- pairs
// .x belongs to the minus system, .y to the plus system.  FP32 pairs use the
// paired instructions (one issue slot for two operations, each component
// rounded as the scalar fused multiply-add); FP64 pairs are two scalars.
template <typename real>
struct Pair;
template <>
struct Pair<float> {
  using t = float2;
};
template <>
struct Pair<double> {
  using t = double2;
};
__device__ __forceinline__ float2 p_set(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ double2 p_set(double a, double b) { return make_double2(a, b); }
__device__ __forceinline__ float2 p_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 p_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 p_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ double2 p_mul(double2 a, double2 b) { return make_double2(a.x * b.x, a.y * b.y); }
__device__ __forceinline__ double2 p_fma(double2 a, double2 b, double2 c) {
  return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y));
}
__device__ __forceinline__ double2 p_neg(double2 a) { return make_double2(-a.x, -a.y); }
__device__ __forceinline__ float2 p_rcp(float2 a) { return make_float2(rcp(a.x), rcp(a.y)); }
__device__ __forceinline__ double2 p_rcp(double2 a) { return make_double2(rcp(a.x), rcp(a.y)); }

// scalars, for code written on either
template <typename real>
__device__ __forceinline__ real p_mul(real a, real b) { return a * b; }
template <typename real>
__device__ __forceinline__ real p_fma(real a, real b, real c) { return fma(a, b, c); }
template <typename real>
__device__ __forceinline__ real p_neg(real a) { return -a; }
template <typename real>
__device__ __forceinline__ real p_rcp(real a) { return rcp(a); }
template <typename real>
__device__ __forceinline__ real p_sel(bool c, bool, real a, real b) { return c ? a : b; }
template <typename real>
__device__ __forceinline__ real p_xor(real v, int d) { return __shfl_xor_sync(0xffffffffu, v, d); }
__device__ __forceinline__ float2 p_sel(bool x, bool y, float2 a, float2 b) {
  return make_float2(x ? a.x : b.x, y ? a.y : b.y);
}
__device__ __forceinline__ double2 p_sel(bool x, bool y, double2 a, double2 b) {
  return make_double2(x ? a.x : b.x, y ? a.y : b.y);
}
__device__ __forceinline__ float2 p_xor(float2 v, int d) {
  return make_float2(__shfl_xor_sync(0xffffffffu, v.x, d), __shfl_xor_sync(0xffffffffu, v.y, d));
}
__device__ __forceinline__ double2 p_xor(double2 v, int d) {
  return make_double2(__shfl_xor_sync(0xffffffffu, v.x, d), __shfl_xor_sync(0xffffffffu, v.y, d));
}

// ---------------------------------------------------------------- weights
// power of two near 1/m (exact scaling): 2^-(exponent of m)
__device__ __forceinline__ double pow2_inv(double m) {
  long long e = (__double_as_longlong(m) >> 52) & 0x7ff;
  return (e > 0 && e < 2046) ? __longlong_as_double((2046 - e) << 52) : 1.0;
}

// S_k of cell j of a window, from the differences D[i] = u[i+1] - u[i] and
// the second differences dd[i] = D[i+1] - D[i]: with G = 4/3 dd^2 (+ eps),
//   beta_0 = G[j] + D[j+1] (D[j+1] + dd[j]),  beta_1 = G[j+1] + D[j+1] D[j+2],
//   beta_2 = G[j+2] + D[j+2] (D[j+2] - dd[j+2])
// (eq. (weight)'s indicators with the squares of their linear parts
// expanded; each is at least 13/16 of its G, so nothing cancels).
//
// FP64: no division, S_k = (d0 d1 d2)^2 + (tau d_l d_m)^2 with d_k = beta_k +
// eps, a common factor (d0 d1 d2)^2 of the row (11 FP64 operations; one
// reciprocal of the product and the ratios would take 14).  d outside
// 2^-80 .. 2^80, where the sixth powers would leave the range, is scaled by a
// power of two first; the test reads exponents with integer instructions
// because every FP64 instruction costs 16 cycles of the SM's FP64 pipe.
__device__ __forceinline__ void z_terms(double d0, double d1, double d2, double &S0, double &S1,
                                        double &S2) {
  double tau = fabs(d2 - d0);
  const int h0 = __double2hiint(d0), h1 = __double2hiint(d1), h2 = __double2hiint(d2);
  const int hx = max(max(h0, h1), h2), hn = min(min(h0, h1), h2);
  if (hx > ((1023 + 80) << 20) || hn < ((1023 - 80) << 20)) {
    const double sc = pow2_inv(hx == h0 ? d0 : (hx == h1 ? d1 : d2));
    d0 *= sc; d1 *= sc; d2 *= sc; tau *= sc;
  }
  const double p01 = d0 * d1, p02 = d0 * d2, p12 = d1 * d2;
  const double P = p01 * d2, P2 = P * P;
  const double t0 = tau * p12, t1 = tau * p02, t2 = tau * p01;
  S0 = fma(t0, t0, P2);
  S1 = fma(t1, t1, P2);
  S2 = fma(t2, t2, P2);
}

// FP32: S_k = 1 + (tau/d_k)^2 by reciprocals (cheap here).  d_k >= 2^-28
// umax^2 (the rounding floor of the indicators) and tau <= 33.4 umax^2 (cells of
// alternating sign: beta <= 13/12 4^2 + 8^2/4), so S_k stays below 2^67.
__device__ __forceinline__ void z_terms(float d0, float d1, float d2, float &S0, float &S1, float &S2) {
  const float tau = d2 - d0;
  const float t0 = tau * rcp(d0), t1 = tau * rcp(d1), t2 = tau * rcp(d2);
  S0 = fmaf(t0, t0, 1.0f);
  S1 = fmaf(t1, t1, 1.0f);
  S2 = fmaf(t2, t2, 1.0f);
}

// differences and S_k of the M cells of a chunk; win holds the cells with a
// two-cell halo.  FP32 lifts eps to the noise floor of the indicators
// (FP32_BETA_FLOOR, physics.cuh) over each five-cell stencil.
template <typename real, int M>
__device__ __forceinline__ void chunk_weights(const real (&win)[M + 4], real eps, real (&D)[M + 3],
                                              real (&S0)[M], real (&S1)[M], real (&S2)[M]) {
  constexpr bool F32 = sizeof(real) == 4;
#pragma unroll
  for (int i = 0; i < M + 3; ++i) D[i] = win[i + 1] - win[i];
  real ddl = D[1] - D[0], ddc = D[2] - D[1];
  const real k43 = real(4.0 / 3.0), e = F32 ? real(0) : eps;
  real Gl = fma(k43 * ddl, ddl, e), Gc = fma(k43 * ddc, ddc, e);
#pragma unroll
  for (int j = 0; j < M; ++j) {
    const real ddr = D[j + 3] - D[j + 2];
    const real Gr = fma(k43 * ddr, ddr, e);
    const real dm = D[j + 1], dp = D[j + 2];
    real d0 = fma(dm, dm + ddl, Gl), d1 = fma(dm, dp, Gc), d2 = fma(dp, dp - ddr, Gr);
    if constexpr (F32) {
      const float um = fmaxf(fmaxf(fmaxf(fabsf(win[j]), fabsf(win[j + 1])),
                                   fmaxf(fabsf(win[j + 2]), fabsf(win[j + 3]))),
                             fabsf(win[j + 4]));
      const float ej = fmaf(FP32_BETA_FLOOR * um, um, eps);
      d0 += ej; d1 += ej; d2 += ej;
    }
    z_terms(d0, d1, d2, S0[j], S1[j], S2[j]);
    ddl = ddc; ddc = ddr;
    Gl = Gc; Gc = Gr;
  }
}

// ---------------------------------------------------------------- runs
template <typename real>
struct Run {
  real A, B, G, D, F, C;
};

// where two neighbouring runs meet: the last unknown of the first run and the
// first unknown of the second, from the unknowns outside both,
//   l = u - p X_in + q X_out,  f = v + r X_in - s X_out
template <typename real>
struct Cut {
  real u, p, q, v, r, s;
};

// X followed (in walk order) by Y; k: their meeting point
template <typename real>
__device__ __forceinline__ Run<real> run_join(const Run<real> &X, const Run<real> &Y, Cut<real> &k) {
  const real i = rcp(fma(-X.C, Y.B, real(1)));
  k.u = fma(-X.C, Y.A, X.D) * i;
  k.p = X.F * i;
  k.s = Y.G * i;
  k.q = X.C * k.s;
  k.v = fma(-Y.B, X.D, Y.A) * i;
  k.r = Y.B * k.p;
  Run<real> o;
  o.A = fma(-X.G, k.v, X.A);
  o.B = fma(X.G, k.r, X.B);
  o.G = -X.G * k.s;
  o.D = fma(-Y.F, k.u, Y.D);
  o.F = -Y.F * k.p;
  o.C = fma(Y.F, k.q, Y.C);
  return o;
}

// the empty run: first = X_out, last = X_in
template <typename real>
__device__ __forceinline__ Run<real> run_empty() {
  Run<real> o;
  o.A = o.B = o.D = o.C = real(0);
  o.G = o.F = real(-1);
  return o;
}

template <typename real>
__device__ __forceinline__ Run<real> run_shfl(const Run<real> &a, int src, int width) {
  Run<real> o;
  o.A = __shfl_sync(0xffffffffu, a.A, src, width);
  o.B = __shfl_sync(0xffffffffu, a.B, src, width);
  o.G = __shfl_sync(0xffffffffu, a.G, src, width);
  o.D = __shfl_sync(0xffffffffu, a.D, src, width);
  o.F = __shfl_sync(0xffffffffu, a.F, src, width);
  o.C = __shfl_sync(0xffffffffu, a.C, src, width);
  return o;
}
template <typename real>
__device__ __forceinline__ Run<real> run_shfl_xor(const Run<real> &a, int m, int width) {
  Run<real> o;
  o.A = __shfl_xor_sync(0xffffffffu, a.A, m, width);
  o.B = __shfl_xor_sync(0xffffffffu, a.B, m, width);
  o.G = __shfl_xor_sync(0xffffffffu, a.G, m, width);
  o.D = __shfl_xor_sync(0xffffffffu, a.D, m, width);
  o.F = __shfl_xor_sync(0xffffffffu, a.F, m, width);
  o.C = __shfl_xor_sync(0xffffffffu, a.C, m, width);
  return o;
}

// ---------------------------------------------------------------- chunks
// Elimination of a chunk's M rows in both systems: x_j = d_j - f_j X_in - c_j
// x_{j+1} for the walk row j.  The minus system's row j is the chunk's cell
// j, the plus system's row j is cell M-1-j.  d and f go to the cells' slots
// of four shared-memory planes (dm, fm minus; dp, fp plus), c of rows
// 0 .. M-2 stays in registers for the back substitution.  Returned per
// system: first = A - B X_in - G last (the chunk's own last unknown), and
// last = D - F X_in - C X_out.
//
// EDGE: the chunk's warp holds cells at or beyond a line end.  On bounded
// lines the first and the last cell take the explicit WENO5-Z value of the
// closure.  Rows beyond the end do not exist: the minus system's state stops
// at the last cell, the plus system's starts there (a chunk without cells
// is never read).
struct EdgeInfo {
  int i0, n;        // line index of the chunk's first cell, line length
  bool periodic;
};

template <typename real, int M, bool EDGE>
__device__ __forceinline__ void chunk_eliminate(const real (&D)[M + 3], const real (&S0)[M],
                                                const real (&S1)[M], const real (&S2)[M],
                                                const EdgeInfo e, real *dm, real *fm, real *dp,
                                                real *fp, typename Pair<real>::t (&cs)[M - 1],
                                                Run<real> &rm, Run<real> &rp) {
  using P = typename Pair<real>::t;
  const auto set1 = [](double v) { return p_set(real(v), real(v)); };
  // the empty chunk: last = X_in, first = last
  P c = set1(0), d = set1(0), f = set1(-1), A = set1(0), B = set1(0), G = set1(-1);
#pragma unroll
  for (int j = 0; j < M; ++j) {
    constexpr int L = M - 1;
    const int jm = j, jp = L - j;
    const P s0 = p_set(S0[jm], S2[jp]), s1 = p_set(S1[jm], S1[jp]), s2 = p_set(S2[jm], S0[jp]);
    // previous / next differences in walk order (the plus system's carry a
    // minus sign, put back in s)
    const P em = p_set(D[jm + 1], -D[jp + 2]), ep = p_set(D[jm + 2], -D[jp + 1]);
    const P t2 = p_mul(set1(2.5), s1), t4 = p_mul(set1(1.25), s1);
    P a = p_fma(set1(2.0), s0, t2);
    P b = p_fma(set1(3.0), s2, p_fma(set1(2.0), t2, s0));
    P cc = p_mul(set1(1.5), s2);
    P s = p_fma(ep, p_fma(set1(2.25), s2, t4), p_mul(em, p_fma(set1(1.5), s0, t2)));
    if constexpr (EDGE) {
      const int im = e.i0 + jm, ip = e.i0 + jp;
      // closure: alpha = (0.1 S0, 0.6 S1, 0.3 S2), the three explicit
      // candidates minus ubar in differences, times 6
      if (!e.periodic && (im == 0 || im == e.n - 1)) {
        const real a0 = real(0.1) * S0[jm], a1 = real(0.6) * S1[jm], a2 = real(0.3) * S2[jm];
        const real D0 = D[jm], D1 = D[jm + 1], D2 = D[jm + 2], D3 = D[jm + 3];
        a.x = real(0); cc.x = real(0);
        b.x = real(6) * (a0 + a1 + a2);
        s.x = a0 * (real(5) * D1 - real(2) * D0) + a1 * (D1 + real(2) * D2) + a2 * (real(4) * D2 - D3);
      }
      if (!e.periodic && (ip == 0 || ip == e.n - 1)) {
        const real a0 = real(0.1) * S2[jp], a1 = real(0.6) * S1[jp], a2 = real(0.3) * S0[jp];
        const real D0 = D[jp], D1 = D[jp + 1], D2 = D[jp + 2], D3 = D[jp + 3];
        a.y = real(0); cc.y = real(0);
        b.y = real(6) * (a0 + a1 + a2);
        s.y = -(a0 * (real(5) * D2 - real(2) * D3) + a1 * (D2 + real(2) * D1) + a2 * (real(4) * D1 - D0));
      }
    }
    if constexpr (EDGE) {
      // one side's row: fold the previous row into the first unknown's
      // expression, then eliminate
      const auto row = [](real a, real b, real cc, real s, bool start, real &c, real &d, real &f,
                          real &A, real &B, real &G) {
        if (!start) {
          A = fma(-G, d, A);
          B = fma(-G, f, B);
          G = -(G * c);
        }
        const real inv = rcp(fma(-a, c, b));
        d = fma(-a, d, s) * inv;
        f = -(a * f) * inv;
        c = cc * inv;
      };
      const int im = e.i0 + jm, ip = e.i0 + jp;
      if (im < e.n) row(a.x, b.x, cc.x, s.x, j == 0, c.x, d.x, f.x, A.x, B.x, G.x);
      if (ip < e.n) row(a.y, b.y, cc.y, s.y, j == 0 || ip == e.n - 1, c.y, d.y, f.y, A.y, B.y, G.y);
    } else if (j == 0) {
      const P inv = p_rcp(b);
      d = p_mul(s, inv);
      f = p_mul(a, inv);
      c = p_mul(cc, inv);
      A = d; B = f; G = c;
    } else {
      const P na = p_neg(a);
      const P inv = p_rcp(p_fma(na, c, b));
      d = p_mul(p_fma(na, d, s), inv);
      f = p_mul(p_mul(na, f), inv);
      c = p_mul(cc, inv);
      if (j < L) {
        const P ng = p_neg(G);
        A = p_fma(ng, d, A);
        B = p_fma(ng, f, B);
        G = p_mul(ng, c);
      }
    }
    if (j < L) {
      dm[jm] = d.x; fm[jm] = f.x;
      dp[jp] = d.y; fp[jp] = f.y;
      cs[j] = c;
    }
  }
  rm.A = A.x; rm.B = B.x; rm.G = G.x; rm.D = d.x; rm.F = f.x; rm.C = c.x;
  rp.A = A.y; rp.B = B.y; rp.G = G.y; rp.D = d.y; rp.F = f.y; rp.C = c.y;
}

// Back substitution of a chunk from X_in and its own last unknown; the face
// values ubar + y overwrite d in dm, dp.  len (RAGGED): cells of the chunk.
template <typename real, int M, bool RAGGED>
__device__ __forceinline__ void chunk_back(const real *u, real *dm, const real *fm, real *dp,
                                           const real *fp,
                                           const typename Pair<real>::t (&cs)[M - 1],
                                           typename Pair<real>::t xin, typename Pair<real>::t x,
                                           int len) {
  using P = typename Pair<real>::t;
  const P nin = p_neg(xin);
  dm[M - 1] = u[M - 1] + x.x;
  dp[0] = u[0] + x.y;
#pragma unroll
  for (int j = M - 2; j >= 0; --j) {
    const int jm = j, jp = M - 1 - j;
    const P g = p_fma(p_set(fm[jm], fp[jp]), nin, p_set(dm[jm], dp[jp]));
    const P y = p_fma(p_neg(cs[j]), x, g);
    // the minus system of a ragged chunk starts at its last cell
    x = RAGGED ? p_set(jm + 1 < len ? y.x : x.x, y.y) : y;
    dm[jm] = u[jm] + x.x;
    dp[jp] = u[jp] + x.y;
  }
}

// The same elimination of one system alone (SIDE 0 minus, 1 plus), d and f to
// its two planes: a warp per side where a launch waits for its FP64
// instructions one after another (short chunks).
template <int SIDE, int M>
__device__ __forceinline__ void side_eliminate(const double (&D)[M + 3], const double (&S0)[M],
                                               const double (&S1)[M], const double (&S2)[M],
                                               const EdgeInfo e, double *dd, double *ff,
                                               double (&cs)[M - 1], Run<double> &r) {
  double c = 0.0, d = 0.0, f = -1.0, A = 0.0, B = 0.0, G = -1.0;
#pragma unroll
  for (int j = 0; j < M; ++j) {
    constexpr int L = M - 1;
    const int jc = SIDE ? L - j : j, i = e.i0 + jc;
    const double s0 = SIDE ? S2[jc] : S0[jc], s1 = S1[jc], s2 = SIDE ? S0[jc] : S2[jc];
    // differences in walk order: before the previous cell, previous, next, after
    const double e0 = SIDE ? -D[jc + 3] : D[jc], em = SIDE ? -D[jc + 2] : D[jc + 1];
    const double ep = SIDE ? -D[jc + 1] : D[jc + 2], e3 = SIDE ? -D[jc] : D[jc + 3];
    const double t2 = 2.5 * s1, t4 = 1.25 * s1;
    double a = fma(2.0, s0, t2), b = fma(3.0, s2, fma(2.0, t2, s0)), cc = 1.5 * s2;
    double s = fma(ep, fma(2.25, s2, t4), em * fma(1.5, s0, t2));
    if (!e.periodic && (i == 0 || i == e.n - 1)) {   // closure
      const double a0 = 0.1 * s0, a1 = 0.6 * s1, a2 = 0.3 * s2;
      a = cc = 0.0;
      b = 6.0 * (a0 + a1 + a2);
      s = a0 * (5.0 * em - 2.0 * e0) + a1 * (em + 2.0 * ep) + a2 * (4.0 * ep - e3);
    }
    if (i < e.n) {
      if (!(j == 0 || (SIDE && i == e.n - 1))) {
        A = fma(-G, d, A);
        B = fma(-G, f, B);
        G = -(G * c);
      }
      const double inv = rcp(fma(-a, c, b));
      d = fma(-a, d, s) * inv;
      f = -(a * f) * inv;
      c = cc * inv;
    }
    if (j < L) {
      dd[jc] = d;
      ff[jc] = f;
      cs[j] = c;
    }
  }
  r.A = A; r.B = B; r.G = G; r.D = d; r.F = f; r.C = c;
}

template <int SIDE, int M>
__device__ __forceinline__ void side_back(const double *u, double *dd, const double *ff,
                                          const double (&cs)[M - 1], double xin, double x, int len) {
  dd[SIDE ? 0 : M - 1] = u[SIDE ? 0 : M - 1] + x;
#pragma unroll
  for (int j = M - 2; j >= 0; --j) {
    const int jc = SIDE ? M - 1 - j : j;
    const double y = fma(-cs[j], x, fma(-ff[jc], xin, dd[jc]));
    x = SIDE || jc + 1 < len ? y : x;   // the minus system of a ragged chunk starts at its last cell
    dd[jc] = u[jc] + x;
  }
}

// ---------------------------------------------------------------- trees
// Runs of the lanes of a warp joined by a butterfly: 5 levels of a few dozen
// instructions on every warp and no barrier.  The way of the FP32 form, and of
// FP64 with short chunks, where a line has its SMs to itself and latency is
// the cost; otherwise the FP64 pipe is, and one warp walks the chunks of the
// segment with a fifth of the instructions.  At each level a lane sees its
// own run and its partner's from the end that faces the other: inner (facing)
// and outer ends as end = a - b X_near - g X_far.  With i = 1/(1 - b b'), the
// partner's inner unknown is u + r X_o - s X_o' (X_o, X_o': outside the own
// and the partner's outer end), kept for the way down.  A lane extends its own
// outer end only and receives the partner's: as many shuffles as reading the
// partner's inputs, six operations fewer (a 200-cell FP64 line, four CTAs of
// two-row chunks, 0.0258 ms instead of 0.0288).
template <typename P>
struct Ends {
  P a, b, g;
};
template <typename P>
struct Step {
  P u, r, s;
};

// F, L: the run's first and last unknown in walk order (L.b belongs to X_out,
// L.g to X_in); rx, ry: this lane is the later of the two in walk order (for
// the minus and the plus component)
template <typename P>
__device__ __forceinline__ void tree_up(int d, bool rx, bool ry, P one, Ends<P> &F, Ends<P> &L,
                                        Step<P> &st) {
  Ends<P> in, out, in2, o, o2;
  in.a = p_sel(rx, ry, F.a, L.a); in.b = p_sel(rx, ry, F.b, L.b); in.g = p_sel(rx, ry, F.g, L.g);
  out.a = p_sel(rx, ry, L.a, F.a); out.b = p_sel(rx, ry, L.b, F.b); out.g = p_sel(rx, ry, L.g, F.g);
  in2.a = p_xor(in.a, d); in2.b = p_xor(in.b, d); in2.g = p_xor(in.g, d);
  const P i = p_rcp(p_fma(p_neg(in.b), in2.b, one));
  st.u = p_mul(p_fma(p_neg(in2.b), in.a, in2.a), i);
  st.r = p_mul(in2.b, p_mul(in.g, i));
  st.s = p_mul(in2.g, i);
  const P nf = p_neg(out.g);
  o.a = p_fma(nf, st.u, out.a);
  o.b = p_fma(out.g, st.r, out.b);
  o.g = p_mul(nf, st.s);
  o2.a = p_xor(o.a, d); o2.b = p_xor(o.b, d); o2.g = p_xor(o.g, d);
  F.a = p_sel(rx, ry, o2.a, o.a); F.b = p_sel(rx, ry, o2.b, o.b); F.g = p_sel(rx, ry, o2.g, o.g);
  L.a = p_sel(rx, ry, o.a, o2.a); L.b = p_sel(rx, ry, o.b, o2.b); L.g = p_sel(rx, ry, o.g, o2.g);
}
template <typename P>
__device__ __forceinline__ void tree_down(bool rx, bool ry, const Step<P> &st, P &xl, P &xr) {
  const P xo = p_sel(rx, ry, xr, xl), xo2 = p_sel(rx, ry, xl, xr);
  const P v = p_fma(p_neg(st.s), xo2, p_fma(st.r, xo, st.u));
  xl = p_sel(rx, ry, v, xl);
  xr = p_sel(rx, ry, xr, v);
}

// the ring of a periodic line closed on itself, X_in = last and X_out =
// first: (1 + G) f + B l = A, C f + (1 + F) l = D, in FP64
template <typename real>
__device__ __forceinline__ void ring_close(const Ends<real> &F, const Ends<real> &L, real &xl,
                                           real &xr) {
  const double A = F.a, B = F.b, G = 1.0 + F.g, D = L.a, C = L.b, E = 1.0 + L.g;
  const double idet = rcp(G * E - B * C);
  xr = real((A * E - B * D) * idet);
  xl = real((G * D - C * A) * idet);
}

}  // namespace ppk
