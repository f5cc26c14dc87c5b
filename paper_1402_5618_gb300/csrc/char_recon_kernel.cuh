// char_recon_kernel.cuh -- kernel of the characteristic-wise reconstruction
// (Sec. 2.3) in the arithmetic of the line: real = double is the plain
// form; real = float the mixed form, reading the FP32 hi parts of the state.
// The method and the layout are described in char_recon.cuh.
#pragma once

#include <cooperative_groups.h>

#include "char_recon.cuh"
#include "compact_solve.cuh"
#include "physics.cuh"

namespace ppk {
namespace chr {

namespace cg = cooperative_groups;

// Sec. 2.3: the Roe average of Ua and Ub, reduced to the four scalars the
// left eigenvectors depend on: u, v (2-D), 1/a and c1 = (gamma - 1)/a^2
template <typename real, int NV>
__device__ __forceinline__ void roe_scalars(const real *Ua, const real *Ub, real gamma,
                                            real (&rs)[4]) {
  const real one = real(1), half = real(0.5);
  const real sa = root(Ua[0]), sb = root(Ub[0]);
  const real isa = rcp(sa), isb = rcp(sb), isab = rcp(sa + sb);
  const real ia = isa * isa, ib = isb * isb;   // 1 / rho
  const real g1 = gamma - one;
  const real pa = g1 * (Ua[NV - 1] - half * kin2<real, NV>(Ua) * ia);
  const real pb = g1 * (Ub[NV - 1] - half * kin2<real, NV>(Ub) * ib);
  const real u = (Ua[1] * isa + Ub[1] * isb) * isab;
  const real v = NV == 4 ? (Ua[2] * isa + Ub[2] * isb) * isab : real(0);
  const real H = ((Ua[NV - 1] + pa) * isa + (Ub[NV - 1] + pb) * isb) * isab;
  const real a2 = g1 * (H - half * (u * u + v * v));
  const real ia2 = rcp(a2);
  rs[0] = u;
  rs[1] = v;
  rs[2] = root(ia2);
  rs[3] = g1 * ia2;
}

// The rows l^(k) of L (eqs. (eigen), (leigenv)), ordered by the eigenvalues
// u - a, u, (u,) u + a, with c1 = (gamma - 1)/a^2 and c2 = c1 |u|^2 / 2: the
// acoustic rows are h + d and h - d, the entropy row e_0 - 2 h and in 2-D the
// shear row (-v, 0, 1, 0), with h = (c2, -c1 u, [-c1 v,] c1)/2 and d = (u, -1,
// [0,] 0)/(2 a).  L x from the two inner products takes 10 operations in 2-D.
template <typename real, int NV>
struct LeftEig {
  real h[NV], d0, d1, v;
  __device__ __forceinline__ explicit LeftEig(const real (&rs)[4]) {
    const real half = real(0.5), hc = half * rs[3];
    h[0] = half * (rs[0] * rs[0] + rs[1] * rs[1]) * hc;
    h[1] = -hc * rs[0];
    if (NV == 4) h[2] = -hc * rs[1];
    h[NV - 1] = hc;
    d1 = -half * rs[2];
    d0 = -d1 * rs[0];
    v = rs[1];
  }
  __device__ __forceinline__ void mul(const real (&x)[NV], real (&y)[NV]) const {
    real H = h[0] * x[0];
#pragma unroll
    for (int m = 1; m < NV; ++m) H += h[m] * x[m];
    const real D = d0 * x[0] + d1 * x[1];
    y[0] = H + D;
    y[1] = x[0] - real(2) * H;
    if (NV == 4) y[2] = x[2] - v * x[0];
    y[NV - 1] = H - D;
  }
  // entry (k, m) with k, m known at compile time
  __device__ __forceinline__ real at(int k, int m) const {
    const real d = m == 0 ? d0 : (m == 1 ? d1 : real(0));
    if (k == 0) return h[m] + d;
    if (k == NV - 1) return h[m] - d;
    if (k == 1) return (m == 0 ? real(1) : real(0)) - real(2) * h[m];
    return m == 0 ? -v : (m == 2 ? real(1) : real(0));
  }
};

// |a| > |b| for a pivot search; FP64 by the high words (an FP64 comparison
// takes a slot of the FP64 pipe; a pivot within 2^-20 of the largest is as good)
__device__ __forceinline__ bool larger(float a, float b) { return fabsf(a) > fabsf(b); }
__device__ __forceinline__ bool larger(double a, double b) {
  return (__double2hiint(a) & 0x7fffffff) > (__double2hiint(b) & 0x7fffffff);
}

// X <- M^{-1} X for an NV x NV block M and NCOL columns: Gaussian
// elimination with partial pivoting, all indices fixed at compile time; the
// pivots' reciprocals serve both passes (row c is final once column c is done)
template <typename real, int NV, int NCOL>
__device__ __forceinline__ void gauss_solve(real (&M)[NV][NV], real (&X)[NV][NCOL]) {
  real inv[NV];
#pragma unroll
  for (int c = 0; c < NV; ++c) {
    real best = M[c][c];
    int piv = c;
#pragma unroll
    for (int r = c + 1; r < NV; ++r) {
      if (larger(M[r][c], best)) { best = M[r][c]; piv = r; }
    }
#pragma unroll
    for (int r = c + 1; r < NV; ++r) {
      const bool sw = piv == r;
#pragma unroll
      for (int j = c; j < NV; ++j) {
        const real t = M[c][j];
        M[c][j] = sw ? M[r][j] : t;
        M[r][j] = sw ? t : M[r][j];
      }
#pragma unroll
      for (int j = 0; j < NCOL; ++j) {
        const real t = X[c][j];
        X[c][j] = sw ? X[r][j] : t;
        X[r][j] = sw ? t : X[r][j];
      }
    }
    inv[c] = rcp(M[c][c]);
#pragma unroll
    for (int r = c + 1; r < NV; ++r) {
      const real f = M[r][c] * inv[c];
#pragma unroll
      for (int j = c + 1; j < NV; ++j) M[r][j] -= f * M[c][j];
#pragma unroll
      for (int j = 0; j < NCOL; ++j) X[r][j] -= f * X[c][j];
    }
  }
#pragma unroll
  for (int c = NV - 1; c >= 0; --c) {
#pragma unroll
    for (int j = 0; j < NCOL; ++j) {
      real s = X[c][j];
#pragma unroll
      for (int q = c + 1; q < NV; ++q) s -= M[c][q] * X[q][j];
      X[c][j] = s * inv[c];
    }
  }
}

// geometry of one line: its first cell's offset in the planes, cell stride,
// plane size, length and boundary kinds
struct LineGeo {
  long long base, cs, ncell;
  int n, bclo, bchi;
};

__device__ __forceinline__ LineGeo line_geo(const CharArgs &a, long long line) {
  LineGeo g;
  if (a.lines) {   // a batched line
    const LineDesc d = a.lines[line];
    g.base = d.off + d.base;
    g.cs = d.cs;
    g.ncell = d.ncell;
    g.n = d.n;
    g.bclo = d.bclo;
    g.bchi = d.bchi;
    return g;
  }
  g.base = line * a.line_stride;
  g.cs = a.cell_stride;
  g.ncell = a.ncell;
  g.n = a.n;
  g.bclo = a.bclo;
  g.bchi = a.bchi;
  return g;
}

// ghost-aware read of the line variables of line cell i
template <typename real, int NV>
__device__ __forceinline__ void line_cell(const LineGeo &g, const real *U, const int (&gv)[NV],
                                          int i, real (&out)[NV]) {
  const int n = g.n;
  bool neg = false;
  if (i < 0 || i >= n) {
    const int bc = i < 0 ? g.bclo : g.bchi;
    if (bc == 0) {
      i = i < 0 ? i + n : i - n;
    } else if (bc == 1) {
      i = i < 0 ? 0 : n - 1;
    } else {
      i = i < 0 ? -i - 1 : 2 * n - 1 - i;
      neg = true;
    }
  }
  const real *src = U + g.base + (long long)i * g.cs;
#pragma unroll
  for (int k = 0; k < NV; ++k) out[k] = src[gv[k] * g.ncell];
  if (neg) out[1] = -out[1];
}

// ---------------------------------------------------------------- runs
// A run of block rows by its two end unknowns (see compact_solve.cuh, with
// blocks): end = a - B X_near - G X_far, X_near the unknown next to that end
// outside the run, X_far the one at its other end.
template <typename real, int NV>
struct End {
  real a[NV], B[NV][NV], G[NV][NV];
};

template <typename real, int NV>
__device__ __forceinline__ void end_empty(End<real, NV> &e) {   // the unknown at the other end
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    e.a[i] = real(0);
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      e.B[i][j] = real(0);
      e.G[i][j] = i == j ? real(-1) : real(0);
    }
  }
}
template <typename real, int NV>
__device__ __forceinline__ void end_select(bool c, const End<real, NV> &x, const End<real, NV> &y,
                                           End<real, NV> &o) {
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    o.a[i] = c ? x.a[i] : y.a[i];
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      o.B[i][j] = c ? x.B[i][j] : y.B[i][j];
      o.G[i][j] = c ? x.G[i][j] : y.G[i][j];
    }
  }
}
template <typename real, int NV>
__device__ __forceinline__ void end_xor(const End<real, NV> &x, int d, End<real, NV> &o) {
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    o.a[i] = __shfl_xor_sync(0xffffffffu, x.a[i], d);
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      o.B[i][j] = __shfl_xor_sync(0xffffffffu, x.B[i][j], d);
      o.G[i][j] = __shfl_xor_sync(0xffffffffu, x.G[i][j], d);
    }
  }
}

// o <- e - M [x | r | -s] columnwise: the end e of a run whose far unknown is
// u + r X_o - s X_o' (e.G multiplies it): a - G u, B + G r, -G s with B the
// coefficient of X_o and the new far coefficient that of X_o'
template <typename real, int NV>
__device__ __forceinline__ void end_extend(const End<real, NV> &e, const real (&u)[NV],
                                           const real (&r)[NV][NV], const real (&s)[NV][NV],
                                           End<real, NV> &o) {
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    real t = e.a[i];
#pragma unroll
    for (int m = 0; m < NV; ++m) t -= e.G[i][m] * u[m];
    o.a[i] = t;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      real p = e.B[i][j], q = real(0);
#pragma unroll
      for (int m = 0; m < NV; ++m) {
        p += e.G[i][m] * r[m][j];
        q -= e.G[i][m] * s[m][j];
      }
      o.B[i][j] = p;
      o.G[i][j] = q;
    }
  }
}

// One level of the butterfly over lanes d apart: F, L the run's first and last
// unknown (walk order), later: this lane's run is the later of the two.  st
// (u, r, s): the partner's facing unknown u + r X_o - s X_o' from the
// unknowns outside the joined run (X_o on this lane's side), for the way down.
template <typename real, int NV>
struct BStep {
  real u[NV], r[NV][NV], s[NV][NV];
};

template <typename real, int NV>
__device__ __forceinline__ void block_up(int d, bool later, End<real, NV> &F, End<real, NV> &L,
                                         BStep<real, NV> &st) {
  End<real, NV> in, out, in2;
  end_select(later, F, L, in);
  end_select(later, L, F, out);
  end_xor(in, d, in2);
  // (I - b' b) [u | r | s] = [a' - b' a | b' g | g']
  real M[NV][NV], X[NV][2 * NV + 1];
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    real t = in2.a[i];
#pragma unroll
    for (int m = 0; m < NV; ++m) t -= in2.B[i][m] * in.a[m];
    X[i][0] = t;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      real p = i == j ? real(1) : real(0), q = real(0);
#pragma unroll
      for (int m = 0; m < NV; ++m) {
        p -= in2.B[i][m] * in.B[m][j];
        q += in2.B[i][m] * in.G[m][j];
      }
      M[i][j] = p;
      X[i][1 + j] = q;
      X[i][1 + NV + j] = in2.G[i][j];
    }
  }
  gauss_solve<real, NV, 2 * NV + 1>(M, X);
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    st.u[i] = X[i][0];
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      st.r[i][j] = X[i][1 + j];
      st.s[i][j] = X[i][1 + NV + j];
    }
  }
  // each lane extends its own outer end; the partner's comes back by shuffles
  // (as many as its inputs would take, and 292 operations fewer in 2-D)
  End<real, NV> o, o2;
  end_extend(out, st.u, st.r, st.s, o);
  end_xor(o, d, o2);
  end_select(later, o2, o, F);
  end_select(later, o, o2, L);
}

template <typename real, int NV>
__device__ __forceinline__ void block_down(bool later, const BStep<real, NV> &st, real (&xl)[NV],
                                           real (&xr)[NV]) {
  real v[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    real t = st.u[i];
#pragma unroll
    for (int m = 0; m < NV; ++m) {
      const real xo = later ? xr[m] : xl[m], xo2 = later ? xl[m] : xr[m];
      t += st.r[i][m] * xo;
      t -= st.s[i][m] * xo2;
    }
    v[i] = t;
  }
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    if (later) xl[i] = v[i];
    else xr[i] = v[i];
  }
}

// the ring of a periodic line closed on itself, X_in = last and X_out = first:
// (I + G_F) f + B_F l = a_F, B_L f + (I + G_L) l = a_L
template <typename real, int NV>
__device__ __forceinline__ void block_ring(const End<real, NV> &F, const End<real, NV> &L,
                                           real (&xl)[NV], real (&xr)[NV]) {
  real M[NV][NV], X[NV][NV + 1], N[NV][NV], Y[NV][1];
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    X[i][0] = F.a[i];
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      M[i][j] = F.G[i][j] + (i == j ? real(1) : real(0));
      X[i][1 + j] = F.B[i][j];
    }
  }
  gauss_solve<real, NV, NV + 1>(M, X);   // f = X_0 - X_1 l
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    real t = L.a[i];
#pragma unroll
    for (int m = 0; m < NV; ++m) t -= L.B[i][m] * X[m][0];
    Y[i][0] = t;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      real p = L.G[i][j] + (i == j ? real(1) : real(0));
#pragma unroll
      for (int m = 0; m < NV; ++m) p -= L.B[i][m] * X[m][1 + j];
      N[i][j] = p;
    }
  }
  gauss_solve<real, NV, 1>(N, Y);
#pragma unroll
  for (int i = 0; i < NV; ++i) xl[i] = Y[i][0];
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    real t = X[i][0];
#pragma unroll
    for (int m = 0; m < NV; ++m) t -= X[i][1 + m] * xl[m];
    xr[i] = t;
  }
}

// ---------------------------------------------------------------- rows
// The block row of a cell, normalised by b: L y_p + diag(a) L y_{p-1} +
// diag(c) L y_{p+1} = s in the deviations y from the cell averages, walk
// order.  win: the five cells of the stencil in walk order.
template <typename real, int NV>
__device__ __forceinline__ void char_row(const real (&win)[5][NV], real gamma, real eps,
                                         bool closure, real (&rs)[4], real (&ca)[NV],
                                         real (&cc)[NV], real (&s)[NV]) {
  constexpr bool F32 = sizeof(real) == 4;
  roe_scalars<real, NV>(win[2], win[3], gamma, rs);
  const LeftEig<real, NV> L(rs);
  real dW[4][NV], top[NV];
#pragma unroll
  for (int w = 0; w < 4; ++w) {
    real dU[NV];
#pragma unroll
    for (int m = 0; m < NV; ++m) dU[m] = win[w + 1][m] - win[w][m];
    L.mul(dU, dW[w]);
  }
  if (F32) {
#pragma unroll
    for (int m = 0; m < NV; ++m) {
      top[m] = fabs(win[0][m]);
#pragma unroll
      for (int w = 1; w < 5; ++w) top[m] = fmax(top[m], fabs(win[w][m]));
    }
  }
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    real D[4], mag = real(0);
#pragma unroll
    for (int w = 0; w < 4; ++w) D[w] = dW[w][k];
    const real k43 = real(4.0 / 3.0);
    const real g0 = D[1] - D[0], g1 = D[2] - D[1], g2 = D[3] - D[2];
    real e = eps;
    if constexpr (F32) {
      // the rounding floor of the indicators on the size of the terms the
      // characteristic variable is summed from
#pragma unroll
      for (int m = 0; m < NV; ++m) mag += fabsf(L.at(k, m)) * top[m];
      e = fmaf(FP32_BETA_FLOOR * mag, mag, eps);
    }
    const real d0 = fma(k43 * g0, g0, e) + D[1] * (D[1] + g0);
    const real d1 = fma(k43 * g1, g1, e) + D[1] * D[2];
    const real d2 = fma(k43 * g2, g2, e) + D[2] * (D[2] - g2);
    real S0, S1, S2;
    z_terms(d0, d1, d2, S0, S1, S2);
    if (closure) {
      const real a0 = real(0.1) * S0, a1 = real(0.6) * S1, a2 = real(0.3) * S2;
      ca[k] = cc[k] = real(0);
      s[k] = (a0 * (real(5) * D[1] - real(2) * D[0]) + a1 * (D[1] + real(2) * D[2]) +
              a2 * (real(4) * D[2] - D[3])) * rcp(real(6) * (a0 + a1 + a2));
    } else {
      const real t2 = real(2.5) * S1, t4 = real(1.25) * S1;
      const real ib = rcp(fma(real(3), S2, fma(real(2), t2, S0)));
      ca[k] = fma(real(2), S0, t2) * ib;
      cc[k] = real(1.5) * S2 * ib;
      s[k] = (D[1] * fma(real(1.5), S0, t2) + D[2] * fma(real(2.25), S2, t4)) * ib;
    }
  }
}

// ---------------------------------------------------------------- kernel
// One warp per (segment of 32 M cells, side); lane k holds the M cells of
// chunk k; a cluster of R CTAs covers the line.  Kept per row of every lane
// until the back substitution: the multipliers Y, F and g (x = g - F X_in - Y
// x_next), in shared memory or, with many lines, in global scratch.  Bound by
// FP64 instructions, in FP32 by instruction fetch and by latency (12 warps per
// SM, 168 registers each).
template <typename real, int NV>
struct CharSmem {
  static constexpr int E = 2 * NV * NV + NV;   // multipliers of a row
  static constexpr int RC = 4 + 3 * NV;        // numbers of a row before its elimination
  // this segment's first and last unknown, then per lane the multipliers of
  // every row, or (scratch: they go to global memory) the numbers of T rows
  static size_t bytes(const CharArgs &a) {
    return sizeof(End<real, NV>) * 2 +
           sizeof(real) * 32 * (a.scr ? RC * (size_t)a.T : E * (size_t)a.M);
  }
};

template <typename real, int NV>
__global__ void __launch_bounds__(32) char_solve_kernel(const CharArgs a) {
  constexpr int E = CharSmem<real, NV>::E;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  End<real, NV> *seg = reinterpret_cast<End<real, NV> *>(smem_raw);
  real *rows = reinterpret_cast<real *>(smem_raw + 2 * sizeof(End<real, NV>));
  cg::cluster_group cluster = cg::this_cluster();
  const int M = a.M, R = a.R, T = a.T, shT = __ffs(T) - 1;
  const int rank = (int)cluster.block_rank(), lane = threadIdx.x, side = blockIdx.y;
  const LineGeo geo = line_geo(a, blockIdx.x / R);
  const int n = geo.n;
  const bool per = geo.bclo == 0;
  const int lo = rank * 32 * M, i0 = lo + lane * M;
  const int cnt = max(0, min(M, n - i0));
  const int dir = side == 0 ? 1 : -1;
  const int first = side == 0 ? i0 : i0 + cnt - 1;   // the chunk's first cell in walk order
  const real *U = reinterpret_cast<const real *>(a.U);
  int gv[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) gv[k] = k == 0 ? 0 : (k == NV - 1 ? NV - 1 : (k == 1 ? a.vn : a.vt));
  const real gam = real(a.gamma), eps = real(a.eps_weno);
  // a row's numbers, and its multipliers over them or in the scratch
  const int RS = a.scr ? CharSmem<real, NV>::RC : E;
  real *mult = rows;
  if (a.scr)
    mult = reinterpret_cast<real *>(a.scr) +
           ((long long)blockIdx.y * gridDim.x + blockIdx.x) * ((long long)32 * E * M);
  // (a lane's column moves with the row: lanes on consecutive cells of a chunk
  // are then in different banks)
  auto at = [&](int t, int e, int k) -> real & { return rows[(t * RS + e) * 32 + ((k + 4 * t) & 31)]; };
  auto mt = [&](int t, int e) -> real & { return mult[(t * E + e) * 32 + ((lane + 4 * t) & 31)]; };
  // the q-th cell of the rows [t0, t0 + T) of all chunks, consecutive q on
  // consecutive cells: its chunk and row; false where the chunk has no such row
  auto tile_cell = [&](int q, int t0, int &ch, int &t, long long &o) {
    ch = q >> shT;
    t = q & (T - 1);
    const int c0 = lo + ch * M, m = min(M, n - c0);
    o = geo.base + (long long)(c0 + (side == 0 ? t0 + t : m - 1 - t0 - t)) * geo.cs;
    return t0 + t < m;
  };

  End<real, NV> F, L;
  end_empty(F);
  end_empty(L);
  // T rows at a time: first the 4 + 3 NV numbers of each, then their
  // elimination -- two loops whose bodies stay in the instruction caches instead
  // of one that does not.  The cells come in with consecutive lanes on
  // consecutive cells, each into its row's slots (read as a stencil cell before
  // the row overwrites them); the two cells on either side are a lane's own.
#pragma unroll 1
  for (int t0 = 0; t0 < M; t0 += T) {
    __syncwarp();
#pragma unroll 4
    for (int q = lane; q < 32 * T; q += 32) {
      int ch, t;
      long long o;
      if (tile_cell(q, t0, ch, t, o)) {
#pragma unroll
        for (int k = 0; k < NV; ++k) at(t, k, ch) = __ldg(U + o + gv[k] * geo.ncell);
      }
    }
    __syncwarp();
    const int tc = min(T, cnt - t0), f0 = first + t0 * dir;
    real win[5][NV], after[2][NV];
    if (tc > 0) {
      line_cell<real, NV>(geo, U, gv, f0 - 2 * dir, win[1]);
      line_cell<real, NV>(geo, U, gv, f0 - dir, win[2]);
      line_cell<real, NV>(geo, U, gv, f0 + tc * dir, after[0]);
      line_cell<real, NV>(geo, U, gv, f0 + (tc + 1) * dir, after[1]);
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        win[3][k] = at(0, k, lane);
        win[4][k] = tc > 1 ? at(1, k, lane) : after[0][k];
      }
    }
#pragma unroll 1
    for (int t = 0; t < tc; ++t) {
      const int c = f0 + t * dir;
#pragma unroll
      for (int w = 0; w < 4; ++w)
#pragma unroll
        for (int k = 0; k < NV; ++k) win[w][k] = win[w + 1][k];
#pragma unroll
      for (int k = 0; k < NV; ++k)
        win[4][k] = t + 2 < tc ? at(min(t + 2, T - 1), k, lane)
                               : (t + 2 == tc ? after[0][k] : after[1][k]);
      real rs[4], ca[NV], cc[NV], s[NV];
      char_row<real, NV>(win, gam, eps, !per && (c == 0 || c == n - 1), rs, ca, cc, s);
#pragma unroll
      for (int i = 0; i < 4; ++i) at(t, i, lane) = rs[i];
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        at(t, 4 + i, lane) = ca[i];
        at(t, 4 + NV + i, lane) = cc[i];
        at(t, 4 + 2 * NV + i, lane) = s[i];
      }
    }
    // elimination of the chunk: last = g - F X_in - Y x_next after every row,
    // first = a - B X_in - G x_next folded along
#pragma unroll 1
    for (int t = 0; t < tc; ++t) {
      real ca[NV], cc[NV], s[NV], rs[4];
      {
#pragma unroll
        for (int i = 0; i < 4; ++i) rs[i] = at(t, i, lane);
#pragma unroll
        for (int i = 0; i < NV; ++i) {
          ca[i] = at(t, 4 + i, lane);
          cc[i] = at(t, 4 + NV + i, lane);
          s[i] = at(t, 4 + 2 * NV + i, lane);
        }
      }
      const LeftEig<real, NV> Lk(rs);
      // (L - diag(a) L Y) [Y' | g' | F'] = [diag(c) L | s - diag(a) L g | -diag(a) L F]
      real B[NV][NV], X[NV][2 * NV + 1];
      {
        real tg[NV];
        Lk.mul(L.a, tg);
#pragma unroll
        for (int i = 0; i < NV; ++i) X[i][NV] = s[i] - ca[i] * tg[i];
      }
#pragma unroll
      for (int j = 0; j < NV; ++j) {
        real y[NV], f[NV], ty[NV], tf[NV];
#pragma unroll
        for (int m = 0; m < NV; ++m) {
          y[m] = L.B[m][j];
          f[m] = L.G[m][j];
        }
        Lk.mul(y, ty);
        Lk.mul(f, tf);
#pragma unroll
        for (int i = 0; i < NV; ++i) {
          const real l = Lk.at(i, j);
          B[i][j] = l - ca[i] * ty[i];
          X[i][j] = cc[i] * l;
          X[i][NV + 1 + j] = -(ca[i] * tf[i]);
        }
      }
      gauss_solve<real, NV, 2 * NV + 1>(B, X);
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        L.a[i] = X[i][NV];
        mt(t0 + t, i) = X[i][NV];
#pragma unroll
        for (int j = 0; j < NV; ++j) {
          L.B[i][j] = X[i][j];
          L.G[i][j] = X[i][NV + 1 + j];
          mt(t0 + t, NV + i * NV + j) = X[i][j];
          mt(t0 + t, NV + NV * NV + i * NV + j) = X[i][NV + 1 + j];
        }
      }
      // first = a - B X_in - G x_p with x_p = g - F X_in - Y x_{p+1}
      real G2[NV][NV];
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        real p = F.a[i];
#pragma unroll
        for (int m = 0; m < NV; ++m) p -= F.G[i][m] * L.a[m];
        F.a[i] = p;
#pragma unroll
        for (int j = 0; j < NV; ++j) {
          real q = F.B[i][j], r = real(0);
#pragma unroll
          for (int m = 0; m < NV; ++m) {
            q -= F.G[i][m] * L.G[m][j];
            r -= F.G[i][m] * L.B[m][j];
          }
          F.B[i][j] = q;
          G2[i][j] = r;
        }
      }
#pragma unroll
      for (int i = 0; i < NV; ++i)
#pragma unroll
        for (int j = 0; j < NV; ++j) F.G[i][j] = G2[i][j];
    }
  }

  // trees over the warp's chunks, then over the segments of the cluster
  BStep<real, NV> st[5], sg[4];
#pragma unroll 1
  for (int h = 0; h < 5; ++h) {
    const bool up = (lane >> h) & 1;
    block_up(1 << h, side == 0 ? up : !up, F, L, st[h]);
  }
  real xl[NV], xr[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) xl[i] = xr[i] = real(0);
  if (R > 1) {
    if (lane == 0) {
      seg[0] = F;
      seg[1] = L;
    }
    cluster.sync();
    const int q = lane & 15;
    end_empty(F);
    end_empty(L);
    if (q < R) {
      const End<real, NV> *o = cluster.map_shared_rank(seg, side == 0 ? q : R - 1 - q);
      F = o[0];
      L = o[1];
    }
#pragma unroll 1
    for (int h = 0; (1 << h) < R; ++h) block_up(1 << h, (q >> h) & 1, F, L, sg[h]);
    // Arrive now, wait before exit: a CTA's shared memory must outlive the
    // reads of its run.  Only here, where every lane's reads have been used
    // (the joins need them all): an arrival does not wait for loads in flight.
    __syncwarp();
    cluster_arrive_relaxed();
  }
  if (per) block_ring(F, L, xl, xr);
  if (R > 1) {
    const int q = lane & 15, own = side == 0 ? rank : R - 1 - rank;
#pragma unroll 1
    for (int h = 3; h >= 0; --h)
      if ((1 << h) < R) block_down((q >> h) & 1, sg[h], xl, xr);
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      xl[i] = __shfl_sync(0xffffffffu, xl[i], own);
      xr[i] = __shfl_sync(0xffffffffu, xr[i], own);
    }
  }
#pragma unroll 1
  for (int h = 4; h >= 0; --h) {
    const bool up = (lane >> h) & 1;
    block_down(side == 0 ? up : !up, st[h], xl, xr);
  }

  // back substitution, the multipliers of the two rows before the current one
  // loading meanwhile; the deviations go where the row's numbers were
  real nx[2][E];
#pragma unroll
  for (int d = 0; d < 2; ++d)
    if (cnt > d) {
#pragma unroll
      for (int e = 0; e < E; ++e) nx[d][e] = mt(cnt - 1 - d, e);
    }
  real *out = reinterpret_cast<real *>(side == 0 ? a.Um : a.Up);
#pragma unroll 1
  for (int t0 = (M - 1) & ~(T - 1); t0 >= 0; t0 -= T) {
    __syncwarp();
#pragma unroll 1
    for (int t = min(T, cnt - t0) - 1; t >= 0; --t) {
      real m[E], x[NV];
#pragma unroll
      for (int e = 0; e < E; ++e) {
        m[e] = nx[0][e];
        nx[0][e] = nx[1][e];
      }
      if (t0 + t > 1) {
#pragma unroll
        for (int e = 0; e < E; ++e) nx[1][e] = mt(t0 + t - 2, e);
      }
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        real p = m[i];
#pragma unroll
        for (int j = 0; j < NV; ++j) {
          p -= m[NV + NV * NV + i * NV + j] * xl[j];
          p -= m[NV + i * NV + j] * xr[j];
        }
        x[i] = p;
      }
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        xr[i] = x[i];
        at(t, i, lane) = x[i];
      }
    }
    __syncwarp();
    // out: consecutive lanes on consecutive cells
#pragma unroll 4
    for (int q = lane; q < 32 * T; q += 32) {
      int ch, t;
      long long o;
      if (tile_cell(q, t0, ch, t, o)) {
#pragma unroll
        for (int k = 0; k < NV; ++k)
          out[o + gv[k] * geo.ncell] = __ldg(U + o + gv[k] * geo.ncell) + at(t, k, ch);
      }
    }
  }
  if (R > 1) cluster_wait();
}

template <typename real, int NV>
cudaError_t launch_nv(const CharArgs &a, cudaStream_t st, bool attrs_only) {
  auto kern = char_solve_kernel<real, NV>;
  if (attrs_only) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(sizeof(End<real, NV>) * 2 + sizeof(real) * 32 * 16 * CharSmem<real, NV>::E));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                               (int)cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.nlines * a.R), 2, 1);
  cfg.blockDim = dim3(32, 1, 1);
  cfg.dynamicSmemBytes = CharSmem<real, NV>::bytes(a);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)a.R;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a);
}

template <typename real>
cudaError_t launch_char_recon_t(const CharArgs &a, int nv, cudaStream_t st, bool attrs_only) {
  return nv == 3 ? launch_nv<real, 3>(a, st, attrs_only) : launch_nv<real, 4>(a, st, attrs_only);
}

}  // namespace chr
}  // namespace ppk
