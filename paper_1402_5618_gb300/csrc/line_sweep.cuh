// line_sweep.cuh -- the fused per-stage line operator of the FVCW scheme.
//
// One thread-block cluster of R CTAs owns one grid line of n cells; CTA r
// holds the contiguous segment [r*SEG, min((r+1)*SEG, n)) of it in shared
// memory and runs, in order:
//   load     cell averages of the segment plus a two-cell halo (ghost cells
//            from the boundary condition at the line ends);
//   solve    for each conserved variable the minus and plus compact-WENO
//            systems (eq. (CWENO-FV)), exactly and in partitioned form
//            (compact_solve.cuh): every thread eliminates a chunk of M rows of
//            one variable in both systems as a function of the unknowns
//            outside it, the chunks of the segment are joined within a warp,
//            the segments of the cluster through distributed shared memory,
//            and every thread substitutes back in its chunk.  A periodic line
//            is the same with the ring closed where the segments are joined;
//   limit    Zhang-Shu limiter per cell (Sec. 2.4);
//   flux     HLLC at every face of the segment (the CTA limits the cell on
//            either side of its segment itself: no exchange of faces; both
//            CTAs at a seam come to the same bits, see Exch::ends);
//   update   flux difference (eq. (1DEulerFV-b)) and either the x-sweep
//            output D = L_x, or the SSP-RK3 stage combination (eq. (RK3))
//            with L = D + L_y (2-D) / L (1-D), plus the grid-wide reductions
//            that fix the next stage's limiter epsilon and the next dt.
//
// real = double: the plain form (FP64 state and arithmetic).
// real = float: the mixed form -- FP32 line arithmetic, the state stored as
// FP32 hi + lo pairs combined with compensated (double-float) arithmetic,
// FP64 only for the limiter factors of cells that need limiting and for the
// closing of a periodic ring.
//
// What bounds it: in FP64 the FP64 pipe (70-77% busy on large grids; a line
// alone waits for its own chain of FP64 instructions), in the mixed form
// instruction issue (47%) and fixed latencies, barriers and instruction
// fetch, with 16 warps per SM; HBM is at 14%.  Per sweep of 4096^2 cells (corner
// blast), against a scan over projective chunk maps with divisions in every
// row and an exchange of limited faces: mixed 1.63 -> 0.83 ms, FP64 48.0 -> 16.4
// (x) and 51.6 -> 18.1 ms (y with the stage update).
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "batch_lines.cuh"
#include "compact_solve.cuh"
#include "dfloat.cuh"
#include "physics.cuh"

namespace cg = cooperative_groups;

namespace ppk {

// device-side control block of one problem (time, dt, reductions, flags)
struct Ctl {
  double t, t_final, dt, cfl, dt_cap;
  long long step, step_limit;
  int active, done, err_steps, err_rate;
  double eps0;                         // limiter epsilon for stage 1
  unsigned long long minrho[3];        // min density after stage k (double bits; +inf init)
  unsigned long long rate;             // max rate after stage 3 (double bits)
  unsigned long long nviol;            // cells outside G
  unsigned long long first_bad;        // min flat index of a bad cell (~0 none)
  unsigned long long theta1, theta2;   // limiter activations
  double last_dt;
  double eps_pos;
  // eq. (CFL-CD) on the limited face values (face_cfl > 0): the largest
  // (|u| + a)/h over the face values of this step's stages per direction
  // (double bits; NaN propagates), the rate of the last accepted step, and
  // what a step that is redone restores
  unsigned long long frate[2];
  double face_cfl;
  double frate_prev;
  double t_prev;
  unsigned long long rate_n, minrho_n;
  long long nreject;
  int nrej_run;
};

enum { MODE_XSWEEP = 0, MODE_FINAL = 1, MODE_OPERATOR = 2 };

struct SweepArgs {
  // plain form: FP64 planes [nv][ncell]
  const double *U;    // stage input
  const double *U0;   // U^n
  double *Uout;       // FINAL: stage output
  // mixed form: FP32 hi / lo planes of the same states
  const float *Uh, *Ul, *U0h, *U0l;
  float *Uoh, *Uol;
  const void *Din;    // flux difference of the other direction (2-D), real
  void *Dout;         // x-sweep output, real
  double *Lout;       // OPERATOR: L (FP64 planes)
  long long ncell;    // cells per variable plane
  int n;              // cells per line
  int R;              // CTAs per line (cluster size)
  long long cell_stride, line_stride;
  int vn, vt;         // grid index of the normal / tangential momentum (vt < 0 in 1-D)
  int bclo, bchi;
  double h, h_other;  // cell size along the line / across (0 in 1-D)
  double ih;          // 1 / h (from the host: no FP64 division per thread)
  double ih_other;    // 1 / h_other (0 in 1-D)
  // FP32 copies for the mixed form's kernels (converting a double costs a
  // slot of GB300's FP64 pipe per warp): gamma, wgl, eps_weno, 1/h,
  // 1/h_other, gamma (gamma - 1), and the limiter epsilon of eps_fixed
  float gamma_f, wgl_f, eps_weno_f, ih_f, ih_other_f, gg1_f, eps_fixed_f;
  double gamma, wgl, eps_weno;
  int stage;          // 0, 1, 2
  double eps_fixed;   // > 0: fixed limiter epsilon, no control-block checks (operator evaluation)
  int limiter;
  int flux;           // 0 HLLC, 1 local Lax-Friedrichs
  int fcheck;         // 1: reduce the face speeds into ctl->frate[fdir]
  int fdir;           // 0: x faces, 1: y faces
  // face values U^-, U^+ computed by another kernel (planes of the line's
  // arithmetic in the state's layout); nullptr: the kernel reconstructs them
  const void *Fm_pre, *Fp_pre;
  Ctl *ctl;
  // batched launch: line table (nullptr: one problem)
  const LineDesc *lines;
};

// resolve the line a cluster works on: for a batched launch, take the
// problem's grid, boundaries, control block and its slice of every buffer.
// Returns the offset of the line's first cell in a plane.
template <typename real>
__device__ __forceinline__ long long bind_line(SweepArgs &a, long long line) {
  if (!a.lines) return line * a.line_stride;
  const LineDesc d = a.lines[line];
  a.ctl = a.ctl + d.prob;
  a.ncell = d.ncell;
  a.n = d.n;
  a.cell_stride = d.cs;
  a.bclo = d.bclo;
  a.bchi = d.bchi;
  a.ih = d.ih;
  a.ih_other = d.ih_other;
  a.ih_f = d.ih_f;
  a.ih_other_f = d.ih_other_f;
  const long long o = d.off;
  if (a.U) a.U += o;
  if (a.U0) a.U0 += o;
  if (a.Uout) a.Uout += o;
  if (a.Uh) a.Uh += o;
  if (a.Ul) a.Ul += o;
  if (a.U0h) { a.U0h += o; a.U0l += o; }
  if (a.Uoh) { a.Uoh += o; a.Uol += o; }
  if (a.Lout) a.Lout += o;
  if (a.Din) a.Din = reinterpret_cast<const real *>(a.Din) + o;
  if (a.Dout) a.Dout = reinterpret_cast<real *>(a.Dout) + o;
  if (a.Fm_pre) {   // face values of the characteristic-wise reconstruction, same layout
    a.Fm_pre = reinterpret_cast<const real *>(a.Fm_pre) + o;
    a.Fp_pre = reinterpret_cast<const real *>(a.Fp_pre) + o;
  }
  return d.base;
}

template <typename real>
__device__ __forceinline__ real shfl_down_r(real v, int d, int width = 32) {
  return __shfl_down_sync(0xffffffffu, v, d, width);
}

// ---------------------------------------------------------------- smem
template <typename real, int NV>
struct Exch {
  Run<real> seg[2 * NV];         // this segment as a run, per variable and side
  // Per variable and side, for every segment of the line the unknowns before
  // (x) and after it (y, walk order); the own segment's first and last are the
  // one after the previous and the one before the next.  A face between two
  // segments is evaluated by both CTAs, and the line's flux differences
  // telescope only if they get the same number: every CTA computes the entries
  // at its ends by the same operations on the same runs.
  typename Pair<real>::t ends[2 * NV][16];
  // mixed form, the line's reference state R (difference form): per
  // variable the hi / lo pair of the median of five sampled cells, R in
  // FP32, the reference fluxes F(R), (u_R, v_R, p_R, E_R + p_R), whether
  // the sampled densities and energies lie within a factor 2 of R (gate)
  float rh[NV], rl[NV], rf[NV], rF[NV], rp[4];
  int rgate[NV];
  float rspread[NV];             // largest |sample - R| per variable (hi parts)
  float hend[2][NV];             // hi parts of the cells before and after the segment
  float epsf;                    // mixed form: the limiter epsilon of this stage
  dfl dt;                        // mixed form: the time step
};

// Segment planes in shared memory carry one pad word per 128 bytes: segment
// cell c (c >= -2) sits at pad(c) = c + (c >> PSH) of its plane.  Lanes of a
// warp then hit distinct banks both when each lane walks its own chunk of M
// cells (lane stride M) and when consecutive lanes take consecutive cells;
// a chunk (M divides 128 bytes) never straddles a pad word.
template <typename real, int NV, int M, int KCHUNK>
struct Smem {
  static constexpr int KC = KCHUNK;       // chunks per conserved variable
  static constexpr int SEG = M * KC;      // cells per CTA segment
  // the chunks of a segment are joined by trees over the lanes (see
  // compact_solve.cuh), or by LPS lanes of one warp per system, eight each
  static constexpr bool TREE = sizeof(real) == 4 || M <= 4;
  static constexpr int LPS = KC / 8;
  // FP64 with short chunks: a warp per variable and side (a warp's FP64
  // instructions take 64 cycles each, and these launches wait for them)
  static constexpr int SIDES = sizeof(real) == 8 && M <= 4 ? 2 : 1;
  static constexpr int THREADS = NV * KC * SIDES;
  static constexpr int PSH = sizeof(real) == 4 ? 5 : 4;
  __host__ __device__ static constexpr int pad(int c) { return c + (c >> PSH); }
  static constexpr int UH = 3;                         // pad(-2) = -3
  static constexpr int UWP = UH + pad(SEG + 1) + 1;    // cells -2 .. SEG+1
  static constexpr int WP = pad(SEG - 1) + 1;          // cells 0 .. SEG-1
  static_assert(((32 * 4 / (int)sizeof(real)) % M) == 0, "a chunk must not straddle a pad word");
  static_assert(KC % 32 == 0, "whole warps per variable");
  // per system: six run values per chunk, and the last unknown of every chunk
  // in walk order (entry 0: the unknown before the segment); one pad entry
  // per eight, so that lanes walking eight chunks each hit distinct banks
  static constexpr int KCP = KC + KC / 8;
  static constexpr int XP = KC + 1 + KC / 8;
  static constexpr int FH = 2;                         // pad(-1) = -2
  static constexpr int FWP = FH + pad(SEG) + 1;        // face values of cells -1 .. SEG
  static constexpr int FLS = SEG + 4;                  // fluxes of a variable, rows on 16 bytes
  static constexpr size_t up16(size_t x) { return (x + 15) / 16 * 16; }
  static constexpr size_t u_off = 0;                                     // real Us[NV][UWP]
  static constexpr size_t fm_off = u_off + sizeof(real) * NV * UWP;      // real Fm, Fp[NV][FWP]
  static constexpr size_t fp_off = fm_off + sizeof(real) * NV * FWP;
  static constexpr size_t zm_off = up16(fp_off + sizeof(real) * NV * FWP);   // real Zm, Zp[NV][WP]
  static constexpr size_t zp_off = zm_off + sizeof(real) * NV * WP;
  static constexpr size_t fl_off = zm_off;     // real Fl[NV][FLS], after Zm and Zp are done with
  static_assert(FLS <= 2 * WP, "the fluxes must fit the two planes they reuse");
  static constexpr size_t cr_off = zp_off + sizeof(real) * NV * WP;      // real Cr[2 NV][6][KCP]
  static constexpr size_t xs_off = cr_off + (TREE ? 0 : sizeof(real) * 2 * NV * 6 * KCP);   // real Xs[2 NV][XP]
  static constexpr size_t ex_off = up16(xs_off + (TREE ? 0 : sizeof(real) * 2 * NV * XP));
  // mixed form: one byte per cell (its face values stored in full, not as
  // differences from R) and one per face (its flux stored as F - F(R))
  static constexpr size_t cf_off = ex_off + sizeof(Exch<real, NV>);
  static constexpr size_t ff_off = cf_off + SEG + 2;   // (flags of cells -1 .. SEG)
  static constexpr size_t bytes = up16(ff_off + SEG + 2);
};

// line-variable k -> grid variable
__device__ __forceinline__ int gvar(int k, int nv, int vn, int vt) {
  return k == 0 ? 0 : (k == nv - 1 ? nv - 1 : (k == 1 ? vn : vt));
}

__device__ __forceinline__ unsigned long long double_bits(double x) {
  return (unsigned long long)__double_as_longlong(x);
}
__device__ __forceinline__ double bits_double(unsigned long long b) {
  return __longlong_as_double((long long)b);
}

// grid-wide extrema on a few control-block words: every warp of every CTA
// reports, so an atomic whose value cannot change the word is skipped (the
// words only move one way during a launch; a stale read only costs an atomic)
__device__ __forceinline__ void atomic_max_bits(unsigned long long *w, unsigned long long v) {
  if (v > *reinterpret_cast<volatile unsigned long long *>(w)) atomicMax(w, v);
}
__device__ __forceinline__ void atomic_min_bits(unsigned long long *w, unsigned long long v) {
  if (v < *reinterpret_cast<volatile unsigned long long *>(w)) atomicMin(w, v);
}

// ---------------------------------------------------------------- kernel
// Resident CTAs per SM the kernel is compiled for (CTAS_*): see sweeps.cuh.
// PRE: the face values come from another kernel (args.Fm_pre / Fp_pre) and
// the reconstruction phases are compiled out.
template <typename real, int NV, int M, int KC, int MODE, bool PRE, int CTAS>
__global__ void __launch_bounds__(Smem<real, NV, M, KC>::THREADS, CTAS) line_sweep(SweepArgs args_in) {
  constexpr bool MIXED = sizeof(real) == 4;
  using S = Smem<real, NV, M, KC>;
  constexpr int SEG = S::SEG;
  constexpr int T = S::THREADS;
  constexpr int UH = S::UH, UWP = S::UWP, WP = S::WP, FH = S::FH, FWP = S::FWP, FLS = S::FLS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  real *Us = reinterpret_cast<real *>(smem_raw + S::u_off);
  real *Fm = reinterpret_cast<real *>(smem_raw + S::fm_off);
  real *Fp = reinterpret_cast<real *>(smem_raw + S::fp_off);
  real *Fl = reinterpret_cast<real *>(smem_raw + S::fl_off);
  Exch<real, NV> &ex = *reinterpret_cast<Exch<real, NV> *>(smem_raw + S::ex_off);

  cg::cluster_group cluster = cg::this_cluster();
  SweepArgs args = args_in;
  const int R = args.R;
  const int rank = (int)cluster.block_rank();
  const long long lbase = bind_line<real>(args, blockIdx.x / R);
  const int n = args.n;
  const int lo = rank * SEG;
  const int hi = min(lo + SEG, n);
  const int tid = threadIdx.x;
  const int v = tid / KC % NV;
  const int sidew = tid / (NV * KC);   // (SIDES == 2: the system this warp solves)
  const int k = tid % KC;
  const int lane = tid & 31;
  const bool per = args.bclo == 0;
  Ctl *ctl = args.ctl;

  // a finished problem skips the launch (uniform over the grid)
  if (args.eps_fixed <= 0.0 && !ctl->active) return;

  const real eps_w = MIXED ? real(args.eps_weno_f) : real(args.eps_weno);
  const real gam = MIXED ? real(args.gamma_f) : real(args.gamma);
  const real wgl = MIXED ? real(args.wgl_f) : real(args.wgl);
  real eps_pos;
  if constexpr (MIXED) {
    // one thread takes the FP64 minimum; the others read it after the
    // load phase's barrier (the limiter comes later)
    if (tid == 0) {
      double e = args.eps_fixed > 0.0 ? args.eps_fixed
                 : (args.stage == 0 ? ctl->eps0
                                    : fmin(ctl->eps_pos, bits_double(ctl->minrho[args.stage - 1])));
      ex.epsf = (float)e;
      if (MODE == MODE_FINAL) {
        const double t = ctl->dt;
        ex.dt.hi = (float)t;
        ex.dt.lo = (float)(t - (double)ex.dt.hi);
      }
    }
    eps_pos = real(0);   // set after the barrier
  } else {
    if (args.eps_fixed > 0.0) eps_pos = real(args.eps_fixed);
    else if (args.stage == 0) eps_pos = real(ctl->eps0);
    else eps_pos = real(fmin(ctl->eps_pos, bits_double(ctl->minrho[args.stage - 1])));
  }

  const long long cs = args.cell_stride;
  unsigned char *cfull = smem_raw + S::cf_off + 1;   // mixed: cell's faces stored in full
  unsigned char *fdel = smem_raw + S::ff_off;    // mixed: face flux stored as F - F(R)

  if constexpr (MIXED && !PRE) {
    for (int c = tid; c < SEG + 2; c += T) cfull[c - 1] = 0;
  }
  // difference form possible: the reference samples and the lo parts load
  // with the hi parts
  const bool two = MIXED && !PRE && args.Ul != nullptr;
  float sh[5], sl[5];
  if constexpr (MIXED && !PRE) {
    if (two && tid < NV) {
      const int g = gvar(tid, NV, args.vn, args.vt);
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        const int i = (int)(((long long)(2 * q + 1) * n) / 10);
        const long long a = g * args.ncell + lbase + (long long)i * cs;
        sh[q] = args.Uh[a];
        sl[q] = args.Ul[a];
      }
    }
  }
  (void)sh; (void)sl;

  // ---------------------------------------------------------------- load
  // line cell i (any i; ghosts by the boundary condition): its address and
  // whether the ghost negates the value (reflective, normal momentum)
  auto cell_addr = [&](int kv, int i, bool &neg) -> long long {
    int g = gvar(kv, NV, args.vn, args.vt);
    neg = false;
    if (i < 0 || i >= n) {
      if (per) {
        i = i < 0 ? i + n : i - n;
      } else {
        int bc = i < 0 ? args.bclo : args.bchi;
        if (bc == 1) {
          i = i < 0 ? 0 : n - 1;
        } else {  // reflective mirror
          i = i < 0 ? -i - 1 : 2 * n - 1 - i;
          neg = kv == 1;
        }
      }
    }
    return g * args.ncell + lbase + (long long)i * cs;
  };
  // Thread (v, k) brings in M cells of the segment of variable v, hi and lo
  // parts, all its loads in flight together in registers until the reference
  // state is known: (hi, lo) -> U or U - R on the way to shared memory, one
  // pass.  Segments on 16-byte boundaries take float4 loads, others one value
  // at a time, lanes on consecutive cells (a fixed stride per thread: no
  // index arithmetic per value).  Threads k < 4 also take a halo cell, the
  // next three a cell left over from the float4.
  constexpr int NQ = (SEG / 4 + KC - 1) / KC;    // float4 of a thread
  constexpr int NH = MIXED && 4 * NQ > M ? 4 * NQ : M;
  real hv[NH], hr = real(0);
  float lv[MIXED ? NH : 1], lr = 0.0f;
  const int len = hi - lo;
  const long long plane = gvar(v, NV, args.vn, args.vt) * args.ncell + lbase;
  const real *src;
  if constexpr (MIXED) src = args.Uh + plane;
  else src = args.U + plane;
  const float *srl = MIXED && two ? args.Ul + plane : nullptr;
  const bool vec = MIXED && cs == 1 &&
                   ((reinterpret_cast<unsigned long long>(src + lo) |
                     reinterpret_cast<unsigned long long>(two ? srl + lo : nullptr)) & 15) == 0;
  const int nq = len >> 2;               // whole float4 of the segment
  // the extra cell of this thread: segment cell cx, or none (k >= 7 or past a tail)
  const int cx = k < 2 ? k - 2 : (k < 4 ? len + k - 2 : 4 * nq + k - 4);
  const bool extra = k < 4 || (vec && k < 7 && cx < len);
  const bool loads = S::SIDES == 1 || sidew == 0;
  if (loads && extra) {
    const int i = lo + cx;
    bool neg = false;
    long long a = (long long)i * cs;
    if (i < 0 || i >= n) a = cell_addr(v, i, neg) - plane;   // ghost cell
    hr = src[a];
    if (MIXED && two) lr = srl[a];
    if (neg) { hr = -hr; lr = -lr; }
  }
  if (MIXED && vec) {
    if constexpr (MIXED) {
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        if (k + q * KC < nq) {
          const float4 x = *reinterpret_cast<const float4 *>(src + lo + 4 * (k + q * KC));
          hv[4 * q] = x.x; hv[4 * q + 1] = x.y; hv[4 * q + 2] = x.z; hv[4 * q + 3] = x.w;
          if (two) {
            const float4 y = *reinterpret_cast<const float4 *>(srl + lo + 4 * (k + q * KC));
            lv[4 * q] = y.x; lv[4 * q + 1] = y.y; lv[4 * q + 2] = y.z; lv[4 * q + 3] = y.w;
          }
        }
      }
    }
  } else if (loads && cs == 1) {
    const real *s1 = src + lo + k;
    const float *s2 = MIXED && two ? srl + lo + k : nullptr;
#pragma unroll
    for (int q = 0; q < M; ++q) {
      if (k + q * KC < len) {
        hv[q] = s1[q * KC];
        if constexpr (MIXED) lv[q] = two ? s2[q * KC] : 0.0f;
      }
    }
  } else if (loads) {
    const long long step = KC * cs;
    long long a = (lo + k) * cs;
#pragma unroll
    for (int q = 0; q < M; ++q, a += step) {
      if (k + q * KC < len) {
        hv[q] = src[a];
        if constexpr (MIXED) lv[q] = two ? srl[a] : 0.0f;
      }
    }
  }

  // ------------------------------------------------ reference state (mixed)
  // The mixed form reconstructs the differences ubar - R from a reference
  // state R of the line (shift invariance of eq. (CWENO-FV): every row's
  // coefficients and right-hand side weights sum to one, the indicators of
  // eq. (weight) see differences only) and evaluates the fluxes as F - F(R)
  // where the face states lie near R, so that FP32 rounding is relative to
  // |U - R| rather than |U|.  R: per variable the median of five sampled
  // cells (hi parts), the same in every CTA of the line.  The plain FP32 form
  // on the hi parts (R = 0) stays where the difference form cannot help:
  // lines whose sampled densities or energies spread beyond a factor 4 of R
  // (strong jumps, vacuum), and lines flat to FP32 precision (every
  // variable's samples within 2^-20 of its scale: R's magnitude, for the
  // momenta at least sqrt(rho_R E_R)).  A face whose states are farther than
  // half of R's density or energy from R is evaluated in full.  The
  // characteristic-wise path (PRE) takes its face values from outside and
  // keeps R = 0.  All in FP32: FP64 instructions here would cost each CTA
  // thousands of cycles on GB300's FP64 pipe while its other warps wait.
  bool dlt = false;
  if constexpr (MIXED && !PRE) {
    if (two && tid < NV) {
      const int kv = tid;
      // the median of the hi parts by rank (ties by index), picked by
      // unrolled selects (no run-time indexing of the arrays)
      float mh = 0.0f, ml = 0.0f;
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        int below = 0;
#pragma unroll
        for (int r = 0; r < 5; ++r) below += (sh[r] < sh[q]) || (sh[r] == sh[q] && r < q);
        if (below == 2) { mh = sh[q]; ml = sl[q]; }
      }
      bool gate = true;
      float spread = 0.0f;
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        if (kv == 0 || kv == NV - 1) gate = gate && sh[q] >= 0.25f * mh && sh[q] <= 4.0f * mh;
        spread = fmaxf(spread, fabsf(sh[q] - mh));
      }
      if (kv == 0 || kv == NV - 1) gate = gate && mh > 0.0f;
      ex.rh[kv] = mh;
      ex.rl[kv] = ml;
      ex.rf[kv] = mh + ml;
      ex.rgate[kv] = gate ? 1 : 0;
      ex.rspread[kv] = spread;
    }
  }
  if constexpr (MIXED) __syncthreads();   // the samples' verdict
  if constexpr (MIXED) eps_pos = ex.epsf;
  if constexpr (MIXED && !PRE) {
    if (two) {
      const float mom = sqrtf(fabsf(ex.rf[0] * ex.rf[NV - 1]));
      bool flat = true;
#pragma unroll
      for (int kv = 0; kv < NV; ++kv) {
        const float scale = (kv == 0 || kv == NV - 1) ? fabsf(ex.rf[kv]) : fmaxf(fabsf(ex.rf[kv]), mom);
        flat = flat && ex.rspread[kv] <= 9.5367432e-07f * scale;   // 2^-20
      }
      dlt = ex.rgate[0] && ex.rgate[NV - 1] && !flat;
    }
    if (dlt && tid == 0) {
      // F(R) and (u_R, v_R, p_R, E_R + p_R), FP32 (O(1) factors of the
      // difference terms; F(R) only meets fluxes of full-form faces)
      const float r0 = ex.rf[0], m = ex.rf[1], t = NV == 4 ? ex.rf[2] : 0.0f;
      const float E = ex.rf[NV - 1];
      const float ir = 1.0f / r0;
      const float u = m * ir, vv = t * ir;
      const float pr = (args.gamma_f - 1.0f) * (E - 0.5f * (m * u + t * vv));
      ex.rF[0] = m;
      ex.rF[1] = m * u + pr;
      if (NV == 4) ex.rF[2] = t * u;
      ex.rF[NV - 1] = (E + pr) * u;
      ex.rp[0] = u;
      ex.rp[1] = vv;
      ex.rp[2] = pr;
      ex.rp[3] = E + pr;
    }
  }
  if (loads) {
    real *dst = Us + v * UWP + UH;
    float rh = 0.0f, rl = 0.0f;
    if (dlt) { rh = ex.rh[v]; rl = ex.rl[v]; }
    // (hi - R_hi) + (lo - R_lo), exact where hi and R_hi are within a
    // factor of two of each other
    auto val = [&](real x, float l) -> real {
      if constexpr (MIXED) return dlt ? (x - rh) + (l - rl) : x;
      else return x;
    };
    if (MIXED && vec) {
      if constexpr (MIXED) {
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          if (k + q * KC < nq) {
            float *d = dst + S::pad(4 * (k + q * KC));
#pragma unroll
            for (int e = 0; e < 4; ++e) d[e] = val(hv[4 * q + e], lv[4 * q + e]);
          }
        }
      }
    } else {
#pragma unroll
      for (int q = 0; q < M; ++q)
        if (k + q * KC < len) dst[S::pad(k + q * KC)] = val(hv[q], lv[MIXED ? q : 0]);
    }
    if (extra) dst[S::pad(cx)] = val(hr, lr);
    if constexpr (MIXED && !PRE) {
      if (k == 1 || k == 2) ex.hend[k - 1][v] = hr;
    }
    for (int c = len + 2 + k; c < SEG + 2; c += KC) dst[S::pad(c)] = real(0);   // past the line
  }
  __syncthreads();
  (void)dlt;
  // epsilon of eq. (weight) for this thread's variable v.  The difference
  // form's indicators see U - R, but the rounding noise the FP32 stages
  // leave in the state scales with |U| wherever a line or a face took the
  // plain form; the floor therefore keeps the reference's share,
  // 2^20 u^2 (R^2 + max|U - R|^2) >= 2^19 u^2 max|U|^2 over the stencil
  real eps_v = eps_w;
  if constexpr (MIXED) {
    if (dlt) eps_v = eps_w + FP32_BETA_FLOOR * ex.rf[v] * ex.rf[v];
  }


  // face values computed outside (the characteristic-wise reconstruction):
  // U^- and U^+ of the segment's cells in the state's layout
  if constexpr (PRE) {
    // A stage may update the state in place, and the halo cells loaded above are
    // the neighbours' cells: no CTA of the line writes before all have loaded
    // (arrive here, wait before the update; the other kernels meet at the joins).
    if (MODE != MODE_XSWEEP && R > 1) cluster_arrive();
    const real *pm = reinterpret_cast<const real *>(args.Fm_pre);
    const real *pp = reinterpret_cast<const real *>(args.Fp_pre);
    const int c0 = lo > 0 || per ? -1 : 0, c1 = hi - lo + (hi < n || per ? 1 : 0);
    for (int c = c0 + k; c < c1; c += KC) {
      bool neg;
      const long long o = cell_addr(v, lo + c, neg);
      Fm[v * FWP + FH + S::pad(c)] = pm[o];
      Fp[v * FWP + FH + S::pad(c)] = pp[o];
    }
  } else {
    // ---------------------------------------------------------------- solve
    // this thread's chunk: cells lo + k M .. of variable v
    real *Zm = reinterpret_cast<real *>(smem_raw + S::zm_off);
    real *Zp = reinterpret_cast<real *>(smem_raw + S::zp_off);
    real *Cr = reinterpret_cast<real *>(smem_raw + S::cr_off);
    real *Xs = reinterpret_cast<real *>(smem_raw + S::xs_off);
    const real *uv = Us + v * UWP + UH;         // u of segment cell c at uv[pad(c)], c in [-2, SEG+2)
    const int cb = S::pad(k * M);               // padded offset of the chunk's first cell
    const int w0 = lo + (k & ~31) * M;          // first cell of the warp's chunks
    const bool wlive = w0 < n;                  // (uniform over the warp)
    constexpr bool TREE = S::TREE;
    using P = typename Pair<real>::t;
    P cs[M - 1];
    // The last segment of a periodic line may hold one cell, whose unknown is
    // its first and its last: both seams then take the one of the ring's closure.
    const bool lone = per && R > 1 && n % SEG == 1;
    // After the back substitution: the face values of the two cells next to the
    // segment are known here as well (the unknowns outside its ends), so this CTA
    // limits those cells itself and needs nothing more from its neighbours; and
    // the segment's own end cells take the same numbers as there.  A lane per
    // value (out: the cell outside, right: that end, plus: that system).
    auto seam_faces = [&](bool act, bool out, bool right, bool plus) {
      if (KC > 32 && (k & ~31) != (right ? ((len - 1) / M & ~31) : 0)) return;
      if (!act || !(per || (right ? hi < n : lo > 0))) return;
      int r = rank;
      if (!out) r = right ? (rank == R - 1 ? 0 : rank + 1) : (rank == 0 ? R - 1 : rank - 1);
      bool y = (right == plus) != out;
      if (TREE && lone && r == R - 2 && y != plus) { r = 0; y = plus; }
      const real *x = reinterpret_cast<const real *>(&ex.ends[2 * v + plus][r]);
      const int at = S::pad((right ? len - 1 : 0) + (out ? (right ? 1 : -1) : 0));
      (plus ? Fp : Fm)[v * FWP + FH + at] = uv[at] + x[y];
    };
    if constexpr (S::SIDES == 2) {
      auto solve = [&](auto side_c) {
        constexpr int SD = decltype(side_c)::value;
        real *dd = (SD ? Fp : Fm) + v * FWP + FH, *ff = (SD ? Zp : Zm) + v * WP + cb;
        double c1[M - 1];
        Run<real> r = run_empty<real>();
        if (wlive) {
          real D[M + 3], S0[M], S1[M], S2[M], win[M + 4];
          win[0] = uv[S::pad(k * M - 2)];
          win[1] = uv[S::pad(k * M - 1)];
#pragma unroll
          for (int q = 0; q < M; ++q) win[q + 2] = uv[cb + q];
          win[M + 2] = uv[S::pad(k * M + M)];
          win[M + 3] = uv[S::pad(k * M + M + 1)];
          chunk_weights<real, M>(win, eps_v, D, S0, S1, S2);
          side_eliminate<SD, M>(D, S0, S1, S2, {lo + k * M, n, per}, dd + cb, ff, c1, r);
        }
        Ends<real> F, L;
        if (lo + k * M < n) {
          L.a = r.D; L.b = r.C; L.g = r.F;
          F.a = fma(-r.G, L.a, r.A);
          F.b = fma(-r.G, L.g, r.B);
          F.g = -r.G * L.b;
        } else {
          F.a = F.b = L.a = L.b = real(0);
          F.g = L.g = real(-1);
        }
        const Ends<real> own = L;
        Step<real> st[5];
#pragma unroll
        for (int h = 0; h < 5; ++h) {
          const bool up = lane & (1 << h);
          tree_up(1 << h, SD ? !up : up, false, real(1), F, L, st[h]);
        }
        real xl = real(0), xr = real(0);
        if (R > 1) {
          if (lane == 0) {
            Run<real> &a = ex.seg[2 * v + SD];
            a.A = F.a; a.B = F.b; a.G = F.g; a.D = L.a; a.C = L.b; a.F = L.g;
          }
          cluster.sync();
          const int q = lane & 15;
          Run<real> o = run_empty<real>();
          if (q < R) o = cluster.map_shared_rank(&ex, SD ? R - 1 - q : q)->seg[2 * v + SD];
          F.a = o.A; F.b = o.B; F.g = o.G;
          L.a = o.D; L.b = o.C; L.g = o.F;
          Step<real> sg[4];
#pragma unroll
          for (int h = 0; h < 4; ++h)
            if ((1 << h) < R) tree_up(1 << h, (q & (1 << h)) != 0, false, real(1), F, L, sg[h]);
          if (per) ring_close(F, L, xl, xr);
#pragma unroll
          for (int h = 3; h >= 0; --h)
            if ((1 << h) < R) tree_down((q & (1 << h)) != 0, false, sg[h], xl, xr);
          if (lane < R) ex.ends[2 * v + SD][SD ? R - 1 - q : q] = p_set(xl, xr);
          __syncwarp();
          const P x = ex.ends[2 * v + SD][rank];
          xl = x.x;
          xr = x.y;
        } else if (per) {
          ring_close(F, L, xl, xr);
          if (lane == 0) ex.ends[2 * v + SD][0] = p_set(xl, xr);
        }
#pragma unroll
        for (int h = 4; h >= 0; --h) {
          const bool up = lane & (1 << h);
          tree_down(SD ? !up : up, false, st[h], xl, xr);
        }
        if (wlive) {
          const real xo = fma(-own.b, xr, fma(-own.g, xl, own.a));
          side_back<SD, M>(uv + cb, dd + cb, ff, c1, xl, xo, n - (lo + k * M));
          __syncwarp();
          seam_faces(lane < 4, lane & 1, lane & 2, SD);
        }
      };
      if (sidew) solve(std::integral_constant<int, 1>());
      else solve(std::integral_constant<int, 0>());
    } else {
    Run<real> rm = run_empty<real>(), rp = run_empty<real>();
    if (wlive) {
      {
        real D[M + 3], S0[M], S1[M], S2[M];
        {
          real win[M + 4];   // the chunk's cells with a two-cell halo
          win[0] = uv[S::pad(k * M - 2)];
          win[1] = uv[S::pad(k * M - 1)];
#pragma unroll
          for (int q = 0; q < M; ++q) win[q + 2] = uv[cb + q];
          win[M + 2] = uv[S::pad(k * M + M)];
          win[M + 3] = uv[S::pad(k * M + M + 1)];
          chunk_weights<real, M>(win, eps_v, D, S0, S1, S2);
        }
        const EdgeInfo e = {lo + k * M, n, per};
        real *dm = Fm + v * FWP + FH + cb, *dp = Fp + v * FWP + FH + cb;
        real *zm = Zm + v * WP + cb, *zp = Zp + v * WP + cb;
        // a warp without a line end skips the edge rows' tests
        if (w0 + 32 * M >= n || (w0 == 0 && !per))
          chunk_eliminate<real, M, true>(D, S0, S1, S2, e, dm, zm, dp, zp, cs, rm, rp);
        else
          chunk_eliminate<real, M, false>(D, S0, S1, S2, e, dm, zm, dp, zp, cs, rm, rp);
      }
      if constexpr (!TREE) {
      real *cm = Cr + (2 * v) * 6 * S::KCP + k + (k >> 3), *cp = cm + 6 * S::KCP;
      cm[0] = rm.A; cm[S::KCP] = rm.B; cm[2 * S::KCP] = rm.G;
      cm[3 * S::KCP] = rm.D; cm[4 * S::KCP] = rm.F; cm[5 * S::KCP] = rm.C;
      cp[0] = rp.A; cp[S::KCP] = rp.B; cp[2 * S::KCP] = rp.G;
      cp[3 * S::KCP] = rp.D; cp[4 * S::KCP] = rp.F; cp[5 * S::KCP] = rp.C;
      }
    }

    P xin, xown;   // the unknown before the chunk, its own last one
    if constexpr (TREE) {
      // ----------------------------------------- a warp per variable: trees
      // over the warp's 32 chunks, then (16 lanes per side) over the
      // segments of the cluster
      Ends<P> F, L;
      if (lo + k * M < n) {   // from first in terms of the chunk's own last to both ends
        const P g = p_set(-rm.G, -rp.G);
        const P f = p_set(rm.F, rp.F), c = p_set(rm.C, rp.C);
        L.a = p_set(rm.D, rp.D); L.b = c; L.g = f;
        F.a = p_fma(g, L.a, p_set(rm.A, rp.A));
        F.b = p_fma(g, f, p_set(rm.B, rp.B));
        F.g = p_mul(g, c);
      } else {
        F.a = F.b = L.a = L.b = p_set(real(0), real(0));
        F.g = L.g = p_set(-real(1), -real(1));
      }
      const Ends<P> own = L;
      const P one = p_set(real(1), real(1));
      Step<P> st[5];
#pragma unroll
      for (int h = 0; h < 5; ++h) {
        const bool r = lane & (1 << h);
        tree_up(1 << h, r, !r, one, F, L, st[h]);
      }
      P xl = p_set(real(0), real(0)), xr = p_set(real(0), real(0));
      if (R > 1) {
        if (lane == 0) {
          Run<real> &a = ex.seg[2 * v], &b = ex.seg[2 * v + 1];
          a.A = F.a.x; a.B = F.b.x; a.G = F.g.x; a.D = L.a.x; a.C = L.b.x; a.F = L.g.x;
          b.A = F.a.y; b.B = F.b.y; b.G = F.g.y; b.D = L.a.y; b.C = L.b.y; b.F = L.g.y;
        }
        cluster.sync();
        // lane: side sd, walk position q among the segments
        const int sd = lane >> 4, q = lane & 15;
        Run<real> o = run_empty<real>();
        if (q < R) o = cluster.map_shared_rank(&ex, sd ? R - 1 - q : q)->seg[2 * v + sd];
        Ends<real> f, l;
        f.a = o.A; f.b = o.B; f.g = o.G;
        l.a = o.D; l.b = o.C; l.g = o.F;
        Step<real> sg[4];
#pragma unroll
        for (int h = 0; h < 4; ++h)
          if ((1 << h) < R) tree_up(1 << h, (q & (1 << h)) != 0, false, real(1), f, l, sg[h]);
        real yl = real(0), yr = real(0);
        if (per) ring_close(f, l, yl, yr);
#pragma unroll
        for (int h = 3; h >= 0; --h)
          if ((1 << h) < R) tree_down((q & (1 << h)) != 0, false, sg[h], yl, yr);
        if (q < R) ex.ends[2 * v + sd][sd ? R - 1 - q : q] = p_set(yl, yr);
        __syncwarp();
        const P xm = ex.ends[2 * v][rank], xp = ex.ends[2 * v + 1][rank];
        xl = p_set(xm.x, xp.x);
        xr = p_set(xm.y, xp.y);
      } else if (per) {
        Ends<real> f, l;
        const bool p = lane & 1;   // even lanes close the minus ring, odd lanes the plus ring
        f.a = p ? F.a.y : F.a.x; f.b = p ? F.b.y : F.b.x; f.g = p ? F.g.y : F.g.x;
        l.a = p ? L.a.y : L.a.x; l.b = p ? L.b.y : L.b.x; l.g = p ? L.g.y : L.g.x;
        real yl, yr;
        ring_close(f, l, yl, yr);
        if (lane < 2) ex.ends[2 * v + lane][0] = p_set(yl, yr);
        xl = p_set(__shfl_sync(0xffffffffu, yl, 0), __shfl_sync(0xffffffffu, yl, 1));
        xr = p_set(__shfl_sync(0xffffffffu, yr, 0), __shfl_sync(0xffffffffu, yr, 1));
      }
#pragma unroll
      for (int h = 4; h >= 0; --h) {
        const bool r = lane & (1 << h);
        tree_down(r, !r, st[h], xl, xr);
      }
      xin = xl;
      xown = p_fma(p_neg(own.b), xr, p_fma(p_neg(own.g), xl, own.a));
    } else {
      __syncthreads();
    // ------------------------------------------- the segment's chunks
    // LPS lanes per system (variable and side), eight chunks each in walk
    // order.  Within a lane the chunks' last unknowns l_q are eliminated one
    // after another, l_q = Dt - Ft X_in - Ct l_{q+1}; the lanes' runs are
    // joined by a butterfly, every lane keeping the meeting points on its
    // path, so that the way down needs no exchange.  Serial work on one or
    // two warps (the other CTAs of the SM fill the pipes meanwhile): a
    // parallel cyclic reduction over the 32 chunks of a warp would take 4
    // times the instructions.  Chunks beyond the line end (the last segment's)
    // are left out: q0 .. q1 are the lane's chunks with cells; a lane without
    // any is the empty run.
    constexpr int LPS = S::LPS;
    constexpr int NCOMB = (2 * NV * LPS + 31) / 32 * 32;
    // (which warps: in turn by CTA, as an FP64 instruction of a warp holds the
    // FP64 unit of its SM quarter for 64 cycles, whatever the others do)
    const int ct = (tid + T - (NCOMB == 32 ? (int)(blockIdx.x % NV) * 32 : 0)) % T;
    const bool comb = ct < NCOMB;
    const bool on = ct < 2 * NV * LPS;
    const int sys = on ? ct / LPS : 0, cl = ct % LPS, sd = sys & 1;
    real Dt[7], Ft[7], Ct[7];
    Run<real> run = run_empty<real>(), seg;
    Cut<real> cut[3];
    const int nlive = (hi - lo + M - 1) / M;
    const int q0 = sd ? max(0, KC - nlive - 8 * cl) : 0;
    const int q1 = sd ? 7 : min(8, nlive - 8 * cl) - 1;
    if (comb) {
      const real *cr = Cr + sys * 6 * S::KCP;
      real al = real(0), be = real(0), ga = real(-1);
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (q < q0 || q > q1) continue;
        const int kw = 8 * cl + q, kk = sd ? KC - 1 - kw : kw;
        const real *c = cr + kk + (kk >> 3);
        const real cA = c[0], cB = c[S::KCP], cG = c[2 * S::KCP];
        const real cD = c[3 * S::KCP], cF = c[4 * S::KCP], cC = c[5 * S::KCP];
        if (q == q0) {
          run.D = cD; run.F = cF; run.C = cC;
          al = cA; be = cB; ga = cG;
        } else {
          const real i1 = rcp(fma(-run.C, cB, real(1)));
          const real dt_ = fma(-run.C, cA, run.D) * i1, ft = run.F * i1, ct = -(run.C * cG) * i1;
          if (q > 0) { Dt[q - 1] = dt_; Ft[q - 1] = ft; Ct[q - 1] = ct; }
          al = fma(-ga, dt_, al);
          be = fma(-ga, ft, be);
          ga = -(ga * ct);
          const real i2 = rcp(fma(-cF, ct, real(1)));
          run.D = fma(-cF, dt_, cD) * i2;
          run.F = -(cF * ft) * i2;
          run.C = cC * i2;
        }
      }
      if (q0 <= q1) {
        run.A = fma(-ga, run.D, al);
        run.B = fma(-ga, run.F, be);
        run.G = -(ga * run.C);
      }
      seg = run;
#pragma unroll
      for (int d = 1, h = 0; d < LPS; d <<= 1, ++h) {
        const Run<real> o = run_shfl_xor(seg, d, LPS);
        const bool rt = cl & d;
        seg = run_join(rt ? o : seg, rt ? seg : o, cut[h]);
      }
      if (on && cl == 0) ex.seg[sys] = seg;
      __syncwarp();
    }
    if (R > 1) cluster.sync();
    if (comb) {
      // The seams at either end of the segment: the runs before and after a
      // seam from the ends of the line, lane 0 joining the segments forwards,
      // lane 1 backwards, so that the neighbour comes to the same two runs.
      // Needed of them is the end at the seam alone (t: its value, the
      // coefficient of the line's far end and of the unknown across the seam),
      // without (e) and with this segment (w).  Periodic: both lanes go on to the
      // whole line, whose ring gives the unknowns at its two ends.
      const int wpos = sd ? R - 1 - rank : rank;
      real e1 = real(0), e2 = real(-1), e3 = real(0), w1 = e1, w2 = e2, w3 = e3;
      real el = real(0), er = real(0);   // before the first and after the last cell (bounded: no weight)
      {
        real t1 = e1, t2 = e2, t3 = e3;
        const int cnt = cl > 1 ? 0 : (per ? R : (cl == 0 ? wpos + 1 : R - wpos));
#pragma unroll 1
        for (int q = 0; q < cnt; ++q) {
          const int at = cl == 0 ? q : R - 1 - q;
          const Run<real> &o = cluster.map_shared_rank(&ex, sd ? R - 1 - at : at)->seg[sys];
          if (at == wpos) { e1 = t1; e2 = t2; e3 = t3; }
          // the next segment's end facing the seam, a - b (across) - g (beyond),
          // and its other one, a2 - f (across) - c (beyond)
          const real a2 = cl == 0 ? o.D : o.A, f = cl == 0 ? o.F : o.G, c = cl == 0 ? o.C : o.B;
          if (q == 0) {
            t1 = a2; t2 = f; t3 = c;
          } else {
            const real a = cl == 0 ? o.A : o.D, b = cl == 0 ? o.B : o.C, g = cl == 0 ? o.G : o.F;
            const real i = rcp(fma(-t3, b, real(1))), fi = f * i;
            t1 = fma(-fi, fma(-t3, a, t1), a2);
            t2 = -(fi * t2);
            t3 = fma(fi, t3 * g, c);
          }
          if (at == wpos) { w1 = t1; w2 = t2; w3 = t3; }
        }
        if (per) {
          Ends<real> f, l;
          l.a = __shfl_sync(0xffffffffu, t1, 0, LPS); l.g = __shfl_sync(0xffffffffu, t2, 0, LPS);
          l.b = __shfl_sync(0xffffffffu, t3, 0, LPS);
          f.a = __shfl_sync(0xffffffffu, t1, 1, LPS); f.g = __shfl_sync(0xffffffffu, t2, 1, LPS);
          f.b = __shfl_sync(0xffffffffu, t3, 1, LPS);
          ring_close(f, l, el, er);
        }
      }
      // lane 0: the seam before the segment, lane 1: the one after it; (o) the
      // run across it; last of the earlier run and first of the later one
      const real o1 = __shfl_xor_sync(0xffffffffu, w1, 1, LPS), o2 = __shfl_xor_sync(0xffffffffu, w2, 1, LPS);
      const real o3 = __shfl_xor_sync(0xffffffffu, w3, 1, LPS);
      const real ea = fma(-e2, cl == 0 ? el : er, e1), oa = fma(-o2, cl == 0 ? er : el, o1);
      const real i1 = rcp(fma(-e3, o3, real(1)));
      const real ye = fma(-e3, oa, ea) * i1, yo = fma(-o3, ea, oa) * i1;
      real sl = cl == 0 ? ye : yo, sf = cl == 0 ? yo : ye;
      if (wpos == (cl == 0 ? 0 : R - 1)) { sl = el; sf = er; }
      // a last segment of one cell (see lone)
      if (lone) {
        if (sd == 0 && wpos == (cl == 0 ? R - 1 : R - 2)) sf = el;
        if (sd == 1 && wpos == (cl == 0 ? 1 : 0)) sl = er;
      }
      real xl = __shfl_sync(0xffffffffu, sl, 0, LPS), xr = __shfl_sync(0xffffffffu, sf, 1, LPS);
      if (on && cl < 2) {
        const int w = (cl == 0) == (sd != 0) ? rank + 1 : rank - 1, rw = w < 0 ? R - 1 : (w == R ? 0 : w);
        ex.ends[sys][cl == 0 ? rank : rw].x = sl;
        ex.ends[sys][cl == 0 ? rw : rank].y = sf;
        if (cl == 0) Xs[sys * S::XP] = xl;
      }
#pragma unroll
      for (int h = 2; h >= 0; --h) {
        if ((1 << h) < LPS) {
          const Cut<real> &c = cut[h];
          const real l = fma(c.q, xr, fma(-c.p, xl, c.u)), f = fma(-c.s, xr, fma(c.r, xl, c.v));
          if (cl & (1 << h)) xl = l;
          else xr = f;
        }
      }
      real x = fma(-run.C, xr, fma(-run.F, xl, run.D));
      real *xs = Xs + sys * S::XP;
#pragma unroll
      for (int q = 7; q >= 0; --q) {
        if (q < 7 && q < q1 && q >= q0) x = fma(-Ct[q], x, fma(-Ft[q], xl, Dt[q]));
        if (q < q0) x = xl;   // what the first chunk with cells sees before it
        const int pos = 8 * cl + q + 1;
        if (on) xs[pos + (pos >> 3)] = x;
      }
    }
      __syncthreads();
      const real *xm = Xs + (2 * v) * S::XP, *xp = xm + S::XP;
      const int m0 = k, m1 = k + 1, p0 = KC - 1 - k, p1 = KC - k;
      xin = p_set(xm[m0 + (m0 >> 3)], xp[p0 + (p0 >> 3)]);
      xown = p_set(xm[m1 + (m1 >> 3)], xp[p1 + (p1 >> 3)]);
    }

    // ------------------------------------------- back substitution
    if (wlive) {
      const int o = v * WP + cb, of = v * FWP + FH + cb, mine = n - (lo + k * M);
      if (w0 + 32 * M > n)
        chunk_back<real, M, true>(uv + cb, Fm + of, Zm + o, Fp + of, Zp + o, cs, xin, xown, mine);
      else
        chunk_back<real, M, false>(uv + cb, Fm + of, Zm + o, Fp + of, Zp + o, cs, xin, xown, mine);
      __syncwarp();   // (a lane past a ragged end may have written its idle slots)
      if (R > 1 || per) seam_faces(lane < 8, lane & 1, lane & 4, lane & 2);
    }
    }
    // This CTA has read its neighbours' runs: arrive now, wait before exit (a
    // CTA's shared memory must outlive the reads of its run).  A relaxed arrival
    // does not wait for loads in flight, so it has to follow the use of every
    // value read from another CTA: each passes a join's shuffle or arithmetic
    // above, whose result the back substitution has consumed.
    if (R > 1) cluster_arrive_relaxed();
  }
  __syncthreads();

  // ---------------------------------------------------------------- limit
  // Cells of the segment and, where the line goes on, the two next to it
  // (their theta counts belong to the neighbours).
  unsigned int t1 = 0, t2 = 0;
  const real inv12 = rcp(real(1) - real(2) * wgl);
  // difference form: the face values hold U - R until a cell is limited,
  // then the limited values in full (cfull[c] = 1)
  float rf[NV];
#pragma unroll
  for (int kv = 0; kv < NV; ++kv) rf[kv] = dlt ? ex.rf[kv] : 0.0f;
  int anyfull = 0;   // this thread limited a cell (difference form)
  if (args.limiter) {
    // FP32 pretest of every cell of this thread (a superset of the cells
    // the exact test limits: its thresholds carry twice the FP32 round-off
    // allowance, which covers the FP32 evaluation and, in the FP64 form, the
    // rounding of the inputs to FP32); the flagged cells (rare) are limited
    // exactly in a second loop, so the pretest loop carries no FP64 state
    static_assert(SEG + 2 <= 32 * T, "one mask bit per cell of a thread");
    const int c0 = tid - (lo > 0 || per ? 1 : 0), c1 = hi - lo + (hi < n || per ? 1 : 0);
    unsigned int mask = 0;
    const float wgl_f = float(wgl), inv12_f = float(inv12), eps_f = float(eps_pos);
#pragma unroll 1
    for (int q = 0, c = c0; c < c1; ++q, c += T) {
      float ub[NV], a[NV], b[NV];
      const int pc = S::pad(c);
#pragma unroll
      for (int kv = 0; kv < NV; ++kv) {
        ub[kv] = to_f32(Us[kv * UWP + UH + pc]);
        a[kv] = to_f32(Fm[kv * FWP + FH + pc]);
        b[kv] = to_f32(Fp[kv * FWP + FH + pc]);
      }
      float full[NV], dm[NV], dp[NV];
#pragma unroll
      for (int kv = 0; kv < NV; ++kv) {
        full[kv] = ub[kv] + rf[kv];
        dm[kv] = a[kv] - ub[kv];
        dp[kv] = b[kv] - ub[kv];
      }
      if (limit_box_free<NV>(full, dm, dp, wgl_f, eps_f)) continue;
#pragma unroll
      for (int kv = 0; kv < NV; ++kv) {
        a[kv] += rf[kv];
        b[kv] += rf[kv];
      }
      if (limit_need_mixed<NV>(full, a, b, wgl_f, inv12_f, eps_f)) mask |= 1u << q;
    }
#pragma unroll 1
    while (mask) {
      const int q = __ffs(mask) - 1;
      mask &= mask - 1;
      const int c = c0 + q * T, pc = S::pad(c);
      real ub[NV], a[NV], b[NV];
#pragma unroll
      for (int kv = 0; kv < NV; ++kv) {
        ub[kv] = Us[kv * UWP + UH + pc];
        a[kv] = Fm[kv * FWP + FH + pc];
        b[kv] = Fp[kv * FWP + FH + pc];
      }
      if constexpr (MIXED) {
        if (dlt) {
          // the average as the plain form has it (the FP32 hi part, not
          // R + (ubar - R): exact relative to ubar however far it is from R)
          // and the face values in full.  A neighbour's cell comes from the
          // load phase: its owner may have updated it in place by now.
          const long long o = lbase + (long long)(lo + c) * cs;
#pragma unroll
          for (int kv = 0; kv < NV; ++kv) {
            ub[kv] = c < 0 ? ex.hend[0][kv]
                     : c >= len ? ex.hend[1][kv]
                                : args.Uh[gvar(kv, NV, args.vn, args.vt) * args.ncell + o];
            a[kv] += rf[kv];
            b[kv] += rf[kv];
          }
        }
      }
      int f;
      if constexpr (MIXED) f = limit_cell_mixed_fp64<NV>(ub, a, b, wgl, eps_pos);
      else f = limit_cell<real, NV>(ub, a, b, wgl, eps_pos, unit_roundoff<real>());
      if (f) {
#pragma unroll
        for (int kv = 0; kv < NV; ++kv) {
          Fm[kv * FWP + FH + pc] = a[kv];
          Fp[kv * FWP + FH + pc] = b[kv];
        }
        if constexpr (MIXED) {
          if (dlt) { cfull[c] = 1; anyfull = 1; }
        }
        if (c >= 0 && c < hi - lo) {
          t1 += f & 1;
          t2 += (f >> 1) & 1;
        }
      }
    }
  }
  // ---------------------------------------------------------------- flux
  // HLLC (or local Lax-Friedrichs) at face f (between cells f-1 and f): the
  // left state is U^- of cell f-1, the right state U^+ of cell f, both in this
  // CTA's shared memory; at the end of a bounded line the exterior state
  // follows from the interior one.  fsmax: the largest |u| + a over this
  // thread's face states; farface: a face of this thread is stored in full.
  real fsmax = real(0);
  int farface = 0;
  if constexpr (MIXED) anyfull = __syncthreads_or(anyfull);
  else __syncthreads();
#pragma unroll 1
  for (int f = lo + tid; f <= hi; f += T) {
    real Ul[NV], Ur[NV], F[NV];
    const int c = f - lo;   // the right cell
    const bool bl = f == 0 && !per, br = f == n && !per;
    {
      const int il = FH + S::pad(c - 1), ir = FH + S::pad(c);
      const real *L = bl ? Fp + ir : Fm + il, *Rr = br ? Fm + il : Fp + ir;
#pragma unroll
      for (int kv = 0; kv < NV; ++kv) {
        Ul[kv] = L[kv * FWP];
        Ur[kv] = Rr[kv * FWP];
      }
    }
    const bool wl = bl && args.bclo == 2, wr = br && args.bchi == 2;   // a wall's mirror state
    real sf;
    bool near = false;
    if constexpr (MIXED) {
      if (dlt) {
        // stored values are U - R (or the limited U in full): both forms of
        // each state
        float dl[NV], dr[NV];
        const bool fulL = anyfull && cfull[bl ? c : c - 1], fulR = anyfull && cfull[br ? c - 1 : c];
#pragma unroll
        for (int kv = 0; kv < NV; ++kv) {
          dl[kv] = Ul[kv];
          dr[kv] = Ur[kv];
          Ul[kv] = fulL ? Ul[kv] : Ul[kv] + rf[kv];
          Ur[kv] = fulR ? Ur[kv] : Ur[kv] + rf[kv];
        }
        if (wl) { Ul[1] = -Ul[1]; dl[1] = -dl[1] - 2.0f * rf[1]; }
        if (wr) { Ur[1] = -Ur[1]; dr[1] = -dr[1] - 2.0f * rf[1]; }
        near = !args.flux && !fulL && !fulR &&
               fabsf(dl[0]) <= 0.5f * rf[0] && fabsf(dr[0]) <= 0.5f * rf[0] &&
               fabsf(dl[NV - 1]) <= 0.5f * rf[NV - 1] && fabsf(dr[NV - 1]) <= 0.5f * rf[NV - 1];
        if (near) hllc_delta<NV>(Ul, Ur, dl, dr, rf, ex.rp, gam, F, sf);
        fdel[c] = near ? 1 : 0;
        farface |= near ? 0 : 1;
      } else {
        if (wl) Ul[1] = -Ul[1];
        if (wr) Ur[1] = -Ur[1];
      }
    } else {
      if (wl) Ul[1] = -Ul[1];
      if (wr) Ur[1] = -Ur[1];
    }
    if (!near) {
      if (args.flux) llf<real, NV>(Ul, Ur, gam, F, sf);
      else hllc<real, NV>(Ul, Ur, gam, F, sf, MIXED || args.fcheck);
    }
    if ((MIXED || args.fcheck) && (sf > fsmax || sf != sf)) fsmax = sf;   // a NaN speed stays
#pragma unroll
    for (int kv = 0; kv < NV; ++kv) Fl[kv * FLS + c] = F[kv];
  }
  // any face of the CTA in full form: only then the update compares the forms
  bool mixedforms = false;
  if constexpr (MIXED) mixedforms = __syncthreads_or(farface) && dlt;
  else __syncthreads();
  (void)mixedforms;

  // ---------------------------------------------------------------- update
  if (PRE && MODE != MODE_XSWEEP && R > 1) cluster_wait();
  // the stage's extrema in the line's arithmetic (converted once per warp)
  real mymin = real(sizeof(real) == 4 ? 3.0e38 : 1.0e300), mymax = real(0);
  unsigned int nbad = 0;
  unsigned long long firstbad = ~0ull;
  const real ih = MIXED ? real(args.ih_f) : real(args.ih);
  const double dt = (MODE == MODE_FINAL && !MIXED) ? ctl->dt : 0.0;
  (void)dt;
  const double gg1 = MIXED ? 0.0 : args.gamma * (args.gamma - 1.0);
  (void)gg1;
  const real *Din = reinterpret_cast<const real *>(args.Din);
  // x-sweep output: thread (v, k) writes cells of its own variable, four at a
  // time on 16-byte boundaries
  int cdone = 0;
  if (MODE == MODE_XSWEEP && !mixedforms) {
    cdone = len;
    if (loads) {
    real *D = reinterpret_cast<real *>(args.Dout) + plane + lo * cs;
    const real *Fv = Fl + v * FLS;
    bool vst = false;
    if constexpr (MIXED) {
      vst = cs == 1 && (reinterpret_cast<unsigned long long>(D) & 15) == 0;
      if (vst) {
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          const int c = 4 * (k + q * KC);
          if (c + 4 <= len) {
            const float4 f = *reinterpret_cast<const float4 *>(Fv + c);
            const float g = Fv[c + 4];
            *reinterpret_cast<float4 *>(D + c) =
                make_float4((f.x - f.y) * ih, (f.y - f.z) * ih, (f.z - f.w) * ih, (f.w - g) * ih);
          }
        }
      }
    }
    const int c0 = vst ? len & ~3 : 0;
    D += (c0 + k) * cs;
    const long long step = KC * cs;
    for (int c = c0 + k; c < len; c += KC, D += step) *D = (Fv[c] - Fv[c + 1]) * ih;
    }
  }
  if (MIXED && MODE == MODE_FINAL) cdone = len;
  for (int c = cdone + tid; c < len; c += T) {
    int i = lo + c;
    long long addr = lbase + (long long)i * cs;
    real Lv[NV];
    // difference form: a face flux stored as F - F(R) next to one stored as F
    // (a limited or distant face state) is put on the same footing
    int fmix = 0;   // 1: only the left face is F - F(R), 2: only the right one
    if constexpr (MIXED) {
      if (mixedforms) fmix = (fdel[c] != fdel[c + 1]) ? (fdel[c] ? 2 : 1) : 0;
    }
#pragma unroll
    for (int kv = 0; kv < NV; ++kv) {
      real fa = Fl[kv * FLS + c], fb = Fl[kv * FLS + c + 1];
      if constexpr (MIXED) {
        if (fmix == 2) fb -= ex.rF[kv];
        else if (fmix == 1) fa -= ex.rF[kv];
      }
      Lv[kv] = (fa - fb) * ih;
      if (MODE != MODE_XSWEEP && Din) Lv[kv] += Din[gvar(kv, NV, args.vn, args.vt) * args.ncell + addr];
    }
    if (MODE == MODE_XSWEEP) {
      real *D = reinterpret_cast<real *>(args.Dout);
#pragma unroll
      for (int kv = 0; kv < NV; ++kv) D[gvar(kv, NV, args.vn, args.vt) * args.ncell + addr] = Lv[kv];
    } else if (MODE == MODE_OPERATOR) {
#pragma unroll
      for (int kv = 0; kv < NV; ++kv) args.Lout[gvar(kv, NV, args.vn, args.vt) * args.ncell + addr] = double(Lv[kv]);
    } else if constexpr (!MIXED) {
      double Ut[NV];
#pragma unroll
      for (int kv = 0; kv < NV; ++kv) {
        int g = gvar(kv, NV, args.vn, args.vt);
        double L = Lv[kv];
        double uk = args.U[g * args.ncell + addr];
        double un;
        if (args.stage == 0) un = uk + dt * L;
        else if (args.stage == 1) un = 0.75 * args.U0[g * args.ncell + addr] + 0.25 * uk + 0.25 * dt * L;
        else un = args.U0[g * args.ncell + addr] * (1.0 / 3.0) + 2.0 / 3.0 * uk + 2.0 / 3.0 * dt * L;
        args.Uout[g * args.ncell + addr] = un;
        Ut[kv] = un;   // line-variable order (no run-time register index)
      }
      // grid momenta: line variable 1 is the normal one (grid index vn)
      double rho = Ut[0], E = Ut[NV - 1];
      double mx = NV == 4 && args.vn != 1 ? Ut[2] : Ut[1];
      double my = NV == 4 ? (args.vn != 1 ? Ut[1] : Ut[2]) : 0.0;
      // one division per cell: 1/rho (1/h from the host)
      const double irho = rcp(rho);
      double e = (E - 0.5 * (mx * mx + my * my) * irho) * irho;
      bool ok = positive(rho) && positive(e) && is_finite(E) && is_finite(mx) && is_finite(my);
      if (!ok) {
        ++nbad;
        firstbad = min(firstbad, (unsigned long long)addr);
      } else {
        mymin = less(rho, mymin) ? rho : mymin;
        double a = root(gg1 * e);
        double rate;
        if (NV == 4) {
          const double ihx = args.vn == 1 ? args.ih : args.ih_other;
          const double ihy = args.vn == 1 ? args.ih_other : args.ih;
          rate = (fabs(mx) * irho + a) * ihx + (fabs(my) * irho + a) * ihy;
        } else {
          rate = (fabs(mx) * irho + a) * args.ih;
        }
        mymax = less(mymax, rate) ? rate : mymax;
      }
    }
  }
  if constexpr (MIXED && MODE == MODE_FINAL) {
    // mixed form in 1-D (2-D combines the two sweeps in a kernel of its own):
    // compensated stage combination on hi + lo pairs; the states of a
    // thread's next cell load while this one is combined
    static_assert(NV == 3, "the 2-D mixed form has no final sweep");
    const dfl third = {0.333333343f, -9.93410776e-09f};
    const dfl two3 = {0.666666687f, -1.98682155e-08f};
    const dfl dtd = ex.dt;
    dfl nk[NV], n0[NV];
    auto fetch = [&](int c) {
#pragma unroll
      for (int kv = 0; kv < NV; ++kv) {
        const long long a = kv * args.ncell + lbase + lo + c;
        nk[kv] = {args.Uh[a], args.Ul[a]};
        if (args.stage != 0) n0[kv] = {args.U0h[a], args.U0l[a]};
      }
    };
    if (tid < len) fetch(tid);
    for (int c = tid; c < len; c += T) {
      dfl uk[NV], u0[NV], un[NV];
#pragma unroll
      for (int kv = 0; kv < NV; ++kv) {
        uk[kv] = nk[kv];
        u0[kv] = n0[kv];
      }
      if (c + T < len) fetch(c + T);
      const int fmix = mixedforms && fdel[c] != fdel[c + 1] ? (fdel[c] ? 2 : 1) : 0;
#pragma unroll
      for (int kv = 0; kv < NV; ++kv) {
        float fa = Fl[kv * FLS + c], fb = Fl[kv * FLS + c + 1];
        if (fmix == 2) fb -= ex.rF[kv];
        else if (fmix == 1) fa -= ex.rF[kv];
        const float L = (fa - fb) * ih;
        const dfl s = df_add(uk[kv], df_mul_f(dtd, L));          // U_k + dt L
        if (args.stage == 0) un[kv] = s;
        else if (args.stage == 1) un[kv] = df_add(df_mul_f(u0[kv], 0.75f), df_mul_f(s, 0.25f));
        else un[kv] = df_add(df_mul(u0[kv], third), df_mul(s, two3));
        const long long a = kv * args.ncell + lbase + lo + c;
        args.Uoh[a] = un[kv].hi;
        args.Uol[a] = un[kv].lo;
      }
      const float rho = un[0].hi, mx = un[1].hi, E = un[2].hi;
      // g = rho E - |m|^2/2 with the compensated parts (its sign decides G)
      const dfl rE = df_mul(un[0], un[2]), m2 = df_mul(un[1], un[1]);
      const dfl gq = df_add(rE, {-0.5f * m2.hi, -0.5f * m2.lo});
      if (!((rho > 0.0f) && (gq.hi > 0.0f) && isfinite(E) && isfinite(mx))) {
        ++nbad;
        firstbad = min(firstbad, (unsigned long long)(lbase + lo + c));
      } else {
        mymin = fminf(mymin, rho);
        const float ir = rcp(rho);
        mymax = fmaxf(mymax, (fabsf(mx) * ir + sqrtf(args.gg1_f * gq.hi) * ir) * ih);
      }
    }
  }

  // ---------------------------------------------------------------- reduce
  // eq. (CFL-CD) checked on the face values: the stage's largest face rate
  // of this direction (max over the step's stages; NaN wins the bit max)
  // (in the line's arithmetic: FP64 instructions cost the FP32 form 1/64 of
  // an issue slot's worth each, and one conversion per warp suffices)
  if (MODE != MODE_OPERATOR && args.fcheck && args.eps_fixed <= 0.0) {
    real fr = fsmax * (MIXED ? real(args.ih_f) : real(args.ih));
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      const real o = shfl_down_r(fr, d);
      if (o > fr || o != o) fr = o;
    }
    if (lane == 0) atomic_max_bits(&ctl->frate[args.fdir], double_bits(double(fr)));
  }
  if (MODE == MODE_FINAL) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      mymin = fmin(mymin, shfl_down_r(mymin, d));
      mymax = fmax(mymax, shfl_down_r(mymax, d));
      nbad += __shfl_down_sync(0xffffffffu, nbad, d);
      t1 += __shfl_down_sync(0xffffffffu, t1, d);
      t2 += __shfl_down_sync(0xffffffffu, t2, d);
      unsigned long long fb = __shfl_down_sync(0xffffffffu, firstbad, d);
      firstbad = fb < firstbad ? fb : firstbad;
    }
    if (lane == 0) {
      atomic_min_bits(&ctl->minrho[args.stage], double_bits(double(mymin)));
      if (args.stage == 2) atomic_max_bits(&ctl->rate, double_bits(double(mymax)));
      if (nbad) {
        atomicAdd(&ctl->nviol, (unsigned long long)nbad);
        atomicMin(&ctl->first_bad, firstbad);
      }
      if (t1) atomicAdd(&ctl->theta1, (unsigned long long)t1);
      if (t2) atomicAdd(&ctl->theta2, (unsigned long long)t2);
    }
  } else if (MODE == MODE_XSWEEP && __any_sync(0xffffffffu, t1 | t2)) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      t1 += __shfl_down_sync(0xffffffffu, t1, d);
      t2 += __shfl_down_sync(0xffffffffu, t2, d);
    }
    if (lane == 0) {
      if (t1) atomicAdd(&ctl->theta1, (unsigned long long)t1);
      if (t2) atomicAdd(&ctl->theta2, (unsigned long long)t2);
    }
  }
  if (!PRE && R > 1) cluster_wait();
}

}  // namespace ppk
