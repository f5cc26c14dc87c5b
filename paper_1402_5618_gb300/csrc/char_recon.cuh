// char_recon.cuh -- the characteristic-wise compact-WENO reconstruction of
// one sweep direction (Sec. 2.3, steps 1-4, eqs. (cha-1), (1DEuler-FVC)).
//
// For every line and each side (minus: U^-_{i+1/2}, plus: U^+_{i-1/2}) the
// block tridiagonal system of the line is assembled and solved in one kernel.
// Row of a cell: the Roe average of the two cells adjacent to its face, its
// left eigenvectors l^(k) (eq. (leigenv); the 4 x 4 system with the shear
// field in 2-D), the differences of the characteristic variables l^(k) ubar
// over the five-cell stencil, and per field the WENO-Z weights and the scalar
// row (a, b, c, s); the block row is diag(a, b, c) L.  As in the
// component-wise form the unknowns are the deviations of the face values from
// the cell averages, and bounded lines close the first and last unknown with
// the explicit WENO5-Z value of each characteristic variable at that face.
//
// The solve is partitioned (compact_solve.cuh with blocks): a thread builds
// and eliminates the M rows of a chunk in walk order (minus left to right,
// plus right to left) as a function of the unknowns just outside it, the
// chunks of a warp and the segments of a cluster are joined by trees, and
// every thread substitutes back from its rows' multipliers.  Nothing but the
// state is read and nothing but the face values written, apart from the
// multipliers of many lines.  A walk of each line by one thread, the alternative
// with half the arithmetic, is bound by its own chain wherever the lines are
// not many thousands: per pass, walk against this, 800 positions in FP64 (38
// steps) 664 ms and 18.5, 512^2 FP64 38.4 and 6.9, 2048^2 FP64 207 and 92.5, 4096^2
// mixed 35.5 and 28.8, 2048^2 mixed (three steps) 37.0 and 20.6, 4096 lines of
// 256-8192 cells mixed 186 and 13.3.
//
// The output planes hold U^- and U^+ of every cell in the state's layout and
// grid variable order; the line kernel limits them, evaluates the face
// fluxes and forms the stage update.
#pragma once

#include <cuda_runtime.h>

#include "batch_lines.cuh"

namespace ppk {

struct CharArgs {
  const void *U;            // stage input: planes [nv][ncell] of the line's arithmetic
                            // (FP64, or the FP32 hi parts of the mixed form)
  void *Um, *Up;            // out: U^-_{i+1/2}, U^+_{i-1/2} of every cell, same layout and type
  long long ncell;          // cells per variable plane
  long long nlines;
  long long cell_stride, line_stride;
  int n;                    // cells per line; batched: the longest line
  int vn, vt;               // grid index of the normal / tangential momentum (vt < 0 in 1-D)
  int bclo, bchi;
  int M, R;                 // rows per chunk, one-warp CTAs per line and side (n <= 32 M R)
  int T;                    // rows of every chunk held in shared memory at a time: a power of
                            // two that divides M, M itself without scratch (M <= 16)
  void *scr;                // multipliers, char_scratch_values() values of the line's type, or
                            // nullptr: in shared memory
  double gamma, eps_weno;
  const LineDesc *lines;    // batched launch: the group's lines (nullptr: one problem)
};

// scratch values: per row of every chunk the blocks Y and F and the vector g
inline long long char_scratch_values(const CharArgs &a, int nv) {
  return a.nlines * 2 * a.R * 32 * a.M * (2 * nv * nv + nv);
}

// one entry per precision, each in its own translation unit (the FP32 one
// is compiled with the mixed form's fast division and square root);
// attrs_only sets the kernels' attributes and launches nothing
cudaError_t launch_char_recon_f64(const CharArgs &a, int nv, cudaStream_t st, bool attrs_only);
cudaError_t launch_char_recon_f32(const CharArgs &a, int nv, cudaStream_t st, bool attrs_only);

}  // namespace ppk
