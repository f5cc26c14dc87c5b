// batch_lines.cuh -- descriptors of a batch of independent problems, shared
// by the line kernels and the characteristic-wise reconstruction.
#pragma once

namespace ppk {

// one problem of a batch: its block of the concatenated state (values
// [off, off + nv*ncell), variable planes of ncell cells) and grid
struct ProbDesc {
  long long off, ncell;
  int nx, ny;
  double dx, dy;
  double idx, idy;    // 1/dx, 1/dy
  int bc[4];
};

// one line of a batched launch, resolved (the kernels read one record instead
// of a chain of two): offset of its problem's block, first cell in a plane, cell stride,
// plane size, length, boundaries, inverse cell sizes along and across
struct LineDesc {
  long long off, base, ncell;
  double ih, ih_other;
  float ih_f, ih_other_f;   // FP32 copies (a conversion takes a slot of the FP64 pipe)
  int n, cs, prob;
  short bclo, bchi;
};

}  // namespace ppk
