// sweeps.cuh -- launch helpers shared by the host library and the
// per-precision translation units that instantiate the line kernel.
#pragma once

#include <cuda_runtime.h>

#include "line_sweep.cuh"

namespace ppk {

// Thread layout by chunk length M: a warp per variable, 32 chunks, 32 M cells
// per CTA and at most 16 CTAs (a cluster) per line; and the resident CTAs per
// SM asked for.
constexpr int seg_cells(int m) { return 32 * m; }
//
// FP32 (issue and latency bound): registers of a 16-row chunk allow 4 CTAs of
// four variables without spills (16 warps an SM; 5 CTAs: 2048^2 x sweep 0.32
// against 0.29 ms), 5 of three (1-D Riemann batch step 2.2 against 2.4 ms with
// 4).  FP64 (bound by the FP64 units, one per SM quarter, each held for 64
// cycles by an instruction of one of its warps): warps in multiples of four.
// Three variables with 16-row chunks would put two CTAs of three warps on an
// SM, so they take 8-row chunks on two warps per variable instead (Riemann
// batch 53.2 against 55.8 ms).
template <typename real, int NV, int M>
struct Layout {
  static constexpr bool F32 = sizeof(real) == 4;
  static constexpr bool WIDE = !F32 && NV == 3 && M == 16;
  static constexpr int MM = WIDE ? 8 : M;
  static constexpr int KC = WIDE ? 64 : 32;
  static constexpr int CTAS = F32 ? (M != 16 ? 6 : (NV == 4 ? 4 : 5))
                                  : (M != 8 ? 2 : (NV == 4 ? 3 : 4));
};

struct LaunchCfg {
  int precision;   // 0 fp64, 1 mixed (fp32 line arithmetic)
  int nv;          // 3 or 4
  int mode;        // MODE_*
  bool attrs_only; // set the kernel's attributes, launch nothing
  int m;           // rows per thread chunk: 2, 4, 8 or 16
};

// Launch one sweep over nlines lines with R CTAs per line (cluster of R);
// one entry per (precision, chunk length), in its own translation unit except
// the two short ones.
cudaError_t launch_sweep_f64_short(const LaunchCfg &c, const SweepArgs &a, long long nlines,
                                   cudaStream_t st);
cudaError_t launch_sweep_f64_m8(const LaunchCfg &c, const SweepArgs &a, long long nlines,
                                cudaStream_t st);
cudaError_t launch_sweep_f64_m16(const LaunchCfg &c, const SweepArgs &a, long long nlines,
                                 cudaStream_t st);
cudaError_t launch_sweep_f32_short(const LaunchCfg &c, const SweepArgs &a, long long nlines,
                                   cudaStream_t st);
cudaError_t launch_sweep_f32_m8(const LaunchCfg &c, const SweepArgs &a, long long nlines,
                                cudaStream_t st);
cudaError_t launch_sweep_f32_m16(const LaunchCfg &c, const SweepArgs &a, long long nlines,
                                 cudaStream_t st);

inline cudaError_t launch_sweep(const LaunchCfg &c, const SweepArgs &a, long long nlines,
                                cudaStream_t st) {
  if (c.precision == 0)
    return c.m == 16 ? launch_sweep_f64_m16(c, a, nlines, st)
         : c.m == 8 ? launch_sweep_f64_m8(c, a, nlines, st) : launch_sweep_f64_short(c, a, nlines, st);
  return c.m == 16 ? launch_sweep_f32_m16(c, a, nlines, st)
       : c.m == 8 ? launch_sweep_f32_m8(c, a, nlines, st) : launch_sweep_f32_short(c, a, nlines, st);
}

template <typename real, int NV, int M, int MODE, bool PRE>
cudaError_t launch_m(const SweepArgs &a, long long nlines, cudaStream_t st, bool attrs_only) {
  using Y = Layout<real, NV, M>;
  using S = Smem<real, NV, Y::MM, Y::KC>;
  auto kern = line_sweep<real, NV, Y::MM, Y::KC, MODE, PRE, Y::CTAS>;
  if (attrs_only) {   // called at handle creation, outside any stream capture
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)S::bytes);
    if (e != cudaSuccess) return e;
    // the largest shared-memory carveout, so that the resident-CTA count the
    // kernel is compiled for is not cut by the L1 split
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                             (int)cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(nlines * a.R), 1, 1);
  cfg.blockDim = dim3(S::THREADS, 1, 1);
  cfg.dynamicSmemBytes = S::bytes;
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

// the reconstructing kernel, or the one taking precomputed face values; attrs_only sets the attributes of both
template <typename real, int NV, int M, int MODE>
cudaError_t launch_pre(const LaunchCfg &c, const SweepArgs &a, long long nlines, cudaStream_t st) {
  if (c.attrs_only) {
    cudaError_t e = launch_m<real, NV, M, MODE, true>(a, nlines, st, true);
    if (e != cudaSuccess) return e;
  } else if (a.Fm_pre) {
    return launch_m<real, NV, M, MODE, true>(a, nlines, st, false);
  }
  return launch_m<real, NV, M, MODE, false>(a, nlines, st, c.attrs_only);
}

template <typename real, int M>
cudaError_t launch_dispatch(const LaunchCfg &c, const SweepArgs &a, long long nlines,
                            cudaStream_t st) {
  if (c.nv == 3) {
    if (c.mode == MODE_FINAL)
      return launch_pre<real, 3, M, MODE_FINAL>(c, a, nlines, st);
    if (c.mode == MODE_OPERATOR)
      return launch_pre<real, 3, M, MODE_OPERATOR>(c, a, nlines, st);
    return cudaErrorInvalidValue;
  }
  if (c.nv == 4) {
    if (c.mode == MODE_XSWEEP)
      return launch_pre<real, 4, M, MODE_XSWEEP>(c, a, nlines, st);
    if constexpr (sizeof(real) == 8) {   // (the mixed form combines its two sweeps separately)
      if (c.mode == MODE_FINAL) return launch_pre<real, 4, M, MODE_FINAL>(c, a, nlines, st);
    }
    if (c.mode == MODE_OPERATOR)
      return launch_pre<real, 4, M, MODE_OPERATOR>(c, a, nlines, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace ppk
