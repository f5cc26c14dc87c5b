// FP64 instantiations of the fused line kernel with 2- and 4-row thread
// chunks: short lines, and few lines spread over more SMs.
#include "sweeps.cuh"

namespace ppk {
cudaError_t launch_sweep_f64_short(const LaunchCfg &c, const SweepArgs &a, long long nlines,
                                   cudaStream_t st) {
  return c.m == 2 ? launch_dispatch<double, 2>(c, a, nlines, st)
                  : launch_dispatch<double, 4>(c, a, nlines, st);
}
}  // namespace ppk
