"""The FP64 reciprocal and square root of physics.cuh against the correctly
rounded operators, compiled from the header into a small library."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1402_5618_gb300 import build

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SRC = r'''
#include "physics.cuh"
__global__ void apply(const double *x, double *r, double *s, long n) {
  const long i = blockIdx.x * 256l + threadIdx.x;
  if (i < n) { r[i] = ppk::rcp(x[i]); s[i] = ppk::root(x[i]); }
}
extern "C" int run(const double *x, double *r, double *s, long n) {
  apply<<<(unsigned)((n + 255) / 256), 256>>>(x, r, s, n);
  return (int)cudaDeviceSynchronize();
}
'''


def test_rcp_and_root(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    (tmp_path / "a.cu").write_text(SRC)
    so = str(tmp_path / "a.so")
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", "-o", so,
                    str(tmp_path / "a.cu")], check=True)
    g = np.random.default_rng(5)
    n = 1 << 20
    x = np.ldexp(g.uniform(1.0, 2.0, n), g.integers(-1000, 1000, n))
    x[:2200] = np.ldexp(1.0, np.arange(2200) % 2000 - 1000)          # powers of two
    x[2200:4200] = np.nextafter(x[200:2200], 0.0)
    special = np.array([0.0, 5e-324, 1e-310, 2.0 ** -1022, 2.0 ** -1021])
    both = torch.from_numpy(np.concatenate([x, special, -x[:1000]])).cuda()
    r, s = torch.zeros_like(both), torch.zeros_like(both)
    lib = ctypes.CDLL(so)
    assert lib.run(*(ctypes.c_void_p(t.data_ptr()) for t in (both, r, s)), ctypes.c_long(both.numel())) == 0
    r, s = r.cpu().numpy(), s.cpu().numpy()
    # third-order steps on 2^-20 approximations: truncation below 2^-58, and at most
    # a quarter more than the final rounding
    ref = 1.0 / x
    assert np.all(np.abs(r[:n] - ref) <= np.spacing(ref))
    ref = np.sqrt(x)
    assert np.all(np.abs(s[:n] - ref) <= np.spacing(ref))
    assert np.array_equal(r[:2000], 1.0 / x[:2000])                  # exact for powers of two
    assert np.array_equal(s[n:n + 5], np.sqrt(special))              # operands the approximation flushes
    assert np.array_equal(-r[-1000:], r[:1000]) and np.all(np.isnan(s[-1000:]))
