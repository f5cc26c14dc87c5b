"""FP64 states whose products, or themselves, lie below FP32's range: the
limiter's FP32 pretest cannot judge them and has to leave them to the exact
limiter.  Jumps at which the limiter acts, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1402_5618_gb300 import workloads as W

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ndim", [1, 2])
@pytest.mark.parametrize("e", [-16, -18, -20, -22, -25, -30, -35, -38, -40, -45, -60])
def test_limited_tiny_states(e, ndim):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_5618_gb300 import binding as B
    B.lib()
    n, k = 200, 40
    g = W.rng(77)
    cell = np.minimum((np.arange(n) * k) // n, k - 1)
    rho, u, p = ((10.0 ** g.uniform(-2, 0, k))[cell], g.uniform(-2, 2, k)[cell], (10.0 ** g.uniform(-2, 0, k))[cell])
    U = W.prim_to_cons_1d(rho, u, p, 1.4) if ndim == 1 else \
        np.repeat(W.prim_to_cons_2d(rho, u, 0.3 * u, p, 1.4)[:, None, :], 12, axis=1)
    U = np.ascontiguousarray(U * 10.0 ** e)
    ny = 1 if ndim == 1 else 12
    bc = (1, 1, 1, 1)
    eps = min(1e-13, U[0].min())
    Lo, cnt = oracle.operator(oracle.make_grid(ndim, n, ny, 1.0 / n, 1.0 / ny, 1.4, bc), U, eps)
    assert cnt.theta1_active > 10 and cnt.theta2_active > 10
    s = B.Solver(B.make_config(ndim, n, ny, 0.0, 1.0, 0.0, 1.0, bc=bc))
    Ud = torch.from_numpy(U.ravel()).cuda()
    L = torch.zeros_like(Ud)
    s.operator(Ud, L, eps)
    s.close()
    # (roundings reach a limited face state through a pressure near zero: 1e-16
    # there is 1e-8 of its sound speed at worst)
    assert np.abs(L.cpu().numpy().reshape(U.shape) - Lo).max() <= 1e-8 * np.abs(Lo).max()
