"""Lines on several CTAs where their segments meet.

Stage 2 of a step updates the stage buffer in place while every CTA also reads
cells of its neighbours.  A step must therefore equal the same step composed of
operator evaluations, which write to a buffer of their own.
"""
import numpy as np
import pytest

from paper_1402_5618_gb300 import workloads as W

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1402_5618_gb300 import binding
    binding.lib()
    return binding


def _blocks(n, stream):
    """random blocks of about ten cells: the limiter acts at many cells, those
    next to the segments' ends among them"""
    g = W.rng(stream)
    k = n // 10
    cell = np.minimum((np.arange(n) * k) // n, k - 1)
    rho, p = 10.0 ** g.uniform(-2, 1, k), 10.0 ** g.uniform(-2, 1, k)
    u = g.uniform(-2, 2, k)
    U = W.prim_to_cons_1d(rho[cell], u[cell], p[cell], 1.4)
    return W.Problem(1, n, 1, 0.0, 1.0, 0.0, 1.0, 1.4, (0, 0, 0, 0), 1.0 / 24.0, 1.0,
                     np.ascontiguousarray(U))


@pytest.mark.parametrize("recon", [0, 1])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("ndim,n", [(1, 65), (1, 800), (1, 4097), (1, 8192), (2, 300)])
def test_step_in_place_equals_operator_steps(B, ndim, n, prec, recon):
    """(2-D: FP64 alone updates in place, its y lines on several CTAs)"""
    p = _blocks(n, 500 + n) if ndim == 1 else W.random_jumps_2d(40, n, stream=500 + n)
    s = B.Solver(B.config_from_problem(p, prec, recon=recon))
    s.set_state(p.U0.ravel().copy())
    dt = s.step()
    got, _, _ = s.get_state()
    L = torch.zeros(p.U0.size, dtype=torch.float64, device="cuda")

    def stage(U):
        s.operator(U, L)
        torch.cuda.synchronize()
        return U + dt * L

    U0 = torch.from_numpy(p.U0.ravel().copy()).cuda()
    U1 = stage(U0)
    U2 = 0.75 * U0 + 0.25 * stage(U1)
    U3 = U0 / 3.0 + 2.0 / 3.0 * stage(U2)
    s.close()
    ref = U3.cpu().numpy().reshape(p.U0.shape[0], -1)
    got = got.reshape(ref.shape)
    # The stage states differ in their last bits (FP64 1e-16, hi parts of the
    # mixed form 6e-8), which the nonlinear weights at jumps raise by up to 1e7 in
    # FP64, and in FP32, whose indicators have a floor, by less than 1e3.
    tol = 1e-8 if prec == 0 else 1e-4
    for v in range(ref.shape[0]):
        err = np.abs(got[v] - ref[v]).max() / np.abs(ref[v]).max()
        assert err <= tol, (v, err)
