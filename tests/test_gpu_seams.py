"""Lines on several CTAs where their segments meet.

Stage 2 of a step updates the stage buffer in place while every CTA also reads
cells of its neighbours.  A step must therefore equal the same step composed of
operator evaluations, which write to a buffer of their own.
"""
import math

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


def _telescoping(n, stream, periodic):
    """1-D noise of a few percent about a moving base state: with a positive
    velocity every flux component stays within a factor of two of its mean, so
    the difference of two face fluxes is exact (Sterbenz), and so is its product
    with 1/h, a power of two.  Bounded lines: the noise stays 120 cells away
    from the ends, where the solve's influence (a factor of four per cell) is below
    rounding, so that the fluxes at both ends are the base state's."""
    g = W.rng(stream)
    amp = np.where((np.arange(n) >= 120) & (np.arange(n) < n - 120), 0.02, 0.0)
    if periodic:
        amp[:] = 0.02
    rho, u, p = (1.0 + amp * g.uniform(-1, 1, n), 2.0 + amp * g.uniform(-1, 1, n),
                 1.0 + amp * g.uniform(-1, 1, n))
    return rho, u, p


# (n, the other side): every chunk length, one segment and many, whole, ragged
# and one-cell last segments; 1-D first
SHAPES = [(40, 0), (128, 0), (200, 0), (513, 0), (577, 0), (1025, 0), (2049, 0), (4097, 0), (8192, 0),
          (60, 400), (200, 160), (300, 257), (1025, 40), (1024, 200), (2049, 200), (4097, 8), (4700, 24)]


@pytest.mark.parametrize("recon", [0, 1])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("periodic", [True, False])
@pytest.mark.parametrize("n,across", SHAPES)
def test_flux_differences_telescope(B, n, across, periodic, prec, recon):
    """Both CTAs at a seam evaluate its face: the sum of L over a line is the
    difference of the end fluxes, exactly, only if they find the same number."""
    if not periodic and n < 400:
        pytest.skip("no room for quiet ends")
    rho, u, p = _telescoping(n, 600 + n, periodic)
    bc = 0 if periodic else 1
    h = 2.0 ** -10
    if across == 0:
        dirs = [(1, W.prim_to_cons_1d(rho, u, p, 1.4)[:, None, :], (n, 1))]
    else:   # constant across: the other direction's fluxes cancel exactly
        Ux = W.prim_to_cons_2d(rho, u, np.ones(n), p, 1.4)
        Uy = W.prim_to_cons_2d(rho, np.ones(n), u, p, 1.4)
        dirs = [(2, np.repeat(Ux[:, None, :], across, axis=1), (n, across)),
                (2, np.repeat(Uy[:, :, None], across, axis=2), (across, n))]
    # LLF in the mixed form: its difference form of HLLC (F - F(R)) rounds the
    # differences of faces near a zero of F - F(R)
    for flux in ((0, 1) if prec == 0 else (1,)):
        for d, (ndim, U, (nx, ny)) in enumerate(dirs):
            s = B.Solver(B.make_config(ndim, nx, ny, 0.0, nx * h, 0.0, ny * h, bc=(bc,) * 4,
                                       precision=prec, flux=flux, recon=recon))
            Ud = torch.from_numpy(np.ascontiguousarray(U).ravel()).cuda()
            L = torch.zeros_like(Ud)
            s.operator(Ud, L, 1e-13)
            s.close()
            Lg = L.cpu().numpy().reshape(U.shape)
            lines = Lg if d == 0 else Lg.transpose(0, 2, 1)
            assert np.abs(lines).max() > 1.0
            for v in range(lines.shape[0]):
                for j in (0, lines.shape[1] // 2, lines.shape[1] - 1):
                    assert math.fsum(lines[v, j]) == 0.0, (flux, d, v, j)
