"""Layouts and branches that the sizes of test_gpu_layouts.py do not reach:
16-row chunks with four variables, the characteristic solve with scratch on a
cluster of several CTAs and on the largest one, bounded mixed lines on several
CTAs, and the rescaled weights of FP64 indicators beyond 2^-80 .. 2^80.
"""
import numpy as np
import pytest

import oracle
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


def _smooth_2d(nx, ny, bc, stream=800):
    """a few Fourier modes per field, at least eight cells to a wave"""
    g = W.rng(stream)
    X, Y = np.meshgrid((np.arange(nx) + 0.5) / nx, (np.arange(ny) + 0.5) / ny)

    def field(base, amp):
        out = np.full((ny, nx), base)
        for _ in range(3):
            kx, ky = int(g.integers(0, max(1, min(4, nx // 8)) + 1)), int(g.integers(0, max(1, min(4, ny // 8)) + 1))
            out += g.uniform(-amp, amp) / 3 * np.sin(2 * np.pi * (kx * X + ky * Y) + g.uniform(0, 2 * np.pi))
        return out

    U = W.prim_to_cons_2d(field(1.0, 0.3), field(0.5, 0.3), field(-0.4, 0.3), field(1.0, 0.3), 1.4)
    return W.Problem(2, nx, ny, 0.0, nx / max(nx, ny), 0.0, ny / max(nx, ny), 1.4, bc, 0.4, 0.1,
                     np.ascontiguousarray(U))


def _error(B, p, prec, recon):
    """largest difference of L from the oracle's over the variable's flux scale"""
    U = torch.from_numpy(np.ascontiguousarray(p.U0).ravel()).cuda()
    L = torch.zeros_like(U)
    s = B.Solver(B.config_from_problem(p, prec, recon=recon))
    s.operator(U, L, 1e-13)
    s.close()
    bc = tuple(p.bc) + (0,) * (4 - len(p.bc))
    g = oracle.make_grid(p.ndim, p.nx, p.ny, p.dx, p.dy, p.gamma, bc, recon=recon)
    Lo, _ = oracle.operator(g, p.U0, 1e-13)
    flat = p.U0.reshape(p.U0.shape[0], -1)
    vel = np.sqrt(np.sum(flat[1:-1] ** 2, axis=0)) / flat[0]
    pr = (p.gamma - 1) * (flat[-1] - 0.5 * flat[0] * vel ** 2)
    smax = np.max(vel + np.sqrt(p.gamma * pr / flat[0]))
    h = min(p.dx, p.dy) if p.ndim == 2 else p.dx
    scale = (np.abs(flat).max(axis=1) * smax).max() / h
    return np.abs(L.cpu().numpy().reshape(Lo.shape) - Lo).max() / scale


@pytest.mark.parametrize("recon", [0, 1])
@pytest.mark.parametrize("bc", [(0, 0, 0, 0), (1, 1, 1, 1)])
@pytest.mark.parametrize("nx,ny", [(2048, 200), (1100, 300), (4097, 9), (4608, 12), (8191, 9), (8192, 8),
                                   (9, 4097)])
def test_long_lines_2d(B, nx, ny, bc, recon):
    """Over 4096 cells: 16-row chunks and clusters up to 16 CTAs.  2048 x 200 and
    1100 x 300: the characteristic solve's scratch on clusters of three and two CTAs
    (8192 x 8: its multipliers in shared memory, 16 CTAs)."""
    p = _smooth_2d(nx, ny, bc)
    # (mixed: the indicators' FP32 floor, 2^20 u^2 |U|^2, is 1e-5 of the fluxes on
    # such data; a layout fault is an error of order one)
    tol = {0: 1e-12, 1: 1e-4}
    for prec in (0, 1):
        assert _error(B, p, prec, recon) <= tol[prec], prec


@pytest.mark.parametrize("recon", [0, 1])
@pytest.mark.parametrize("n", [257, 511, 513, 1025, 2047, 4097, 8191])
def test_bounded_mixed_lines(B, n, recon):
    """A layout fault is an error of order one; the wall's velocity jump leaves 1e-5."""
    assert _error(B, W.random_smooth_1d(n, stream=300 + n, periodic=False), 1, recon) <= 1e-4


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("bc", [(0, 0, 0, 0), (1, 1, 1, 1)])
def test_batch_2d_16_rows(B, bc, prec):
    """Mixed batches take 16-row chunks at these lengths by rule (FP64: 8), one
    step against the oracle's with the same dt."""
    probs = [_smooth_2d(nx, ny, bc, 810 + nx) for nx, ny in ((511, 20), (24, 512), (513, 40), (1025, 16), (300, 264))]
    s = B.Solver(None, batch=[B.config_from_problem(p, prec) for p in probs])
    s.set_state(np.concatenate([p.U0.ravel() for p in probs]))
    s.step()
    out, off = s.get_state()[0], 0
    for k, p in enumerate(probs):
        dt = s.problem_stats(k).last_dt
        g = oracle.make_grid(2, p.nx, p.ny, p.dx, p.dy, p.gamma, p.bc)
        ref = oracle.rk3_step(g, p.U0, dt)
        got = out[off:off + ref.size].reshape(ref.shape)
        off += ref.size
        # dt L in FP32 (mixed): CFL 0.4 of the bound on L above
        assert np.abs(got - ref).max() / np.abs(ref).max() <= (1e-12 if prec == 0 else 1e-4), k
    s.close()


@pytest.mark.parametrize("recon", [0, 1])
@pytest.mark.parametrize("k", [50, -50])
@pytest.mark.parametrize("nx,ny", [(200, 1), (1300, 1), (517, 60)])
def test_rescaled_weights(B, nx, ny, k, recon):
    """FP64: with U scaled by 2^k and the weights' epsilon by 4^k every operation of
    the scheme scales exactly, and so must L; indicators of order 4^k leave
    2^-80 .. 2^80, where the weights rescale them.  (The limiter's epsilon bounds
    the specific energy too, which does not scale: too small to enter a sum.)"""
    p = W.random_smooth_1d(nx, stream=850 + nx) if ny == 1 else W.random_jumps_2d(nx, ny, stream=850 + nx)
    out = []
    for e in (0, k):
        U = torch.from_numpy(np.ascontiguousarray(p.U0).ravel() * 2.0 ** e).cuda()
        L = torch.zeros_like(U)
        s = B.Solver(B.config_from_problem(p, 0, recon=recon, eps_weno=1e-13 * 4.0 ** e))
        s.operator(U, L, 1e-80)
        s.close()
        out.append(L.cpu().numpy() * 2.0 ** -e)
    assert np.array_equal(out[0], out[1])
