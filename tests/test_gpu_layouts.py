"""The line kernels' thread layouts at their edges: line lengths around the
chunk, warp and segment boundaries of every chunk length, few lines and many,
bounded and periodic, both reconstructions and both arithmetics, one operator
evaluation against the oracle.

Bounds as stated for operator evaluations elsewhere: FP64 1e-12 of each
variable's flux scale; mixed form 2e-6 on resolved smooth data, 1e-4 where the
data are not resolved (jumps, a few cells per wave).
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


def _scale(p):
    """per-variable flux scale (max |F_v| + max |U_v| max(|u|+a)) / h"""
    flat = p.U0.reshape(p.U0.shape[0], -1)
    rho, E = flat[0], flat[-1]
    vel = np.sqrt(np.sum(flat[1:-1] ** 2, axis=0)) / rho
    pr = (p.gamma - 1) * (E - 0.5 * rho * vel ** 2)
    smax = np.max(vel + np.sqrt(p.gamma * pr / rho))
    mom = np.abs(rho * vel * vel + pr).max()
    F = [np.abs(rho * vel).max()] + [mom] * (flat.shape[0] - 2) + [np.abs(vel * (E + pr)).max()]
    h = min(p.dx, p.dy) if p.ndim == 2 else p.dx
    return np.array([(f + np.abs(u).max() * smax) / h for f, u in zip(F, flat)])


def _check(B, p, tol32):
    eps = min(1e-13, p.U0[0].min())
    U = torch.from_numpy(np.ascontiguousarray(p.U0).ravel()).cuda()
    scale = _scale(p)
    for recon in (B.RECON_COMPONENT, B.RECON_CHARACTERISTIC):
        g = oracle.make_grid(p.ndim, p.nx, p.ny, p.dx, p.dy, p.gamma, p.bc, recon=recon)
        Lo, _ = oracle.operator(g, p.U0, eps)
        for prec, tol in ((B.PREC_FP64, 1e-12), (B.PREC_MIXED, tol32)):
            if tol is None:
                continue
            s = B.Solver(B.config_from_problem(p, prec, recon=recon))
            L = torch.zeros_like(U)
            s.operator(U, L, eps)
            s.close()
            Lg = L.cpu().numpy().reshape(p.U0.shape)
            for v in range(Lo.shape[0]):
                err = np.abs(Lg[v] - Lo[v]).max() / scale[v]
                assert err <= tol, (recon, prec, v, err)


SIZES_1D = [8, 9, 16, 17, 31, 33, 63, 64, 65, 127, 129, 255, 257, 511, 513, 1025, 2047, 2049, 4095,
            4097, 7681, 8191]


@pytest.mark.parametrize("n", SIZES_1D)
@pytest.mark.parametrize("periodic", [True, False])
def test_single_lines(B, n, periodic):
    """One line: the shortest chunks its cluster of 16 CTAs allows."""
    # (not the mixed form on long bounded lines: the velocity at a wall is a jump)
    tol32 = 1e-4 if n < 256 else (2e-6 if periodic else None)
    _check(B, W.random_smooth_1d(n, stream=300 + n, periodic=periodic), tol32)


@pytest.mark.parametrize("nx,ny", [(33, 640), (65, 200), (130, 170), (300, 257), (513, 180), (1031, 40)])
@pytest.mark.parametrize("periodic", [True, False])
def test_many_lines(B, nx, ny, periodic):
    """Enough lines for the long chunks in one direction or both."""
    bc = (0, 0, 0, 0) if periodic else (1, 2, 2, 1)
    _check(B, W.random_jumps_2d(nx, ny, stream=400 + nx, bc=bc), 1e-4)
