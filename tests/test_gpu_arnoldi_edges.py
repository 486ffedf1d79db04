"""Arnoldi kernels at their edges: projections on one to many basis vectors (the inner
products go in chunks of eight, the projection in eights, fours and ones), vectors of odd
length (n odd: no 16-byte packs in FP32), several right-hand sides, and the rotations
of a full cycle.

Each solve's answer is checked with an apply of its own: |b - A J| <= 1.01 tol |b| in
FP64 (the solver stops on its own residual, computed to about 1e-13).
"""
import pytest

import vie_inputs as vi

from gpu_common import eps_dev, mu_dev, vie  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,with_mu,nrhs", [(7, False, 1), (9, True, 3), (10, False, 2), (24, False, 1)])
@pytest.mark.parametrize("restart", [1, 4, 8, 9, 17, 40])
@pytest.mark.parametrize("mode", ["mixed", "fp64"])
def test_solve_residual(vie, n, with_mu, nrhs, restart, mode):
    import torch

    p = vi.maxwell_problem(n=n, wavelengths=1.0, with_mu=with_mu, seed=9, ndirs=nrhs)
    P = vie.Problem("maxwell", n, p.lo, p.hi, p.omega, eps_dev(p), mu_dev(p))
    b = torch.empty((nrhs, P.ncomp, n, n, n), dtype=torch.complex128, device="cuda:0")
    P.rhs(p.directions, p.polarisations, nrhs, b)
    J = torch.zeros_like(b)
    tol = 1e-9
    P.solve(b, J, tol=tol, restart=restart, max_outer=400, max_inner=4000, nrhs=nrhs,
            mode=vie.VIE_SOLVE_MIXED if mode == "mixed" else vie.VIE_SOLVE_FP64)
    y = torch.empty_like(b)
    P.apply(J, y, vie.VIE_FP64, nrhs=nrhs)
    for r in range(nrhs):
        assert float(torch.linalg.vector_norm(b[r] - y[r]) / torch.linalg.vector_norm(b[r])) <= 1.01 * tol
    P.close()
