"""Set-up of the discrete kernels by one line operator per axis on octants.

Every symbol comes from four base octants by exchanging axes, so an operator
apply and a scattered field with all symbols in play are compared with the
oracle, which transforms each symbol on the whole cube.  Sizes: the smallest,
odd (no Nyquist entry), partial line tiles (n + 1 no multiple of the eight lines
of a tile), one more than a 32-wide combine tile, Bluestein lines (3n = 69),
and a padded convolution grid (n = 23 runs on 2 x 24).

Tolerance 1e-12: the transforms carry about 2^-47 per double-word operation over
some 40 butterfly levels, near 3e-13, and the FP64 parity tests of the apply hold
the same bound.
"""
import numpy as np
import pytest

import vie_inputs as vi
from oracle import operators

from gpu_common import eps_dev, mu_dev, rel, to_dev, vie  # noqa: F401

pytestmark = pytest.mark.gpu

CASES = [("maxwell", n, True, 0) for n in (4, 5, 15, 16, 23, 32)] + [
    ("maxwell", 16, False, 1), ("helmholtz", 21, False, 0), ("laplace", 32, False, 1), ("laplace", 7, False, 0)]


@pytest.mark.parametrize("kind,n,with_mu,fp64", CASES)
def test_apply_and_field_match_oracle(vie, monkeypatch, kind, n, with_mu, fp64):
    import torch

    if fp64:
        monkeypatch.setenv("VIE_SETUP_FP64", "1")
    if kind == "laplace":
        p = vi.laplace_bump_problem(n=n, seed=3)
    elif kind == "helmholtz":
        p = vi.helmholtz_problem(n=n, wavelengths=2.0, seed=3)
    else:
        p = vi.maxwell_problem(n=n, wavelengths=2.0, with_mu=with_mu, seed=3)
    P = vie.Problem(kind, n, p.lo, p.hi, p.omega, eps_dev(p), mu_dev(p))
    op = operators.OracleProblem.from_problem(p)
    x = vi.random_field(n, P.ncomp, 5)[0]
    xd = to_dev(x)
    y = torch.empty_like(xd)
    P.apply(xd, y, vie.VIE_FP64)
    f = torch.empty((6 if kind == "maxwell" else 1, n, n, n), dtype=torch.complex128, device=xd.device)
    P.eval_scattered(xd, f)
    torch.cuda.synchronize()
    assert rel(y.cpu().numpy(), op.apply(x)) < 1e-12
    assert rel(f.cpu().numpy(), op.scattered(x)) < 1e-12
    P.close()
