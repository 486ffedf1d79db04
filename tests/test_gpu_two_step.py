"""Two-step passes (M = R1 R2 with run-time radices): every radix, both radix
classes, the half-line z pass, padded grids and the lengths without a split.

Sizes by convolution grid M: 16 = 4 4, 50 = 10 5, 66 = 11 6, 70 = 10 7, 88 = 11 8,
126 = 14 9, 162 = 18 9 (half lines 9 9), 180 = 15 12, 210 = 15 14; 22 and 26 -> 28
without a split or padded; larger: 200 = 20 10, 220 = 20 11, 242 = 22 11, 294 =
21 14 (halves 21 7: no half-line pass), 300 = 20 15 from n = 149 (padded).
Tolerances are the parity tests': 1e-12 of the oracle in FP64 and double-word
arithmetic (about 2^-47 and 50 operations deep), 2e-5 in FP32.
"""
import numpy as np
import pytest

import vie_inputs as vi
from oracle import operators

from gpu_common import eps_dev, mu_dev, rel, to_dev, vie  # noqa: F401

pytestmark = pytest.mark.gpu


def _apply(P, x, prec, nrhs):
    import torch

    y = torch.empty_like(x)
    P.apply(x, y, prec, nrhs=nrhs)
    torch.cuda.synchronize()
    return y


@pytest.mark.parametrize("kind,n,with_mu", [
    ("maxwell", 8, True), ("helmholtz", 11, False), ("maxwell", 13, True), ("laplace", 25, False),
    ("maxwell", 33, True), ("helmholtz", 35, False), ("maxwell", 44, False), ("helmholtz", 63, False),
    ("maxwell", 32, True), ("helmholtz", 48, False), ("laplace", 81, False), ("helmholtz", 90, False),
    ("laplace", 105, False)])
def test_against_oracle(vie, kind, n, with_mu):
    import torch

    if kind == "laplace":
        p = vi.laplace_bump_problem(n=n, seed=5)
    elif kind == "helmholtz":
        p = vi.helmholtz_problem(n=n, wavelengths=2.0, seed=5)
    else:
        p = vi.maxwell_problem(n=n, wavelengths=2.0, with_mu=with_mu, seed=5)
    P = vie.Problem(kind, n, p.lo, p.hi, p.omega, eps_dev(p), mu_dev(p))
    op = operators.OracleProblem.from_problem(p)
    nrhs = 2 if n <= 35 else 1
    x = vi.random_field(n, P.ncomp, 7, nrhs=nrhs)
    x32 = x.astype(np.complex64)
    y = {k: _apply(P, to_dev(v), prec, nrhs).cpu().numpy() for k, v, prec in
         (("fp64", x, vie.VIE_FP64), ("df64", x, vie.VIE_DF64), ("fp32", x32, vie.VIE_FP32))}
    for r in range(nrhs):
        yo = op.apply(x[r])
        assert rel(y["fp64"][r], yo) < 1e-12
        assert rel(y["df64"][r], yo) < 1e-12
        assert rel(y["fp32"][r], op.apply(x32[r].astype(np.complex128))) < 2e-5
    f = torch.empty((6 if kind == "maxwell" else 1, n, n, n), dtype=torch.complex128, device="cuda:0")
    P.eval_scattered(to_dev(x[0]), f)
    assert rel(f.cpu().numpy(), op.scattered(x[0])) < 1e-12
    P.close()


@pytest.mark.parametrize("kind,n,with_mu", [("helmholtz", 100, False), ("maxwell", 100, True), ("laplace", 110, False),
                                            ("helmholtz", 121, False), ("maxwell", 147, False),
                                            ("helmholtz", 149, False), ("maxwell", 110, True)])
def test_precisions_agree(vie, kind, n, with_mu):
    """Large grids: the FP32 and double-word applies against the FP64 one, and the FP64
    one against an apply that runs other kernels on the same data (symmetry: the discrete
    kernels are even in the offset, so mirroring x and the medium mirrors y)."""
    import torch

    if kind == "laplace":
        p = vi.laplace_bump_problem(n=n, seed=6)
    elif kind == "helmholtz":
        p = vi.helmholtz_problem(n=n, wavelengths=2.0, seed=6)
    else:
        p = vi.maxwell_problem(n=n, wavelengths=2.0, with_mu=with_mu, seed=6)
    eps, mu = eps_dev(p), mu_dev(p)
    P = vie.Problem(kind, n, p.lo, p.hi, p.omega, eps, mu)
    x = to_dev(vi.random_field(n, P.ncomp, 8)[0])
    y = _apply(P, x, vie.VIE_FP64, 1)

    def off(a, b):
        return float(torch.linalg.vector_norm(a - b) / torch.linalg.vector_norm(b))

    assert off(_apply(P, x, vie.VIE_DF64, 1), y) < 1e-12
    assert off(_apply(P, x.to(torch.complex64), vie.VIE_FP32, 1).to(torch.complex128), y) < 2e-5
    P.close()
    # x and y exchanged (grid axes and components): the x-lines of one run are the y-lines of the other
    perm = [1, 0, 2]
    e2 = eps.reshape(3, 3, n, n, n)[perm][:, perm].transpose(-1, -2).contiguous().reshape(9, -1)
    m2 = None if mu is None else mu.reshape(3, 3, n, n, n)[perm][:, perm].transpose(-1, -2).contiguous().reshape(9, -1)
    P2 = vie.Problem(kind, n, p.lo, p.hi, p.omega, e2, m2)
    v = x.reshape(-1, 3, n, n, n)[:, perm].transpose(-1, -2).contiguous()
    if v.shape[0] == 2:
        v[1].neg_()  # M is an axial vector: a reflection changes its sign
    y2 = _apply(P2, v.reshape(x.shape), vie.VIE_FP64, 1).reshape(-1, 3, n, n, n)
    if v.shape[0] == 2:
        y2[1].neg_()
    assert off(y2.transpose(-1, -2)[:, perm].reshape(y.shape), y) < 1e-12
    P2.close()
