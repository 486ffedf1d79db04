"""The double-word apply against the FP64 apply of the same handle.

Both use the same tables (to the 2^-49 of their double-word copies), so the
difference is the double-word arithmetic of the convolution alone: about u^2 =
2^-48 per operation, growing with the square root of some 50 operations on the
way of a value, 2.5e-14 relative to the convolution's part; the identity part is
added in FP64.  Tolerance: 3e-14 of the norm of y - x.  Sizes: the register-resident
double-word kernels (2n = 256), other 2n, odd radices, a long line.
"""
import pytest

import vie_inputs as vi

from gpu_common import eps_dev, mu_dev, to_dev, vie  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,n,with_mu", [("helmholtz", 128, False), ("maxwell", 48, True), ("laplace", 35, False),
                                            ("maxwell", 21, False), ("helmholtz", 11, False), ("helmholtz", 5, False),
                                            ("laplace", 150, False)])
def test_df64_against_fp64(vie, kind, n, with_mu):
    import torch

    if kind == "laplace":
        p = vi.laplace_bump_problem(n=n, seed=4)
    elif kind == "helmholtz":
        p = vi.helmholtz_problem(n=n, wavelengths=2.0, seed=4)
    else:
        p = vi.maxwell_problem(n=n, wavelengths=2.0, with_mu=with_mu, seed=4)
    P = vie.Problem(kind, n, p.lo, p.hi, p.omega, eps_dev(p), mu_dev(p))
    x = to_dev(vi.random_field(n, P.ncomp, 6)[0])
    y64, ydf = torch.empty_like(x), torch.empty_like(x)
    P.apply(x, y64, vie.VIE_FP64)
    P.apply(x, ydf, vie.VIE_DF64)
    torch.cuda.synchronize()
    assert float(torch.linalg.vector_norm(ydf - y64) / torch.linalg.vector_norm(y64 - x)) < 3e-14
    P.close()
