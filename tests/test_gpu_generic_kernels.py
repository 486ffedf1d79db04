"""VIE_GENERIC_FFT takes every apply to the Stockham kernels: other kernels than without
it (other bits), the same operator.

Lines of 64, 70, 96, 126 and 256 points; tolerances of the parity tests (1e-12 in FP64 and
double-word arithmetic, 2e-5 in FP32).
"""
import pytest

import vie_inputs as vi

from gpu_common import eps_dev, mu_dev, to_dev, vie  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,n,with_mu", [("helmholtz", 32, False), ("helmholtz", 35, False), ("laplace", 48, False),
                                            ("maxwell", 63, True), ("maxwell", 128, False)])
def test_generic_kernels_run(vie, kind, n, with_mu, monkeypatch):
    import torch

    if kind == "laplace":
        p = vi.laplace_bump_problem(n=n, seed=3)
    elif kind == "helmholtz":
        p = vi.helmholtz_problem(n=n, wavelengths=2.0, seed=3)
    else:
        p = vi.maxwell_problem(n=n, wavelengths=2.0, with_mu=with_mu, seed=3)
    P = vie.Problem(kind, n, p.lo, p.hi, p.omega, eps_dev(p), mu_dev(p))
    x = to_dev(vi.random_field(n, P.ncomp, 4)[0])
    cout = 6 if kind == "maxwell" else 1

    def run():
        out = {}
        for prec, dt in ((vie.VIE_FP64, torch.complex128), (vie.VIE_DF64, torch.complex128),
                         (vie.VIE_FP32, torch.complex64)):
            v = x.to(dt)
            out[prec] = torch.empty_like(v)
            P.apply(v, out[prec], prec)
        out["field"] = torch.empty((cout, n, n, n), dtype=torch.complex128, device="cuda:0")
        P.eval_scattered(x, out["field"])
        torch.cuda.synchronize()
        return out

    usual = run()
    monkeypatch.setenv("VIE_GENERIC_FFT", "1")
    generic = run()
    monkeypatch.delenv("VIE_GENERIC_FFT")
    for k, y in usual.items():
        g = generic[k].to(torch.complex128)
        y = y.to(torch.complex128)
        assert not torch.equal(g, y), k
        off = float(torch.linalg.vector_norm(g - y) / torch.linalg.vector_norm(y))
        assert off < (2e-5 if k == vie.VIE_FP32 else 1e-12), k
    P.close()
