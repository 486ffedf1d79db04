"""Two-step passes on long lines: every radix from 16 to 24 in either step, half lines,
the largest grids, several right-hand sides, and the z pass next to the line passes.

Convolution grids: 324 = 18 18, 336 = 21 16, 360 = 20 18, 384 = 24 16 (double-word; the
FP32 and FP64 kernels there are register-resident), 420 = 21 20, 432 = 24 18, 440 = 22 20,
462 = 22 21, 480 = 24 20, 504 = 24 21, 576 = 24 24 (four pencils of six FP64 lines do not fit
in shared memory, so the z pass takes two).  In double-word arithmetic the z pass has no
two-step kernel at 324, 400 to 440, 462, 504 and 576 (neither the length nor its half splits
into radices up to 16) and runs the Stockham kernel; the other passes do.

The reference is the FP64 Stockham path (VIE_GENERIC_FFT), whose codelets, index maps and
kernels are others; it is compared with the oracle at small sizes by the parity tests.
Tolerances are those tests': 1e-12 in FP64 and double-word arithmetic, 2e-5 in FP32.
"""
import pytest

import vie_inputs as vi

from gpu_common import vie  # noqa: F401

pytestmark = pytest.mark.gpu


def _problem(vie, kind, n, with_mu):
    import torch

    dev = torch.device("cuda:0")
    eps = vi.bump_medium_torch(n, 3, dev)
    mu = vi.bump_medium_torch(n, 4, dev, amp=0.3) if with_mu else None
    return vie.Problem(kind, n, -1.0, 1.0, 0.0 if kind == "laplace" else 9.0, eps, mu)


def _field(shape, seed):
    import torch

    g = torch.Generator(device="cuda:0").manual_seed(seed)
    return torch.randn(shape, dtype=torch.complex128, device="cuda:0", generator=g)


def _apply(P, x, prec, nrhs=1):
    import torch

    y = torch.empty_like(x)
    P.apply(x, y, prec, nrhs=nrhs)
    torch.cuda.synchronize()
    return y


def _off(a, b):
    import torch

    return float(torch.linalg.vector_norm(a.to(b.dtype) - b) / torch.linalg.vector_norm(b))


@pytest.mark.parametrize("kind,n,with_mu,nrhs", [
    ("helmholtz", 162, False, 1), ("maxwell", 168, True, 1), ("maxwell", 180, False, 1), ("helmholtz", 192, False, 2),
    ("laplace", 210, False, 1), ("maxwell", 216, True, 1), ("helmholtz", 220, False, 2), ("helmholtz", 231, False, 1),
    ("maxwell", 240, True, 1), ("helmholtz", 252, False, 1), ("maxwell", 288, True, 1), ("maxwell", 48, True, 3),
    ("helmholtz", 81, False, 3)])
def test_against_stockham(vie, kind, n, with_mu, nrhs, monkeypatch):
    import torch

    P = _problem(vie, kind, n, with_mu)
    x = _field((nrhs, P.ncomp, n, n, n), n)
    cout = 6 if kind == "maxwell" else 1
    field = torch.empty((cout, n, n, n), dtype=torch.complex128, device="cuda:0")
    monkeypatch.setenv("VIE_GENERIC_FFT", "1")
    ref = _apply(P, x, vie.VIE_FP64, nrhs)
    P.eval_scattered(x[0], field)
    torch.cuda.synchronize()
    ref_field = field.clone()
    monkeypatch.delenv("VIE_GENERIC_FFT")
    assert _off(_apply(P, x, vie.VIE_FP64, nrhs), ref) < 1e-12
    assert _off(_apply(P, x, vie.VIE_DF64, nrhs), ref) < 1e-12
    assert _off(_apply(P, x.to(torch.complex64), vie.VIE_FP32, nrhs), ref) < 2e-5
    P.eval_scattered(x[0], field.zero_())
    torch.cuda.synchronize()
    assert _off(field, ref_field) < 1e-12
    P.close()


@pytest.mark.parametrize("kind,n,with_mu", [("helmholtz", 81, False), ("maxwell", 100, True), ("maxwell", 150, False)])
def test_axes_exchanged(vie, kind, n, with_mu):
    """z, x, y in place of x, y, z (grid axes and components): the z pass of one run works on
    the x-lines of the other, so an error of one of the passes does not cancel."""
    import torch

    perm = [1, 2, 0]  # new axis a is old axis perm[a]: new x = old y, new y = old z, new z = old x

    def turn(t):  # [..., 3, z, y, x] -> the same field in the new axes
        return t[..., perm, :, :, :].permute(*range(t.dim() - 3), -1, -3, -2).contiguous()

    dev = torch.device("cuda:0")
    eps = vi.bump_medium_torch(n, 3, dev)
    mu = vi.bump_medium_torch(n, 4, dev, amp=0.3) if with_mu else None

    def tensor(t):
        return None if t is None else turn(t.reshape(3, 3, n, n, n)[perm]).reshape(9, -1)

    args = (n, -1.0, 1.0, 9.0)
    P, Q = vie.Problem(kind, *args, eps, mu), vie.Problem(kind, *args, tensor(eps), tensor(mu))
    x = _field((P.ncomp // 3, 3, n, n, n), 5)
    for prec, dt, tol in ((vie.VIE_FP64, torch.complex128, 1e-12), (vie.VIE_DF64, torch.complex128, 1e-12),
                          (vie.VIE_FP32, torch.complex64, 2e-5)):
        v = x.to(dt)
        assert _off(_apply(Q, turn(v), prec), turn(_apply(P, v, prec))) < tol, prec
    P.close()
    Q.close()


@pytest.mark.parametrize("kind,n,with_mu", [("helmholtz", 81, False), ("maxwell", 99, True), ("helmholtz", 149, False)])
def test_half_lines_stay_inside_their_buffers(vie, kind, n, with_mu):
    """Guard bands of 4096 elements around x and y (half-line z pass; 149 on a grid of 300)."""
    import torch

    P = _problem(vie, kind, n, with_mu)
    size = P.ncomp * n ** 3
    for prec, dt in ((vie.VIE_FP64, torch.complex128), (vie.VIE_DF64, torch.complex128), (vie.VIE_FP32, torch.complex64)):
        xb = torch.full((size + 8192,), 12345.25 - 678.5j, dtype=dt, device="cuda:0")
        yb = xb.clone()
        xb[4096:-4096] = _field((size,), 6).to(dt)
        before = xb.clone()
        P.apply(xb[4096:-4096], yb[4096:-4096], prec)
        torch.cuda.synchronize()
        assert torch.equal(xb, before)
        for edge in (yb[:4096], yb[-4096:]):
            assert bool((edge == 12345.25 - 678.5j).all()), prec
        assert bool(torch.isfinite(torch.view_as_real(yb)).all()), prec
    P.close()
