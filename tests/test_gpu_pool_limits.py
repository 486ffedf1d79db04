"""The library's pool on the device: what it keeps between problems is at most a
thirty-second of the device, also after problems that held more than that together, and
all of it goes back on request.  The give-back when an allocation fails or the
device is nearly full is tested on the host (test_host_memory.py)."""
import pytest

import vie_inputs as vi

from gpu_common import eps_dev, vie  # noqa: F401

pytestmark = pytest.mark.gpu


def _problems(vie, count, n):
    """`count` problems that have each run a solve, alive together."""
    import torch

    p = vi.helmholtz_problem(n=n, wavelengths=1.5, seed=2)
    eps = eps_dev(p)
    out = []
    for _ in range(count):
        P = vie.Problem("helmholtz", n, p.lo, p.hi, p.omega, eps)
        P._eps = None
        b = torch.empty((3, n, n, n), dtype=torch.complex128, device="cuda:0")
        P.rhs(p.directions[0], None, 1, b)
        P.solve(b, torch.zeros_like(b), tol=1e-6, restart=50, mode=vie.VIE_SOLVE_MIXED)
        out.append(P)
    return out


def _free():
    import torch

    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def test_kept_memory_after_more_than_the_bound(vie):
    import torch

    for P in _problems(vie, 1, 96):  # kernels loaded, schedules chosen
        P.close()
    vie.vie_release_memory()
    base = _free()
    bound = torch.cuda.get_device_properties(0).total_memory // 32
    problems = _problems(vie, 9, 96)
    assert base - _free() > bound
    for P in problems:
        P.close()
    kept = base - _free()
    assert 0 < kept <= bound + (64 << 20)
    vie.vie_release_memory()
    assert base - _free() <= 4 << 20
