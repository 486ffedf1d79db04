"""The library's memory pool: bounded, reused by the next problem, safe with several
threads and streams (each request's answer is bitwise the same alone and among others)."""
import threading

import pytest

import vie_inputs as vi

from gpu_common import eps_dev, vie  # noqa: F401

pytestmark = pytest.mark.gpu


def _request(vie, n, seed, stream=None):
    import torch

    p = vi.helmholtz_problem(n=n, wavelengths=1.5, seed=seed)
    with torch.cuda.stream(stream or torch.cuda.current_stream()):
        eps = eps_dev(p)
        P = vie.Problem("helmholtz", n, p.lo, p.hi, p.omega, eps)
        b = torch.empty((3, n, n, n), dtype=torch.complex128, device="cuda:0")
        P.rhs(p.directions[0], None, 1, b)
        J = torch.zeros_like(b)
        P.solve(b, J, tol=1e-8, restart=30, mode=vie.VIE_SOLVE_MIXED)
        torch.cuda.current_stream().synchronize()
        P.close()
    return J


def test_kept_memory_is_bounded_and_reused(vie):
    import torch

    _request(vie, 16, 1)
    total = torch.cuda.get_device_properties(0).total_memory
    free = []
    for n in (64, 96, 64, 96, 96):
        _request(vie, n, 2)
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        free.append(torch.cuda.mem_get_info()[0])
    assert free[0] - min(free) <= total // 32 + (64 << 20)
    assert free[-1] == free[-2]  # the same request again maps nothing new


def test_threads_and_streams(vie):
    import torch

    sizes = [(16, 1), (24, 2), (20, 3), (32, 4)]
    for n, seed in sizes:  # the z-pass schedules are chosen on an idle device
        _request(vie, n, seed)
    alone = [_request(vie, n, seed) for n, seed in sizes]
    got, errors = {}, []

    def work(t):
        try:
            st = torch.cuda.Stream()
            for k in range(3):
                n, seed = sizes[(t + k) % len(sizes)]
                got[(t, k)] = ((t + k) % len(sizes), _request(vie, n, seed, st))
        except Exception as e:  # reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(t,)) for t in range(6)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not errors, errors
    torch.cuda.synchronize()
    for i, J in got.values():
        assert torch.equal(J, alone[i])
