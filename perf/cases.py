"""Performance cases: the work users of this library have it do, through its Python binding.

``listed()`` names the fixed cases, ``draw(rng)`` gives more of the same ranges.  A case is a
dict of plain values: ``op`` (what is called), ``kind``, ``n``, ``mu``, ``wavelengths`` across the
box and, where they apply, ``prec``, ``nrhs``, ``mode``.

* ``apply``      one operator apply y = (I + B + K) x on a problem that exists: every solver
                 iteration, the library's and a user's own, is one of these.
* ``solve``      one solve on a problem that exists, from the right-hand sides to the densities.
* ``scattered``  the scattered field of a density.
* ``request``    a whole scattering request with a medium of its own: create the problem, form the
                 right-hand side, solve, release it (what each request of the serving loop does).

Inputs are made from the seed on the GPU: the media of the repository's workloads (one
anisotropic bump for Laplace and Maxwell, four complex-symmetric bumps for Helmholtz), plane
waves of random direction and polarisation, Gaussian vectors for plain applies.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1805_04791_gb300 as vie

LO, HI = -1.0, 1.0
PREC = {"fp32": vie.VIE_FP32, "fp64": vie.VIE_FP64, "df64": vie.VIE_DF64}
MODE = {"mixed": vie.VIE_SOLVE_MIXED, "fp64": vie.VIE_SOLVE_FP64, "bicgstab": vie.VIE_SOLVE_BICGSTAB}


def _case(op, kind, n, mu=False, wavelengths=4.0, name=None, **more):
    c = {"op": op, "kind": kind, "n": n, "mu": mu, "wavelengths": 0.0 if kind == "laplace" else wavelengths, **more}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: an FP32 apply of the electrostatic workload's grid, bound by launches and latency
        _case("apply", "laplace", 32, name="apply_fp32_32", prec="fp32", nrhs=1),
        # the step of the repository's benchmark: the FP32 apply inside a Helmholtz solve
        _case("apply", "helmholtz", 128, name="apply_fp32_128", prec="fp32", nrhs=1),
        # the paper's 150-point mesh, no power of two: what its media are run on
        _case("apply", "maxwell", 150, wavelengths=5.0, name="apply_fp32_150", prec="fp32", nrhs=1),
        # the largest workload: [J; M] with mu at 256^3, ten wavelengths
        _case("apply", "maxwell", 256, mu=True, wavelengths=10.0, name="apply_fp32_256_mu", prec="fp32", nrhs=1),
        # a refinement residual of the mixed solve at a serving size: FP64 vectors, double-word arithmetic
        _case("apply", "helmholtz", 96, name="apply_df64_96", prec="df64", nrhs=1),
        # the electrostatic workload's solve: small grid, many short steps
        _case("solve", "laplace", 32, name="solve_32", mode="mixed", nrhs=1),
        # the acoustic workload's solve
        _case("solve", "helmholtz", 128, name="solve_128", mode="mixed", nrhs=1),
        # several incident waves on one medium with mu, in one lockstep group
        _case("solve", "maxwell", 64, mu=True, name="solve_64_mu_rhs8", mode="mixed", nrhs=8),
        # the paper's solver on its 70-point mesh, FP64 throughout
        _case("solve", "helmholtz", 70, wavelengths=1.0, name="bicgstab_70", mode="bicgstab", nrhs=1),
        # E and H of a solved density at a serving size
        _case("scattered", "maxwell", 64, name="scattered_64", nrhs=1),
        # a mid-sized and the largest request of the serving mix
        _case("request", "helmholtz", 64, wavelengths=3.0, name="request_64", mode="mixed", nrhs=1),
        _case("request", "maxwell", 192, name="request_192", mode="mixed", nrhs=1),
    ]


def _size(rng, lo, hi):
    """A third of the draws are a size of the repository's workloads and the paper's meshes, the others any integer."""
    known = [m for m in (30, 32, 42, 48, 50, 64, 70, 96, 100, 120, 128, 150, 180, 192, 220) if lo <= m <= hi]
    if rng.random() < 1 / 3:
        return rng.choice(known)
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["laplace", "helmholtz", "helmholtz", "maxwell", "maxwell"])
    mu = kind == "maxwell" and rng.random() < 0.4
    op = rng.choice(["apply", "apply", "solve", "solve", "scattered", "request", "request"])

    def waves(most):
        return round(rng.uniform(1.0, most), 2)

    if op == "apply":
        prec = rng.choice(["fp32", "fp32", "df64", "fp64"])
        n = _size(rng, 24, 220 if prec == "fp32" else 128)
        return _case(op, kind, n, mu, waves(5.0), prec=prec, nrhs=rng.choice([1, 1, 2, 3]))
    if op == "solve":
        mode = rng.choice(["mixed", "mixed", "mixed", "fp64", "bicgstab"])
        n = _size(rng, 24, 128 if mode == "mixed" else 72)
        return _case(op, kind, n, mu, waves(4.0 if mode == "mixed" else 2.0), mode=mode,
                     nrhs=rng.choice([1, 1, 4]) if n <= 64 else 1)
    if op == "scattered":
        return _case(op, kind, _size(rng, 24, 128), mu, waves(5.0), nrhs=1)
    return _case(op, kind, _size(rng, 24, 128), mu, waves(4.0), mode="mixed", nrhs=1)


# ------------------------------------------------------------------- inputs


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _nodes(n, dev):
    return LO + (torch.arange(n, dtype=torch.float64, device=dev) + 0.5) * ((HI - LO) / n)


def _rotation(r):
    q, t = np.linalg.qr(r.standard_normal((3, 3)))
    return q * np.sign(np.diag(t))


def _medium(n, bumps, dev):
    """I + sum of g_j S_j, g_j a Gaussian of centre c and squared width w2: [9][n^3] complex128."""
    t = _nodes(n, dev)
    eps = torch.zeros((9, n, n, n), dtype=torch.complex128, device=dev)
    eps[::4] = 1.0
    for c, w2, S in bumps:
        g = [torch.exp(-((t - float(v)) ** 2) / w2) for v in c]
        w = g[2][:, None, None] * g[1][None, :, None] * g[0][None, None, :]
        for k in range(9):
            eps[k] += complex(S[k // 3, k % 3]) * w
    return eps.reshape(9, -1)


def _inputs(case, seed):
    r = np.random.default_rng([int(seed), 7])
    kind, n, dev = case["kind"], case["n"], _device()
    mu = None
    if kind == "helmholtz":
        bumps = []
        for _ in range(4):
            d = r.standard_normal(3)
            c = d / np.linalg.norm(d) * 0.5 * r.random() ** (1 / 3)
            Q = _rotation(r)
            lam = r.uniform(0.5, 2.0, 3) + 1j * r.uniform(0.0, 0.05, 3)
            bumps.append((c, r.uniform(0.15, 0.3) ** 2, r.uniform(0.5, 1.0) * (Q @ np.diag(lam) @ Q.T)))
        eps = _medium(n, bumps, dev)
    else:
        loss = 0.0 if kind == "laplace" else 1.0

        def bump(amp):
            Q = _rotation(r)
            lam = np.array([1.0, 2.0, 3.0]) + 1j * loss * r.uniform(0.0, 0.05, 3)
            return [((0.0, 0.0, 0.0), 0.1, amp * (Q @ np.diag(lam) @ Q.T))]

        eps = _medium(n, bump(0.5), dev)
        if case["mu"]:
            mu = _medium(n, bump(0.3), dev)
    dirs, pols = [], []
    for _ in range(case["nrhs"]):
        d = r.standard_normal(3)
        d /= np.linalg.norm(d)
        p = np.cross(d, r.standard_normal(3))
        dirs.append(d)
        pols.append(p / np.linalg.norm(p))
    return eps, mu, np.array(dirs), np.array(pols)


def _omega(case):
    return 2.0 * math.pi * case["wavelengths"] / (HI - LO)


def _ncomp(case):
    return 6 if case["mu"] else 3


def _vector(case, seed, dtype):
    """Gaussian test vectors (real-valued for electrostatics)."""
    n, dev = case["n"], _device()
    g = torch.Generator(device=dev).manual_seed(int(seed) * 1000003 + 17)
    x = torch.empty((case["nrhs"], _ncomp(case), n, n, n), dtype=dtype, device=dev)
    real = torch.float32 if dtype == torch.complex64 else torch.float64
    for v in x:
        v.copy_(torch.complex(torch.randn(v.shape, generator=g, device=dev, dtype=real),
                              torch.randn(v.shape, generator=g, device=dev, dtype=real)))
    if case["kind"] == "laplace":
        x = torch.complex(x.real, torch.zeros_like(x.real))
    return x


def _density(case, seed):
    """A smooth density with the medium's support, as a solve gives it."""
    t = _nodes(case["n"], _device())
    g = torch.exp(-(t ** 2) / 0.1)
    return _vector(case, seed, torch.complex128) * (g[:, None, None] * g[None, :, None] * g[None, None, :])


def prepare(case, seed):
    eps, mu, d, p = _inputs(case, seed)
    s = {"case": case, "d": d, "p": p if case["kind"] == "maxwell" else None}
    n, c, r = case["n"], _ncomp(case), case["nrhs"]
    if case["op"] == "request":
        s.update(eps=eps, mu=mu)
        return s
    P = vie.Problem(case["kind"], n, LO, HI, _omega(case), eps, mu)
    P._eps = None  # the handle holds what it needs of the medium
    s["P"] = P
    if case["op"] == "apply":
        s["x"] = _vector(case, seed, torch.complex64 if case["prec"] == "fp32" else torch.complex128)
        s["y"] = torch.empty_like(s["x"])
        P.apply(s["x"], s["y"], PREC[case["prec"]], r)  # chooses the schedule, allocates the scratch
    elif case["op"] == "solve":
        s["b"] = torch.empty((r, c, n, n, n), dtype=torch.complex128, device=eps.device)
        P.rhs(d, s["p"], r, s["b"])
        s["J"] = torch.zeros_like(s["b"])
    else:
        s["J"] = _density(case, seed)
        s["f"] = torch.empty((r, 6 if case["kind"] == "maxwell" else 1, n, n, n), dtype=torch.complex128,
                             device=eps.device)
        P.eval_scattered(s["J"], s["f"], r)  # builds the field kernels
    return s


def run(s):
    case = s["case"]
    if case["op"] == "apply":
        s["P"].apply(s["x"], s["y"], PREC[case["prec"]], case["nrhs"])
        return s["y"]
    if case["op"] == "scattered":
        s["P"].eval_scattered(s["J"], s["f"], case["nrhs"])
        return s["f"]
    if case["op"] == "solve":
        s["J"].zero_()
        s["P"].solve(s["b"], s["J"], tol=1e-10, restart=50, mode=MODE[case["mode"]], nrhs=case["nrhs"])
        return s["J"]
    n = case["n"]
    P = vie.Problem(case["kind"], n, LO, HI, _omega(case), s["eps"], s["mu"])
    try:
        b = torch.empty((case["nrhs"], P.ncomp, n, n, n), dtype=torch.complex128, device=s["eps"].device)
        P.rhs(s["d"], s["p"], case["nrhs"], b)
        J = torch.zeros_like(b)
        P.solve(b, J, tol=1e-10, restart=30, mode=MODE[case["mode"]], nrhs=case["nrhs"])
    finally:
        P.close()
    return J


# --------------------------------------------------------------------- work


def _apply_work(case, esz, nrhs):
    """One apply: x and y, the kernel octants and H once; line transforms of the nonzero lines only."""
    n, c = case["n"], _ncomp(case)
    N, M = n ** 3, 2 * n
    narr, nh = (9, 12) if case["mu"] else (6, 6)
    line = 5.0 * M * math.log2(M)
    flops = nrhs * (2 * c * 7 * n * n * line + 8.0 * M ** 3 * (30 if case["mu"] else 9) + 8.0 * N * 3 * c)
    return esz * (2.0 * c * N * nrhs + narr * (n + 1.0) ** 3 + nh * N), flops


def work(case):
    n, c, r = case["n"], _ncomp(case), case["nrhs"]
    if case["op"] == "apply":
        b, f = _apply_work(case, 8 if case["prec"] == "fp32" else 16, r)
        return {"bytes": b, "flops": f}
    if case["op"] == "scattered":
        b, f = _apply_work(case, 16, r)
        return {"bytes": b, "flops": f}
    # a solve takes a few tens of applies (twenty are counted) on tables that are read once
    b, f = _apply_work(case, 8 if case["mode"] == "mixed" else 16, r)
    b, f = max(b, 32.0 * c * r * n ** 3), 20.0 * f
    if case["op"] == "request":
        # the medium is read once; the kernel transforms of the distinct symbols on one octant
        nsym = {"laplace": 2, "helmholtz": 2}.get(case["kind"], 4 if case["mu"] else 3)
        b += 144.0 * (2 if case["mu"] else 1) * n ** 3
        f += nsym * 5.0 * n * n * ((2.25 + 1.5 + 1.0) * 3 * n * math.log2(3 * n) + 3 * 2 * n * math.log2(2 * n))
    return {"bytes": b, "flops": f}


# -------------------------------------------------------------------- exact


class _Exact:
    """The discrete operators in 64 bits with library FFTs: truncated kernels from their Fourier
    series on the (3n)^3 grid, convolutions on the zero-padded (2n)^3 grid."""

    def __init__(self, case, seed):
        eps, mu, self.d, self.p = _inputs(case, seed)
        self.case, self.n, self.w, self.dev = case, case["n"], _omega(case), eps.device
        self.H = [self._h(m) for m in ([eps] if mu is None else [eps, mu])]
        n, sn, D = self.n, 3 * self.n, HI - LO
        m = torch.fft.fftfreq(sn, 1.0 / sn, dtype=torch.float64, device=self.dev)
        self.k = 2.0 * math.pi * m / (3.0 * D)
        self.ko = self.k.clone()
        if sn % 2 == 0:
            self.ko[sn // 2] = 0.0  # the odd factors' mean over both signs of the Nyquist frequency
        j = torch.arange(3 * (sn // 2) ** 2 + 1, dtype=torch.float64, device=self.dev)
        self.table = self._ghat(2.0 * math.pi / (3.0 * D) * torch.sqrt(j), self.w, math.sqrt(3.0) * D)
        mi = m.round().long() ** 2
        self.j2 = mi[:, None, None] + mi[None, :, None] + mi[None, None, :]
        self.idx = torch.cat([torch.arange(n), torch.arange(-(n - 1), 0)]).to(self.dev)
        self.kept = {}

    def _h(self, e):
        A = e.reshape(3, 3, -1).permute(2, 0, 1)
        if self.case["kind"] == "laplace":
            A = A.real.to(torch.complex128)
        eye = torch.eye(3, dtype=torch.complex128, device=e.device)
        n = self.n
        H = torch.cat([torch.linalg.solve(B + eye, B - eye) for B in A.split(1 << 20)])
        return H.permute(1, 2, 0).reshape(3, 3, n, n, n)

    @staticmethod
    def _ghat(kappa, w, L):
        def E(a):
            return L * torch.exp(0.5j * a * L) * torch.sinc(0.5 * a * L / math.pi)

        g = (E(w + kappa) - E(w - kappa)) / (2j * torch.where(kappa == 0, torch.ones_like(kappa), kappa))
        t, wt = np.polynomial.legendre.leggauss(64 + int(w * L))
        r = 0.5 * L * (t + 1.0)
        g[0] = complex(np.sum(0.5 * L * wt * r * np.exp(1j * w * r)))
        return g

    def hat(self, sym):
        """DFT on the (2n)^3 grid of the discrete kernel of a symbol: "" is 1, "x" i k_x, "xy" -k_x k_y."""
        sym = "".join(sorted(sym))
        if sym in self.kept:
            return self.kept[sym]
        F = self.table[self.j2]
        for a in set(sym):
            k = self.k if sym.count(a) == 2 else self.ko
            f = -(k ** 2) if sym.count(a) == 2 else 1j * k
            F *= f.reshape([-1 if ax == "zyx".index(a) else 1 for ax in range(3)])
        F = torch.fft.ifftn(F)
        M, i, s = 2 * self.n, self.idx % (2 * self.n), self.idx % (3 * self.n)
        e = torch.zeros((M, M, M), dtype=torch.complex128, device=self.dev)
        e[i[:, None, None], i[None, :, None], i[None, None, :]] = F[s[:, None, None], s[None, :, None], s[None, None, :]]
        del F
        e = torch.fft.fftn(e)
        if 16.0 * M ** 3 * 10 < 60e9 and self.n <= 200:
            self.kept[sym] = e
        return e

    def conv(self, x, want):
        """For each output the sum over (coefficient, symbol, input component) of its terms."""
        n, M = self.n, 2 * self.n
        X = [torch.fft.fftn(v, s=(M, M, M)) for v in x]
        out = [torch.zeros_like(X[0]) for _ in want]
        for sym in sorted({"".join(sorted(t[1])) for w in want for t in w}):
            K = self.hat(sym)
            for o, w in zip(out, want):
                for cf, s, c in w:
                    if "".join(sorted(s)) == sym:
                        o.addcmul_(K, X[c], value=cf)
            del K
        del X
        return torch.stack([torch.fft.ifftn(o)[:n, :n, :n] for o in out])

    def _terms(self, curl):
        """Rows of W (+ w^2 V for Maxwell) and, with `curl`, i w curl V of the other vector."""
        w, ax = self.w, "xyz"
        mx = self.case["kind"] == "maxwell"

        def rows(o, sg, q):
            t = [[(1.0, ax[a] + ax[b], o + b) for b in range(3)] + ([(w * w, "", o + a)] if mx else [])
                 for a in range(3)] if o is not None else [[] for _ in range(3)]
            if q is not None:
                for a in range(3):
                    b, c = (a + 1) % 3, (a + 2) % 3
                    t[a] += [(sg * 1j * w, ax[b], q + c), (-sg * 1j * w, ax[c], q + b)]
            return t

        return rows, curl

    def apply(self, x):
        kind, mu = self.case["kind"], self.case["mu"]
        rows, _ = self._terms(mu)
        u = self.conv(x, rows(0, 1, 3) + rows(3, -1, 0) if mu else rows(0, 1, None)) + 0.5 * x
        sg = 2.0 if kind == "helmholtz" else -2.0  # H of eps^-1 is -H of eps
        y = x.clone()
        for b, H in enumerate(self.H):
            y[3 * b:3 * b + 3] += sg * torch.einsum("ab...,b...->a...", H, u[3 * b:3 * b + 3])
        return y

    def rhs(self, r):
        kind, d, p = self.case["kind"], self.d[r], self.p[r]
        n, t = self.n, _nodes(self.n, self.dev)
        ph = torch.exp(1j * self.w * (d[0] * t[None, None, :] + d[1] * t[None, :, None] + d[2] * t[:, None, None]))
        if kind == "laplace":
            v = [-d]
            ph = torch.ones((n, n, n), dtype=torch.complex128, device=self.dev)
        elif kind == "helmholtz":
            v = [-1j * self.w * d]
        else:
            v = [p, np.cross(d, p)]
        return torch.cat([2.0 * torch.einsum("ab...,b...->a...", H, torch.stack([complex(c) * ph for c in u]))
                          for H, u in zip(self.H, v)])

    def solve(self, b, tol=3e-14, m=60):
        """Restarted GMRES to the accuracy of 64 bits."""
        x, nb = torch.zeros_like(b), float(torch.linalg.vector_norm(b))
        r = b
        for _ in range(6):
            beta = float(torch.linalg.vector_norm(r))
            if beta <= tol * nb:
                break
            V, Hs = [r / beta], np.zeros((m + 1, m), np.complex128)
            for j in range(m):
                w = self.apply(V[j])
                for _pass in range(2):
                    for i, v in enumerate(V):
                        h = torch.vdot(v.reshape(-1), w.reshape(-1))
                        Hs[i, j] += complex(h)
                        w -= h * v
                Hs[j + 1, j] = float(torch.linalg.vector_norm(w))
                e = np.zeros(j + 2, np.complex128)
                e[0] = beta
                y, *_ = np.linalg.lstsq(Hs[:j + 2, :j + 1], e, rcond=None)
                if np.linalg.norm(Hs[:j + 2, :j + 1] @ y - e) <= 0.5 * tol * nb:
                    break
                V.append(w / Hs[j + 1, j].real)
            for c, v in zip(y, V):
                x += complex(c) * v
            r = b - self.apply(x)
        return x

    def scattered(self, x):
        rows, _ = self._terms(True)
        if self.case["kind"] != "maxwell":
            return self.conv(x, [[(1.0, a, c) for c, a in enumerate("xyz")]])
        if self.case["mu"]:
            return self.conv(x, rows(0, 1, 3) + rows(3, -1, 0))
        return self.conv(x, rows(0, 1, None) + rows(None, -1, 0))


def exact(case, seed):
    E = _Exact(case, seed)
    if case["op"] == "apply":
        x = _vector(case, seed, torch.complex64 if case["prec"] == "fp32" else torch.complex128)
        return torch.stack([E.apply(v.to(torch.complex128)) for v in x])
    if case["op"] == "scattered":
        return torch.stack([E.scattered(v) for v in _density(case, seed)])
    return torch.stack([E.solve(E.rhs(r)) for r in range(case["nrhs"])])
