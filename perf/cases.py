"""Cases that stand for what a program has this library do, each through its public entry
points (paper_1508_02363_gb300.dbar).

A case is a dict of plain values.  `kind` says which call it is:

* ``solve``    CGO solves of one potential for nk values of k (Plan.solve_device, or Plan's
               page-locked host route with io = "host"): the library's main path, from one k
               of a small grid in FP64 to a batch of 128 at 1024^2 in mixed precision.
* ``reflect``  the DS II reflection coefficient r(k) (dbar_reflection), by the iterated
               equation or by the two CGO solves per k.
* ``uneven``   solves on grids of several sizes in one dbar_solve_batches call.
* ``serve``    requests of several grid classes, each with its own potential, submitted to a
               running Server and waited for.
* ``apply``    one application of the operator to nk fields (dbar_apply): a caller's own
               Krylov method, or a check of a solution.
* ``field``    m = h(S) of nk fields (dbar_m_from_S).
* ``fft2``     the 2-D transform of nk fields (dbar_fft2).

Potentials are Gaussian mixtures as in the benchmark and serving workloads (1 to 6 terms,
centres U[-3,3]^2, widths U[0.5,2], |c| U[0,5]); every k is resolved by its grid.  A program
makes one plan per grid and uses it for many potentials and lists of k, so the plan (or the
server) of the case in hand is kept between calls of prepare().
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1508_02363_gb300 import dbar

# --------------------------------------------------------------------------- the cases


def listed():
    return [
        # one CGO solution on a coarse grid in FP64: the smallest call, bound by launches
        _solve("fp64_n64_k1", N=64, L=5.0, nk=1, kmax=1.0, prec="fp64"),
        # many k for one potential, all in FP64 (the 512^2 box of the batched FP64 workload)
        _solve("fp64_n512_k48", N=512, L=8.0, nk=48, kmax=3.0, prec="fp64"),
        # one k at the benchmark's grid: an interactive caller waiting for one solution
        _solve("mixed_n1024_k1", N=1024, L=10.0, nk=1, kmax=8.0, prec="mixed"),
        # the benchmark: 128 k at 1024^2, FP32 inner solves refined to 1e-12
        _solve("mixed_n1024_k128", N=1024, L=10.0, nk=128, kmax=8.0, prec="mixed"),
        # a ragged batch on a small grid, with m on the x-grid as well as S
        _solve("mixed_n256_k37_m", N=256, L=6.0, nk=37, kmax=0.6, prec="mixed", want_m=1),
        # the largest grid, a few large |k|
        _solve("mixed_n2048_k5", N=2048, L=12.0, nk=5, kmax=20.0, prec="mixed"),
        # potential and solutions in page-locked host memory
        _solve("host_n512_k64", N=512, L=6.0, nk=64, kmax=11.0, prec="mixed", io="host"),
        # r(k) on part of the k-grid by the iterated equation (Taylor order 11, thousands of small solves)
        {"name": "reflect_n128_k4096", "kind": "reflect", "N": 128, "L": 3.2, "nk": 4096, "iterated": 1},
        # solves on grids of 128^2 to 2048^2 in one call
        {"name": "uneven_150", "kind": "uneven", "n": 150, "nmax": 2048},
        # a burst of requests to a running server, each with its own potential
        {"name": "serve_24", "kind": "serve", "n": 24, "nmax": 1024},
        # one operator application in the inner precision
        {"name": "apply_n1024_k16_f32", "kind": "apply", "N": 1024, "L": 10.0, "nk": 16, "kmax": 8.0, "fp32": 1},
        # plain 2-D transforms of an odd number of FP64 fields
        {"name": "fft2_n512_k33_f64", "kind": "fft2", "N": 512, "nk": 33, "fp32": 0},
    ]


def _solve(name, N, L, nk, kmax, prec, want_m=0, io="device"):
    return {"name": name, "kind": "solve", "N": N, "L": L, "nk": nk, "kmax": kmax, "prec": prec,
            "want_m": want_m, "io": io}


# box and largest |k| per grid size (N/(2L) >= 2 kmax + 20, the radius where a mixture's transform ends)
_BOX = {128: (5.0, 0.5), 256: (6.0, 0.6), 512: (6.0, 11.0), 1024: (10.0, 8.0), 2048: (12.0, 20.0)}


def draw(rng):
    """One more case: sizes over the range of the listed ones, on a logarithmic scale."""
    kind = rng.choice(["mixed", "mixed", "mixed", "mixed", "fp64", "fp64", "reflect", "uneven", "serve",
                       "apply", "field", "fft2"])
    if kind == "mixed":
        N = rng.choice([128, 256, 512, 1024, 2048])
        L, kmax = _BOX[N]
        nk = _log_int(rng, 1, min(400, (1 << 26) // (N * N)))
        io = "host" if rng.random() < 0.25 else "device"
        return _no_name(_solve("", N, L, nk, kmax, "mixed", want_m=int(io == "device" and rng.random() < 0.25),
                               io=io))
    if kind == "fp64":
        N = rng.choice([64, 128, 256, 512])
        nk = _log_int(rng, 1, min(300, (1 << 23) // (N * N)))
        return _no_name(_solve("", N, 5.0 if N < 512 else 8.0, nk, {64: 0.5, 128: 0.5, 256: 2.0, 512: 3.0}[N],
                               "fp64"))
    if kind == "reflect":
        iterated = int(rng.random() < 0.6)
        return {"kind": "reflect", "N": 128, "L": 3.2, "nk": _log_int(rng, 40, 4096 if iterated else 1200),
                "iterated": iterated}
    if kind == "uneven":
        return {"kind": "uneven", "n": _log_int(rng, 20, 150), "nmax": rng.choice([512, 1024, 2048])}
    if kind == "serve":
        return {"kind": "serve", "n": _log_int(rng, 3, 24), "nmax": rng.choice([512, 1024])}
    N = rng.choice([128, 256, 512, 1024, 2048])
    if kind == "apply":
        L, kmax = _BOX[N]
        fp32 = int(rng.random() < 0.7)
        return {"kind": "apply", "N": N, "L": L, "nk": _log_int(rng, 1, min(300, (1 << 24) // (N * N))),
                "kmax": kmax, "fp32": fp32}
    nk = _log_int(rng, 1, min(300, (1 << 23) // (N * N)))
    if kind == "field":
        return {"kind": "field", "N": N, "L": _BOX[N][0], "nk": nk}
    return {"kind": "fft2", "N": N, "nk": nk, "fp32": rng.choice([0, 1])}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(max(lo, hi))))))


def _no_name(c):
    return {k: v for k, v in c.items() if k != "name"}


# --------------------------------------------------------------------------- inputs


def _x(N, L):
    return L * (-np.pi + 2.0 * np.pi * np.arange(N) / N)


def _mixture(rng, N, L):
    """A sum of 1 to 6 Gaussians on the grid, complex128 [y][x]."""
    t = int(rng.integers(1, 7))
    c, w = rng.uniform(-3.0, 3.0, (t, 2)), rng.uniform(0.5, 2.0, t)
    a = rng.uniform(0.0, 5.0, t) * np.exp(2j * np.pi * rng.uniform(size=t))
    x = _x(N, L)
    gx = np.exp(-((x[None] - c[:, :1]) / w[:, None]) ** 2)
    gy = np.exp(-((x[None] - c[:, 1:]) / w[:, None]) ** 2)
    return np.ascontiguousarray((gy.T * a) @ gx)


def _k_list(rng, nk, kmax):
    """nk values with |k| log-uniform over two decades up to kmax."""
    return np.exp(rng.uniform(math.log(0.0125 * kmax), math.log(kmax), nk)) * np.exp(2j * np.pi * rng.uniform(size=nk))


def _uneven_groups(case, seed):
    """[(N, Q, k)]: per grid size the two potentials of the uneven workload (L = 4), each with its k."""
    rng = np.random.default_rng(seed)
    out = []
    for N, share in ((128, 0.3), (256, 0.3), (512, 0.2), (1024, 0.15), (2048, 0.05)):
        if N > case["nmax"]:
            continue
        X, Y = np.meshgrid(_x(N, 4.0), _x(N, 4.0))
        s = rng.uniform(0.9, 1.1)
        r2 = (X * X + Y * Y) / (s * s)
        pots = [(np.exp(-r2).astype(complex), 13.9)]
        if N > 128:  # the second potential is not resolved at 128^2
            pots.append((np.exp(-r2 * r2 / 4.0) * (1.0 + 0.3 * np.cos(3.0 * X)) + 0j, 20.0))
        count = max(len(pots), int(round(case["n"] * share)))
        for i, (Q, xi_q) in enumerate(pots):
            nk = count // len(pots) + (1 if i < count % len(pots) else 0)
            kmax = min(12.0, (N / 8.0 - xi_q) / 2.0)
            out.append((N, Q, kmax * np.sqrt(rng.uniform(size=nk)) * np.exp(2j * np.pi * rng.uniform(size=nk))))
    return out


def _requests(case, seed):
    """[(N, L, Q, k)] of a burst: the grid classes in turn, each k resolved by its class (L = 6)."""
    rng = np.random.default_rng(seed)
    classes = [c for c in ((256, 0.6), (512, 11.0), (1024, 20.0)) if c[0] <= case["nmax"]]
    out = []
    for i in range(case["n"]):
        N, top = classes[i % len(classes)]
        k = math.exp(rng.uniform(math.log(0.1), math.log(top))) * np.exp(2j * np.pi * rng.uniform())
        out.append((N, 6.0, _mixture(rng, N, 6.0), complex(k)))
    return out


def _fields(rng, nk, N, L):
    """Fourier fields S of smooth decaying functions, complex128 [nk][N][N] on the GPU: transforms
    of Gaussians centred near the origin (closed form 0.5 w^2 e^{-w^2 |xi|^2/4 - i xi.x0})."""
    m = np.arange(N)
    m = np.where(m <= N // 2, m, m - N) / L
    xi = torch.from_numpy(m).cuda()
    w = torch.from_numpy(rng.uniform(0.6, 1.4, nk)).cuda()
    c = torch.from_numpy(rng.uniform(-1.5, 1.5, (nk, 2))).cuda()
    a = torch.from_numpy(rng.standard_normal(nk) + 1j * rng.standard_normal(nk)).cuda()

    def axis(x0):
        return torch.exp(-(w[:, None] ** 2) * xi ** 2 / 4.0 - 1j * x0[:, None] * xi)

    return (0.5 * a * w ** 2)[:, None, None] * axis(c[:, 1])[:, :, None] * axis(c[:, 0])[:, None, :]


def _inputs(case, seed):
    """What is random in a case: host arrays, and for apply / field / fft2 the fields on the GPU."""
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "solve":
        return _mixture(rng, case["N"], case["L"]), _k_list(rng, case["nk"], case["kmax"])
    if kind == "reflect":
        N, L = case["N"], case["L"]
        X, Y = np.meshgrid(_x(N, L), _x(N, L))
        s, c = rng.uniform(0.95, 1.05), rng.uniform(-0.1, 0.1, 2)
        Q = rng.uniform(0.7, 1.3) * np.exp(-((X - c[0]) ** 2 + (Y - c[1]) ** 2) / (s * s)) + 0j
        # k on the xi-grid: all of it for the iterated equation, what the grid resolves for the other
        top = N // 2 if case["iterated"] else 24
        m = np.arange(-top + 1, top + 1 if case["iterated"] else top)
        at = rng.choice(m.size * m.size, case["nk"], replace=False)
        return Q, (m[at % m.size] + 1j * m[at // m.size]) / L
    if kind == "apply":
        Q, k = _mixture(rng, case["N"], case["L"]), _k_list(rng, case["nk"], case["kmax"])
        S = _fields(rng, case["nk"], case["N"], case["L"])
        return Q, k, S.to(torch.complex64) if case["fp32"] else S
    if kind == "field":
        return _fields(rng, case["nk"], case["N"], case["L"])
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn((case["nk"], case["N"], case["N"]), generator=g, device="cuda",
                       dtype=torch.complex64 if case["fp32"] else torch.complex128)


# --------------------------------------------------------------------------- plans, prepare, run

_kept = {}  # the plan(s) or server of the case in hand


def _keep(key, make):
    if key not in _kept:
        _kept.clear()
        _kept[key] = make()
    return _kept[key]


def prepare(case, seed):
    kind = case["kind"]
    key = repr(sorted((k, v) for k, v in case.items() if k != "name"))
    st = {"case": case}
    if kind == "serve":
        st["server"] = _keep(key, lambda: dbar.Server(24 << 30, prec="mixed", tol=1e-12, max_batch=32))
        st["requests"] = _requests(case, seed)
        return st
    if kind == "uneven":
        groups = _uneven_groups(case, seed)

        def plans():
            most = {}
            for N, _, k in groups:
                most[N] = max(most.get(N, 0), k.size)
            return {N: dbar.Plan(N, 4.0, prec="mixed", tol=1e-12, max_batch=nk) for N, nk in most.items()}

        st["plans"] = _keep(key, plans)
        st["batches"] = [{"plan": st["plans"][N].handle, "Q": torch.from_numpy(Q).cuda(), "k": k,
                          "S_out": torch.empty((k.size, N, N), dtype=torch.complex128, device="cuda")}
                         for N, Q, k in groups]
        return st
    N, nk = case["N"], case["nk"]
    if kind == "solve":
        Q, st["k"] = _inputs(case, seed)
        st["plan"] = _keep(key, lambda: dbar.Plan(N, case["L"], M=2, prec=case["prec"], tol=1e-12, max_batch=nk))
        shape = (nk, N, N)
        if case["io"] == "host":
            st["Q"] = torch.from_numpy(Q).pin_memory().numpy()
            st["S"] = torch.empty(shape, dtype=torch.complex128, pin_memory=True).numpy()
        else:
            st["Q"] = torch.from_numpy(Q).cuda()
            st["S"] = torch.empty(shape, dtype=torch.complex128, device="cuda")
            st["m"] = torch.empty_like(st["S"]) if case["want_m"] else None
        return st
    if kind == "reflect":
        Q, st["k"] = _inputs(case, seed)
        st["Q"] = torch.from_numpy(Q).cuda()
        kw = dict(iterated=1, restart=16) if case["iterated"] else {}
        st["plan"] = _keep(key, lambda: dbar.Plan(N, case["L"], M=11, prec="mixed", tol=1e-12, max_batch=nk, **kw))
        return st
    if kind == "apply":
        Q, st["k"], st["S"] = _inputs(case, seed)
        st["Q"] = torch.from_numpy(Q).cuda()
    else:
        st["S"] = _inputs(case, seed)
    st["out"] = torch.empty_like(st["S"])
    L = case.get("L", 4.0)
    prec = "mixed" if case.get("fp32") else "fp64"
    st["plan"] = _keep(key, lambda: dbar.Plan(N, L, M=2, prec=prec, restart=4, max_batch=nk))
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "serve":
        srv = st["server"]
        tickets = [srv.submit(*rq) for rq in st["requests"]]
        return [srv.wait(t)["S"] for t in tickets]
    if kind == "uneven":
        dbar.dbar_solve_batches(st["batches"])
        return [b["S_out"] for b in st["batches"]]
    plan = st["plan"]
    if kind == "solve":
        if case["io"] == "host":
            dbar.dbar_solve_cgo(plan.handle, st["Q"], st["k"], st["S"], io_on_device=False)
            return st["S"]
        plan.solve_device(st["Q"], st["k"], st["S"], st["m"])
        return {"S": st["S"], "m": st["m"]} if case["want_m"] else st["S"]
    if kind == "reflect":
        return dbar.dbar_reflection(plan.handle, st["Q"], st["k"])[0]
    if kind == "apply":
        dbar.dbar_apply(plan.handle, st["Q"], st["k"], st["S"], st["out"], bool(case["fp32"]))
    elif kind == "field":
        dbar.dbar_m_from_S(plan.handle, case["nk"], st["S"], st["out"])
    else:
        dbar.dbar_fft2(plan.handle, case["nk"], st["S"], st["out"], -1, bool(case["fp32"]))
    return st["out"]


def work(case):
    """Inputs read once and outputs written once; flops of the transforms: two 2-D FFTs per
    operator application, about 34 applications for a CGO solve to 1e-12 and 16 (8 steps of two)
    for the iterated equation."""
    kind = case["kind"]

    def fft2(N):
        return 5.0 * N * N * 2.0 * math.log2(N)

    if kind in ("solve", "reflect"):
        n = case["N"] ** 2
        apps = 34 if kind == "solve" else (16 if case["iterated"] else 68)
        out = n * (1 + case.get("want_m", 0)) if kind == "solve" else 1
        return {"bytes": 16.0 * (n + case["nk"] * out), "flops": case["nk"] * apps * 2.0 * fft2(case["N"])}
    if kind == "uneven":
        g = _uneven_sizes(case)
        return {"bytes": sum(16.0 * N * N * (q + c) for N, q, c in g), "flops": sum(c * 68.0 * fft2(N) for N, _, c in g)}
    if kind == "serve":
        Ns = [N for N in (256, 512, 1024) if N <= case["nmax"]]
        Ns = [Ns[i % len(Ns)] for i in range(case["n"])]
        return {"bytes": sum(32.0 * N * N for N in Ns), "flops": sum(68.0 * fft2(N) for N in Ns)}
    n, el = case["nk"] * case["N"] ** 2, 8.0 if case.get("fp32") else 16.0
    q = 16.0 * case["N"] ** 2 if kind == "apply" else 0.0
    return {"bytes": 2.0 * n * el + q, "flops": case["nk"] * {"apply": 2.0, "field": 1.0, "fft2": 1.0}[kind] * fft2(case["N"])}


def _uneven_sizes(case):
    """(N, potentials, solves) per grid size of _uneven_groups."""
    out = []
    for N, share in ((128, 0.3), (256, 0.3), (512, 0.2), (1024, 0.15), (2048, 0.05)):
        if N <= case["nmax"]:
            pots = 2 if N > 128 else 1
            out.append((N, pots, max(pots, int(round(case["n"] * share)))))
    return out


# --------------------------------------------------------------------------- the same in 64 bits


def exact(case, seed):
    """What run() returns, by plain torch in FP64: the three-transform operator of the paper's
    Sec. 4.3 (Sec. 5.3 for the iterated equation) and GMRES on the stacked real system."""
    kind = case["kind"]
    if kind == "serve":
        return [_cgo(Q, [k], N, L, 2)[0][0] for N, L, Q, k in _requests(case, seed)]
    if kind == "uneven":
        return [_cgo(Q, k, N, 4.0, 2)[0] for N, Q, k in _uneven_groups(case, seed)]
    if kind == "solve":
        Q, k = _inputs(case, seed)
        S, g = _cgo(Q, k, case["N"], case["L"], 2)
        return {"S": S, "m": torch.cat([g.h(s[None]) for s in S])} if case["want_m"] else S
    if kind == "reflect":
        Q, k = _inputs(case, seed)
        if case["iterated"]:
            return _reflection_iterated(Q, k, case["N"], case["L"], 11)
        plus, _ = _cgo(Q, k / 2, case["N"], case["L"], 11)
        minus, _ = _cgo(-Q, k / 2, case["N"], case["L"], 11)
        return 0.5j * (plus[:, 0, 0] - minus[:, 0, 0])
    if kind == "apply":
        Q, k, S = _inputs(case, seed)
        g = _Grid(case["N"], case["L"], 2)
        Qd = torch.from_numpy(Q).to(g.X.device)
        return torch.cat([_cgo_apply(g, _ekq(g, Qd, k[i:i + 1]), S[i:i + 1].to(torch.complex128)) for i in range(case["nk"])])
    S = _inputs(case, seed)
    if kind == "field":
        g = _Grid(case["N"], case["L"], 2)
        return torch.cat([g.h(S[i:i + 1]) for i in range(case["nk"])])
    return torch.fft.fft2(S.to(torch.complex128))


class _Grid:
    """x_j = L(-pi + 2 pi j/N), xi_m = m/L, m in [-N/2+1, N/2]; F, its inverse, h(S) of order M."""

    def __init__(self, N, L, M):
        self.N, self.L, self.M = N, L, M
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        x = torch.from_numpy(_x(N, L)).to(dev)
        self.X, self.Y = x[None, :].expand(N, N), x[:, None].expand(N, N)
        self.z = self.X + 1j * self.Y
        m = torch.arange(N, device=dev, dtype=torch.float64)
        m = torch.where(m <= N // 2, m, m - N)
        self.m1, self.m2 = m[None, :].expand(N, N), m[:, None].expand(N, N)
        self.sign = 1.0 - 2.0 * ((self.m1 + self.m2) % 2)
        self.sw = 2.0 * math.pi * L * L / (N * N)
        self.W = [_closed_form(n, self.z) for n in range(M + 1)]

    def F(self, f):
        return self.sw * self.sign * torch.fft.fft2(f)

    def Finv(self, S):
        return torch.fft.ifft2(self.sign * S) / self.sw

    def h(self, S, shift=None):
        """F^{-1}(S/(xi - xi0)) regularised at xi0 (eq. Sreg, fourreg5; eq. dbarinvShift with shift =
        (m1, m2) of xi0 per field)."""
        s = self.Finv(S)
        if shift is None:
            s1 = s2 = torch.zeros((1, 1, 1), dtype=torch.float64, device=S.device)
        else:
            s1, s2 = shift[:, 0, None, None], shift[:, 1, None, None]
        ph = torch.exp(-1j * (s1 * self.X + s2 * self.Y) / self.L)
        p1, p2 = self.m1 % self.N, self.m2 % self.N
        wrap = lambda p: torch.where(p <= self.N // 2, p, p - self.N)  # noqa: E731
        dt = torch.complex(wrap((p1 - s1) % self.N) / self.L, wrap((p2 - s2) % self.N) / self.L)  # on the torus
        d = torch.complex((self.m1 - s1) / self.L, (self.m2 - s2) / self.L)  # at the points as they are
        at0 = dt == 0
        gauss = torch.exp(-(dt.abs() ** 2))
        U = S / torch.where(at0, 1.0, d)
        c, term = [], self.sw * ph * s
        for n in range(self.M + 1):
            c.append((-0.5j) ** n / math.factorial(n) * term.sum((-2, -1), keepdim=True))
            term = term * self.z
        G = sum(c[n] * torch.conj(dt) ** n for n in range(self.M + 1)) * gauss
        fill = -0.5j * (self.sw * torch.conj(self.z) * ph * s).sum((-2, -1), keepdim=True)
        U = torch.where(at0, fill, U - G / torch.where(at0, 1.0, dt))
        return self.Finv(U) + torch.conj(ph) * sum(c[n] * self.W[n] for n in range(self.M + 1))


def _closed_form(n, z):
    """W_n(z) = F^{-1}(conj(xi)^n/xi e^{-|xi|^2}) (eq. fourreg5, and its series near the origin)."""
    a = z.abs() ** 2 / 4.0
    pref = 1j * (2j) ** n * math.factorial(n)
    near = a < n + 1
    an, series, term = torch.where(near, a, 0.0), 0.0, 1.0 / math.factorial(n + 1)
    for j in range(120):
        series = series + term
        term = term * an / (j + n + 2)
    part = sum(a ** r / math.factorial(r) for r in range(n + 1))
    far = pref / torch.where(near, 1.0, z) ** (n + 1) * (1.0 - torch.exp(-a) * part)
    return torch.where(near, pref * (torch.conj(z) / 4.0) ** (n + 1) * torch.exp(-a) * series, far)


def _ekq(g, Q, k):
    k = torch.from_numpy(np.asarray(k, dtype=complex)).to(Q.device)[:, None, None]
    return torch.exp(-2j * (k.imag * g.X + k.real * g.Y)) * Q


def _cgo_apply(g, eq, S):
    return S + 1j * g.F(eq * torch.conj(g.h(S)))


def _cgo(Q, k, N, L, M):
    """S [nk][N][N] of A S = -i F(E_k Q), and the grid."""
    g = _Grid(N, L, M)
    Qd = torch.from_numpy(Q).to(g.X.device)
    step = max(1, (1 << 22) // (N * N))
    out = []
    for i in range(0, len(k), step):
        eq = _ekq(g, Qd, k[i:i + step])
        out.append(_gmres(lambda S: _cgo_apply(g, eq, S), -1j * g.F(eq)))
    return torch.cat(out), g


def _reflection_iterated(q, k, N, L, M):
    """r = i h(i conj k), h - K_0(H(h)) = -i F(q) (eq. eqh2 at k/2), xi0 = i conj k."""
    g = _Grid(N, L, M)
    q = torch.from_numpy(q).to(g.X.device)
    s = torch.from_numpy(np.rint(np.stack([k.imag, k.real], 1) * L)).to(q.device)
    step, out = (1 << 23) // (N * N), []
    for i in range(0, len(k), step):
        si = s[i:i + step]

        def apply(h):
            H = -1j * g.F(q * torch.conj(g.h(h, si)))
            return h + 1j * g.F(q * torch.conj(g.h(H)))

        h = _gmres(apply, (-1j * g.F(q)).expand(len(si), N, N).contiguous())
        at = si.long()
        out.append(1j * h[torch.arange(len(si)), at[:, 1] % N, at[:, 0] % N])
    return torch.cat(out)


def _gmres(apply, b, m=24, tol=2e-14, cycles=8):
    """Restarted GMRES on the stacked real and imaginary parts, all fields of b together."""
    nb, shape = b.shape[0], b.shape
    real = lambda v: torch.view_as_real(v.contiguous()).reshape(nb, -1)  # noqa: E731
    x, bn, last = torch.zeros_like(b), torch.linalg.norm(real(b), dim=1), math.inf
    safe = torch.where(bn > 0, bn, 1.0)
    for _ in range(cycles):
        r = real(b - apply(x))
        beta = torch.linalg.norm(r, dim=1)
        now = float((beta / safe).max())
        if now <= tol or now > 0.5 * last:
            break
        last = now
        V = torch.zeros((nb, m + 1, r.shape[1]), dtype=torch.float64, device=b.device)
        H = torch.zeros((nb, m + 1, m), dtype=torch.float64, device=b.device)
        V[:, 0] = r / torch.where(beta > 0, beta, 1.0)[:, None]
        j = 0
        while j < m:
            w = real(apply(torch.view_as_complex(V[:, j].reshape(shape + (2,)).contiguous())))
            for _twice in range(2):
                c = torch.bmm(V[:, : j + 1], w[:, :, None])
                w = w - torch.bmm(c.transpose(1, 2), V[:, : j + 1])[:, 0]
                H[:, : j + 1, j] += c[:, :, 0]
            n = torch.linalg.norm(w, dim=1)
            H[:, j + 1, j] = n
            V[:, j + 1] = w / torch.where(n > 0, n, 1.0)[:, None]
            j += 1
            if j % 4 == 0:
                e = torch.zeros((nb, j + 1, 1), dtype=torch.float64, device=b.device)
                e[:, 0, 0] = beta
                y = torch.linalg.lstsq(H[:, : j + 1, :j], e).solution
                res = torch.linalg.norm((e - H[:, : j + 1, :j] @ y)[:, :, 0], dim=1)
                if float((res / safe).max()) <= 0.1 * tol:
                    break
        x = x + torch.view_as_complex(torch.bmm(y.transpose(1, 2), V[:, :j])[:, 0].reshape(shape + (2,)).contiguous())
    return x
