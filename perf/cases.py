"""Performance cases of the Krylov return-probability library.

Each case is a call that a user's program makes through the public entry points of
paper_1704_02770_gb300: H.v products (`Hamiltonian.apply`), evolutions from a product state or
a dense state (`return_probability`, `autocorrelation`, `evolve`), ensembles of disorder
phases and of initial states (`return_probability_states`), the adjoint gradient (`grad`) and
the sorted-list basis.  Sizes and parameters are those of the repository's workloads, tests
and benchmark, with the evolutions of the large sectors cut to shorter times.

The reference values of `exact` come from a Chebyshev expansion of exp(-iHt) in complex128
with torch gathers over an explicit basis list; it shares no code with the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1704_02770_gb300 as kry

GOLDEN = (math.sqrt(5.0) - 1.0) / 2.0
ELEM = {"c128": 16, "c128e": 16, "c64": 8}
TOL = {"c128": 1e-10, "c128e": 1e-10, "c64": 1e-7}   # error budgets of the repository's workloads


def _case(name, kind, L, N, dtype, K=1, t=0.0, n_times=0, m=30, h=1.5, delta=1.0, pbc=True, lst=False):
    c = dict(kind=kind, L=L, N=N, dtype=dtype, K=K, t=t, n_times=n_times, m=m, h=h, delta=delta, pbc=pbc, list=lst)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one H.v of a small sector: the smallest call, all launch latency
        _case("apply_L16_c128", "apply", 16, 8, "c128", h=2.0),
        # one H.v of a sector whose vector is about the size of L2: a user's own Lanczos or Chebyshev loop
        _case("apply_L26_c64", "apply", 26, 13, "c64"),
        # P(t) of the small workload to t = 100, as run for many parameters: launch-bound
        _case("P_L16_c128", "P", 16, 8, "c128", t=100.0, n_times=40, h=2.0),
        # P(t) and C(t) off half filling, odd length, open chain: an ordinary small study
        _case("C_L19_open_c128e", "C", 19, 8, "c128e", t=20.0, n_times=25, h=1.0, delta=0.7, pbc=False),
        # the benchmark's workload in its three arithmetic forms, cut to shorter times
        _case("P_L24_c64", "P", 24, 12, "c64", t=15.0, n_times=20),
        _case("P_L24_c128", "P", 24, 12, "c128", t=3.0, n_times=12),
        # a dense initial state in, the evolved state out (quench protocols, typicality)
        _case("evolve_L23_c128e", "evolve", 23, 11, "c128e", t=5.0, n_times=8),
        # disorder average: 64 phases at once
        _case("batched_L20_K64_c64", "P", 20, 10, "c64", K=64, t=5.0, n_times=20),
        # ensemble of random product states, each with its own phase, P and C, FP64
        _case("states_L15_K9_c128", "states", 15, 7, "c128", K=9, t=20.0, n_times=15),
        # backward direction: dP/dh_i and dP/dDelta by the adjoint evolution
        _case("grad_L18_c128", "grad", 18, 9, "c128", t=5.0, h=1.0),
        # dilute interacting particles on the Fibonacci ring, sorted-list basis
        _case("P_L55_N4_list_c64", "P", 55, 4, "c64", t=20.0, n_times=15),
        # the largest sector of the workloads: one short-time evolution (one or two Krylov steps)
        _case("P_L30_c64", "P", 30, 15, "c64", t=0.3, n_times=8),
    ]


def _krylov_products(c):
    """H.v products that an evolution to t needs at least, about: the degree at which a polynomial
    of H represents exp(-iHt), with the spectral half-width of an XXZ chain with fields."""
    r = 0.35 * c["L"] + 0.25 * c["L"] * c["h"] / 1.5 if not c["list"] and c["L"] <= 32 else 1.2 * c["N"] + c["h"]
    return max(10.0, r * c["t"] + 10.0)


def _cost(c):
    """A rough cost of one pass, in bytes of Krylov vectors touched (draw keeps it bounded)."""
    D = math.comb(c["L"], c["N"]) * c["K"] * ELEM[c["dtype"]]
    if c["kind"] == "apply":
        return 2.0 * D
    return 40.0 * D * _krylov_products(c) * (3.0 if c["kind"] == "grad" else 1.0) * (3.0 if c["dtype"] == "c128" else 1.0)


def draw(rng):
    while True:
        kind = rng.choice(["apply", "apply", "P", "P", "P", "C", "evolve", "batched", "states", "grad", "list"])
        dtype = rng.choice(["c128", "c64", "c64", "c128e"])
        h = round(rng.uniform(0.2, 3.0), 3)
        delta = round(rng.uniform(0.0, 1.5), 3)
        pbc = rng.random() < 0.7
        m = rng.choice([30, 30, 30, 25, 18])
        t = round(10.0 ** rng.uniform(0.0, 1.5), 4)
        n_times = rng.randint(4, 40)
        if kind == "apply":
            K = rng.choice([1, 1, 1, 5, 32])
            L = rng.randint(10, 27 if K == 1 else 18)
            c = _case(None, "apply", L, L // 2 - rng.randint(0, 2), rng.choice(["c128", "c64"]), K=K, h=h, delta=delta, pbc=pbc)
        elif kind in ("P", "C", "evolve"):
            L = rng.randint(12, 25)
            c = _case(None, kind, L, L // 2 - rng.randint(0, 2), dtype, t=t, n_times=n_times, m=m, h=h, delta=delta, pbc=pbc)
        elif kind == "batched":
            L = rng.randint(10, 20)
            c = _case(None, "P", L, L // 2 - rng.randint(0, 1), dtype, K=rng.choice([3, 16, 31, 64, 100]), t=t, n_times=n_times,
                      m=m, h=h, delta=delta, pbc=pbc)
        elif kind == "states":
            L = rng.randint(10, 18)
            c = _case(None, "states", L, L // 2 - rng.randint(0, 1), dtype, K=rng.choice([2, 9, 33, 64]), t=t, n_times=n_times,
                      m=m, h=h, delta=delta, pbc=pbc)
        elif kind == "grad":
            L = rng.randint(10, 20)
            c = _case(None, "grad", L, L // 2 - rng.randint(0, 1), "c128", t=min(t, 5.0), h=h, delta=delta, pbc=pbc)
        else:
            c = _case(None, "P", rng.randint(33, 60), rng.randint(2, 4), dtype, t=t, n_times=n_times, m=m, h=h, delta=delta, pbc=pbc, lst=True)
        if _cost(c) < 7.0e11:
            return c


# ---------------------------------------------------------------- inputs

def _fields(c, seed):
    """Quasiperiodic fields of K phases drawn from the seed: h_i = h cos(2 pi q i + phi)."""
    rng = np.random.default_rng(seed)
    phi = rng.uniform(0.0, 2.0 * math.pi, size=c["K"])
    i = np.arange(1, c["L"] + 1)
    return c["h"] * np.cos(2.0 * math.pi * GOLDEN * i[None, :] + phi[:, None])


def _spread_state(c):
    """N particles spread evenly over the chain (the Neel state at half filling)."""
    return sum(1 << ((k * c["L"]) // c["N"]) for k in range(c["N"]))


def _states(c, seed):
    if c["kind"] == "states":
        rng = np.random.default_rng(seed + 77)
        return [int(sum(1 << int(p) for p in rng.choice(c["L"], size=c["N"], replace=False))) for _ in range(c["K"])]
    return [_spread_state(c)] * c["K"]


def _times(c):
    if c["kind"] == "grad" or c["n_times"] == 1:
        return [c["t"]]
    t0 = min(0.1, 0.05 * c["t"])
    a, b = math.log(t0), math.log(c["t"])
    return [math.exp(a + (b - a) * k / (c["n_times"] - 1)) for k in range(c["n_times"] - 1)] + [c["t"]]


def _vector(c, seed):
    """A random dense vector (normalised per realisation), the same values in every dtype."""
    D = math.comb(c["L"], c["N"])
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = torch.randn(D * c["K"] * 2, generator=g, device="cuda", dtype=torch.float32)
    x = torch.view_as_complex(x.view(-1, 2))
    if c["dtype"] != "c64":
        x = x.to(torch.complex128)
    x = x.view(D, c["K"])
    return (x / torch.linalg.vector_norm(x, dim=0, keepdim=True)).reshape(-1).contiguous()


def prepare(case, seed):
    basis = kry.Basis(case["L"], case["N"], list=case["list"])
    st = dict(case=case, basis=basis, H=kry.Hamiltonian(basis, 1.0, case["delta"], _fields(case, seed), pbc=case["pbc"]),
              times=np.array(_times(case)) if case["kind"] != "apply" else None, states=_states(case, seed))
    if case["kind"] in ("apply", "evolve"):
        st["x"] = _vector(case, seed)
        st["out"] = torch.empty_like(st["x"])
    return st


def run(state):
    c, H = state["case"], state["H"]
    kw = dict(m=c["m"], tol=TOL[c["dtype"]])
    if c["kind"] == "apply":
        return H.apply(state["x"], out=state["out"])
    if c["kind"] == "evolve":
        P, _ = H.evolve(state["x"], state["times"], psi_out=state["out"], emulated=c["dtype"] == "c128e", **kw)
        return P, state["out"]
    if c["kind"] == "C":
        C, P, _ = H.autocorrelation(state["states"][0], state["times"], dtype=c["dtype"], **kw)
        return C, P
    if c["kind"] == "states":
        P, C, _ = H.return_probability_states(state["states"], state["times"], dtype=c["dtype"], autocorrelation=True, **kw)
        return P, C
    if c["kind"] == "grad":
        P, gh, gd, _ = H.grad(state["states"][0], c["t"], **kw)
        return np.array([P]), gh, np.array([gd])
    P, _ = H.return_probability(state["states"][0], state["times"], dtype=c["dtype"], **kw)
    return P


# ---------------------------------------------------------------- work and tolerance

def work(case):
    """One H.v reads a vector and writes one; every antiparallel bond (about half of them) is a complex
    add.  An evolution needs the products of a polynomial of H; its small results are not counted."""
    n = math.comb(case["L"], case["N"]) * case["K"]
    prods = 1.0 if case["kind"] == "apply" else _krylov_products(case) * (3.0 if case["kind"] == "grad" else 1.0)
    return {"bytes": prods * 2.0 * n * ELEM[case["dtype"]], "flops": prods * n * (case["L"] + 4.0)}


def tolerance(case):
    """H.v: the rounding of a row's sum (measured 2e-16 and 6e-8 against 64 bits).  Evolutions: measured
    against 64 bits P is off by 1e-15 to 6e-14 (FP64 and float-float) and 2e-9 to 5e-7 (complex64) of
    its norm, psi by 2e-12 and 3e-7, the gradient by 4e-12 to 3e-11; the caller's error budgets (1e-10 and 1e-7 on
    P at every time) allow more, since a step that rounding makes a little longer or shorter is as good."""
    if case["kind"] == "apply":
        return {"rel": 1e-15, "max": 1e-14} if case["dtype"] == "c128" else {"rel": 3e-7, "max": 3e-6}
    if case["dtype"] == "c64":
        return {"rel": 2e-6, "max": 2e-5}
    return {"rel": 2e-10, "max": 2e-9} if case["kind"] == "grad" else {"rel": 1e-11, "max": 1e-10}


# ---------------------------------------------------------------- reference in 64 bits

def _popcount(x):
    n = torch.zeros_like(x)
    while bool((x != 0).any()):
        n += x & 1
        x = x >> 1
    return n


class _Reference:
    """H of the sector as gather tables over the explicit sorted basis, complex128 vectors [D, K]."""

    def __init__(self, c, seed):
        L, N, dev = c["L"], c["N"], "cuda"
        if L <= 27:
            parts = [torch.arange(a, min(a + (1 << 24), 1 << L), device=dev) for a in range(0, 1 << L, 1 << 24)]
            s = torch.cat([p[_popcount(p) == N] for p in parts])
        else:
            # every state of N particles in ascending order, highest particle last
            s = torch.zeros(1, dtype=torch.int64, device=dev)
            for k in range(N):
                s = torch.cat([s[s < (1 << p)] | (1 << p) for p in range(k, L)]) if k else \
                    torch.tensor([1 << p for p in range(L)], device=dev)
        self.s, self.D = s, s.numel()
        bonds = [(i, i + 1) for i in range(L - 1)] + ([(L - 1, 0)] if c["pbc"] and L >= 3 else [])
        occ = [((s >> i) & 1).to(torch.float64) - 0.5 for i in range(L)]
        zz = torch.zeros(self.D, dtype=torch.float64, device=dev)
        self.hops = []
        for (i, j) in bonds:
            zz += c["delta"] * occ[i] * occ[j]
            rows = torch.nonzero(occ[i] != occ[j]).squeeze(1)
            to = torch.searchsorted(s, s[rows] ^ ((1 << i) | (1 << j)))
            self.hops.append((rows.to(torch.int32), to.to(torch.int32)))
        f = torch.from_numpy(_fields(c, seed)).to(dev)
        self.diag = zz[:, None] + sum(occ[i][:, None] * f[None, :, i] for i in range(L))
        n_anti = torch.zeros(self.D, dtype=torch.float64, device=dev)
        for rows, _ in self.hops:
            n_anti[rows.long()] += 0.5
        lo, hi = (self.diag - n_anti[:, None]).min().item(), (self.diag + n_anti[:, None]).max().item()
        self.c, self.r = 0.5 * (lo + hi), 0.5 * (hi - lo)

    def apply(self, x):
        y = self.diag * x
        for rows, to in self.hops:
            y.index_add_(0, rows, x.index_select(0, to), alpha=0.5)
        return y

    def index(self, state):
        return int(torch.searchsorted(self.s, torch.tensor([state], device=self.s.device)).item())

    def degree(self, x):
        return int(math.ceil(x + 12.0 * max(x, 1.0) ** (1.0 / 3.0) + 25.0))

    def chebyshev(self, x):
        """T_k((H - c)/r) x for k = 0, 1, ..."""
        scale = lambda v: (self.apply(v) - self.c * v) / self.r   # noqa: E731
        a, b = x, scale(x)
        yield a
        while True:
            yield b
            a, b = b, 2.0 * scale(b) - a

    def coefficients(self, t, deg):
        """exp(-iHt) = sum_k q_k T_k: cosine series of exp(-i r t cos(theta)), [len(t), deg + 1]."""
        t = np.atleast_1d(np.asarray(t, dtype=np.float64))
        n = 1 << int(math.ceil(math.log2(2 * deg + 64)))
        th = 2.0 * math.pi * np.arange(n) / n
        q = np.empty((t.size, deg + 1), dtype=np.complex128)
        for a in range(0, t.size, 512):
            f = np.exp(-1j * self.r * t[a:a + 512, None] * np.cos(th)[None, :])
            q[a:a + 512] = np.fft.fft(f, axis=1)[:, :deg + 1] / n
        q[:, 1:] *= 2.0
        return q * np.exp(-1j * self.c * t)[:, None]

    def evolve(self, x, t):
        deg = self.degree(self.r * abs(t))
        q = self.coefficients([t], deg)[0]
        y = torch.zeros_like(x)
        for k, v in zip(range(deg + 1), self.chebyshev(x)):
            y += complex(q[k]) * v
        return y

    def moments(self, x, deg):
        """<x|T_k|x> per realisation, [deg + 1, K], without a vector kept."""
        return torch.stack([(x.conj() * v).sum(0) for _, v in zip(range(deg + 1), self.chebyshev(x))]).cpu().numpy()

    def P(self, mom, t):
        return np.abs(self.coefficients(t, mom.shape[0] - 1) @ mom) ** 2


def _product_states(ref, c, seed):
    x = torch.zeros(ref.D, c["K"], dtype=torch.complex128, device="cuda")
    for k, s in enumerate(_states(c, seed)):
        x[ref.index(s), k] = 1.0
    return x


def _gradient(ref, c, seed):
    """dA/dtheta = -i int <lambda(s)| dH/dtheta |psi(s)> ds by 16-point Gauss-Legendre on short segments."""
    t, L = c["t"], c["L"]
    gx, gw = np.polynomial.legendre.leggauss(16)
    nseg = max(1, int(math.ceil(2.0 * ref.r * t / 16.0)))
    edges = np.linspace(0.0, t, nseg + 1)
    nodes = np.concatenate([a + 0.5 * (b - a) * (gx + 1.0) for a, b in zip(edges, edges[1:])])
    weights = np.tile(0.5 * (t / nseg) * gw, nseg)
    psi0 = _product_states(ref, c, seed)
    # psi(s_q) and lambda(s_q) = exp(iH(t - s_q)) psi0; H is real and psi0 too, so with the
    # symmetric nodes lambda(s_q) is the conjugate of psi(t - s_q), the mirrored node
    psi, x, now = [], psi0, 0.0
    for q in nodes:
        x, now = ref.evolve(x, q - now), q
        psi.append(x[:, 0])
    A = torch.vdot(psi0[:, 0], ref.evolve(x, t - now)[:, 0])
    dens = torch.zeros(ref.D, dtype=torch.complex128, device="cuda")
    for q in range(len(nodes)):
        dens += float(weights[q]) * psi[len(nodes) - 1 - q] * psi[q]   # conj(lambda) = psi(t - s)
    occ = [((ref.s >> i) & 1).to(torch.float64) - 0.5 for i in range(L)]
    bonds = [(i, i + 1) for i in range(L - 1)] + ([(L - 1, 0)] if c["pbc"] and L >= 3 else [])
    zz = sum(occ[i] * occ[j] for i, j in bonds)
    grad = lambda d: float(2.0 * (A.conj() * (-1j) * (d * dens).sum()).real)   # noqa: E731
    return np.array([float((A.conj() * A).real)]), np.array([grad(o) for o in occ]), np.array([grad(zz)])


def exact(case, seed):
    D = math.comb(case["L"], case["N"])
    if D * case["K"] > 2.2e7 or 27 < case["L"] <= 32:
        return None
    ref = _Reference(case, seed)
    kind = case["kind"]
    if kind == "apply":
        return ref.apply(_vector(case, seed).to(torch.complex128).view(D, case["K"])).reshape(-1)
    # time of the Chebyshev sequence: gathers of 16-byte elements over all bonds
    if ref.degree(ref.r * case["t"]) * case["L"] * (D * case["K"] * 80.0 / 2e12 + 3e-5) > 20.0:
        return None
    if kind == "grad":
        return _gradient(ref, case, seed)
    times = np.array(_times(case))
    deg = ref.degree(ref.r * case["t"])
    x = _vector(case, seed).to(torch.complex128).view(D, -1) if kind == "evolve" else _product_states(ref, case, seed)
    mom = ref.moments(x, deg)
    P = ref.P(mom, times)
    if kind == "evolve":
        return P[:, 0], ref.evolve(x, case["t"]).reshape(-1)
    if kind == "P":
        return P if case["K"] > 1 else P[:, 0]
    # C(t) = (1/t) int_0^t P by 64-point Gauss-Legendre between consecutive output times, split
    gx, gw = np.polynomial.legendre.leggauss(64)
    C, total, last = np.empty_like(P), np.zeros(P.shape[1]), 0.0
    for o, t in enumerate(times):
        n = max(1, int(math.ceil(2.0 * ref.r * (t - last) / 40.0)))
        for a, b in zip(np.linspace(last, t, n + 1), np.linspace(last, t, n + 1)[1:]):
            total = total + 0.5 * (b - a) * (gw @ ref.P(mom, a + 0.5 * (b - a) * (gx + 1.0)))
        last = t
        C[o] = total / t
    return (C[:, 0], P[:, 0]) if kind == "C" else (P, C)
