"""The one-read form (sectors of 65,536 states and more): the update and the dots of its result in one pass
over the Krylov vectors, with coefficients from the recurrence instead of dots of u.

Sectors just above the line (D = 77,520 and 92,378: neither a multiple of the 64 rows of a unit) and a
sorted-list one; m runs over every split of the vectors (1 to 16 in a group, two groups from 17 on)."""
import numpy as np
import pytest
import torch

import workloads
from oracle import basis as ob

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kry():
    import paper_1704_02770_gb300 as k
    k.load()
    return k


def _setup(kry, L, N, lst=False, hh=1.3):
    h = workloads.quasiperiodic_field(L, hh, 0.7)
    return h, kry.Hamiltonian(kry.Basis(L, N, list=lst), 1.0, 0.8, h)


@pytest.fixture(scope="module")
def reference():
    """psi(0.6) of a fixed dense state in the (20, 7) sector from the oracle's Krylov evolution."""
    L, N = 20, 7
    h = workloads.quasiperiodic_field(L, 1.3, 0.7)
    H = ob.CSR(L, N, 1.0, 0.8, h, True)
    rng = np.random.default_rng(8)
    psi0 = rng.normal(size=H.D) + 1j * rng.normal(size=H.D)
    psi0 /= np.linalg.norm(psi0)
    P, psi, _ = _oracle(H, psi0, [0.3, 0.6])
    return psi0, P, psi


def _oracle(H, psi0, times):
    # power series of exp(-iHt) in steps of 0.05: 30 terms of a norm below 0.05 * 20 = 1, to rounding
    P, psi, t = [], psi0.copy(), 0.0
    for tt in times:
        while t < tt - 1e-12:
            dt = min(0.05, tt - t)
            term = psi.copy()
            for n in range(1, 31):
                term = H.matvec(term) * (-1j * dt / n)
                psi = psi + term
            t += dt
        P.append(abs(np.vdot(psi0, psi)) ** 2)
    return np.array(P), psi, None


# each m ends its step in another split: one group of 1 to 16 vectors with and without an empty slot, then two
@pytest.mark.parametrize("m", [5, 7, 9, 12, 15, 16, 17, 18, 23, 29, 31, 32])
@pytest.mark.parametrize("form", ["c128", "c128e", "c64"])
def test_every_split_against_the_power_series(kry, reference, m, form):
    psi0, P0, psi1 = reference
    _, H = _setup(kry, 20, 7)
    x = torch.from_numpy(psi0).cuda()
    if form == "c64":
        x = x.to(torch.complex64)
    out = torch.empty_like(x)
    tol = 1e-6 if form == "c64" else 1e-10
    P, st = H.evolve(x, [0.3, 0.6], m=m, tol=tol, psi_out=out, emulated=form == "c128e")
    err = np.linalg.norm(out.cpu().numpy() - psi1)
    # the budget, and for complex64 the rounding of the stored vectors, 2^-24 per step and operation
    assert err <= (1e-5 if form == "c64" else tol), err
    assert np.max(np.abs(P - P0)) <= (1e-5 if form == "c64" else tol)
    assert st["n_second_pass"] == 0


@pytest.mark.parametrize("form,bound", [("c128", 5e-14), ("c128e", 2e-12), ("c64", 2e-6)])
def test_orthogonality_and_forced_second_pass(kry, form, bound):
    """The coefficients of the recurrence keep every new vector as orthogonal as dots of u do (the bounds are
    about 1e2 units of roundoff of the vector storage), the check and the forced subtraction change nothing
    beyond it, and the conditional node gives the same bits."""
    L, N = 19, 9
    _, H = _setup(kry, L, N)
    s, times, tol = 0, [0.5, 3.0], 1e-6 if form == "c64" else 1e-10
    s = sum(1 << (2 * i) for i in range(N))
    P0, st0 = H.return_probability(s, times, tol=tol, dtype=form)
    H.orth_check(True)
    P1, st1 = H.return_probability(s, times, tol=tol, dtype=form)
    H.orth_check(2)
    P2, st2 = H.return_probability(s, times, tol=tol, dtype=form)
    H.orth_check(False)
    H.second_pass_node(True)
    P3, st3 = H.return_probability(s, times, tol=tol, dtype=form)
    H.second_pass_node(False)
    print(f"[one-read] {form}: max |<v_i, w>|/||w|| = {st1['max_orth_loss']:.2e}")
    assert 0.0 < st1["max_orth_loss"] <= bound and st0["n_second_pass"] == 0
    # (all but those whose dots are exactly zero, as those of a basis state's first vector, are subtracted)
    assert st2["n_second_dots"] == st2["n_hv"] and st2["n_second_pass"] >= st2["n_hv"] - st2["n_krylov_steps"]
    bar = 1e-6 if form == "c64" else 1e-12
    assert np.max(np.abs(P1 - P0)) <= bar and np.max(np.abs(P2 - P0)) <= bar
    assert np.array_equal(P3, P0)
    m = 30
    assert (st0["n_launches"] - 1) % (3 * m + 2) == 0


@pytest.mark.parametrize("form", ["c128", "c128e", "c64"])
def test_invariant_subspaces(kry, form):
    """Sparse fields: a Krylov space that ends early (no hopping: every basis state is an eigenvector; a
    single bond's worth of weight) is found and P stays exact."""
    L, N = 20, 7
    H = kry.Hamiltonian(kry.Basis(L, N), 0.0, 1.0, workloads.quasiperiodic_field(L, 1.0, 0.1))
    s = (1 << N) - 1
    P, st = H.return_probability(s, [1.0, 10.0], tol=1e-6, dtype=form)
    assert np.max(np.abs(P - 1.0)) <= 1e-6 and st["n_breakdowns"] >= 1


def test_list_basis_agrees_with_the_split_tables(kry):
    L, N = 20, 7
    h, H = _setup(kry, L, N)
    _, Hl = _setup(kry, L, N, lst=True)
    s = sum(1 << (2 * i) for i in range(N))
    for form, tol, bar in (("c128", 1e-10, 1e-12), ("c128e", 1e-10, 1e-12), ("c64", 1e-7, 1e-6)):
        P, _ = H.return_probability(s, [0.5, 4.0], tol=tol, dtype=form)
        Pl, _ = Hl.return_probability(s, [0.5, 4.0], tol=tol, dtype=form)
        assert np.max(np.abs(P - Pl)) <= bar


def test_profile_and_shapes(kry):
    """Kind 0 (pass A's dots) stays empty and the update's bytes are one read; shapes give equal results."""
    L, N, m = 20, 7, 30
    _, H = _setup(kry, L, N)
    s = sum(1 << (2 * i) for i in range(N))
    P0, _ = H.return_probability(s, [2.0], m=m)
    H.profile(True)
    P1, st = H.return_probability(s, [2.0], m=m)
    pr = H.profile_read()
    H.profile(False)
    vec = H.basis.dim * 16 * st["n_krylov_steps"]
    assert np.array_equal(P0, P1)
    assert pr["dots"]["launches"] == 0 and pr["update"]["launches"] == m * pr["smallexp"]["launches"]
    assert pr["update"]["bytes"] == pytest.approx(vec * sum(j + 3 for j in range(m)), rel=1e-12)
    assert pr["hv"]["bytes"] == pytest.approx(vec * 2 * m, rel=1e-12)
    for shape in ([0, 1, 0, 2, 0], [0, 2, 0, 2, 0], [0, 3, 1, 4, 0], [77, 0, 0, 1, 0]):
        H.set_shape(shape)
        P, _ = H.return_probability(s, [2.0], m=m)
        assert np.max(np.abs(P - P0)) <= 1e-12


# 32,768 elements and more: groups of 64 threads with one to many states (K = 10, 16, 31, 64), of 128 (33,
# 100, 128), units that do not divide the elements, a thread per element in the H.v up to K = 16
@pytest.mark.parametrize("K", [10, 16, 17, 31, 33, 64, 100, 128])
@pytest.mark.parametrize("form", ["c128", "c128e", "c64"])
def test_batched_against_single_realisations(kry, K, form):
    L, N = 14, 7
    h = np.array([workloads.quasiperiodic_field(L, 1.3, p) for p in workloads.phases(9, K)])
    B = kry.Basis(L, N)
    H = kry.Hamiltonian(B, 1.0, 0.8, h)
    states = workloads.random_basis_states(L, N, 5, K)
    times, tol = [0.4, 1.5, 4.0], 1e-7 if form == "c64" else 1e-10
    # (the common step is the smallest of the realisations', so the errors differ within the budgets)
    bar = 2e-6 if form == "c64" else 1e-11
    P, C, st = H.return_probability_states(states, times, m=30, tol=tol, dtype=form, autocorrelation=True)
    P18, _ = H.return_probability_states(states, times, m=18, tol=tol, dtype=form)
    assert np.max(np.abs(P18 - P)) <= 10 * bar
    H.orth_check(True)
    P2, st2 = H.return_probability_states(states, times, m=30, tol=tol, dtype=form)
    H.orth_check(False)
    assert st["n_second_pass"] == 0 and np.max(np.abs(P2 - P)) <= bar
    assert 0.0 < st2["max_orth_loss"] <= (2e-6 if form == "c64" else 2e-12)
    for k in (0, K // 2, K - 1):
        Hk = kry.Hamiltonian(B, 1.0, 0.8, h[k])
        Ck, Pk, _ = Hk.autocorrelation(states[k], times, m=30, tol=tol, dtype=form)
        assert np.max(np.abs(P[:, k] - Pk)) <= bar and np.max(np.abs(C[:, k] - Ck)) <= bar


@pytest.mark.parametrize("K", [12, 40])
@pytest.mark.parametrize("form", ["c128", "c128e", "c64"])
def test_batched_general_state_and_idle_realisations(kry, K, form):
    """Dense initial states with psi_out, and realisations whose Krylov space ends at once beside others that
    run on (their vectors stay zero)."""
    L, N = 14, 7
    h = np.array([workloads.quasiperiodic_field(L, 1.3, p) for p in workloads.phases(9, K)])
    B = kry.Basis(L, N)
    H = kry.Hamiltonian(B, 1.0, 0.8, h)
    D = B.dim
    rng = np.random.default_rng(2)
    x = rng.normal(size=(D, K)) + 1j * rng.normal(size=(D, K))
    x /= np.linalg.norm(x, axis=0)
    dt = torch.complex64 if form == "c64" else torch.complex128
    tol = 1e-6 if form == "c64" else 1e-10
    xs = torch.from_numpy(x.reshape(-1)).cuda().to(dt)
    out = torch.empty_like(xs)
    P, _ = H.evolve(xs, [0.5, 1.0], tol=tol, psi_out=out, emulated=form == "c128e")
    got = out.cpu().numpy().reshape(D, K)
    for k in (0, K - 1):
        Hk = kry.Hamiltonian(B, 1.0, 0.8, h[k])
        o1 = torch.empty(D, dtype=dt, device="cuda")
        P1, _ = Hk.evolve(xs.view(D, K)[:, k].contiguous(), [0.5, 1.0], tol=tol, psi_out=o1, emulated=form == "c128e")
        assert np.linalg.norm(got[:, k] - o1.cpu().numpy()) <= (1e-5 if form == "c64" else tol)
        assert np.max(np.abs(P[:, k] - P1)) <= (1e-5 if form == "c64" else tol)
    # the ferromagnetic state of N = L is an eigenstate; in this sector a state of one domain with J = 0
    H0 = kry.Hamiltonian(B, 0.0, 1.0, h)
    P0, st0 = H0.return_probability((1 << N) - 1, [1.0, 5.0], tol=1e-6, dtype=form)
    assert np.max(np.abs(P0 - 1.0)) <= 1e-6 and st0["n_breakdowns"] >= K


@pytest.mark.parametrize("exponent", [133, 60, -30])
@pytest.mark.parametrize("K", [1, 10])
def test_recurrence_is_free_of_the_scale_of_H(kry, K, exponent):
    """2^e H over times 2^-e t is the same evolution (2^133 is beyond the range of FP32): the coefficients of
    the recurrence are kept over beta_i, so P, the orthogonality of the vectors and the number of subtractions
    do not notice.  (Below about 2^-40 the absolute floor of the small exponential's half-width, 1e-12, would
    shorten the steps.)"""
    L, N = (20, 7) if K == 1 else (14, 7)
    s = sum(1 << (2 * i) for i in range(N))
    h = np.array([workloads.quasiperiodic_field(L, 1.3, p) for p in workloads.phases(9, K)])
    B = kry.Basis(L, N)
    f = 2.0**exponent
    times = np.array([0.5, 2.0])
    out = []
    for J, hh, t in ((1.0, h, times), (f, f * h, times / f)):
        H = kry.Hamiltonian(B, J, 0.8, hh if K > 1 else hh[0])
        H.orth_check(True)
        out.append(H.return_probability(s, t, tol=1e-10))
    (P1, st1), (P2, st2) = out
    print(f"[scale 2^{exponent}] K={K}: |dP| {np.max(np.abs(P2 - P1)):.1e}, loss {st1['max_orth_loss']:.1e} and {st2['max_orth_loss']:.1e}")
    assert np.max(np.abs(P2 - P1)) <= 1e-10
    assert st2["n_second_pass"] == 0 and 0.0 < st2["max_orth_loss"] <= (5e-14 if K == 1 else 2e-12)


@pytest.mark.parametrize("K", [10, 40, 64])
@pytest.mark.parametrize("form,eps,tol", [("c128", 1e-8, 1e-10), ("c128e", 1e-8, 1e-10), ("c64", 5e-5, 2e-5)])
def test_batched_second_pass_of_some_realisations(kry, K, form, eps, tol):
    """States within eps of an eigenvector: the first update cancels all but eps of H v, so its dots exceed the
    threshold and pass C2 subtracts them, in these realisations alone (0, 3 and K - 1); realisation 1 is the
    eigenvector itself, whose Krylov space ends at once, and the others are random.  Where the corrected
    coefficients were wrong the part of size eps would be, above the tolerance.  (complex64: the rounding of
    H v leaves ||w|| = 4e-7 for the eigenvector, and the step's budget, 0.05 tol / t_end, has to be above it.)"""
    from scipy.sparse import csr_matrix
    from scipy.sparse.linalg import eigsh
    L, N = 14, 7
    h = np.array([workloads.quasiperiodic_field(L, 1.3, p) for p in workloads.phases(9, K)])
    H = kry.Hamiltonian(kry.Basis(L, N), 1.0, 0.8, h)
    D = H.basis.dim
    rng = np.random.default_rng(6)
    x = rng.normal(size=(D, K)) + 1j * rng.normal(size=(D, K))
    x /= np.linalg.norm(x, axis=0)
    csr, near = {}, (0, 3, K - 1)
    for k in near + (1,):
        csr[k] = ob.CSR(L, N, 1.0, 0.8, h[k], True)
        A = csr_matrix((csr[k].val, csr[k].col, csr[k].rowptr), shape=(D, D))
        v = eigsh(A, k=1, which="SA", tol=1e-15, v0=np.ones(D))[1][:, 0]
        x[:, k] = v + (eps * x[:, k] if k != 1 else 0.0)
        x[:, k] /= np.linalg.norm(x[:, k])
    xs = torch.from_numpy(x.reshape(-1)).cuda()
    if form == "c64":
        xs = xs.to(torch.complex64)
    out = torch.empty_like(xs)
    P, st = H.evolve(xs, [0.3, 0.6], tol=tol, psi_out=out, emulated=form == "c128e")
    got = out.cpu().numpy().reshape(D, K)
    print(f"[second pass] K={K} {form}: {st['n_second_pass']} of {st['n_hv'] * K} updates")
    assert 3 * st["n_krylov_steps"] <= st["n_second_pass"] < 3 * st["n_hv"] and st["n_breakdowns"] >= st["n_krylov_steps"]
    csr[2] = ob.CSR(L, N, 1.0, 0.8, h[2], True)
    x0 = xs.cpu().numpy().reshape(D, K).astype(np.complex128)
    for k in csr:
        Pk, psi, _ = _oracle(csr[k], x0[:, k].copy(), [0.3, 0.6])
        err = np.linalg.norm(got[:, k] - psi)
        assert err <= tol and np.max(np.abs(P[:, k] - Pk)) <= tol, (k, err)


@pytest.mark.parametrize("L,N,hh", [(8, 4, 0.5), (10, 5, 1.5), (20, 7, 1.3)])
def test_complex64_keeps_psi_over_many_steps(kry, L, N, hh):
    """The real inner product leaves Im <v_i, v_j> to itself, which rounding lets grow where Ritz values converge
    (small sectors).  Over many steps in complex64 the norm of psi and psi itself must not notice: the reference
    is the spectral exponential, in the largest sector the FP64 evolution.  The bar: every step rounds its 31
    vectors' combination and each product by 2^-24 (an error that turns with the state, so the steps' add up
    at worst linearly), and the budget tol."""
    h = workloads.quasiperiodic_field(L, hh, 0.3)
    H = kry.Hamiltonian(kry.Basis(L, N), 1.0, 1.0, h)
    D = H.basis.dim
    rng = np.random.default_rng(3)
    psi0 = rng.normal(size=D) + 1j * rng.normal(size=D)
    psi0 /= np.linalg.norm(psi0)
    x = torch.from_numpy(psi0).cuda()
    t, out = 200.0 if D < 1000 else 40.0, torch.empty_like(x)
    if D < 1000:
        lam, Q = np.linalg.eigh(ob.CSR(L, N, 1.0, 1.0, h, True).dense())
        exact = Q @ (np.exp(-1j * lam * t) * (Q.T @ psi0))
    else:
        H.evolve(x, [t], tol=1e-10, psi_out=out)
        exact = out.cpu().numpy()
    o64 = torch.empty_like(x, dtype=torch.complex64)
    _, st = H.evolve(x.to(torch.complex64), [t], tol=1e-6, psi_out=o64)
    got = o64.cpu().numpy().astype(np.complex128)
    err, drift = np.linalg.norm(got - exact), abs(np.linalg.norm(got) - 1.0)
    print(f"[c64 psi] L={L}: {st['n_krylov_steps']} steps, |dpsi| {err:.2e}, | ||psi|| - 1 | {drift:.2e}")
    assert st["n_krylov_steps"] >= 10
    assert err <= 1e-6 + st["n_hv"] * 2.0**-24 and drift <= 1e-6 + st["n_krylov_steps"] * 2.0**-22


@pytest.mark.parametrize("K", [1, 10, 40])
@pytest.mark.parametrize("lst", [False, True])
@pytest.mark.parametrize("general", [False, True])
def test_complex64_early_P_of_a_basis_state(kry, K, lst, general):
    """P sees the other vectors' components along psi0 at first order.  From a basis state alpha_0 and beta_0 are
    exact in complex64 (sums of a few multiples of J / 2), so 1 - P is right in second order of t and rounding
    enters with the fourth, as a few 2^-24 of (1 - P)^2: given that every update takes off its whole dot with
    psi0, the rounding of H v included.  As a basis state and as the same state in a dense vector."""
    L, N = (20, 7) if K == 1 else (14, 7)
    s = sum(1 << ((k * L) // N) for k in range(N))
    h = np.array([workloads.quasiperiodic_field(L, 0.7, p) for p in workloads.phases(9, K)])
    B = kry.Basis(L, N, list=lst)
    H = kry.Hamiltonian(B, 1.0, 1.0, h if K > 1 else h[0])
    times = [0.02, 0.05, 0.1, 0.2]
    P8, _ = H.return_probability(s, times, tol=1e-10)
    if general:
        x = torch.zeros(B.dim, K, dtype=torch.complex64, device="cuda")
        x[int(B.rank(torch.tensor([s], device="cuda"))[0])] = 1.0
        P4, _ = H.evolve(x.reshape(-1), times, tol=1e-8)
    else:
        P4, _ = H.return_probability(s, times, tol=1e-8, dtype="c64")
    print(f"[early P] K={K} list={lst} general={general}: {np.max(np.abs(P4 - P8) / (1 - P8)**2) * 2**24:.2f} x 2^-24 (1 - P)^2")
    assert np.all(np.abs(P4 - P8) <= 4.0 * 2.0**-24 * (1.0 - P8)**2 + 1e-13)


@pytest.mark.parametrize("K", [1, 10])
@pytest.mark.parametrize("form,eps", [("c128", 2.0**-53), ("c128e", 2.0**-48)])
def test_eigenvector_keeps_its_phase(kry, K, form, eps):
    """From an eigenvector the first update leaves rounding alone.  The Krylov space ends there, and the dots of
    that rest are still taken off: they refine alpha_0, whose error turns the phase by t times as much.  Bar: one
    rounding of the energy, eps |E| t, and what the eigenvector itself is off by (its residual, times t)."""
    from scipy.sparse import csr_matrix
    from scipy.sparse.linalg import eigsh
    L, N = (20, 7) if K == 1 else (14, 7)
    h = workloads.quasiperiodic_field(L, 1.3, 0.7)
    c = ob.CSR(L, N, 1.0, 0.8, h, True)
    A = csr_matrix((c.val, c.col, c.rowptr), shape=(c.D, c.D))
    lam, V = eigsh(A, k=1, which="SA", tol=1e-15, v0=np.ones(c.D))
    E, v = lam[0], V[:, 0] / np.linalg.norm(V[:, 0])
    t, res = 3.0, np.linalg.norm(A @ v - E * v)
    H = kry.Hamiltonian(kry.Basis(L, N), 1.0, 0.8, np.tile(h, (K, 1)) if K > 1 else h)
    x = torch.from_numpy(np.repeat(v[:, None], K, axis=1).astype(np.complex128).reshape(-1)).cuda()
    out = torch.empty_like(x)
    _, st = H.evolve(x, [t], tol=1e-10, psi_out=out, emulated=form == "c128e")
    err = np.linalg.norm(out.cpu().numpy().reshape(-1, K) - (np.exp(-1j * t * E) * v)[:, None], axis=0).max()
    print(f"[eigenvector] K={K} {form}: |dpsi| {err:.1e}, eps |E| t {eps * abs(E) * t:.1e}, residual t {res * t:.1e}")
    assert st["n_breakdowns"] >= K and st["n_second_pass"] >= 1
    assert err <= eps * abs(E) * t + 2.0 * res * t + 1e-14
