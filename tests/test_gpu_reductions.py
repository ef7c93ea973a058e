"""Row splits and sums of the vector kernels at their edges, against the dense oracle.

The dots take 64 threads' rows at a time (128 rows of complex64), one to eight vectors per group
of threads and several units of rows where the vectors are few; the sums over a warp and over the
CTAs are taken on aligned integers.  The sectors here have fewer rows than one unit, odd counts and
counts just beside a multiple of the unit; m runs over every split of the vectors."""
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


def _case(L, N, seed=4):
    h = workloads.quasiperiodic_field(L, 1.2, 0.3)
    H = ob.CSR(L, N, 1.0, 0.8, h, True)
    rng = np.random.default_rng(seed)
    psi0 = rng.normal(size=H.D) + 1j * rng.normal(size=H.D)
    return h, H, psi0 / np.linalg.norm(psi0)


# D = 5, 36, 126, 165, 495, 715: below, beside and above multiples of 64 and 128, odd and even
@pytest.mark.parametrize("L,N", [(5, 1), (9, 2), (9, 4), (11, 3), (12, 4), (13, 4)])
@pytest.mark.parametrize("emulated", [False, True])
def test_general_state_against_eigh(kry, L, N, emulated):
    h, Hc, psi0 = _case(L, N)
    lam, Q = np.linalg.eigh(Hc.dense())
    exact = Q @ (np.exp(-1j * lam * 1.5) * (Q.T @ psi0))
    H = kry.Hamiltonian(kry.Basis(L, N), 1.0, 0.8, h)
    x = torch.from_numpy(psi0).cuda()
    out = torch.empty_like(x)
    for m in (1, 3, 8, 9, 16, 17, 25, 30, 32):
        if m < 3:   # a one- or two-vector Krylov space meets no useful tolerance here
            continue
        tol = 1e-5 if m == 3 else 1e-10
        H.evolve(x, [0.7, 1.5], m=m, tol=tol, psi_out=out, emulated=emulated)
        # the local error budget is tol / 2 per unit of t / t_end
        assert np.linalg.norm(out.cpu().numpy() - exact) <= tol
    out64 = torch.empty_like(x, dtype=torch.complex64)
    for m in (9, 17, 30):
        H.evolve(x.to(torch.complex64), [0.7, 1.5], m=m, tol=1e-6, psi_out=out64)
        # rounding of the storage (2^-24 per operation and step) beside the budget
        assert np.linalg.norm(out64.cpu().numpy() - exact) <= 1e-5


@pytest.mark.parametrize("emulated,scale", [(False, 1e-30), (False, 1e-4), (False, 1.0), (False, 1e4),
                                             (True, 1e-8), (True, 1e4)])
def test_sums_scale_with_the_state(kry, emulated, scale):
    """The integer sums align to the largest value, and the update sums its rounding-level terms in FP32
    only where the vectors' scales fit (2^-40 to 2^40), so an unnormalised state loses nothing: P
    scales with the fourth power of the norm.  (A float-float value below 2^-80 is zero.)"""
    L, N = 11, 5
    h, Hc, psi0 = _case(L, N)
    H = kry.Hamiltonian(kry.Basis(L, N), 1.0, 0.8, h)
    x = torch.from_numpy(psi0).cuda()
    P1, _ = H.evolve(x, [0.5, 2.0], tol=1e-10, emulated=emulated)
    # (the budget is absolute: 1e-10 of the unit state is 1e-10 s of one with norm s, and P is its square)
    P, _ = H.evolve(x * scale, [0.5, 2.0], tol=1e-10 * scale, emulated=emulated)
    assert np.max(np.abs(P / scale**4 - P1)) <= 1e-9


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_non_finite_states_are_refused(kry, bad):
    L, N = 9, 4
    h, _, psi0 = _case(L, N)
    H = kry.Hamiltonian(kry.Basis(L, N), 1.0, 0.8, h)
    x = torch.from_numpy(psi0).cuda()
    x[7] = bad
    with pytest.raises(kry.KryError):
        H.evolve(x, [0.5], tol=1e-10)


@pytest.mark.parametrize("L,N,K", [(11, 5, 1), (11, 5, 3), (20, 7, 1), (14, 7, 10)])
def test_norms_whose_squares_are_subnormal(kry, L, N, K):
    """A state of norm 1e-155 has a squared norm of 1e-310, summed from subnormal squares: it is not zero and the
    evolution runs.  (Both forms of the pass, single and batched.)  The D squares are off by up to half the
    spacing 5e-324 of the subnormal numbers each, so the squared norm by less than D 5e-324 / 1e-310, and psi
    by that times the spectral half-width (below 20) and t."""
    s = 1e-155
    h = np.array([workloads.quasiperiodic_field(L, 1.2, p) for p in workloads.phases(4, K)])
    H = kry.Hamiltonian(kry.Basis(L, N), 1.0, 0.8, h if K > 1 else h[0])
    D = H.basis.dim
    rng = np.random.default_rng(5)
    x = rng.normal(size=(D, K)) + 1j * rng.normal(size=(D, K))
    x = torch.from_numpy((x / np.linalg.norm(x, axis=0)).reshape(-1)).cuda()
    out1, out = torch.empty_like(x), torch.empty_like(x)
    H.evolve(x, [0.5], tol=1e-8, psi_out=out1)
    H.evolve(x * s, [0.5], tol=1e-8 * s, psi_out=out)
    err = torch.linalg.vector_norm((out / s - out1).view(D, K), dim=0).max().item()
    assert err <= 1e-8 + 20.0 * 0.5 * D * 5e-324 / s**2
