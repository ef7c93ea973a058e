"""Full reorthogonalisation in the real inner product Re <a, b> (CPU emulation of the Lanczos pass).

H is real and symmetric, so the Lanczos process of a complex vector is that of H (+) H on its real
and imaginary parts, and only Re <v_i, v_j> = delta_ij has to be enforced.  The emulation runs a few
Krylov steps of a complex state with complex and with real coefficients and compares both with the
spectral exponential: the error and the loss of Re-orthogonality must not grow.  On the smallest
sector the Krylov space nearly exhausts the Ritz values, where Im <v_i, v_j> is free to grow; the
results must not notice.
"""
import numpy as np
import pytest

import workloads
from oracle import basis as ob


def _evolve(H, psi, m, tau, steps, real, store):
    s = np.trace(H) / len(H)
    A = (H - s * np.eye(len(H))).astype(np.float32 if store == np.complex64 else np.float64)
    loss = 0.0
    for _ in range(steps):
        b0 = np.linalg.norm(psi)
        V = np.zeros((m + 1, len(psi)), store)
        V[0] = psi / b0
        al, be = np.zeros(m), np.zeros(m)
        for j in range(m):
            Vd = V[:j + 1].astype(np.complex128)
            u = (A @ V[j]).astype(store)
            c = Vd.conj() @ u.astype(np.complex128)
            if real:
                c = c.real
            al[j] = c[j].real
            w = u.copy()
            for i in range(j + 1):
                w = (w - store(c[i]) * V[i]).astype(store)
            be[j] = np.linalg.norm(w.astype(np.complex128))
            V[j + 1] = (w / be[j]).astype(store)
            loss = max(loss, np.abs((Vd.conj() @ V[j + 1].astype(np.complex128)).real).max())
        T = np.diag(al) + np.diag(be[:m - 1], 1) + np.diag(be[:m - 1], -1)
        lam, Q = np.linalg.eigh(T)
        y = (Q * np.exp(-1j * tau * (lam + s))) @ Q[0]
        psi = b0 * (y @ V[:m].astype(np.complex128))
    return psi, loss


@pytest.mark.parametrize("L,N,hh,m,tau,store,bar", [
    (8, 4, 0.5, 20, 1.0, np.complex128, 1e-12), (12, 6, 1.5, 26, 0.8, np.complex128, 1e-12),
    (8, 4, 0.5, 20, 1.0, np.complex64, 3e-6), (10, 5, 1.5, 24, 0.8, np.complex64, 3e-6)])
def test_real_coefficients_keep_the_error(L, N, hh, m, tau, store, bar):
    h = workloads.quasiperiodic_field(L, hh, workloads.phases(2)[0])
    H = ob.CSR(L, N, 1.0, 1.0, h, True).dense()
    rng = np.random.default_rng(3)
    psi0 = rng.normal(size=len(H)) + 1j * rng.normal(size=len(H))
    psi0 /= np.linalg.norm(psi0)
    lam, Q = np.linalg.eigh(H)
    exact = Q @ (np.exp(-1j * lam * tau * 4) * (Q.T @ psi0))
    out = {r: _evolve(H, psi0, m, tau, 4, r, store) for r in (False, True)}
    err = {r: np.linalg.norm(out[r][0] - exact) for r in out}
    assert err[False] < bar and err[True] < max(2.0 * err[False], bar / 10)
    assert out[True][1] < 4.0 * out[False][1] + 1e-15
    assert abs(np.linalg.norm(out[True][0]) - 1.0) < bar
