"""GPU matrix-free H.v (kry_apply) against the oracle CSR SpMV.

Tolerances: complex128, 1e-13 relative to max|y| (FP64 sums of at most L+1 terms in a
different order); complex64, 2e-6 relative (FP32 rounding of the same sums).
"""
import numpy as np
import pytest
import torch

from oracle import basis as ob
import workloads

pytestmark = pytest.mark.gpu

CASES = [(1, 0, True), (1, 1, True), (2, 1, False), (2, 1, True), (3, 1, True), (4, 2, True),
         (5, 2, False), (10, 3, False), (12, 6, True), (16, 8, True), (17, 5, True),
         (20, 10, True), (22, 11, True), (24, 12, True)]


def _vec(D, seed, dtype=torch.complex128):
    g = torch.Generator().manual_seed(seed)
    x = torch.randn(D, dtype=torch.complex128, generator=g)
    return x.to(dtype).cuda()


@pytest.mark.parametrize("L,N,pbc", CASES)
def test_apply_c128(kry, L, N, pbc):
    rng = np.random.default_rng(L * 100 + N)
    J, Delta = 0.8 + rng.random(), rng.normal()
    h = rng.normal(size=L)
    B = kry.Basis(L, N)
    H = kry.Hamiltonian(B, J, Delta, h, pbc=pbc)
    x = _vec(B.dim, L + N)
    y = H.apply(x).cpu().numpy()
    yo = ob.CSR(L, N, J, Delta, h, pbc).matvec(x.cpu().numpy())
    scale = max(np.max(np.abs(yo)), 1e-300)
    assert np.max(np.abs(y - yo)) <= 1e-13 * scale


@pytest.mark.parametrize("L,N,pbc", [(12, 6, True), (16, 8, True), (24, 12, True)])
def test_apply_c64(kry, L, N, pbc):
    h = workloads.quasiperiodic_field(L, 1.5, 0.3)
    B = kry.Basis(L, N)
    H = kry.Hamiltonian(B, 1.0, 1.0, h, pbc=pbc)
    x = _vec(B.dim, 7, torch.complex64)
    y = H.apply(x).cpu().numpy()
    yo = ob.CSR(L, N, 1.0, 1.0, h, pbc).matvec(x.cpu().numpy().astype(np.complex128))
    assert np.max(np.abs(y - yo)) <= 2e-6 * np.max(np.abs(yo))


def test_apply_is_hermitian(kry):
    L, N = 18, 9
    B = kry.Basis(L, N)
    H = kry.Hamiltonian(B, 1.0, 0.7, workloads.quasiperiodic_field(L, 2.0, 1.0), pbc=True)
    x, y = _vec(B.dim, 1), _vec(B.dim, 2)
    lhs = torch.vdot(x, H.apply(y)).item()
    rhs = torch.vdot(H.apply(x), y).item()
    assert abs(lhs - rhs) < 1e-11 * abs(lhs)


def test_apply_L30_sampled_rows(kry):
    """Full-size sector of the L=30 workload: sampled rows against the oracle row builder."""
    L, N = 30, 15
    h = workloads.quasiperiodic_field(L, 1.5, workloads.phases(5)[0])
    B = kry.Basis(L, N)
    H = kry.Hamiltonian(B, 1.0, 1.0, h, pbc=True)
    x = _vec(B.dim, 30)
    y = H.apply(x)
    b = ob.basis(L, N)
    rng = np.random.default_rng(0)
    rows = np.unique(np.concatenate([rng.integers(0, B.dim, 2000), [0, B.dim - 1]]))
    xs = x.cpu().numpy()
    yo = ob.row_apply(L, 1.0, 1.0, h, True, b, xs, rows)
    yg = y[torch.from_numpy(rows).cuda()].cpu().numpy()
    assert np.max(np.abs(yg - yo)) <= 1e-13 * np.max(np.abs(yo))


def test_apply_rejects_bad_arguments(kry):
    B = kry.Basis(8, 4)
    H = kry.Hamiltonian(B, 1.0, 1.0, [0.0] * 8)
    x = _vec(B.dim, 0)
    with pytest.raises(ValueError):
        H.apply(x[:-1])
    assert kry.load().kry_apply(H._h, 0, x.data_ptr(), x.data_ptr(), None) == kry.KRY_EINVAL


def _largest(Hc, h, x):
    """Per row, the scale of the rounding of H x for a real x: its largest hop term, and the terms that add up
    to its diagonal (fields and bonds, which may cancel)."""
    dmax = 0.5 * np.sum(np.abs(h)) + 0.25 * 0.6 * len(h)
    return np.maximum(np.maximum.reduceat(np.abs(Hc.val) * np.abs(x[Hc.col]), Hc.rowptr[:-1]), dmax * np.abs(x))


@pytest.mark.parametrize("L,N", [(2, 1), (3, 1), (5, 2), (8, 4), (9, 1), (9, 8), (11, 6), (13, 6), (16, 3), (17, 8)])
@pytest.mark.parametrize("pbc", [True, False])
def test_apply_edges_of_items(kry, L, N, pbc):
    """Items of 32 lower parts and up to eight upper parts: sectors whose groups are smaller than a warp,
    not a multiple of it, or leave an item's blocks unfilled, on open and closed chains.  The complex128
    sum on aligned integers is bounded as FP64 adds are, the real and the imaginary part each by its own
    largest term."""
    h = workloads.quasiperiodic_field(L, 1.7, 0.9)
    Hc = ob.CSR(L, N, 1.0, 0.6, h, pbc)
    rng = np.random.default_rng(L * 31 + N)
    # values over 60 binary orders, some zero
    x = (rng.normal(size=Hc.D) + 1j * rng.normal(size=Hc.D)) * 2.0 ** rng.integers(-60, 1, size=Hc.D)
    x[rng.random(Hc.D) < 0.1] = 0.0
    H = kry.Hamiltonian(kry.Basis(L, N), 1.0, 0.6, h, pbc=pbc)
    y = H.apply(torch.from_numpy(x).cuda()).cpu().numpy()
    yo = Hc.matvec(x)
    big = _largest(Hc, h, x.real), _largest(Hc, h, x.imag)
    assert np.all(np.abs(y.real - yo.real) <= (L + 4) * 2.0**-52 * big[0] + 1e-300)
    assert np.all(np.abs(y.imag - yo.imag) <= (L + 4) * 2.0**-52 * big[1] + 1e-300)
    big = np.maximum(*big)
    y32 = H.apply(torch.from_numpy(x.astype(np.complex64)).cuda()).cpu().numpy()
    assert np.all(np.abs(y32 - yo) <= (L + 6) * 2.0**-22 * big + 1e-30)


@pytest.mark.parametrize("special", [float("inf"), float("-inf"), float("nan"), 1e-300])
def test_apply_special_values(kry, special):
    """Rows whose neighbours hold values the integer sum cannot (infinities, NaN, below 2^-895) are summed
    in FP64: the same result as the oracle's, and the other rows are untouched."""
    L, N = 10, 5
    h = workloads.quasiperiodic_field(L, 1.0, 0.2)
    Hc = ob.CSR(L, N, 1.0, 1.0, h, True)
    x = np.zeros(Hc.D, np.complex128) if special == 1e-300 else np.ones(Hc.D, np.complex128)
    x[17] = complex(special, 2.0 * special if special == 1e-300 else 1.0)
    y = kry.Hamiltonian(kry.Basis(L, N), 1.0, 1.0, h).apply(torch.from_numpy(x).cuda()).cpu().numpy()
    with np.errstate(invalid="ignore"):
        yo = Hc.matvec(x)
    for a, b in ((y.real, yo.real), (y.imag, yo.imag)):
        assert np.array_equal(np.isfinite(a), np.isfinite(b))
        ok = np.isfinite(b)
        assert np.allclose(a[ok], b[ok], rtol=1e-14, atol=0.0)


@pytest.mark.parametrize("scale", [1e-4, 1e-8, 1e-12, 1e-20, 1e-120, 1e-290, 1e-318])
@pytest.mark.parametrize("L,N", [(6, 3), (13, 6), (16, 8)])
def test_apply_keeps_the_smaller_part(kry, L, N, scale):
    """H is real: a real or imaginary part far below the other (a complex-step derivative, two real vectors in
    one complex one), down to subnormal values, keeps its own accuracy.  (1e-290 and below: the spacing of the
    subnormal numbers, 2^-1074 per term, is added to the bound.)"""
    h = workloads.quasiperiodic_field(L, 1.7, 0.9)
    Hc = ob.CSR(L, N, 1.0, 0.6, h, True)
    rng = np.random.default_rng(L)
    a, b = rng.normal(size=Hc.D), rng.normal(size=Hc.D) * scale
    H = kry.Hamiltonian(kry.Basis(L, N), 1.0, 0.6, h)
    for re, im in ((a, b), (b, a)):
        y = H.apply(torch.from_numpy(re + 1j * im).cuda()).cpu().numpy()
        for got, part in ((y.real, re), (y.imag, im)):
            want = Hc.matvec(part.astype(np.complex128)).real
            assert np.all(np.abs(got - want) <= (L + 4) * (2.0**-52 * _largest(Hc, h, part) + 2.0**-1074))


@pytest.mark.parametrize("value", [float("inf"), 1e-300, 5e-324])
def test_apply_rows_do_not_depend_on_others(kry, value):
    """A value outside the integer sum's range changes the rows it is a neighbour of and no bit of the others."""
    L, N = 13, 6
    h = workloads.quasiperiodic_field(L, 1.7, 0.9)
    Hc = ob.CSR(L, N, 1.0, 0.6, h, True)
    H = kry.Hamiltonian(kry.Basis(L, N), 1.0, 0.6, h)
    rng = np.random.default_rng(3)
    x = rng.normal(size=Hc.D) + 1j * rng.normal(size=Hc.D)
    y = H.apply(torch.from_numpy(x).cuda()).cpu().numpy()
    touched = np.zeros(Hc.D, bool)
    for r in (5, 700, 1300):
        x[r] = complex(value, -value)
        touched |= np.logical_or.reduceat(Hc.col == r, Hc.rowptr[:-1])
        touched[r] = True
    y2 = H.apply(torch.from_numpy(x).cuda()).cpu().numpy()
    assert touched.sum() < 60 and np.array_equal(y[~touched], y2[~touched])
