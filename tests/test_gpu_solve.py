"""GPU shifted band LU + multi-RHS solves (eq. (10)) against the oracle's
gbtrf-style band LU: pivot rows identical, solutions within tolerance."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import block_from_dev, block_to_dev, dev, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def device():
    return dev()


CASES = [(1, 0, False, 1), (5, 2, True, 3), (70, 3, False, 2), (97, 33, True, 7), (256, 64, True, 33),
         (300, 128, False, 5), (300, 128, True, 40), (129, 31, False, 64)]


@pytest.mark.parametrize("n,b,cplx,nrhs", CASES)
@pytest.mark.parametrize("trans", [0, 1])
def test_fp64_solve_matches_oracle(device, n, b, cplx, nrhs, trans):
    import torch
    import paper_2012_00506_gb300 as pk
    ab = synth.random_band(n, b, 1000 + n + b, cplx)
    lo, hi = oracle.gershgorin(ab)
    c = 0.5 * (lo + hi)
    shifts = np.array([c + 0.05j, lo + 0.3 * (hi - lo) + 0.01j, hi - 0.1 + 0.2j])
    Y = synth.random_subspace(n, nrhs, 2000 + n, True)
    X, ipiv = pk.shifted_solve(to_dev(ab, device), shifts, block_to_dev(Y, device), trans=trans,
                               precision=pk.FP64, return_ipiv=True)
    ipiv = ipiv.cpu().numpy()
    for s, z in enumerate(shifts):
        F, ip, info = oracle.band_lu(ab, z)
        assert info == 0
        Xo = oracle.band_solve(F, ip, b, Y, trans)
        Xg = block_from_dev(X[s])
        assert np.array_equal(ipiv[s], ip)
        err = np.max(np.abs(Xg - Xo)) / np.max(np.abs(Xo))
        assert err < 1e-11, err


@pytest.mark.parametrize("n,b,cplx,nrhs", [(200, 16, True, 40), (300, 64, False, 70), (257, 128, True, 33),
                                           (1000, 128, True, 300), (130, 100, False, 5), (31, 3, True, 129)])
def test_mixed_solve_fp32_class(device, n, b, cplx, nrhs):
    import paper_2012_00506_gb300 as pk
    ab = synth.random_band(n, b, 3000 + n, cplx)
    lo, hi = oracle.gershgorin(ab)
    shifts = np.array([0.5 * (lo + hi) + 0.1j, lo + 0.2 + 0.05j])
    Y = synth.random_subspace(n, nrhs, 4000 + n, True)
    for trans in (0, 1):
        X = pk.shifted_solve(to_dev(ab, device), shifts, block_to_dev(Y, device), trans=trans, precision=pk.MIXED)
        for s, z in enumerate(shifts):
            F, ip, _ = oracle.band_lu(ab, z)
            Xo = oracle.band_solve(F, ip, b, Y, trans)
            err = np.max(np.abs(block_from_dev(X[s]) - Xo)) / np.max(np.abs(Xo))
            assert err < 1e-4, err   # complex64 with FP32 accumulation


def test_band_matmul(device):
    import paper_2012_00506_gb300 as pk
    for cplx in (False, True):
        ab = synth.random_band(333, 21, 55, cplx)
        X = synth.random_subspace(333, 9, 56, cplx)
        Y = block_from_dev(pk.band_matmul(to_dev(ab, device), block_to_dev(X, device)))
        Yo = oracle.band_matvec(ab, X)
        assert np.max(np.abs(Y - (Yo if cplx else Yo.real))) < 1e-13


# The factorization's dispatch: panels of at most 160 rows, of at most 256 (b <= 224) and wider; one CTA per
# system (more systems than clusters), two per SM (more than 152 systems) and clusters of 2, 4 and 8; the last
# block columns and orders that are no multiple of the tile.
@pytest.mark.parametrize("n,b,nshift,precision", [(33, 32, 1, 1), (95, 40, 5, 1), (260, 100, 3, 1), (300, 130, 40, 1),
                                                  (330, 224, 2, 1), (420, 230, 2, 1), (450, 350, 1, 1),
                                                  (129, 31, 160, 1), (100, 33, 80, 1), (64, 64, 50, 1),
                                                  (161, 30, 20, 0), (200, 70, 40, 0), (97, 96, 80, 0), (260, 128, 4, 0)])
def test_factor_dispatch_pivots_and_solutions(device, n, b, nshift, precision):
    import paper_2012_00506_gb300 as pk
    ab = synth.random_band(n, b, 5000 + n + b, True)
    lo, hi = oracle.gershgorin(ab)
    t = (np.arange(nshift) + 0.5) / nshift
    shifts = lo + (hi - lo) * (0.1 + 0.8 * t) + 1j * (hi - lo) * (0.02 + 0.05 * t)
    Y = synth.random_subspace(n, 3, 6000 + n, True)
    for trans in (0, 1):
        X, ipiv = pk.shifted_solve(to_dev(ab, device), shifts, block_to_dev(Y, device), trans=trans,
                                   precision=precision, return_ipiv=True)
        ipiv = ipiv.cpu().numpy()
        for s in sorted({0, nshift // 2, nshift - 1}):
            F, ip, info = oracle.band_lu(ab, shifts[s])
            Xo = oracle.band_solve(F, ip, b, Y, trans)
            err = np.max(np.abs(block_from_dev(X[s]) - Xo)) / np.max(np.abs(Xo))
            if precision == pk.FP64:
                assert np.array_equal(ipiv[s], ip)
            assert err < (1e-11 if precision == pk.FP64 else 1e-4), (s, trans, err)


def test_equal_pivots_take_the_lowest_row(device):
    """Bands whose columns hold entries of equal modulus: the pivot is the first of them, as in gbtrf."""
    import paper_2012_00506_gb300 as pk
    n, b = 150, 40
    ab = np.where(np.arange(b + 1)[None, :] + np.arange(n)[:, None] < n, 1.0, 0.0) * np.where(
        np.arange(b + 1) % 3 == 1, -0.5, 0.5)
    ab[:, 0] = 0.25
    z = np.array([0.25 + 0.5j, 0.75 + 0.0625j])
    Y = synth.random_subspace(n, 2, 77, True)
    for precision in (0, 1):
        X, ipiv = pk.shifted_solve(to_dev(ab, device), z, block_to_dev(Y, device), precision=precision,
                                   return_ipiv=True)
        for s in range(2):
            F, ip, info = oracle.band_lu(ab, z[s])
            k = 33  # while the entries are still exact in both precisions
            assert np.array_equal(ipiv.cpu().numpy()[s][:1], ip[:1])
            if precision == pk.FP64:
                assert np.array_equal(ipiv.cpu().numpy()[s][:k], ip[:k])


# The default column block: 8 (halves of 16-column items), 16, 32 and 64 in FP64, 16 and 32 in complex64 beyond
# the tensor-core solve's bands; column counts at the edges of the blocks.
@pytest.mark.parametrize("precision,b,nshift,nrhs", [(0, 20, 1, 1), (0, 20, 2, 8), (0, 33, 3, 9), (0, 20, 9, 150),
                                                     (0, 20, 70, 33), (0, 20, 152, 65), (1, 140, 2, 17),
                                                     (1, 140, 40, 70)])
def test_default_solve_width(device, precision, b, nshift, nrhs):
    import paper_2012_00506_gb300 as pk
    n = 150
    ab = synth.random_band(n, b, 7000 + b, True)
    lo, hi = oracle.gershgorin(ab)
    t = (np.arange(nshift) + 0.5) / nshift
    shifts = lo + (hi - lo) * t + 0.1j * (hi - lo)
    Y = synth.random_subspace(n, nrhs, 8000 + nrhs, True)
    for trans in (0, 1):
        X = pk.shifted_solve(to_dev(ab, device), shifts, block_to_dev(Y, device), trans=trans, precision=precision)
        for s in sorted({0, nshift - 1}):
            F, ip, _ = oracle.band_lu(ab, shifts[s])
            Xo = oracle.band_solve(F, ip, b, Y, trans)
            err = np.max(np.abs(block_from_dev(X[s]) - Xo)) / np.max(np.abs(Xo))
            assert err < (1e-11 if precision == pk.FP64 else 1e-4), (s, trans, err)


@pytest.mark.parametrize("n,b,cplx", [(70, 5, False), (200, 40, True)])
@pytest.mark.parametrize("s", [-480, 470])
def test_fp64_solve_scales_exactly(device, n, b, cplx, s):
    """Band and shifts times a power of two: the pivots' reciprocals are taken on scaled values, so the
    solution is scaled exactly (no entry of the factors leaves the normal range at these powers)."""
    import paper_2012_00506_gb300 as pk
    ab = synth.random_band(n, b, 77, cplx)
    Y = synth.random_subspace(n, 6, 78, True)
    z = np.array([0.3 + 0.2j, -0.7 + 0.01j])
    f = 2.0 ** s
    X, i0 = pk.shifted_solve(to_dev(ab, device), z, block_to_dev(Y, device), return_ipiv=True)
    Z, i1 = pk.shifted_solve(to_dev(ab * f, device), z * f, block_to_dev(Y, device), return_ipiv=True)
    assert np.array_equal(i0.cpu().numpy(), i1.cpu().numpy())
    assert np.array_equal((Z * f).cpu().numpy(), X.cpu().numpy())


def test_fp64_pivot_reciprocals_are_correctly_rounded(device):
    """Blocks [[z - a, -1], [-1, z - d]] with z = 2^-40 i and d = fl(1 / a): the second pivot is (z - d) minus the
    reciprocal of the first.  In Smith's form the real part of that reciprocal is fl(1 / -a) = -d (the correction
    y^2 / a is below a rounding of a), so the second pivot is imaginary to the last bit, and with it the
    solution's second entry for (0, 1); an error of one unit in the last place would make its real part 1e-4 of it."""
    import paper_2012_00506_gb300 as pk
    nb = 500
    a = 1.0 + np.random.default_rng(2).uniform(size=nb)
    ab = np.zeros((2 * nb, 2))
    ab[0::2, 0] = a
    ab[0::2, 1] = 1.0
    ab[1::2, 0] = 1.0 / a
    Y = np.zeros((2 * nb, 1), dtype=np.complex128)
    Y[1::2] = 1.0
    X = block_from_dev(pk.shifted_solve(to_dev(ab, device), np.array([1j * 2.0 ** -40]), block_to_dev(Y, device))[0])
    assert np.all(X[1::2].real == 0.0) and np.all(X[1::2].imag != 0.0)


# One case per panel kernel: at most 160 rows (with clusters, and two systems per SM), at most 256, wider; complex128.
@pytest.mark.parametrize("b,nshift,precision", [(40, 3, 1), (40, 160, 1), (120, 2, 1), (200, 3, 1), (300, 2, 1),
                                                (40, 2, 0), (70, 40, 0), (128, 80, 0)])
@pytest.mark.parametrize("first", [0, 64])
def test_ties_with_displaced_rows_take_the_lowest_logical_row(device, b, nshift, precision, first):
    """Pairs of columns k, k + 1 of one panel: k takes its pivot (4) from row p, so row k moves down to p; the
    largest entries of column k + 1 are then a 2 in row r and a 2 in the displaced row.  gbtrf takes the one that
    stands higher now, row r if r < p, although the other row was the higher one before.  All numbers are
    dyadic, so pivots and multipliers are exact in both precisions."""
    import paper_2012_00506_gb300 as pk
    rng = np.random.default_rng(b)
    n = first + b + 70
    groups = min(16, (b - 31) // 2)
    rows = first + rng.permutation(np.arange(32, b + 1))[:2 * groups]
    ab = np.zeros((n, b + 1))
    want = first + np.arange(32)
    displaced = 0
    for q in range(groups):
        k, p, r = first + 2 * q, rows[2 * q], rows[2 * q + 1]
        ab[k, p - k] = 4.0
        ab[k, 1] = 2.0
        ab[k + 1, r - k - 1] = 2.0
        want[2 * q:2 * q + 2] = p, min(p, r)
        displaced += r < p
    assert 2 <= displaced < groups
    z = 1j * 0.5 ** (np.arange(nshift) % 3)
    Y = synth.random_subspace(n, 2, 79, True)
    X, ipiv = pk.shifted_solve(to_dev(ab, device), z, block_to_dev(Y, device), precision=precision, return_ipiv=True)
    ipiv = ipiv.cpu().numpy()
    for s in range(nshift):
        assert np.array_equal(ipiv[s][first:first + 32], want)
        if s < 3:
            F, ip, info = oracle.band_lu(ab, z[s])
            assert np.array_equal(ip[first:first + 32], want)
            Xo = oracle.band_solve(F, ip, b, Y, 0)
            assert np.max(np.abs(block_from_dev(X[s]) - Xo)) < (1e-11 if precision == 0 else 1e-4) * np.max(np.abs(Xo))
