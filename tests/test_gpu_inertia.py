"""GPU inertia (Sylvester counts by pivot-free LDL^T, Section 3.2) against the
oracle: counts and every pivot must be bit-identical."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import dev, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def device():
    return dev()


CASES = [(1, 0, False, 1), (2, 1, True, 2), (37, 3, True, 3), (200, 7, False, 4), (257, 32, False, 5),
         (300, 64, True, 6), (333, 128, True, 7), (150, 120, False, 8), (64, 63, True, 9), (500, 1, False, 10),
         # widest bands with the window in shared memory, and past it (window in the workspace)
         (420, 149, True, 11), (450, 194, False, 12), (400, 150, True, 13), (460, 195, False, 14),
         # n not above b: the window is the whole matrix
         (100, 149, True, 15)]


@pytest.mark.parametrize("n,b,cplx,seed", CASES)
def test_counts_and_pivots_bit_exact(device, n, b, cplx, seed):
    import paper_2012_00506_gb300 as pk
    ab = synth.random_band(n, b, 500 + seed, cplx)
    lo, hi = oracle.gershgorin(ab)
    rng = np.random.default_rng(seed)
    sig = np.concatenate([np.linspace(lo - 0.1, hi + 0.1, 7), rng.uniform(lo, hi, 5)])
    neg, piv = pk.inertia(to_dev(ab, device), sig, pivots=True)
    piv = piv.cpu().numpy()
    for s_i, s in enumerate(sig):
        c, d = oracle.inertia(ab, s, return_pivots=True)
        assert neg[s_i] == c
        assert np.array_equal(piv[s_i], d), (s_i, np.max(np.abs(piv[s_i] - d)))


def test_padded_leading_dimension(device):
    import paper_2012_00506_gb300 as pk
    ab = synth.random_band(120, 5, 77, True)
    abp = synth.pad_band(ab, 9)
    sig = [-0.3, 0.0, 0.41]
    assert list(pk.inertia(to_dev(abp, device), sig, b=5)) == [oracle.inertia(ab, s) for s in sig]


def test_laplacian_closed_form_full_size(device):
    import paper_2012_00506_gb300 as pk
    m, k = 63, 32
    ab = synth.laplacian_2d_band(m, k)
    i = np.arange(1, m + 1)[:, None]
    j = np.arange(1, k + 1)[None, :]
    ev = np.sort((4 - 2 * np.cos(i * np.pi / (m + 1)) - 2 * np.cos(j * np.pi / (k + 1))).ravel())
    u = np.unique(np.round(ev, 12))
    sig = 0.5 * (u[:-1] + u[1:])[::37]
    neg = pk.inertia(to_dev(ab, device), sig)
    assert all(neg[t] == np.sum(ev < s) for t, s in enumerate(sig))


def test_zero_pivot_rule(device):
    import paper_2012_00506_gb300 as pk
    d = np.array([0.5, -1.0, 2.0, -1.0, 0.0, 3.0])
    ab = synth.diagonal_band(d, 2)
    neg, piv = pk.inertia(to_dev(ab, device), [-1.0, 0.0], pivots=True)
    assert list(neg) == [oracle.inertia(ab, -1.0), oracle.inertia(ab, 0.0)] == [2, 3]
    assert np.sum(piv.cpu().numpy()[0] == -oracle.pivmin(ab)) == 2


def test_bisection_enclosures(device):
    import paper_2012_00506_gb300 as pk
    ab = synth.random_band(400, 9, 99, True)
    ev = np.linalg.eigvalsh(synth.band_to_dense(ab))
    idx = [0, 57, 200, 399]
    lo, hi = pk.bisect(to_dev(ab, device), idx, rtol=1e-13, fanout=8)
    for t, k in enumerate(idx):
        assert lo[t] <= ev[k] < hi[t] + 1e-15
        assert hi[t] - lo[t] <= 1e-13 * max(1.0, abs(lo[t]), abs(hi[t]))
        assert oracle.inertia(ab, lo[t]) <= k < oracle.inertia(ab, hi[t])
    # same FP64 operations in the same order on both sides: identical bits
    for ab2 in (ab, synth.random_band(301, 17, 98, False), synth.mixture_band(1000, 40, 97, is_complex=True)):
        glo, ghi = pk.gershgorin(to_dev(ab2, device))
        olo, ohi = oracle.gershgorin(ab2)
        assert (glo, ghi) == (olo, ohi), (glo - olo, ghi - ohi)


# The panel kernel eliminates 8 columns per round on a cluster whose size depends on b and the number
# of shifts: orders and bandwidths around multiples of 8, bands narrower than a panel, n <= b, and
# shift counts that reach the largest cluster (1 shift), smaller ones and one CTA per shift.
@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("n,b,nsig", [(7, 2, 1), (8, 8, 1), (9, 9, 40), (17, 16, 2), (63, 5, 1), (64, 24, 90),
                                      (65, 25, 1), (130, 31, 60), (129, 33, 1), (143, 66, 1), (150, 57, 30),
                                      (31, 70, 2), (200, 149, 1), (190, 129, 20), (210, 200, 1)])
def test_panel_edges_bit_exact(device, n, b, nsig, cplx):
    import paper_2012_00506_gb300 as pk
    ab = synth.random_band(n, b, 900 + n + b, cplx)
    lo, hi = oracle.gershgorin(ab)
    sig = np.random.default_rng(n).uniform(lo, hi, nsig)
    neg, piv = pk.inertia(to_dev(ab, device), sig, pivots=True)
    piv = piv.cpu().numpy()
    for i, s in enumerate(sig):
        c, d = oracle.inertia(ab, s, return_pivots=True)
        assert neg[i] == c
        assert np.array_equal(piv[i], d)


def test_panel_zero_pivots_and_nan(device):
    """Exactly zero pivots (a diagonal band whose entries meet the shift, a band of zeros below the
    diagonal) become -pivmin and count as negative; a NaN in the band is reported."""
    import paper_2012_00506_gb300 as pk
    for b in (3, 20):
        ab = np.zeros((100, b + 1))
        ab[:, 0] = np.arange(100) % 7 - 3.0
        sig = [-3.0, 0.0, 0.5, 3.0]
        neg, piv = pk.inertia(to_dev(ab, device), sig, pivots=True)
        for i, s in enumerate(sig):
            c, d = oracle.inertia(ab, s, return_pivots=True)
            assert neg[i] == c and np.array_equal(piv[i].cpu().numpy(), d)
        ab[50, 1] = np.nan
        with pytest.raises(pk.PdeshepError) as e:
            pk.inertia(to_dev(ab, device), sig)
        assert e.value.status == 4


@pytest.mark.parametrize("nsig", [1, 400])
@pytest.mark.parametrize("kind", ["unit", "wide", "near", "edge"])
def test_quotients_are_rounded_to_nearest(device, nsig, kind):
    """The kernels divide in integers: 2 x 2 blocks [[d, a], [a, 0]] on the diagonal give the pivots d and
    -fl(fl(a/d) a), whose bits show the quotient's.  Significands at random, next to each other and at
    the ends of their range (a quotient next to 1, to 2 and to half-way points), exponents whose quotient is
    subnormal, zero or infinite, one call per kernel (1 shift: cluster, 400: one CTA per shift)."""
    import paper_2012_00506_gb300 as pk
    m = 3000
    g = np.random.default_rng(len(kind) + nsig)
    sig = lambda: (1.0 + g.integers(0, 1 << 52, m).astype(np.float64) * 2.0 ** -52) * g.choice([-1.0, 1.0], m)
    d, a = sig(), sig()
    if kind == "wide":
        d, a = np.ldexp(d, g.integers(-480, 480, m)), np.ldexp(a, g.integers(-480, 480, m))
    elif kind == "near":
        a = np.nextafter(d, d * g.choice([1.0, 2.0, 0.5], m)) * 2.0 ** g.integers(-3, 4, m).astype(np.float64)
    elif kind == "edge":
        u = g.integers(0, 4, m) * 2.0 ** -52
        d = np.where(g.random(m) < 0.5, 1.0 + u, 2.0 - 2.0 ** -52 - u)
        v = g.integers(0, 4, m) * 2.0 ** -52
        a = np.where(g.random(m) < 0.5, 1.0 + v, 2.0 - 2.0 ** -52 - v)
        e = g.choice([0, 0, 500, -520, -1040], m)
        a, d = np.ldexp(a, e), np.ldexp(d, np.where(e == 0, g.choice([0, -1074 + 52, 700], m), 500))
    a[::97] = 0.0
    ab = np.zeros((2 * m, 2))
    ab[0::2, 0] = d
    ab[0::2, 1] = a
    neg, piv = pk.inertia(to_dev(ab, device), np.zeros(nsig), pivots=True)
    piv = piv.cpu().numpy()
    with np.errstate(all="ignore"):
        want = 0.0 - (a / d) * a
    want = np.where(want == 0.0, -oracle.pivmin(ab), want)
    for i in (0, nsig - 1):
        assert np.array_equal(piv[i][0::2], d)
        assert np.array_equal(piv[i][1::2], want, equal_nan=True)


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("n,b", [(70, 0), (120, 3), (150, 24), (200, 56)])
def test_counts_of_many_and_few_shifts_agree(device, n, b, cplx):
    """Calls of one shift to several rounds of the chip (900, 1600) take different kernels: the same counts, and
    the oracle's."""
    import paper_2012_00506_gb300 as pk
    ab = synth.random_band(n, b, 4000 + b, cplx)
    lo, hi = oracle.gershgorin(ab)
    sig = lo + (hi - lo) * (np.arange(1600) + 0.5) / 1600
    band = to_dev(ab, device)
    all_ = pk.inertia(band, sig)
    assert np.array_equal(pk.inertia(band, sig[:900]), all_[:900])
    assert np.array_equal(pk.inertia(band, sig[700:830]), all_[700:830])
    for k in (3, 799, 1598):
        assert pk.inertia(band, sig[k:k + 1])[0] == all_[k] == oracle.inertia(ab, sig[k])
