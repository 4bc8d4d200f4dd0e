"""GPU CholQR and small Hermitian eigensolver (Rayleigh-Ritz step of Section
2.2) against the oracle."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import block_from_dev, block_to_dev, dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def device():
    return dev()


@pytest.mark.parametrize("cplx", [False, True])
def test_cholqr_matches_oracle(device, cplx):
    import paper_2012_00506_gb300 as pk
    n = 300
    sizes = [1, 17, 64, 70]
    Q0 = synth.random_subspace(n, sum(sizes), 11, cplx)
    Q, R = pk.cholqr(block_to_dev(Q0, device), sizes, passes=1)
    Qg = block_from_dev(Q)
    off = 0
    for t, m in enumerate(sizes):
        Qo, Ro, info = oracle.cholqr(Q0[:, off:off + m])
        assert info == 0
        Rg = R[t].cpu().numpy()
        assert np.max(np.abs(Rg - Ro)) < 1e-12 * np.max(np.abs(Ro))
        assert np.max(np.abs(Qg[:, off:off + m] - Qo)) < 1e-12
        off += m
    Q2, _ = pk.cholqr(block_to_dev(Q0, device), sizes, passes=2)
    Q2 = block_from_dev(Q2)
    off = 0
    for m in sizes:
        B = Q2[:, off:off + m]
        assert np.max(np.abs(B.conj().T @ B - np.eye(m))) < 1e-14
        off += m


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("sizes", [[1, 31, 32, 33], [63, 64, 65, 2], [159], [97, 100, 3, 128]])
def test_cholqr_at_panel_edges(device, cplx, sizes):
    """Orders around the 32-column panels and tiles, one block and several.  Gaussian columns with
    m <= n/3: the condition number of R stays below 5, its error below 25 m eps."""
    import paper_2012_00506_gb300 as pk
    n = 480
    Q0 = synth.random_subspace(n, sum(sizes), 29, cplx)
    Q, R = pk.cholqr(block_to_dev(Q0, device), sizes, passes=1)
    Qg = block_from_dev(Q)
    off = 0
    for t, m in enumerate(sizes):
        Rg = R[t].cpu().numpy()
        Qo, Ro, info = oracle.cholqr(Q0[:, off:off + m])
        assert info == 0
        assert np.all(np.tril(Rg, -1) == 0)
        assert np.max(np.abs(Rg - Ro)) < 1e-12 * np.max(np.abs(Ro))
        assert np.max(np.abs(Qg[:, off:off + m] - Qo)) < 1e-12
        off += m


def test_cholqr_breakdown(device):
    import paper_2012_00506_gb300 as pk
    Q0 = np.ones((64, 3))
    with pytest.raises(pk.PdeshepError) as e:
        pk.cholqr(block_to_dev(Q0, device), [3], passes=1)
    assert e.value.status == 3


@pytest.mark.parametrize("cplx", [False, True])
def test_eigh_matches_oracle(device, cplx):
    import torch
    import paper_2012_00506_gb300 as pk
    rng = np.random.default_rng(5)
    sizes = [1, 2, 13, 64, 150]
    mats = []
    for m in sizes:
        A = rng.normal(size=(m, m)) + (1j * rng.normal(size=(m, m)) if cplx else 0)
        mats.append(0.5 * (A + A.conj().T))
    out = pk.eigh([torch.from_numpy(A).to(device) for A in mats])
    for A, (lam, V) in zip(mats, out):
        lo, Vo, sw = oracle.jacobi_eig(A)
        lam = lam.cpu().numpy()
        V = V.cpu().numpy()
        nrm = max(1.0, np.linalg.norm(A))
        assert np.max(np.abs(lam - lo)) < 1e-13 * nrm
        assert np.max(np.abs(V.conj().T @ V - np.eye(len(lam)))) < 1e-13
        assert np.linalg.norm(A @ V - V * lam) < 1e-12 * nrm
        gaps = np.min(np.abs(lo[:, None] - lo[None, :]) + np.eye(len(lo)) * 1e9, axis=1)
        for k in range(len(lo)):
            if gaps[k] > 1e-6 * nrm:
                assert np.max(np.abs(V[:, k] - Vo[:, k])) < 1e-10 * nrm / gaps[k]


# The ring form of the Jacobi stage: orders around one and two places per CTA, odd ones (a dummy player),
# uneven blocks in one call, an order whose columns do not fit the cluster (complex 460), and the tiles of the
# products (16 and 32 x 64) at their edges.
@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("sizes", [[1], [2, 3, 4, 5], [15, 16, 17, 31, 33], [65, 7, 66], [129, 128, 200, 1], [271],
                                   [460]])
def test_eigh_orders(device, sizes, cplx):
    import torch
    import paper_2012_00506_gb300 as pk
    rng = np.random.default_rng(sum(sizes))
    mats = []
    for m in sizes:
        A = rng.normal(size=(m, m)) + (1j * rng.normal(size=(m, m)) if cplx else 0)
        mats.append(0.5 * (A + A.conj().T))
    out = pk.eigh([torch.from_numpy(A).to(device) for A in mats])
    for A, (lam, V) in zip(mats, out):
        lam, V = lam.cpu().numpy(), V.cpu().numpy()
        nrm = max(1.0, np.linalg.norm(A))
        assert np.max(np.abs(lam - np.linalg.eigvalsh(A))) < 1e-13 * nrm
        assert np.max(np.abs(A @ V - V * lam)) < 1e-12 * nrm
        assert np.max(np.abs(V.conj().T @ V - np.eye(A.shape[0]))) < 1e-12


def test_eigh_degenerate_spectra(device):
    """Multiple eigenvalues, a diagonal block and one far from the others in scale."""
    import torch
    import paper_2012_00506_gb300 as pk
    rng = np.random.default_rng(3)
    Q, _ = np.linalg.qr(rng.normal(size=(90, 90)))
    mats = [np.eye(40), np.diag(np.arange(33.0) // 3), Q @ np.diag(np.repeat(np.arange(9.0), 10)) @ Q.T,
            1e6 * np.outer(Q[0], Q[0]) + np.diag(np.linspace(0, 1, 90))]
    mats = [0.5 * (A + A.T) for A in mats]
    for A, (lam, V) in zip(mats, pk.eigh([torch.from_numpy(A).to(device) for A in mats])):
        lam, V = lam.cpu().numpy(), V.cpu().numpy()
        nrm = max(1.0, np.linalg.norm(A))
        assert np.max(np.abs(lam - np.linalg.eigvalsh(A))) < 1e-13 * nrm
        assert np.max(np.abs(A @ V - V * lam)) < 1e-12 * nrm
        assert np.max(np.abs(V.T @ V - np.eye(A.shape[0]))) < 1e-12


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("nblk,m", [(16, 130), (40, 33), (150, 20)])
def test_eigh_many_blocks(device, cplx, nblk, m):
    """More blocks than one wave of CTAs holds in the refinement and the sort: every block's eigenvalues and
    vectors stand on their own."""
    import torch
    import paper_2012_00506_gb300 as pk
    rng = np.random.default_rng(3 * nblk + m)
    mats = []
    for t in range(nblk):
        A = rng.normal(size=(m - t % 3, m - t % 3)) + (1j * rng.normal(size=(m - t % 3, m - t % 3)) if cplx else 0)
        mats.append(0.5 * (A + A.conj().T))
    for A, (lam, V) in zip(mats, pk.eigh([torch.from_numpy(A).to(device) for A in mats])):
        lam, V = lam.cpu().numpy(), V.cpu().numpy()
        nrm = max(1.0, np.linalg.norm(A))
        assert np.max(np.abs(lam - np.linalg.eigvalsh(A))) < 1e-13 * nrm
        assert np.max(np.abs(V.conj().T @ V - np.eye(len(lam)))) < 1e-13
        assert np.max(np.abs(A @ V - V * lam)) < 1e-13 * nrm


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("d", [[1e-310, -1e-310], [1.0, -1.0, 3e-310, -3e-310], [5e-324, 0.0, 2.0, -2.0]])
def test_eigh_subnormal_gaps(device, cplx, d):
    """Diagonal matrices with eigenvalues a subnormal distance apart (the mean of the diagonal is 0 or harmless):
    nothing has to be rotated, so eigenvalues and vectors are exact."""
    import torch
    import paper_2012_00506_gb300 as pk
    A = np.diag(np.array(d, dtype=np.complex128 if cplx else np.float64))
    (lam, V), = pk.eigh([torch.from_numpy(A).to(device)])
    lam, V = lam.cpu().numpy(), V.cpu().numpy()
    assert np.all(np.isfinite(V))
    assert np.array_equal(np.abs(V) != 0, np.abs(V) == 1)
    assert np.array_equal(V.conj().T @ V, np.eye(len(d)))
    assert np.max(np.abs(lam - np.sort(d))) <= 2e-16 * np.max(np.abs(d))


# Calls above and below the size from which the refinement's first steps are taken in float-float.
@pytest.mark.parametrize("cplx,nblk,m", [(False, 2, 60), (True, 1, 160), (True, 6, 160), (False, 6, 267), (True, 2, 267)])
@pytest.mark.parametrize("gap", [0.0, 1e-14, 1e-12, 1e-11, 1e-10])
def test_eigh_of_doublets(device, cplx, nblk, m, gap):
    """Blocks of close pairs (gap in units of the spread) and some simple eigenvalues."""
    import torch
    import paper_2012_00506_gb300 as pk
    rng = np.random.default_rng(m + nblk)
    mats = []
    for t in range(nblk):
        Q, _ = np.linalg.qr(rng.normal(size=(m, m)) + (1j * rng.normal(size=(m, m)) if cplx else 0))
        pairs = m // 2 if t % 2 == 0 else 3
        base = rng.uniform(-0.5, 0.5, pairs)
        d = np.concatenate([base, base + gap, rng.uniform(-0.5, 0.5, m - 2 * pairs)])
        A = (Q * d) @ Q.conj().T
        mats.append(0.5 * (A + A.conj().T))
    for A, (lam, V) in zip(mats, pk.eigh([torch.from_numpy(A).to(device) for A in mats])):
        lam, V = lam.cpu().numpy(), V.cpu().numpy()
        nrm = max(1.0, np.linalg.norm(A))
        assert np.max(np.abs(lam - np.linalg.eigvalsh(A))) < 1e-13 * nrm
        assert np.max(np.abs(V.conj().T @ V - np.eye(len(lam)))) < 1e-13
        assert np.max(np.abs(A @ V - V * lam)) < 1e-13 * nrm


@pytest.mark.parametrize("cplx,nblk,m", [(False, 6, 267), (True, 3, 200), (True, 1, 50), (False, 4, 90)])
@pytest.mark.parametrize("scale", [1e-140, 1e-100, 1e-60, 1e-38, 1e-30, 1e18, 1e30, 1e37, 1e39, 1e100, 1e140])
def test_eigh_of_any_scale(device, cplx, nblk, m, scale):
    """Matrices far out of FP32's range or near its ends: the FP32 start is no help, the refinement may diverge
    from it to infinity, and the block then has to be redone, never returned."""
    import torch
    import paper_2012_00506_gb300 as pk
    rng = np.random.default_rng(1)
    mats = []
    for t in range(nblk):
        A = rng.normal(size=(m, m)) + (1j * rng.normal(size=(m, m)) if cplx else 0)
        mats.append(0.5 * (A + A.conj().T))
    for A, (lam, V) in zip(mats, pk.eigh([torch.from_numpy(A * scale).to(device) for A in mats])):
        lam, V = lam.cpu().numpy() / scale, V.cpu().numpy()
        nrm = np.linalg.norm(A)
        assert np.max(np.abs(lam - np.linalg.eigvalsh(A))) < 1e-13 * nrm
        assert np.max(np.abs(V.conj().T @ V - np.eye(m))) < 1e-13
        assert np.max(np.abs(A @ V - V * lam)) < 1e-13 * nrm
