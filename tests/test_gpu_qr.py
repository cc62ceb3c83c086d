"""The blocked Householder QR at the edges of its blocks, slices and clusters.

Blocks of eight reflectors (n around multiples of eight), row slices that end
inside a warp, one to three rows a thread, wide matrices, columns of very
different magnitude, and panels that only the column-by-column kernel holds.
Tolerance, as for the other panels: the rounding of m-term sums, 30 sqrt(m)
units of 1e-6 (complex64) or 1e-14 (complex128).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2603_13304_gb300")


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P.build()
    P.lib()


def gauss(rng, m, n, c64):
    a = rng.standard_normal((m, n)) + 1j * rng.standard_normal((m, n))
    return a.astype(np.complex64 if c64 else np.complex128)


def check(A, Q, R, c64):
    A, Q, R = (x.astype(np.complex128) for x in (A, Q, R))
    m = A.shape[0]
    tol = 30 * np.sqrt(m) * (1e-6 if c64 else 1e-14)
    scale = np.linalg.norm(A, axis=0)
    scale[scale == 0] = 1.0
    k = Q.shape[1]
    assert np.abs(np.tril(R, -1)).max() == 0.0 and np.abs(np.diag(R).imag).max() == 0.0
    assert np.abs(Q.conj().T @ Q - np.eye(k)).max() < tol
    assert np.abs((Q @ R - A) / scale).max() < tol       # column by column


def panel(A, c64, cluster=0):
    m, n = A.shape
    a = torch.from_numpy(A).cuda()
    q, r = torch.empty_like(a), torch.full((n, n), 7.0, dtype=a.dtype, device="cuda")
    P.bbp_k_panel_qr(c64, a, m, n, q, r, 1, cluster)
    return q.cpu().numpy(), r.cpu().numpy()


@pytest.mark.parametrize("c64", [True, False])
@pytest.mark.parametrize("m,n", [(1, 1), (9, 7), (8, 8), (33, 9), (65, 17), (129, 24), (200, 96), (511, 31), (700, 15),
                                 (1025, 8), (1601, 12)])
def test_blocks_and_slices(c64, m, n):
    rng = np.random.default_rng(m + 7 * n)
    A = gauss(rng, m, n, c64)
    cmin = P.bbp_k_panel_cluster(c64, m, n)
    for cluster in sorted({0, cmin, min(16, cmin + 2), 16}):
        q, r = panel(A, c64, cluster)
        check(A, q, r, c64)


@pytest.mark.parametrize("c64", [True, False])
def test_magnitudes(c64):
    """Columns from the bottom to the top of the type's range."""
    rng = np.random.default_rng(3)
    A = gauss(rng, 300, 21, c64)
    e = np.linspace(-30, 30, 21) if c64 else np.linspace(-120, 120, 21)
    A = (A * 10.0 ** rng.permutation(e)[None, :]).astype(A.dtype)
    for cluster in (0, P.bbp_k_panel_cluster(c64, 300, 21), 4):
        q, r = panel(A, c64, cluster)
        check(A, q, r, c64)


@pytest.mark.parametrize("m,n", [(5, 3), (3, 5), (8, 32), (17, 33), (64, 64), (256, 32), (130, 50)])
def test_canonical_moves(m, n):
    rng = np.random.default_rng(m + n)
    A = gauss(rng, m, n, False)
    k = min(m, n)
    a = torch.from_numpy(A.copy()).cuda()
    q = torch.empty((m, k), dtype=a.dtype, device="cuda")
    r = torch.empty((k, n), dtype=a.dtype, device="cuda")
    tau = torch.empty(k, dtype=a.dtype, device="cuda")
    P.bbp_k_qr(a, m, n, q, r, tau)
    check(A, q.cpu().numpy(), r.cpu().numpy(), False)


@pytest.mark.parametrize("c64,m,n", [(True, 2304, 102), (True, 1296, 290), (False, 2048, 92), (False, 256, 106)])
def test_full_clusters(c64, m, n):
    """Panels whose slices leave no room for the block buffers."""
    rng = np.random.default_rng(n)
    A = gauss(rng, m, n, c64)
    assert P.bbp_k_panel_cluster(c64, m, n) > 0
    q, r = panel(A, c64)
    check(A, q, r, c64)
