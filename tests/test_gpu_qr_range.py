"""QR calls at the ends of what the entry points take.

Wide matrices (a canonical move of a short, wide tensor), complex128 columns
whose squares are near the ends of the type's range, and the R factor alone of
panels that just fit the published smallest cluster.  Tolerance as for the
other QR tests: 30 sqrt(m) units of 1e-14 (complex128) or 1e-6 (complex64).
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


def gauss(m, n, dtype=np.complex128):
    rng = np.random.default_rng(m + 3 * n)
    return (rng.standard_normal((m, n)) + 1j * rng.standard_normal((m, n))).astype(dtype)


def qr(A):
    m, n = A.shape
    k = min(m, n)
    a = torch.from_numpy(A.copy()).cuda()
    q, r = a.new_empty((m, k)), a.new_empty((k, n))
    P.bbp_k_qr(a, m, n, q, r, a.new_empty(k))
    return q.cpu().numpy(), r.cpu().numpy()


def check(A, Q, R, tol):
    scale = np.abs(A).max(axis=0) * np.sqrt(A.shape[0])     # (no squares: they may leave the range)
    assert np.abs(np.tril(R, -1)).max(initial=0.0) == 0.0
    assert np.abs(Q.conj().T @ Q - np.eye(Q.shape[1])).max() < tol
    assert (np.abs(Q @ (R / scale) - A / scale)).max() < tol


@pytest.mark.parametrize("m,n", [(8, 735), (8, 736), (17, 736), (17, 737), (12, 820), (7, 1000), (1, 1581), (1, 5000)])
def test_wide(m, n):
    A = gauss(m, n)
    check(A, *qr(A), 30 * np.sqrt(m) * 1e-14)


@pytest.mark.parametrize("m,n", [(32, 8), (40, 17), (9, 12)])
@pytest.mark.parametrize("e", [-150.0, -145.0, 145.0, 150.0])
def test_complex128_range(m, n, e):
    A = gauss(m, n) * 10.0 ** e
    check(A, *qr(A), 30 * np.sqrt(m) * 1e-14)


@pytest.mark.parametrize("c64,m,n", [(True, 251, 214), (True, 319, 171), (True, 1296, 290), (False, 256, 106),
                                     (False, 2048, 92)])
def test_r_alone_on_the_smallest_cluster(c64, m, n):
    A = gauss(m, n, np.complex64 if c64 else np.complex128)
    a = torch.from_numpy(A).cuda()
    r = a.new_empty((n, n))
    cmin = P.bbp_k_panel_cluster(c64, m, n)
    assert cmin > 0
    P.bbp_k_panel_qr(c64, a, m, n, None, r, 1, cmin)
    R, A = r.cpu().numpy().astype(np.complex128), A.astype(np.complex128)
    tol = 30 * np.sqrt(m) * (1e-6 if c64 else 1e-14)
    assert np.abs(np.tril(R, -1)).max() == 0.0
    scale = np.linalg.norm(A, axis=0)
    assert np.abs((R.conj().T @ R - A.conj().T @ A) / np.outer(scale, scale)).max() < tol
