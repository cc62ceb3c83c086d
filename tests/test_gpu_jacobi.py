"""The cluster Jacobi SVD at the edges of its blocks and row layouts.

Row counts that leave blocks short or empty, one CTA and several, rows longer
than a warp's registers hold, repeated and vanishing singular values, and
matrices far from unit norm.  Reference: numpy's SVD of the same matrix in
complex128.  Tolerances, relative to the matrix's norm: 1e-12 (complex128)
and 2e-5 (complex64) as for the other truncations; U^H U - 1 on directions
above the floor, 1e-11 and 1e-4.
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


def svd(Z, chi, c64):
    m, n = Z.shape
    k = min(chi, m, n)
    dt = torch.complex64 if c64 else torch.complex128
    z = torch.from_numpy(np.ascontiguousarray(Z)).to(dt).cuda()
    u = torch.full((m, k), float("nan"), dtype=dt, device="cuda")
    r = torch.full((k, n), float("nan"), dtype=dt, device="cuda")
    work = torch.zeros(max(P.bbp_k_svd_work_bytes_rand(c64, m, n, chi), P.bbp_k_svd_work_bytes(m, n)),
                       dtype=torch.uint8, device="cuda")
    status = torch.zeros(2, dtype=torch.int32, device="cuda")
    if c64:
        P.bbp_k_svd_trunc_rand(True, z, m, n, chi, u, r, work, status, 1)
    else:
        P.bbp_k_svd_trunc(z, m, n, chi, u, r, work, status)
    assert int(status[0].item()) == 0
    return u.cpu().numpy().astype(np.complex128), r.cpu().numpy().astype(np.complex128)


def check(Z, chi, c64):
    Z = np.asarray(Z).astype(np.complex64 if c64 else np.complex128)
    u, r = svd(Z, chi, c64)
    Z = Z.astype(np.complex128)
    k = min(chi, *Z.shape)
    a, s, b = np.linalg.svd(Z, full_matrices=False)
    best = np.linalg.norm(Z - (a[:, :k] * s[:k]) @ b[:k])
    tol = 2e-5 if c64 else 1e-12
    scale = np.linalg.norm(Z)
    assert np.isfinite(u).all() and np.isfinite(r).all()
    assert np.linalg.norm(Z - u @ r) <= best + tol * scale
    live = s[:k] > (1e-3 if c64 else 1e-8) * max(s[0], 1e-300)
    g = (u.conj().T @ u - np.eye(k))[np.ix_(live, live)]
    assert live.sum() == 0 or np.abs(g).max() < (1e-4 if c64 else 1e-11)
    sv = np.sort(np.linalg.norm(r, axis=1))[::-1]
    assert np.abs(sv - s[:k]).max() <= tol * max(scale, 1e-300)


def gauss(rng, m, n):
    return rng.standard_normal((m, n)) + 1j * rng.standard_normal((m, n))


@pytest.mark.parametrize("c64", [True, False])
@pytest.mark.parametrize("m,n", [(1, 1), (1, 9), (2, 2), (3, 3), (5, 4), (7, 9), (8, 8), (9, 33), (15, 15), (17, 16),
                                 (16, 100), (31, 40), (33, 33), (48, 64), (61, 59), (9, 700), (64, 64)])
def test_shapes(c64, m, n):
    rng = np.random.default_rng(100 * m + n)
    check(gauss(rng, m, n), min(m, n), c64)
    check(gauss(rng, m, n) * 0.7 ** np.arange(n)[None, :], max(1, min(m, n) // 2), c64)


@pytest.mark.parametrize("c64", [True, False])
def test_degenerate_and_vanishing(c64):
    rng = np.random.default_rng(5)
    a = np.linalg.qr(gauss(rng, 40, 24))[0]
    b = np.linalg.qr(gauss(rng, 30, 24))[0]
    s = np.array([1.0] * 8 + [0.5] * 8 + [0.0] * 8)
    check((a * s) @ b.conj().T, 16, c64)
    Z = gauss(rng, 20, 24)
    Z[7] = Z[3]
    Z[11] = 0
    check(Z, 18, c64)
    check(np.zeros((12, 12)), 5, c64)


@pytest.mark.parametrize("c64,scale", [(True, 1e-15), (True, 1e12), (False, 1e-120), (False, 1e120)])
def test_scales(c64, scale):
    rng = np.random.default_rng(6)
    check(gauss(rng, 24, 36) * 0.8 ** np.arange(36)[None, :] * scale, 12, c64)


@pytest.mark.parametrize("m,n,chi,plateau", [(400, 380, 32, 8), (400, 380, 32, 0), (260, 300, 21, 3)])
def test_randomised_cut(m, n, chi, plateau):
    """The complex128 finish across the cut: a plateau of equal singular values
    (pairs that are rotated one by one) or none (all at once)."""
    rng = np.random.default_rng(m + chi)
    r = 4 * chi
    a = np.linalg.qr(gauss(rng, m, r))[0]
    b = np.linalg.qr(gauss(rng, n, r))[0]
    s = np.exp(-np.arange(r) * 6.0 / chi)
    if plateau:
        s[chi - plateau // 2:chi + plateau] = s[chi]
    check((a * s) @ b.conj().T, chi, True)
