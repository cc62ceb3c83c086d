"""Exchanges of the panel QR under load.

Panels narrower than their cluster, and ordinary ones.  Many panels a launch, so
that the CTAs of a cluster start apart, and many launches: every panel has to be
factorised (a wait that runs out leaves a NaN) and every launch has to give the
same bits.  Tolerance as for the other panels.
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


def check(c64, m, n, cluster, batch):
    rng = np.random.default_rng(m + n)
    A = (rng.standard_normal((batch, m, n)) + 1j * rng.standard_normal((batch, m, n)))
    A = A.astype(np.complex64 if c64 else np.complex128)
    a = torch.from_numpy(A).cuda()
    first = None
    for _ in range(20):
        q, r = torch.empty_like(a), torch.empty((batch, n, n), dtype=a.dtype, device="cuda")
        P.bbp_k_panel_qr(c64, a, m, n, q, r, batch, cluster)
        got = torch.view_as_real(q), torch.view_as_real(r)
        if first is None:
            first = got
        assert all(torch.equal(x, y) for x, y in zip(got, first))
    tol = 30 * np.sqrt(m) * (1e-6 if c64 else 1e-14)
    q, r = q.to(torch.complex128), r.to(torch.complex128)
    eye = torch.eye(n, dtype=torch.complex128, device="cuda")
    assert (q.mH @ q - eye).abs().max().item() < tol
    assert ((q @ r - a.to(torch.complex128)).norm(dim=1) / a.to(torch.complex128).norm(dim=1)).max().item() < tol


@pytest.mark.parametrize("c64", [True, False])
@pytest.mark.parametrize("m,n,cluster", [(300, 9, 16), (300, 16, 16), (300, 17, 9), (1100, 24, 16), (260, 12, 5)])
def test_fewer_columns_than_ctas(c64, m, n, cluster):
    check(c64, m, n, cluster, 40)


@pytest.mark.parametrize("c64", [True, False])
@pytest.mark.parametrize("m,n,cluster", [(1300, 40, 6), (2000, 33, 9), (520, 48, 0), (1000, 47, 16)])
def test_many_at_once(c64, m, n, cluster):
    """Every SM busy with panels, so that the warps of a CTA drift apart: a column
    or a row read before it is stored shows as other bits."""
    cmin = P.bbp_k_panel_cluster(c64, m, n)
    check(c64, m, n, max(cluster, cmin) if cluster else 0, 48)
