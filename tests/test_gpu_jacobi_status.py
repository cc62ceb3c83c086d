"""A Jacobi run that cannot converge says so.

Rows with a NaN never become orthogonal: the sweeps run out and the status
word is set, on one CTA and on clusters, in both types and in every order of
the pair sums (up to 64 rows, above, and beyond one CTA's shared memory).
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


@pytest.mark.parametrize("c64", [True, False])
@pytest.mark.parametrize("m,n", [(4, 6), (24, 30), (64, 64), (70, 80), (100, 100)])
def test_nan_is_reported(c64, m, n):
    rng = np.random.default_rng(m)
    Z = rng.standard_normal((m, n)) + 1j * rng.standard_normal((m, n))
    for bad in (0.0, np.nan):
        Z[m // 2, n // 3] = bad
        dt = torch.complex64 if c64 else torch.complex128
        z = torch.from_numpy(Z).to(dt).cuda()
        k = min(m, n, 8 if c64 else m)
        u, r = z.new_empty((m, k)), z.new_empty((k, n))
        nbytes = max(P.bbp_k_svd_work_bytes_rand(c64, m, n, 60), P.bbp_k_svd_work_bytes(m, n))
        work = torch.zeros(nbytes, dtype=torch.uint8, device="cuda")
        status = torch.zeros(2, dtype=torch.int32, device="cuda")
        if c64:
            P.bbp_k_svd_trunc_rand(True, z, m, n, 60, u.new_empty((m, min(m, n, 60))), u.new_empty((min(m, n, 60), n)),
                                   work, status, 1)
        else:
            P.bbp_k_svd_trunc(z, m, n, k, u, r, work, status)
        assert (int(status[0].item()) != 0) == bool(np.isnan(bad))
