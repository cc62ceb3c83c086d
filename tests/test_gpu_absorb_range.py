"""The complex128 absorb far from unit scale, and operand rows of every kind.

Operands of 1e-25 and 1e25: the products lie past float's range, their sums are
taken near one and scaled back in complex128.  P = 9, 18, 25: rows whose limbs are
not whole MMAs in either, one or no type; r odd and one.  Tolerances of the other
absorb tests: 2e-5 (TF32) and 3e-4 (BF16) of sum |x s|.
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


def absorb(X, S, bf16, c64):
    (Pd, Q), (l, _, r) = X.shape, S.shape
    ct = torch.complex64 if c64 else torch.complex128
    x, s = torch.from_numpy(X).to("cuda", ct), torch.from_numpy(S).to("cuda", ct)
    out = torch.full((l, Q, r), float("nan"), dtype=ct, device="cuda")
    work = torch.zeros(P.bbp_k_tc_absorb_bytes(bf16, Pd, Q, l, r), dtype=torch.uint8, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    P.bbp_k_tc_absorb(bf16, c64, x, Pd, Q, s, l, r, out, work, err)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    return out.cpu().numpy().astype(np.complex128)


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("c64,ex,es", [(False, -25, -20), (False, 25, 20), (False, -30, 30), (True, 0, 0)])
@pytest.mark.parametrize("Pd,Q,l,r", [(9, 30, 5, 7), (18, 70, 3, 64), (25, 33, 4, 1), (36, 40, 2, 12)])
def test_scales_and_rows(Pd, Q, l, r, c64, ex, es, bf16):
    rng = np.random.default_rng(Pd + Q + l + r)
    X = rng.standard_normal((Pd, Q)) + 1j * rng.standard_normal((Pd, Q))
    S = rng.standard_normal((l, Pd, r)) + 1j * rng.standard_normal((l, Pd, r))
    got = absorb(X * 10.0 ** ex, S * 10.0 ** es, bf16, c64)
    ref, scale = np.einsum("pq,apr->aqr", X, S), np.einsum("pq,apr->aqr", np.abs(X), np.abs(S))
    assert np.isfinite(got).all()
    assert (np.abs(got / 10.0 ** (ex + es) - ref) / scale).max() < (3e-4 if bf16 else 2e-5)
