"""The tile table tells a real product from an absorb of the same shape.

An absorb reads its operands otherwise (limbs once or per segment) and writes
complex entries, so each form is recorded, timed and kept by itself; a table
without form numbers, as written before, is read, and serves both.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2603_13304_gb300")


@pytest.fixture(autouse=True)
def clean():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P.build()
    P.lib()
    P.bbp_autotune_clear()
    yield
    P.bbp_autotune_record(False)
    P.bbp_autotune_clear()


def absorb(Pd, Q, l, r, c64):
    g = torch.Generator(device="cuda").manual_seed(1)
    ct = torch.complex64 if c64 else torch.complex128
    x = torch.randn((Pd, Q), generator=g, device="cuda", dtype=torch.complex128).to(ct)
    s = torch.randn((l, Pd, r), generator=g, device="cuda", dtype=torch.complex128).to(ct)
    out = torch.empty((l, Q, r), dtype=ct, device="cuda")
    work = torch.zeros(P.bbp_k_tc_absorb_bytes(False, Pd, Q, l, r), dtype=torch.uint8, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    P.bbp_k_tc_absorb(False, c64, x, Pd, Q, s, l, r, out, work, err)
    assert int(err.item()) == 0
    return torch.view_as_real(out).cpu().numpy()


def plain(M, N, K):
    a = torch.zeros((M, K), device="cuda")
    b = torch.zeros((N, K), device="cuda")
    c = torch.zeros((M, N), device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    P.bbp_k_tc_gemm(False, a, K, b, K, c, N, M, N, K, 1.0, err)
    assert int(err.item()) == 0


@pytest.mark.parametrize("Pd,K", [(16, 96), (25, 160)])          # limbs once; every segment
def test_forms(tmp_path, Pd, K):
    Q, l, r = 40, 6, 10
    P.bbp_autotune_record(True)
    before = [absorb(Pd, Q, l, r, c64) for c64 in (True, False)]
    plain(2 * Q, l * r, K)
    P.bbp_autotune_record(False)
    assert P.bbp_autotune_info()[1] == 3
    cache = tmp_path / "tiles.txt"
    assert P.bbp_autotune_run(str(cache)) == 3
    forms = sorted(int(ln.split()[8]) for ln in open(cache) if ln.startswith("tc "))
    assert forms == ([0, 3, 4] if Pd == 16 else [0, 1, 2])
    P.bbp_autotune_clear()
    assert P.bbp_autotune_load(str(cache)) == 3
    old = tmp_path / "old.txt"
    old.write_text("tc 0 %d %d %d 64 1 3.000\n" % (2 * Q, l * r, K))
    after = [absorb(Pd, Q, l, r, c64) for c64 in (True, False)]
    P.bbp_autotune_clear()
    assert P.bbp_autotune_load(str(old)) == 1
    again = [absorb(Pd, Q, l, r, c64) for c64 in (True, False)]
    for a, b, c in zip(before, after, again):                    # the tile does not change the sums
        assert np.array_equal(a, b) and np.array_equal(a, c)
