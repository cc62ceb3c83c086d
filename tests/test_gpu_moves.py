"""Canonical moves in place and the centre normalisation, through whole
iterations: networks whose boundary tensors are taller, wider and larger than
one CTA holds, against the same networks run eagerly on one stream (the same
kernels, another schedule) and, for the centre norms, log-norms that must not
depend on the schedule.  Equality of the dense messages to 1e-10 (complex128)
and 2e-5 (complex64), the agreement asked of the two precisions elsewhere.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
P = pytest.importorskip("paper_2603_13304_gb300")
syn = pytest.importorskip("synthetic")


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P.build()
    P.lib()


def dense(ctx, block, face):
    v = None
    for x in P.bbp_get_message(ctx, block, face):
        l, p, r = x.shape
        v = x.reshape(l * p, r) if v is None else (v @ x.reshape(l, p * r)).reshape(-1, r)
    return v.reshape(-1)


@pytest.mark.parametrize("D,chi,prec", [(2, 5, "FP64"), (3, 33, "FP64"), (2, 8, "TF32"), (3, 64, "FP32"),
                                        (4, 27, "TF32")])
def test_schedules_agree(D, chi, prec):
    nb = syn.square_neighbours(6, 6, False)
    t = syn.dimer_singlet_peps(nb, 2, D, seed=3, noise=1e-2, noise_seed=4)
    em = syn.initial_edge_matrices(36, D, seed=5)
    got = []
    for graphs, streams in ((True, 16), (False, 1)):
        ctx = P.bbp_create_peps(P.SQUARE, 6, 6, 0, 2, D, t)
        try:
            P.bbp_partition_blocks(ctx, 3, 3)
            P.bbp_set_options(ctx, chi, getattr(P, prec))
            P.bbp_set_execution(ctx, graphs, streams)
            P.bbp_init_messages(ctx, em)
            P.bbp_iterate(ctx, 0.0, 4)
            m = [dense(ctx, b, f) for b in range(4) for f in range(4)]
            got.append((m, P.bbp_norm(ctx)))
        finally:
            P.bbp_destroy(ctx)
    tol = 1e-10 if prec == "FP64" else 2e-5
    for a, b in zip(got[0][0], got[1][0]):
        assert np.isfinite(a).all() and np.linalg.norm(a - b) <= tol * np.linalg.norm(b)
    assert abs(got[0][1] - got[1][1]) <= tol * max(1.0, abs(got[1][1]))
