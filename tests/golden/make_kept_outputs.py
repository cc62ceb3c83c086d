"""Entries of messages that later builds have to reproduce (run on a GPU).

    python tests/golden/make_kept_outputs.py > tests/golden/kept_outputs.json

Networks whose truncations follow the rounding of everything before them: full
precision on flat spectra (Gaussian tensors), where the randomised truncation
has not converged, and the mixed mode at D = 6, chi = 64.
"""
import json
import os
import sys

import numpy as np

sys.path.insert(0, os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", ".."))

NETWORKS = {
    "gaussian-D3-chi9-fp64": dict(size=4, block=2, D=3, chi=9, precision="FP64", seed=31),
    "gaussian-D3-chi20-fp64": dict(size=6, block=3, D=3, chi=20, precision="FP64", seed=11),
    "kagome-D3-chi32-tf32": dict(size=2, block=2, D=3, chi=32, precision="TF32", seed=12),
    "kagome-D6-chi64-tf32": dict(size=2, block=2, D=6, chi=64, precision="TF32", seed=21),
}
ITERATIONS, ENTRIES = 2, 24


def messages(size, block, D, chi, precision, seed, places=None):
    """The messages after ITERATIONS iterations: (block, face) -> places, the dense vector's entries there, its norm and
    its length.  places: (block, face) -> the places (chosen here when None)."""
    import torch

    import paper_2603_13304_gb300 as P
    import synthetic as syn

    kagome = precision != "FP64"
    nb, Lx = (syn.kagome_neighbours(3 * size, size), 3 * size) if kagome else (syn.square_neighbours(size, size, False), size)
    n = len(nb)
    if kagome:
        t = syn.dimer_singlet_peps(nb, 2, D, seed=seed, noise=1e-2, noise_seed=seed + 1)
    else:
        t = syn.gaussian_peps(n, 2, D, seed=seed)
    ctx = P.bbp_create_peps(P.KAGOME if kagome else P.SQUARE, Lx, size, int(kagome), 2, D, t)
    P.bbp_partition_blocks(ctx, block, block)
    P.bbp_set_options(ctx, chi, getattr(P, precision))
    P.bbp_init_messages(ctx, syn.initial_edge_matrices(n, D, seed=seed + 2))
    P.bbp_iterate(ctx, 0.0, ITERATIONS)
    legs = 2 * block if kagome else block
    out = {}
    for b in range(P.bbp_info(ctx)[0]):
        for f in range(4):
            v = None
            for x in P.bbp_get_message(ctx, b, f, cap=2 * legs * chi * chi * D * D):
                x = torch.from_numpy(x).cuda().to(torch.complex128)
                l, p, r = x.shape
                v = x.reshape(l * p, r) if v is None else (v @ x.reshape(l, p * r)).reshape(-1, r)
            v = v.reshape(-1)
            if v.numel() < ENTRIES:
                continue
            # half of them the largest (a stable order), half spread over the vector
            if places is None:
                big = torch.argsort(v.abs(), descending=True, stable=True)[:4 * ENTRIES:8]
                at = torch.cat([big, torch.arange(ENTRIES // 2, device="cuda") * (v.numel() // (ENTRIES // 2))])
            else:
                at = torch.tensor(places[(b, f)], device="cuda")
            out[(b, f)] = (at.cpu().numpy(), v[at].cpu().numpy(), float(v.norm()), v.numel())
    P.bbp_destroy(ctx)
    return out


if __name__ == "__main__":
    import paper_2603_13304_gb300 as P

    P.build()
    P.lib()
    doc = {}
    for name, net in NETWORKS.items():
        doc[name] = [{"block": b, "face": f, "at": [int(i) for i in at], "re": [float(x) for x in v.real],
                      "im": [float(x) for x in v.imag], "norm": norm, "size": size}
                     for (b, f), (at, v, norm, size) in messages(**net).items()]
    print(json.dumps(doc))
