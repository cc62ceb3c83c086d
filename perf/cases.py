"""Workloads that time the BlockBP engine through its public entry points.

A case is a dict of plain values; ``prepare`` builds what a program holds
before the call (site tensors uploaded, blocks cut, messages iterated past
their bond-1 start), ``run`` is one pass of the call and returns its results,
``work`` states what a pass cannot do without, ``exact`` gives the results in
64 bits by plain torch where a call has a closed form.

Kinds of case:

* ``iterate``  one synchronous BlockBP iteration (Alg. 1) of a network, the
  call a solver repeats until the messages stop changing.  The messages come
  back as dense vectors over their fused legs (their matrix-product form is
  unique up to gauge only).
* ``batch``    one round over several networks of uneven size.
* ``rdm``      the reduced density matrix of sites of a block.
* ``core``     the pair density matrix of a bond from the core's periodic MPS
  (Edge tensor network).
* ``split``    truncated SVD of one split of a swallow; U and Rem come back as
  the kept part U Rem and the Gram matrix U^H U, both free of the phases of
  the singular vectors.
* ``panel``, ``qr``  Householder QR with a real diagonal of R: tall panels on
  a cluster of CTAs, small canonical moves on one.
* ``absorb``   the contraction of a site tensor into the boundary MPS.

Values of the mixed-precision modes are returned in their 32-bit type.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2603_13304_gb300 as P
import synthetic as syn

PRECISION = {"fp64": P.FP64, "tf32": P.TF32, "bf16": P.BF16, "fp32": P.FP32}


def listed():
    return [
        # the smallest factorisation: a canonical move at D = 2, chi = 8 (launch latency)
        {"name": "qr-c128-32x8", "kind": "qr", "m": 32, "n": 8},
        # a canonical move of the largest boundary tensors, 64 x 36 rows at D = 6, chi = 64
        {"name": "panel-c64-2304x64", "kind": "panel", "dtype": "c64", "m": 2304, "n": 64},
        # the bulk split of the FP64 path at D = 4, chi = 32
        {"name": "split-c128-512x512-chi32", "kind": "split", "dtype": "c128", "m": 512, "n": 512, "chi": 32,
         "power": 6},
        # the bulk split of the mixed modes at D = 6, chi = 64
        {"name": "split-c64-2304x2304-chi64", "kind": "split", "dtype": "c64", "m": 2304, "n": 2304, "chi": 64,
         "power": 1},
        # the bulk swallow at D = 5, chi = 64: two fused legs of 25 in, two out
        {"name": "absorb-tf32-625x625-64x64", "kind": "absorb", "mode": "tf32", "P": 625, "Q": 625, "l": 64,
         "r": 64},
        # a small open network in full precision: every message a few kilobytes, bound by launches
        {"name": "iterate-square-D2-chi8-fp64", "kind": "iterate", "lattice": "square", "size": 6, "block": 3,
         "periodic": 0, "D": 2, "chi": 8, "precision": "fp64", "alpha": 1.0, "hermitise": 0, "settle": 2},
        # odd sizes on a torus with the learning step and Hermitised messages
        {"name": "iterate-torus-D3-chi21-bf16", "kind": "iterate", "lattice": "square", "size": 6, "block": 3,
         "periodic": 1, "D": 3, "chi": 21, "precision": "bf16", "alpha": 0.8, "hermitise": 1, "settle": 2},
        # the parity path: Kagome super-cell at D = 4, chi = 32 in full precision
        {"name": "iterate-kagome-D4-chi32-fp64", "kind": "iterate", "lattice": "kagome", "size": 2, "block": 2,
         "periodic": 1, "D": 4, "chi": 32, "precision": "fp64", "alpha": 1.0, "hermitise": 0, "settle": 1},
        # the headline: Kagome super-cell at D = 6, chi = 64, mixed precision
        {"name": "iterate-kagome-D6-chi64-tf32", "kind": "iterate", "lattice": "kagome", "size": 2, "block": 2,
         "periodic": 1, "D": 6, "chi": 64, "precision": "tf32", "alpha": 1.0, "hermitise": 0, "settle": 2},
        # several small jobs at once: uneven D, chi, lattice and block size
        {"name": "batch-6-tf32", "kind": "batch", "count": 6, "mix": 4, "precision": "tf32", "settle": 2},
        # observables of a converged state, ordinary size with an odd chi
        {"name": "rdm-kagome-D4-chi27-tf32", "kind": "rdm", "D": 4, "chi": 27, "precision": "tf32", "sites": 2,
         "settle": 2},
        # the bond environment an imaginary-time step starts from
        {"name": "core-kagome-D4-chi32-tf32", "kind": "core", "D": 4, "chi": 32, "precision": "tf32", "settle": 2},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["qr", "panel", "split", "split", "absorb", "iterate", "iterate", "batch", "rdm", "core"])
    if kind == "qr":
        n = rng.randint(3, 32)
        return {"kind": kind, "m": _log(rng, n, 256), "n": n}
    if kind == "panel":
        c64 = rng.random() < 0.7
        n = rng.randint(16, 96 if c64 else 48)
        return {"kind": kind, "dtype": "c64" if c64 else "c128", "m": _log(rng, 600, 2304 if c64 else 1100), "n": n}
    if kind == "split":
        c64 = rng.random() < 0.7
        chi = rng.randint(16, 64) if c64 else rng.randint(8, 32)
        lo, hi = (6 * chi, 36 * chi) if c64 else (6 * chi, 16 * chi)
        return {"kind": kind, "dtype": "c64" if c64 else "c128", "m": _log(rng, lo, hi), "n": _log(rng, lo, hi),
                "chi": chi, "power": 1 if c64 else 6}
    if kind == "absorb":
        return {"kind": kind, "mode": rng.choice(["tf32", "tf32", "bf16"]), "P": _log(rng, 16, 625),
                "Q": _log(rng, 16, 625), "l": rng.randint(5, 64), "r": rng.randint(5, 64)}
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(2, 6), "mix": rng.randint(5, 1 << 20), "precision": "tf32",
                "settle": 2}
    if kind == "rdm":
        return {"kind": kind, "D": rng.randint(2, 4), "chi": rng.randint(8, 27), "precision": "tf32",
                "sites": rng.randint(1, 2), "settle": 2}
    if kind == "core":
        return {"kind": kind, "D": rng.randint(2, 4), "chi": rng.randint(8, 32), "precision": "tf32", "settle": 2}
    precision = rng.choice(["fp64", "tf32", "tf32", "bf16", "fp32"])
    kagome = rng.random() < 0.5
    D = rng.randint(2, 3 if precision == "fp64" else 4)
    chi = rng.randint(8, 20 if precision == "fp64" else 32)
    block = 2 if kagome else rng.randint(2, 3)
    return {"kind": kind, "lattice": "kagome" if kagome else "square", "size": 2 if kagome else 2 * block,
            "block": block, "periodic": 1 if kagome else rng.randint(0, 1), "D": D, "chi": chi,
            "precision": precision, "alpha": rng.choice([1.0, 1.0, 0.75]), "hermitise": rng.choice([0, 0, 1]),
            "settle": 2}


# ------------------------------------------------------------------ networks

class Network:
    """A context that a program keeps: created, partitioned, settled."""

    def __init__(self, kagome, size, block, periodic, D, chi, precision, seed, alpha=1.0, hermitise=0, settle=2,
                 streams=16):
        if kagome:
            nb, Lx, Ly = syn.kagome_neighbours(3 * size, size), 3 * size, size
        else:
            nb, Lx, Ly = syn.square_neighbours(size, size, bool(periodic)), size, size
        n = len(nb)
        if precision == "fp64" and not kagome:      # generic tensors
            t = syn.gaussian_peps(n, 2, D, seed=seed)
        else:                                        # near a product of singlets, as after a few time steps
            t = syn.dimer_singlet_peps(nb, 2, D, seed=seed, noise=1e-2, noise_seed=seed + 1)
        edges = syn.initial_edge_matrices(n, D, seed=seed + 2)
        self.kagome, self.precision = kagome, precision
        self.ctx = P.bbp_create_peps(P.KAGOME if kagome else P.SQUARE, Lx, Ly, int(periodic), 2, D, t)
        P.bbp_partition_blocks(self.ctx, block, block)
        P.bbp_set_options(self.ctx, chi, PRECISION[precision], alpha)
        if hermitise:
            P.bbp_set_hermitise(self.ctx, True)
        P.bbp_set_execution(self.ctx, True, streams)
        P.bbp_init_messages(self.ctx, edges)
        if settle:
            P.bbp_iterate(self.ctx, 0.0, settle)
        self.blocks = P.bbp_info(self.ctx)[0]
        legs = 2 * block if kagome else block
        self.cap = 2 * legs * chi * chi * D * D
        self.large = precision != "fp64" and D ** (2 * legs) > 100000     # put together on the device

    def messages(self):
        """The incoming messages as dense vectors, one row each (open faces carry none)."""
        rows = []
        for b in range(self.blocks):
            for f in range(4):
                v = None
                for x in P.bbp_get_message(self.ctx, b, f, cap=self.cap):
                    if self.large:
                        x = torch.from_numpy(x).to("cuda", torch.complex64)
                    l, p, r = x.shape
                    v = x.reshape(l * p, r) if v is None else (v @ x.reshape(l, p * r)).reshape(-1, r)
                if v.shape[0] > 1:
                    rows.append(v.reshape(-1))
        if self.large:
            return torch.stack(rows)
        m = np.stack(rows)
        return m if self.precision == "fp64" else m.astype(np.complex64)

    def __del__(self):
        ctx, self.ctx = getattr(self, "ctx", None), None
        if ctx is not None:
            P.bbp_destroy(ctx)


def _mix(case):
    """(kagome, size, block, D, chi) of the networks of a batch: the shapes belong to the case, the entries to the seed."""
    rng = np.random.default_rng(case["mix"])
    out = []
    for _ in range(case["count"]):
        kagome = bool(rng.integers(2))
        block = 2 if kagome else int(rng.integers(2, 4))
        out.append((kagome, 2 if kagome else 2 * block, block, int(rng.integers(2, 5)), int(rng.choice([8, 16, 27, 32]))))
    return out


# -------------------------------------------------------------------- inputs

_ready = False


def _setup():
    global _ready
    if not _ready:
        P.lib()
        P.use_torch_allocator()
        _ready = True


def _gauss(shape, seed, dtype=torch.complex128):
    g = torch.Generator(device="cuda").manual_seed(seed)
    re = torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)
    im = torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)
    return torch.complex(re, im).to(dtype).contiguous()


def _matrices(case, seed):
    """Device inputs of the kernel-level kinds."""
    kind = case["kind"]
    dtype = torch.complex128 if case.get("dtype", "c128") == "c128" else torch.complex64
    if kind in ("qr", "panel"):
        return _gauss((case["m"], case["n"]), seed, dtype)
    if kind == "split":
        # singular values fall by e every chi / 6, as across the cuts of a PEPS with a finite correlation length
        m, n, chi = case["m"], case["n"], case["chi"]
        k = min(m, n, 4 * chi)
        a = torch.linalg.qr(_gauss((m, k), seed))[0]
        b = torch.linalg.qr(_gauss((n, k), seed + 1))[0]
        s = torch.exp(-torch.arange(k, device="cuda", dtype=torch.float64) * 6.0 / chi)
        return ((a * s) @ b.mH).to(dtype).contiguous()
    x = _gauss((case["P"], case["Q"]), seed, torch.complex64)
    s = _gauss((case["l"], case["P"], case["r"]), seed + 1, torch.complex64)
    return x / math.sqrt(case["P"]), s


def prepare(case, seed):
    _setup()
    kind = case["kind"]
    state = {"case": case}
    if kind in ("qr", "panel", "split", "absorb"):
        state["in"] = _matrices(case, seed)
        byte = torch.uint8
        if kind == "qr":
            m, n = case["m"], case["n"]
            state["a"] = torch.empty_like(state["in"])
            state["tau"] = torch.empty(min(m, n), dtype=torch.complex128, device="cuda")
        if kind == "split":
            c64 = case["dtype"] == "c64"
            nbytes = P.bbp_k_svd_work_bytes_rand(c64, case["m"], case["n"], case["chi"])
            state["work"] = torch.empty(nbytes, dtype=byte, device="cuda")
            state["status"] = torch.zeros(4, dtype=torch.int32, device="cuda")
        if kind == "absorb":
            nbytes = P.bbp_k_tc_absorb_bytes(case["mode"] == "bf16", case["P"], case["Q"], case["l"], case["r"])
            state["work"] = torch.empty(nbytes, dtype=byte, device="cuda")
            state["status"] = torch.zeros(4, dtype=torch.int32, device="cuda")
        return state
    if kind == "iterate":
        state["net"] = Network(case["lattice"] == "kagome", case["size"], case["block"], case["periodic"], case["D"],
                               case["chi"], case["precision"], seed, case["alpha"], case["hermitise"], case["settle"])
    elif kind == "batch":
        state["nets"] = [Network(kagome, size, block, int(kagome), D, chi, case["precision"], seed + 10 * i,
                                 settle=case["settle"], streams=2)
                         for i, (kagome, size, block, D, chi) in enumerate(_mix(case))]
    else:
        state["net"] = Network(True, 2, 2, 1, case["D"], case["chi"], case["precision"], seed, settle=case["settle"])
    return state


# ---------------------------------------------------------------------- runs

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "qr":                     # the call overwrites its input: a program copies what it keeps
        m, n = case["m"], case["n"]
        k = min(m, n)
        a, x = state["a"], state["in"]
        a.copy_(x)
        q, r = x.new_empty((m, k)), x.new_empty((k, n))
        P.bbp_k_qr(a, m, n, q, r, state["tau"])
        return {"q": q, "r": r}
    if kind == "panel":
        m, n, x = case["m"], case["n"], state["in"]
        q, r = torch.empty_like(x), x.new_empty((n, n))
        P.bbp_k_panel_qr(case["dtype"] == "c64", x, m, n, q, r)
        return {"q": q, "r": r}
    if kind == "split":
        m, n, x = case["m"], case["n"], state["in"]
        k = min(case["chi"], m, n)
        u, rem = x.new_empty((m, k)), x.new_empty((k, n))
        P.bbp_k_svd_trunc_rand(case["dtype"] == "c64", x, m, n, case["chi"], u, rem, state["work"], state["status"],
                               case["power"])
        return {"kept": u @ rem, "gram": u.mH @ u}
    if kind == "absorb":
        x, s = state["in"]
        out = s.new_empty((case["l"], case["Q"], case["r"]))
        P.bbp_k_tc_absorb(case["mode"] == "bf16", True, x, case["P"], case["Q"], s, case["l"], case["r"], out,
                          state["work"], state["status"])
        return out
    if kind == "batch":
        nets = state["nets"]
        _, iters, _, _ = P.bbp_batch_iterate([x.ctx for x in nets], 0.0, 1)
        return {"iters": iters, "messages": [x.messages() for x in nets]}
    net = state["net"]
    if kind == "iterate":
        iters, _, _ = P.bbp_iterate(net.ctx, 0.0, 1)
        return {"iters": iters, "messages": net.messages()}
    if kind == "rdm":
        return P.bbp_block_rdm(net.ctx, 0, [0, 1][:case["sites"]]).astype(np.complex64)
    # <a c| rho |b d> = <|b><a| (x) |d><c|> on the A-B bond of a block's first unit cell
    unit = np.eye(4).reshape(2, 2, 2, 2)
    ops = [[unit[b, a], unit[d, c]] for a in (0, 1) for c in (0, 1) for b in (0, 1) for d in (0, 1)]
    return P.bbp_core_expect(net.ctx, 0, [0, 1], ops).reshape(4, 4).astype(np.complex64)


# ---------------------------------------------------------------------- work

def _network_work(kagome, size, block, D, chi, precision, updates=None):
    """Absorbs of one iteration: each of a block's sites swallowed once for every outgoing message, 8 chi^2 D^8 real
    flops at full bonds; half of that, since the boundary's bonds are shorter near a block's corners."""
    sites = 9 * size * size if kagome else size * size
    faces = 4 if updates is None else updates
    z = 16 if precision == "fp64" else 8
    legs = 2 * block if kagome else block
    blocks = 3 if kagome else (size // block) ** 2
    flops = 0.5 * faces * sites * 8.0 * chi ** 2 * float(D) ** 8
    moved = sites * 2 * 16.0 * D ** 4 + 2.0 * blocks * faces * legs * z * chi * chi * D * D
    return moved, flops


def work(case):
    kind = case["kind"]
    z = 16.0 if case.get("dtype", "c128") == "c128" else 8.0
    if kind in ("qr", "panel"):
        m, n = case["m"], case["n"]
        k, t = min(m, n), max(m, n)
        return {"bytes": z * (m * n + m * k + k * n), "flops": 16.0 * (t * k * k - k ** 3 / 3.0)}
    if kind == "split":
        # one product with the matrix from each side and the kept factors
        m, n, k = case["m"], case["n"], case["chi"]
        return {"bytes": z * (m * n + m * k + k * n), "flops": 16.0 * m * n * k}
    if kind == "absorb":
        p, q, l, r = case["P"], case["Q"], case["l"], case["r"]
        return {"bytes": 8.0 * (p * q + l * p * r + l * q * r), "flops": 8.0 * l * p * q * r}
    if kind == "batch":
        parts = [_network_work(kagome, size, block, D, chi, case["precision"], 4 if kagome else 2)
                 for kagome, size, block, D, chi in _mix(case)]
        return {"bytes": sum(x[0] for x in parts), "flops": sum(x[1] for x in parts)}
    if kind == "iterate":
        moved, flops = _network_work(case["lattice"] == "kagome", case["size"], case["block"], case["D"], case["chi"],
                                     case["precision"], 4 if case["periodic"] else 2)
        return {"bytes": moved, "flops": flops}
    moved, flops = _network_work(True, 2, 2, case["D"], case["chi"], case["precision"])
    one = flops / 12                      # one block contracted once
    return {"bytes": moved / 3, "flops": one * ((1, 4, 16)[case["sites"]] if kind == "rdm" else 1)}


# --------------------------------------------------------------------- exact

def exact(case, seed):
    kind = case["kind"]
    if kind not in ("qr", "panel", "split", "absorb"):
        return None                       # a truncated iteration has no closed form
    x = _matrices(case, seed)
    if kind == "absorb":
        x, s = (v.to(torch.complex128) for v in x)
        return torch.stack([x.mT @ a for a in s])
    x = x.to(torch.complex128)
    if kind in ("qr", "panel"):           # LAPACK's convention: reflectors that leave a real diagonal
        q, r = torch.linalg.qr(x.cpu())
        return {"q": q, "r": r}
    tall = x if x.shape[0] >= x.shape[1] else x.mH
    v = torch.linalg.eigh((tall.mH @ tall).cpu())[1][:, -case["chi"]:].to(tall.device)
    kept = (tall @ v) @ v.mH
    return {"kept": kept if tall is x else kept.mH.contiguous(), "gram": torch.eye(case["chi"], dtype=x.dtype)}
