"""Workloads the library's speed is measured on, through the Python binding.

Each case is a dict of plain values. listed() gives the standing ones, draw()
more of the same kinds and ranges, prepare() the inputs and buffers a program
holds before the call, run() one pass, work() the traffic and operations a
pass cannot do without, exact() the result in plain FP64 PyTorch.

Kinds:
  hpl      FP64 LU with partial pivoting and the solve of one right-hand side
           (with emulation: the trailing update on the BF16 tensor cores)
  solve    several right-hand sides against a factor in hand, A X = B and
           A^T X = B
  mxp      mixed-precision solve of a diagonally dominant system
  batch    many uneven small systems in one launch, half of them general with
           pivoting in FP64, half dominant in mixed precision
  layer    the differentiable solve, forward and backward
"""
import numpy as np
import torch

import paper_2604_09517_gb300 as hpl

PREC = {"bf16": hpl.PREC_BF16, "fp8": hpl.PREC_FP8_E4M3, "fp16": hpl.PREC_FP16, "tf32": hpl.PREC_TF32}


def listed():
    return [
        # the small benchmark system: a program that solves one dense system at
        # a time, bound by the latency of 1024 dependent pivot searches
        {"name": "hpl_1024", "kind": "hpl", "n": 1024, "nb": 64, "lookahead": 0, "emulation": 0},
        # an ordinary system of odd order with the default options
        {"name": "hpl_3001", "kind": "hpl", "n": 3001, "nb": 256, "lookahead": 1, "emulation": 0},
        # the large FP64 system of the test suite, where the update dominates
        {"name": "hpl_12800", "kind": "hpl", "n": 12800, "nb": 256, "lookahead": 1, "emulation": 0},
        # FP64 accuracy from the tensor cores, the fast way to a pivoted FP64 factor
        {"name": "hpl_emulated_8192", "kind": "hpl", "n": 8192, "nb": 256, "lookahead": 1, "emulation": 1},
        # a factor reused for new right-hand sides, and its transpose as an adjoint needs it
        {"name": "solve_4096x64", "kind": "solve", "n": 4096, "nrhs": 64},
        # a small mixed-precision system, a single panel wide: launches and host reads count
        {"name": "mxp_2000", "kind": "mxp", "n": 2000, "nb": 3072, "prec": "bf16", "stored": True, "bf16_storage": False,
         "inner32": False, "ns_iters": 2},
        # an ordinary mixed-precision system with the default options
        {"name": "mxp_16384", "kind": "mxp", "n": 16384, "nb": 3072, "prec": "bf16", "stored": True,
         "bf16_storage": False, "inner32": False, "ns_iters": 2},
        # a large one with FP8 operands and the benchmark's options
        {"name": "mxp_fp8_49152", "kind": "mxp", "n": 49152, "nb": 4096, "prec": "fp8", "stored": True,
         "bf16_storage": False, "inner32": True, "ns_iters": 1},
        # the matrix regenerated from its seed and kept in BF16 only: the way to
        # the largest orders a GPU's memory holds
        {"name": "mxp_regen_65536", "kind": "mxp", "n": 65536, "nb": 4096, "prec": "bf16", "stored": False,
         "bf16_storage": True, "inner32": False, "ns_iters": 1},
        # a small batch: fewer systems than two per SM, so the longest one counts
        {"name": "batch_256", "kind": "batch", "count": 256},
        # the benchmark's batch
        {"name": "batch_4096", "kind": "batch", "count": 4096},
        # the benchmark's differentiable layer, one training step's forward and backward
        {"name": "layer_4096x64", "kind": "layer", "n": 4096, "nrhs": 64, "nb": 2048},
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["hpl", "hpl", "emulated", "solve", "mxp", "mxp", "mxp", "batch", "layer"])
    if kind == "hpl":
        n = _log(rng, 300, 12800)
        return {"kind": "hpl", "n": n, "nb": rng.choice([64, 128] if n < 2048 else [128, 256]),
                "lookahead": rng.choice([0, 1]) if n < 4096 else 1, "emulation": 0}
    if kind == "emulated":
        return {"kind": "hpl", "n": _log(rng, 2048, 16384), "nb": 256, "lookahead": 1, "emulation": 1}
    if kind == "solve":
        return {"kind": "solve", "n": _log(rng, 300, 8192), "nrhs": _log(rng, 2, 128)}
    if kind == "batch":
        return {"kind": "batch", "count": _log(rng, 64, 4096)}
    if kind == "layer":
        return {"kind": "layer", "n": _log(rng, 256, 6144), "nrhs": _log(rng, 1, 128), "nb": rng.choice([1024, 2048])}
    stored = rng.random() < 0.75
    n = _log(rng, 1000, 49152 if stored else 65536)
    prec = rng.choice(["bf16", "bf16", "fp8", "fp16", "tf32"])
    big = n >= 24576
    storage = prec == "bf16" and rng.random() < 0.4
    return {"kind": "mxp", "n": n, "nb": rng.choice([3072, 4096]) if big else rng.choice([1024, 2048, 3072]), "prec": prec,
            "stored": stored, "bf16_storage": storage, "inner32": not storage and rng.random() < 0.5,
            "ns_iters": 1 if big else 2}


# --------------------------------------------------------------------------
# Inputs: from the seed alone, column-major, uniform[-0.5, 0.5).

def _rng(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _uniform(g, m, n):
    return (torch.rand((n, m), generator=g, dtype=torch.float64, device="cuda").sub_(0.5)).t()


def _dominant(g, n):
    """Uniform entries, the diagonal replaced by its row's sum of magnitudes."""
    A = _uniform(g, n, n)
    rows = torch.zeros(n, dtype=torch.float64, device="cuda")
    for c in range(0, n, 4096):
        rows += A[:, c:c + 4096].abs().sum(dim=1)
    A.diagonal().copy_(rows)
    return A


def _batch_sizes(count):
    """n ~ U{32..512}: the first half general, the second dominant."""
    return np.random.default_rng(1).integers(32, 513, size=count), (np.arange(count) >= count // 2).astype(np.uint8)


def _batch_data(seed, n, kind):
    g = _rng(seed)
    a = torch.rand(int((n * n).sum()), generator=g, dtype=torch.float64, device="cuda").sub_(0.5)
    b = torch.rand(int(n.sum()), generator=g, dtype=torch.float64, device="cuda").sub_(0.5)
    off = 0
    for s in range(len(n)):
        k = int(n[s])
        if kind[s]:
            A = a[off:off + k * k].view(k, k).t()
            A.diagonal().copy_(A.abs().sum(dim=1))
        off += k * k
    return a, b


def prepare(case, seed):
    lib = hpl.load()
    kind = case["kind"]
    if kind == "batch":
        n, k = _batch_sizes(case["count"])
        a, b = _batch_data(seed, n, k)
        bt = hpl.Batch(n, k)
        bt.plan()
        return {"kind": kind, "batch": bt, "A": a, "B": b}
    n = case["n"]
    g = _rng(seed)
    if kind == "hpl":
        A0, b0 = _uniform(g, n, n), _uniform(g, n, 1)[:, 0]
        opts = hpl.make_opts(nb=case["nb"], lookahead=case["lookahead"], fp64_emulation=case["emulation"])
        return {"kind": kind, "case": case, "A0": A0, "b0": b0, "A": hpl.colmajor(n, n), "x": torch.empty_like(b0),
                "ipiv": torch.empty(n, dtype=torch.int32, device="cuda"), "info": hpl.Info(),
                "ws": hpl.workspace(lib.lu_factor_workspace_size(n, opts)),
                "sws": hpl.workspace(lib.lu_solve_workspace_size(n, 1))}
    if kind == "solve":
        LU, r = _uniform(g, n, n), case["nrhs"]
        ipiv, _ = hpl.lu_factor(LU)
        return {"kind": kind, "LU": LU, "ipiv": ipiv, "B0": _uniform(g, n, r), "X": hpl.colmajor(n, r),
                "Y": hpl.colmajor(n, r), "ws": hpl.workspace(lib.lu_solve_workspace_size(n, r))}
    if kind == "mxp":
        A = _dominant(g, n) if case["stored"] else None
        opt = dict(nb=case["nb"], prec=PREC[case["prec"]], ns_iters=case["ns_iters"],
                   storage=hpl.STORAGE_BF16 if case["bf16_storage"] else hpl.STORAGE_FP32,
                   inner=hpl.INNER_FP32 if case["inner32"] else hpl.INNER_FP64)
        need = lib.mxp_workspace_size(n, 1, hpl.make_opts(**opt))
        return {"kind": kind, "A": A, "b": _uniform(g, n, 1)[:, 0], "seed": seed, "opt": opt, "ws": hpl.workspace(need),
                "X": hpl.colmajor(n, 1), "info": hpl.Info()}
    A, B = _dominant(g, n).requires_grad_(), _uniform(g, n, case["nrhs"]).requires_grad_()
    G = torch.randn((case["nrhs"], n), generator=g, dtype=torch.float64, device="cuda").t()
    return {"kind": kind, "A": A, "B": B, "G": G, "nb": case["nb"]}


def run(state):
    kind = state["kind"]
    if kind == "hpl":
        # the factorization is in place and the program keeps A for the residual check
        c, A, x = state["case"], state["A"], state["x"]
        A.copy_(state["A0"])
        x.copy_(state["b0"])
        ipiv, _ = hpl.lu_factor(A, nb=c["nb"], lookahead=c["lookahead"], fp64_emulation=c["emulation"],
                                ipiv=state["ipiv"], ws=state["ws"], info=state["info"])
        hpl.lu_solve(A, ipiv, x, ws=state["sws"])
        return {"lu": A, "ipiv": ipiv, "x": x}
    if kind == "solve":
        X, Y = state["X"].copy_(state["B0"]), state["Y"].copy_(state["B0"])
        hpl.lu_solve(state["LU"], state["ipiv"], X, ws=state["ws"])
        hpl.lu_solve(state["LU"], state["ipiv"], Y, trans=1, ws=state["ws"])
        return {"x": X, "xt": Y}
    if kind == "mxp":
        X, _, _ = hpl.mxp_solve(state["A"], state["b"], X=state["X"], ws=state["ws"], info=state["info"],
                                seed=state["seed"], **state["opt"])
        return {"x": X}
    if kind == "batch":
        # general systems are factored in place, every solution replaces its right-hand side
        bt = state["batch"]
        bt.A.copy_(state["A"])
        bt.B.copy_(state["B"])
        bt.run()
        return {"lu": bt.A, "ipiv": bt.ipiv, "x": bt.B}
    X = hpl.solve(state["A"], state["B"], state["nb"])
    gA, gB = torch.autograd.grad(X, (state["A"], state["B"]), state["G"])
    return {"x": X, "grad_a": gA, "grad_b": gB}


def work(case):
    """Bytes: every input read once, every output written once. Flops: 2n^3/3
    per factorization, 2n^2 per right-hand side and triangular solve pair; the
    layer's backward adds the transposed solves and the outer product."""
    if case["kind"] == "batch":
        n, kind = _batch_sizes(case["count"])
        n, gen = n.astype(float), kind == 0
        return {"bytes": 8 * float((n * n).sum() + (n * n)[gen].sum() + 2 * n.sum()) + 4 * float(n[gen].sum()),
                "flops": float((2 * n ** 3 / 3 + 2 * n * n).sum())}
    n = float(case["n"])
    lu = 2 * n ** 3 / 3
    if case["kind"] == "hpl":
        return {"bytes": 16 * n * n + 20 * n, "flops": lu + 2 * n * n}
    if case["kind"] == "solve":
        return {"bytes": 8 * n * n + 24 * n * case["nrhs"], "flops": 4 * n * n * case["nrhs"]}
    if case["kind"] == "mxp":
        return {"bytes": (8 * n * n if case["stored"] else 0) + 16 * n, "flops": lu + 2 * n * n}
    r = case["nrhs"]
    return {"bytes": 16 * n * n + 32 * n * r, "flops": lu + 6 * n * n * r}


def _solve(A, B):
    """A X = B by LU with partial pivoting and one step of refinement."""
    LU, piv = torch.linalg.lu_factor(A)
    X = torch.linalg.lu_solve(LU, piv, B)
    return LU, X + torch.linalg.lu_solve(LU, piv, B - A @ X)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        n, k = _batch_sizes(case["count"])
        a, b = _batch_data(seed, n, k)
        off = boff = 0
        for s in range(len(n)):
            m = int(n[s])
            A, x = a[off:off + m * m].view(m, m).t(), b[boff:boff + m].view(m, 1)
            LU, X = _solve(A, x)
            x.copy_(X)
            if not k[s]:
                A.copy_(LU)
            off, boff = off + m * m, boff + m
        return {"lu": a, "ipiv": None, "x": b}
    n = case["n"]
    if n > 20000 or (kind == "mxp" and not case["stored"]):
        return None         # too long, or a matrix that only the library's generator defines
    g = _rng(seed)
    if kind == "hpl":
        LU, x = _solve(_uniform(g, n, n), _uniform(g, n, 1))
        return {"lu": LU, "ipiv": None, "x": x[:, 0]}
    if kind == "solve":
        A = _uniform(g, n, n)
        B = _uniform(g, n, case["nrhs"])
        return {"x": _solve(A, B)[1], "xt": _solve(A.t(), B)[1]}
    A = _dominant(g, n)
    if kind == "mxp":
        return {"x": _solve(A, _uniform(g, n, 1))[1]}
    B = _uniform(g, n, case["nrhs"])
    G = torch.randn((case["nrhs"], n), generator=g, dtype=torch.float64, device="cuda").t()
    X, gB = _solve(A, B)[1], _solve(A.t(), G)[1]
    return {"x": X, "grad_a": -gB @ X.t(), "grad_b": gB}
