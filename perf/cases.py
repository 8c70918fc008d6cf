"""The workloads whose speed is watched: what a user of the library runs, from
one Krylov step on a tiny grid to batches of uneven matrices and a serving
burst.

A case is a dict of plain values:

  op     what is called: "spmv", "spmmv", "dot" (sell_spmv_dot), "batch"
         (a plan of many products), "build" (CRS -> SELL-C-sigma, one product,
         release) or "serve" (a burst of requests through the server)
  kind   the matrix recipe of paper_1307_6209_gb300/synth.py: "laplace",
         "stencil", "lognormal", "banded", "dense", "longrow", or "mixed"
         (banded and lognormal in turn, the batch recipe)
  n      grid side (laplace, stencil), side (dense) or rows (the others)
  C, sigma, store, k   chunk height, sorting scope, value storage ("f64",
         "f32", "bf16") and number of right-hand sides
  comp   accumulation of reduced-precision products: "plain", "all"
         (compensated) or "long" (compensated on rows over 64 entries)
  block, unroll, pipeline   launch shape (0, 0, -1: the library's own)
  count  matrices of a batch, requests of a burst
"""
import math

import numpy as np
import torch

from paper_1307_6209_gb300 import sell, serving, synth

STORE = {"f64": sell.SELL_F64, "f32": sell.SELL_F32, "bf16": sell.SELL_BF16}
STORE_DTYPE = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
VECTOR_DTYPE = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.float32}
VALUE_BYTES = {"f64": 8, "f32": 4, "bf16": 2}
COMP = {"plain": 0, "all": sell.SELL_SPMV_COMPENSATED, "long": sell.SELL_SPMV_COMPENSATED_LONG}
N_SORT = 1 << 30  # a sorting scope no smaller than any matrix here: a global sort
SERVE_MATRICES = 8


def _case(op, kind, n, *, C=32, sigma=1, store="f64", k=1, comp="plain", block=0, unroll=0, pipeline=-1, count=1,
          name=None):
    c = dict(op=op, kind=kind, n=n, C=C, sigma=sigma, store=store, k=k, comp=comp, block=block, unroll=unroll,
             pipeline=pipeline, count=count)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one conjugate-gradient step (p, Ap, p . Ap) on the 5-point Laplacian of a 64 x 64 grid: the smallest
        # call, where launches and latency are all there is
        _case("dot", "laplace", 64, name="krylov_laplace64_f64"),
        # the 27-point stencil on 200^3, binary64, with the launch the autotuner picks for it: the large regular
        # matrix of a structured-grid solver
        _case("spmv", "stencil", 200, C=128, block=128, unroll=2, pipeline=1, name="spmv_stencil200_f64"),
        # the same kind of matrix with bfloat16 values (mixed-precision preconditioner), an odd grid, no tuning
        _case("spmv", "stencil", 187, store="bf16", name="spmv_stencil187_bf16"),
        # a block solver: eight right-hand sides at once, binary32
        _case("spmmv", "stencil", 150, store="f32", k=8, name="spmmv_stencil150_f32_k8"),
        # the irregular matrix of the C x sigma sweep: random columns, lognormal row lengths
        _case("spmv", "lognormal", 2_000_000, sigma=N_SORT, name="spmv_lognormal2M_f64"),
        # four right-hand sides on an irregular matrix of odd size, compensated long rows, the sigma of the sweep
        _case("spmmv", "lognormal", 999_983, C=64, sigma=4096, store="f32", k=4, comp="long",
              name="spmmv_lognormal1M_f32_k4"),
        # the two pathological shapes of the paper: a dense matrix stored as sparse, and short rows with one of 10^6
        _case("spmv", "dense", 8000, name="spmv_dense8000_f64"),
        _case("spmv", "longrow", 1_000_000, name="spmv_longrow1M_f64"),
        # many uneven matrices in one plan (rows uniform in 1,000..200,000, half banded, half lognormal), at one
        # and at eight right-hand sides
        _case("batch", "mixed", 200_000, sigma=N_SORT, store="f32", count=96, name="batch96_mixed_f32_k1"),
        _case("batch", "mixed", 200_000, sigma=4096, store="f32", k=8, count=48, name="batch48_mixed_f32_k8"),
        # a matrix that changes: conversion from CRS on the device, its first product, release
        _case("build", "lognormal", 2_000_000, sigma=N_SORT, name="build_lognormal2M_f64"),
        # requests of 1-8 right-hand sides against resident matrices, through the server, host to host
        _case("serve", "lognormal", 300_000, sigma=N_SORT, count=32, name="serve_burst32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["spmv", "spmv", "spmv", "spmmv", "spmmv", "dot", "batch", "batch", "build", "build", "serve"])
    C = rng.choice([32, 32, 64, 128])
    sigma = rng.choice([1, 256, 4096, N_SORT])
    store = rng.choice(["f64", "f64", "f32", "f32", "bf16"])
    comp = "plain" if store == "f64" else rng.choice(["plain", "plain", "all", "long"])
    if op == "batch":
        return _case(op, rng.choice(["mixed", "mixed", "banded", "lognormal"]), _log_int(rng, 2_000, 200_000), C=C,
                     sigma=max(256, sigma), store=store, k=rng.choice([1, 1, 2, 4, 5, 8]), comp=comp,
                     count=rng.randint(4, 64))
    if op == "serve":
        return _case(op, "lognormal", _log_int(rng, 10_000, 300_000), C=32, sigma=N_SORT, count=rng.randint(4, 32))
    kind = rng.choice(["stencil", "lognormal", "banded"] if op == "build" else
                      ["laplace", "stencil", "stencil", "lognormal", "lognormal", "banded", "dense", "longrow"])
    k = rng.choice([2, 3, 4, 5, 7, 8, 8, 16]) if op == "spmmv" else 1
    if kind == "laplace":
        n = _log_int(rng, 16, 512)
    elif kind == "stencil":
        n = _log_int(rng, 10, 120 if op == "build" else 200 if k <= 2 else 150)
    elif kind == "dense":
        n = _log_int(rng, 100, 8000 if k <= 2 else 4000)
    elif kind == "longrow":
        n = _log_int(rng, 10_000, 1_000_000)
    else:
        n = _log_int(rng, 1_000, 2_000_000 if k <= 4 else 1_000_000)
    return _case(op, kind, n, C=C, sigma=sigma, store=store, k=k, comp=comp)


# ------------------------------------------------------------------ inputs
def _matrix(kind, n, store, seed):
    """The CRS matrix on the device, its values already those of the storage type."""
    if kind == "laplace":
        A = synth.laplace2d(n)
        A = synth.CSR(A.nrows, A.ncols, *(torch.from_numpy(v).cuda() for v in (A.rpt, A.col, A.val)))
    elif kind == "stencil":
        A = synth.stencil27_device(n, 0.1, seed=seed)
    elif kind == "lognormal":
        A = synth.lognormal_device(n, seed=seed)
    elif kind == "banded":
        A = synth.banded_device(n, seed=seed)
    elif kind == "dense":
        A = synth.dense_device(n, seed=seed)
    else:
        A = synth.long_row_device(n, n, seed=seed)
    A.val = A.val.to(STORE_DTYPE[store]).to(torch.float64)
    return A


def _vectors(n, k, dtype, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.rand((n, k) if k > 1 else (n,), generator=g, dtype=dtype, device="cuda") * 2 - 1


def _parts(case, seed):
    """(kind, rows, seed) of each matrix of a batch: the batch recipe scaled to at most n rows (the sizes are the
    case's own, the entries come from the seed)."""
    rng = np.random.default_rng([case["n"], case["count"]])
    rows = rng.integers(max(1, case["n"] // 200), case["n"] + 1, case["count"])
    kinds = ["banded", "lognormal"] if case["kind"] == "mixed" else [case["kind"]] * 2
    return [(kinds[i % 2], int(r), seed * 1000 + i) for i, r in enumerate(rows)]


def _serve_parts(case, seed):
    """Resident matrices (rows log-uniform up to n, half f64, half f32) and the requests (matrix, k, seed); sizes
    and request mix are the case's own."""
    rng = np.random.default_rng([case["n"], case["count"]])
    rows = np.exp(rng.uniform(math.log(max(1000, case["n"] // 30)), math.log(case["n"]), SERVE_MATRICES)).astype(int)
    mats = [(int(r), "f64" if i % 2 == 0 else "f32", seed * 1000 + i) for i, r in enumerate(rows)]
    reqs = [(int(rng.integers(0, SERVE_MATRICES)), int(rng.integers(1, 9)), seed * 1000 + 500 + i)
            for i in range(case["count"])]
    return mats, reqs


def _build(case, A, store=None):
    h = sell.sell_build(A, C=case["C"], sigma=min(case["sigma"], max(1, A.nrows)), store_type=STORE[store or case["store"]])
    if case["block"] or case["unroll"] or case["pipeline"] >= 0:
        sell.sell_set_launch(h, case["block"], case["unroll"], case["pipeline"])
    return h


def _padded(rows, k):
    """Elements that one matrix's block takes in a buffer shared by a batch (blocks start 256-byte aligned)."""
    return (rows * k + 63) // 64 * 64


def prepare(case, seed):
    op, k, dtype = case["op"], case["k"], VECTOR_DTYPE[case["store"]]
    flags = COMP[case["comp"]]
    if op == "serve":
        mats, reqs = _serve_parts(case, seed)
        hs = [_build(case, _matrix(case["kind"], r, st, sd), st) for r, st, sd in mats]
        X = [_vectors(mats[m][0], kk, VECTOR_DTYPE[mats[m][1]], sd).cpu().pin_memory() for m, kk, sd in reqs]
        srv = serving.Server(hs, sum(h.info.device_bytes for h in hs) + (1 << 30), max_batch=64, streams=6)
        return {"op": op, "srv": srv, "reqs": [(m, x) for (m, _, _), x in zip(reqs, X)]}
    if op == "batch":
        parts = _parts(case, seed)
        y = torch.zeros(sum(_padded(r, k) for _, r, _ in parts), dtype=dtype, device="cuda")
        items, at = [], 0
        for kind, r, sd in parts:
            h = _build(case, _matrix(kind, r, case["store"], sd))
            Y = y[at:at + r * k].view((r, k) if k > 1 else (r,))
            items.append((h, _vectors(r, k, dtype, sd), Y, flags))
            at += _padded(r, k)
        return {"op": op, "plan": sell.sell_batch_create(items), "y": y}
    A = _matrix(case["kind"], case["n"], case["store"], seed)
    x = _vectors(A.ncols, k, dtype, seed + 1)
    y = torch.empty((A.nrows, k) if k > 1 else (A.nrows,), dtype=dtype, device="cuda")
    if op == "build":
        return {"op": op, "case": case, "A": A, "x": x, "y": y, "flags": flags}
    dot = torch.empty(1, dtype=torch.float64, device="cuda")
    return {"op": op, "h": _build(case, A), "x": x, "y": y, "dot": dot, "flags": flags}


def run(state):
    op = state["op"]
    if op == "spmv":
        return sell.sell_spmv(state["h"], state["x"], state["y"], state["flags"])
    if op == "spmmv":
        return sell.sell_spmmv(state["h"], state["x"], state["y"], state["flags"])
    if op == "dot":
        sell.sell_spmv_dot(state["h"], state["x"], state["y"], state["dot"], state["flags"])
        return [state["y"], state["dot"]]
    if op == "batch":
        state["plan"].run()
        return state["y"]
    if op == "build":
        h = _build(state["case"], state["A"])
        sell.sell_spmv(h, state["x"], state["y"], state["flags"])
        info = h.info
        h.free()
        return [state["y"], info.stored, info.max_row_len, info.beta, info.zeta]
    pending = [state["srv"].submit(m, x) for m, x in state["reqs"]]
    return [r.wait().Y for r in pending]


# ------------------------------------------------------------------ the least work
def _entries(kind, n):
    """Rows and (expected) entries of a recipe."""
    if kind == "laplace":
        return n * n, 5 * n * n - 4 * n
    if kind == "stencil":
        return n ** 3, (3 * n - 2) ** 3
    if kind == "dense":
        return n, n * n
    if kind == "longrow":
        return n, 3 * (n - 1) + n
    if kind == "banded":
        return n, 18.5 * n
    return n, 16 * n


def _product(rows, entries, store, k):
    """Values and columns once, a length per row, x once, y once."""
    v = 8 if store == "f64" else 4
    return {"bytes": entries * (VALUE_BYTES[store] + 4) + 4 * rows + 2 * rows * k * v, "flops": 2 * entries * k}


def work(case):
    op, k, store = case["op"], case["k"], case["store"]
    if op == "serve":
        mats, reqs = _serve_parts(case, 1)
        w = [_product(*_entries("lognormal", mats[m][0]), mats[m][1], kk) for m, kk, _ in reqs]
    elif op == "batch":
        w = [_product(*_entries(kind, r), store, k) for kind, r, _ in _parts(case, 1)]
    else:
        rows, entries = _entries(case["kind"], case["n"])
        w = [_product(rows, entries, store, k)]
        if op == "build":  # CRS read (binary64 values), the format written, then read by the product
            w.append({"bytes": entries * (12 + VALUE_BYTES[store] + 4) + 12 * rows, "flops": 0})
        if op == "dot":
            w.append({"bytes": 8, "flops": 2 * rows})
    return {"bytes": sum(p["bytes"] for p in w), "flops": sum(p["flops"] for p in w)}


# ------------------------------------------------------------------ the same in 64 bits
def _exact_product(A, x):
    rows = torch.repeat_interleave(torch.arange(A.nrows, device="cuda"), A.rpt[1:] - A.rpt[:-1])
    col = A.col.long()
    x = x.double().view(A.ncols, -1)
    y = torch.zeros((A.nrows, x.shape[1]), dtype=torch.float64, device="cuda")
    for q in range(x.shape[1]):
        y[:, q].index_add_(0, rows, A.val * x[:, q][col])
    return y


def exact(case, seed):
    op, k, dtype = case["op"], case["k"], VECTOR_DTYPE[case["store"]]
    if op == "serve":
        mats, reqs = _serve_parts(case, seed)
        A = [_matrix(case["kind"], r, st, sd) for r, st, sd in mats]
        out = []
        for m, kk, sd in reqs:
            y = _exact_product(A[m], _vectors(mats[m][0], kk, VECTOR_DTYPE[mats[m][1]], sd))
            out.append((y if kk > 1 else y[:, 0]).cpu())
        return out
    if op == "batch":
        parts = _parts(case, seed)
        y = torch.zeros(sum(_padded(r, k) for _, r, _ in parts), dtype=torch.float64, device="cuda")
        at = 0
        for kind, r, sd in parts:
            A = _matrix(kind, r, case["store"], sd)
            y[at:at + r * k] = _exact_product(A, _vectors(r, k, dtype, sd)).reshape(-1)
            at += _padded(r, k)
        return y
    A = _matrix(case["kind"], case["n"], case["store"], seed)
    x = _vectors(A.ncols, k, dtype, seed + 1)
    y = _exact_product(A, x)
    y = y if k > 1 else y[:, 0]
    if op == "dot":
        return [y, torch.dot(x.double(), y).view(1)]
    if op == "build":
        return [y, None, None, None, None]
    return y
