"""What users of this framework have it do, as cases that can be timed and compared.

A case is a plain dict; `prepare` builds its inputs on the GPU from a seed and the plan a program
keeps, `run` makes one pass through the public entry points and returns every output core, `work`
says what the pass cannot do without, and `exact` gives the outputs in 64-bit numpy where they are
unique (left-orthogonal results of an untruncated recompression, inner products). Truncated
results are unique up to the signs of their singular directions only, so they have no `exact`.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2410_04385_gb300 import binding, costmodel, power_iteration

PRECISION = {"fp64": binding.TT_FP64, "fp32": binding.TT_MIXED_FP32, "tf32": binding.TT_MIXED_TF32,
             "bf16": binding.TT_MIXED_BF16, "fp64_tc": binding.TT_FP64_TC}

# A drawn case's predicted flops stay below the largest listed one's.
MAX_FLOPS = 9.0e10


def listed():
    return [
        # One pointwise product of two small functions on an 8^6 grid, through the one-line call
        # that plans, runs and returns the cores: an interactive user's or a loop's smallest unit.
        {"name": "small_call", "kind": "product", "form": "call", "d": 6, "n": 8, "ry": 2, "rz": 5,
         "sketch": 12, "max_rank": 10, "tol": 1e-12, "precision": "fp64", "variant": 1, "ep": 0.0,
         "ragged": False},
        # The inner product behind every relative error and norm: order 20, rank 50 operands.
        {"name": "dot_d20", "kind": "dot", "d": 20, "n": 32, "ry": 50, "rz": 50},
        # Largest-entry search: two iterations on a rank-50, order-50 tensor with sketch rank 5, a
        # chain of very small recompressions and inner products issued from Python.
        {"name": "power_d50", "kind": "power", "d": 50, "n": 10, "ry": 50, "rank": 5, "iters": 2},
        # HaTT-2 (truncated sketches) at the size of the Fourier-series experiment, as a graph.
        {"name": "hatt2_d7", "kind": "product", "form": "graph", "d": 7, "n": 20, "ry": 20, "rz": 18,
         "sketch": 30, "max_rank": 0, "tol": 0.0, "precision": "fp64", "variant": 2, "ep": 0.01,
         "ragged": False},
        # The headline workload: random pair, order 20, modes 32, ranks 20 (Kronecker rank 400),
        # sketch 50, target rank 40, planned once and replayed as a CUDA graph.
        {"name": "hatt_d20", "kind": "product", "form": "graph", "d": 20, "n": 32, "ry": 20, "rz": 20,
         "sketch": 50, "max_rank": 40, "tol": 0.0, "precision": "fp64", "variant": 1, "ep": 0.0,
         "ragged": False},
        # Uneven modes and ranks, planned once and called eagerly, no truncation (every core has an
        # exact value): the shapes real tensors have.
        {"name": "hatt_ragged", "kind": "product", "form": "eager", "d": 15, "n": 33, "ry": 29, "rz": 17,
         "sketch": 45, "max_rank": 0, "tol": 0.0, "precision": "fp64", "variant": 1, "ep": 0.0,
         "ragged": True},
        # Large modes and ranks at the size of the smooth order-50 configuration (n = 64, ranks
        # 40, sketch 90, target 80, tol 1e-8), fewer cores: one big recompression, called eagerly.
        {"name": "hatt_n64", "kind": "product", "form": "eager", "d": 12, "n": 64, "ry": 40, "rz": 40,
         "sketch": 90, "max_rank": 80, "tol": 1e-8, "precision": "fp64", "variant": 1, "ep": 0.0,
         "ragged": False},
        # The same size with TF32 sketch products (FP64 everywhere else), as a graph.
        {"name": "hatt_n64_tf32", "kind": "product", "form": "graph", "d": 12, "n": 64, "ry": 40, "rz": 40,
         "sketch": 90, "max_rank": 80, "tol": 0.0, "precision": "tf32", "variant": 1, "ep": 0.0,
         "ragged": False},
        # FP64-accurate products on the tensor cores, no truncation.
        {"name": "hatt_n64_tc", "kind": "product", "form": "eager", "d": 10, "n": 64, "ry": 40, "rz": 36,
         "sketch": 80, "max_rank": 0, "tol": 0.0, "precision": "fp64_tc", "variant": 1, "ep": 0.0,
         "ragged": False},
        # A sum of four tensors (what a time step or a Krylov update leaves) as one TT of rank 96 on
        # a 64^8 grid, rounded back to the rank-24 cap; shapes fixed, called eagerly.
        {"name": "round_r96", "kind": "round", "form": "eager", "d": 8, "n": 64, "ry": 24, "max_rank": 24,
         "tol": 1e-8},
        # The nonlinear half: u * u at the solver's rank cap and tolerance, replayed as a graph
        # (every truncation level is in the graph, the host reads nothing back).
        {"name": "square_graph", "kind": "square", "form": "graph", "d": 8, "n": 64, "ry": 24,
         "max_rank": 24, "tol": 1e-10, "precision": "fp64"},
        # Many independent uneven pairs in one persistent launch of the task engine.
        {"name": "batch_12", "kind": "batch", "count": 12, "dmin": 10, "dmax": 20, "n": 32, "rmin": 8,
         "rmax": 40, "precision": "fp64", "shapes": 7},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_any(rng):
    kind = rng.choice(["call", "eager", "eager", "graph", "graph", "trunc", "tc", "tf32", "hatt2", "dot", "power",
                       "round", "square", "batch"])
    if kind == "dot":
        return {"kind": "dot", "d": rng.randint(2, 40), "n": _log(rng, 4, 64), "ry": _log(rng, 2, 100),
                "rz": _log(rng, 2, 100)}
    if kind == "power":
        return {"kind": "power", "d": rng.randint(6, 50), "n": rng.randint(5, 16), "ry": _log(rng, 6, 50),
                "rank": rng.randint(3, 8), "iters": rng.randint(1, 3)}
    if kind == "round":
        r = _log(rng, 5, 32)
        return {"kind": "round", "form": "eager", "d": rng.randint(3, 12), "n": rng.randint(9, 64), "ry": r,
                "max_rank": r, "tol": 1e-8}
    if kind == "square":
        return {"kind": "square", "form": rng.choice(["graph", "eager"]), "d": rng.randint(4, 10),
                "n": rng.randint(16, 64), "ry": _log(rng, 8, 32), "max_rank": _log(rng, 8, 32),
                "tol": 1e-10, "precision": "fp64"}
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(4, 12), "dmin": 6, "dmax": rng.randint(8, 20),
                "n": rng.choice([16, 21, 32]), "rmin": 8, "rmax": rng.randint(12, 40), "precision": "fp64",
                "shapes": rng.randint(0, 999)}
    case = {"kind": "product", "form": rng.choice(["eager", "graph"]), "d": rng.randint(4, 24),
            "n": rng.randint(7, 64), "ry": _log(rng, 4, 40), "rz": _log(rng, 4, 40), "sketch": _log(rng, 8, 96),
            "max_rank": 0, "tol": 0.0, "precision": "fp64", "variant": 1, "ep": 0.0,
            "ragged": rng.random() < 0.5}
    if kind == "call":
        case.update(form="call", d=rng.randint(3, 8), n=rng.randint(4, 16), ry=rng.randint(2, 6),
                    rz=rng.randint(2, 6), sketch=rng.randint(6, 16))
    elif kind in ("eager", "graph"):
        case.update(form=kind)
    elif kind == "trunc":
        case.update(sketch=rng.randint(12, 96))
        case.update(max_rank=max(4, int(0.8 * case["sketch"])), tol=rng.choice([0.0, 1e-8]))
    elif kind == "tc":
        case.update(precision="fp64_tc", n=rng.randint(24, 64), ry=rng.randint(16, 40), rz=rng.randint(16, 40),
                    sketch=rng.randint(32, 96))
    elif kind == "tf32":
        case.update(precision=rng.choice(["tf32", "bf16", "fp32"]), n=rng.randint(24, 64), ry=rng.randint(16, 40),
                    rz=rng.randint(16, 40), sketch=rng.randint(32, 96))
    elif kind == "hatt2":
        case.update(variant=2, ep=0.01, d=rng.randint(4, 10), sketch=_log(rng, 8, 40))
    return case


def draw(rng):
    while True:
        case = _draw_any(rng)
        if work(case)["flops"] <= MAX_FLOPS:
            return case


# ------------------------------------------------------------------ shapes ---

def _shapes(case):
    """Mode sizes and the operands' bond ranks of a product (uneven with `ragged`: drawn between
    the half and the whole of the named sizes from the case alone)."""
    d, n = case["d"], case["n"]
    if not case.get("ragged"):
        ry, rz = [case["ry"]] * (d - 1), [case["rz"]] * (d - 1)
        return [n] * d, [1] + ry + [1], [1] + rz + [1]
    r = np.random.RandomState(1000 * d + 10 * n + case["ry"])
    ns = [int(v) for v in r.randint((n + 1) // 2, n + 1, size=d)]
    ry = [int(v) for v in r.randint((case["ry"] + 1) // 2, case["ry"] + 1, size=d - 1)]
    rz = [int(v) for v in r.randint((case["rz"] + 1) // 2, case["rz"] + 1, size=d - 1)]
    return ns, [1] + ry + [1], [1] + rz + [1]


def _batch_shapes(case):
    r = np.random.RandomState(case["shapes"])
    out = []
    for _ in range(case["count"]):
        d = int(r.randint(case["dmin"], case["dmax"] + 1))
        ry = [1] + [int(v) for v in r.randint(case["rmin"], case["rmax"] + 1, size=d - 1)] + [1]
        rz = [1] + [int(v) for v in r.randint(case["rmin"], case["rmax"] + 1, size=d - 1)] + [1]
        out.append(([case["n"]] * d, ry, rz, 2 * max(max(ry), max(rz))))
    return out


def _sketch_ranks(n, r, s, want):
    """The clamped sketch ranks of a plan (no rank above what its unfolding or neighbours allow)."""
    d = len(n)
    ell = [1] * (d + 1)
    for k in range(1, d):
        ell[k] = min(want, r[k] * s[k], math.prod(n[:k]), math.prod(n[k:]))
    for k in range(1, d):
        ell[k] = min(ell[k], ell[k - 1] * n[k - 1])
    for k in range(d - 1, 0, -1):
        ell[k] = min(ell[k], n[k] * ell[k + 1])
    return ell


def _size(n, r):
    return sum(r[k] * n[k] * r[k + 1] for k in range(len(n)))


def _product_work(n, r, s, want, cap, truncated):
    ell = _sketch_ranks(n, r, s, want)
    hp, sw = costmodel.hatt1_flops(n, r, s, ell)
    out = [min(v, cap) for v in ell] if cap else ell
    flops = hp + sw + (costmodel.truncation_flops(n, ell) if truncated else 0.0)
    return 8.0 * (_size(n, r) + _size(n, s) + _size(n, out)), flops


def _dot_flops(n, a, b):
    return sum(2.0 * a[k] * b[k] * n[k] * b[k + 1] + 2.0 * a[k] * n[k] * a[k + 1] * b[k + 1] for k in range(len(n)))


def work(case):
    kind = case["kind"]
    if kind == "product":
        n, r, s = _shapes(case)
        trunc = case["tol"] > 0 or (case["max_rank"] > 0 and case["sketch"] > case["max_rank"])
        byt, flops = _product_work(n, r, s, case["sketch"], case["max_rank"], trunc)
    elif kind == "square":
        n = [case["n"]] * case["d"]
        r = [1] + [case["ry"]] * (case["d"] - 1) + [1]
        byt, flops = _product_work(n, r, r, case["max_rank"] + 10, case["max_rank"], True)
        byt -= 8.0 * _size(n, r)                     # both operands are the one tensor
    elif kind == "dot":
        n = [case["n"]] * case["d"]
        a = [1] + [case["ry"]] * (case["d"] - 1) + [1]
        b = [1] + [case["rz"]] * (case["d"] - 1) + [1]
        byt, flops = 8.0 * (_size(n, a) + _size(n, b) + 1), _dot_flops(n, a, b)
    elif kind == "power":
        n = [case["n"]] * case["d"]
        r = [1] + [case["ry"]] * (case["d"] - 1) + [1]
        x = [1] * (case["d"] + 1)
        byt = flops = 0.0
        for _ in range(case["iters"]):
            ell = _sketch_ranks(n, r, x, case["rank"])
            b, f = _product_work(n, r, x, case["rank"], 0, False)
            byt += b
            flops += f + _dot_flops(n, ell, x) + _dot_flops(n, ell, ell)
            x = ell
    elif kind == "round":
        d, r = case["d"], case["ry"]
        n = [case["n"]] * d
        w = [1] + [4 * r] * (d - 1) + [1]
        b = [1] * (d + 1)
        for k in range(d - 1):
            b[k + 1] = min(w[k + 1], b[k] * n[k])
        flops = costmodel.truncation_flops(n, b)
        for k in range(d - 1):
            rows = b[k] * n[k]
            flops += 4.0 * rows * b[k + 1] * w[k + 1] + 2.0 * b[k + 1] * w[k + 1] * n[k + 1] * w[k + 2]
        byt = 8.0 * (4 * _size(n, [1] + [r] * (d - 1) + [1]) + _size(n, [1] + [case["max_rank"]] * (d - 1) + [1]))
    else:
        byt = flops = 0.0
        for n, r, s, want in _batch_shapes(case):
            b, f = _product_work(n, r, s, want, 0, False)
            byt += b
            flops += f
    return {"bytes": byt, "flops": flops}


# ------------------------------------------------------------------ inputs ---

def _gaussian(n, r, gen):
    """Gaussian cores N(0, 1/(n r_right)) on the GPU: a tensor of unit expected norm."""
    return [torch.randn((r[k], n[k], r[k + 1]), dtype=torch.float64, device="cuda", generator=gen)
            / math.sqrt(n[k] * r[k + 1]) for k in range(len(n))]


def _generator(seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    return gen


def _options(case, seed):
    return dict(sketch_rank=case["sketch"], max_rank=case["max_rank"], tol=case["tol"], seed=seed % 100003,
                precision=PRECISION[case["precision"]], variant=case["variant"], ep=case["ep"])


def _inputs(case, seed):
    """The operands of a product, an inner product or a power iteration, and its sketch seed."""
    gen = _generator(seed)
    if case["kind"] == "product":
        n, r, s = _shapes(case)
        return _gaussian(n, r, gen), _gaussian(n, s, gen)
    n = [case["n"]] * case["d"]
    r = [1] + [case["ry"]] * (case["d"] - 1) + [1]
    if case["kind"] == "dot":
        s = [1] + [case["rz"]] * (case["d"] - 1) + [1]
        return _gaussian(n, r, gen), _gaussian(n, s, gen)
    return [torch.rand((r[k], n[k], r[k + 1]), dtype=torch.float64, device="cuda", generator=gen)
            for k in range(case["d"])]               # a nonnegative tensor


def prepare(case, seed):
    kind = case["kind"]
    if kind == "product":
        Y, Z = _inputs(case, seed)
        opts = _options(case, seed)
        state = {"case": case, "Y": Y, "Z": Z, "opts": opts}
        if case["form"] != "call":
            rec = binding.HadamardRecompressor(Y, Z, fixed_ranks=1, **opts)
            if case["form"] == "graph":
                rec.capture()
            state["rec"] = rec
        return state
    if kind == "square":
        n = [case["n"]] * case["d"]
        u = _gaussian(n, [1] + [case["ry"]] * (case["d"] - 1) + [1], _generator(seed))
        rec = binding.HadamardRecompressor(u, u, max_rank=case["max_rank"], tol=case["tol"], seed=seed % 100003,
                                           precision=PRECISION[case["precision"]], fixed_ranks=1)
        if case["form"] == "graph":
            rec.capture()
        return {"case": case, "u": u, "rec": rec}
    if kind == "dot":
        A, B = _inputs(case, seed)
        return {"case": case, "A": A, "B": B}
    if kind == "power":
        return {"case": case, "Y": _inputs(case, seed), "seed": seed % 100003}
    if kind == "round":
        gen = _generator(seed)
        n = [case["n"]] * case["d"]
        r = [1] + [case["ry"]] * (case["d"] - 1) + [1]
        terms = [_gaussian(n, r, gen) for _ in range(4)]
        coef = [1.0, 0.03, -0.02, 0.01]
        w = binding.tt_lincomb(terms, coef)
        rnd = binding.Rounder(w, max_rank=case["max_rank"], tol=case["tol"], fixed_ranks=1)
        return {"case": case, "terms": terms, "coef": coef, "w": w, "rnd": rnd}
    gen = _generator(seed)
    pairs = []
    for j, (n, r, s, want) in enumerate(_batch_shapes(case)):
        pairs.append((_gaussian(n, r, gen), _gaussian(n, s, gen),
                      dict(sketch_rank=want, max_rank=want, oversample=0, seed=(seed + j) % 100003,
                           precision=PRECISION[case["precision"]])))
    return {"case": case, "batch": binding.BatchedRecompressor(pairs)}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("product", "square"):
        if case["form"] == "call":
            return binding.tt_hadamard_recompress(state["Y"], state["Z"], **state["opts"])
        rec = state["rec"]
        if case["form"] == "graph":
            rec.replay()
        else:
            rec.run()
        return rec.result()
    if kind == "dot":
        return binding.tt_dot(state["A"], state["B"])
    if kind == "power":
        lams, X = power_iteration.largest_entry(state["Y"], iters=case["iters"], rank=case["rank"],
                                                seed=state["seed"])
        return [lams] + list(X)
    if kind == "round":
        binding.tt_lincomb(state["terms"], state["coef"], out=state["w"])
        state["rnd"].run()
        return state["rnd"].result()
    batch = state["batch"]
    batch.run()
    return [torch.cat([c.reshape(-1) for c in batch.result(j)]) for j in range(batch.count)]


# ------------------------------------------------------------------- exact ---

def _philox(counter, key0, key1):
    """Philox4x32-10 (Salmon et al., SC'11) on counters (count, 4), in numpy."""
    mask = np.uint64(0xFFFFFFFF)
    x = [counter[:, j].astype(np.uint64) for j in range(4)]
    k0, k1 = np.uint64(key0), np.uint64(key1)
    for rnd in range(10):
        if rnd:
            k0, k1 = (k0 + np.uint64(0x9E3779B9)) & mask, (k1 + np.uint64(0xBB67AE85)) & mask
        p0, p1 = np.uint64(0xD2511F53) * x[0], np.uint64(0xCD9E8D57) * x[2]
        x = [(p1 >> np.uint64(32)) ^ x[1] ^ k0, p1 & mask, (p0 >> np.uint64(32)) ^ x[3] ^ k1, p0 & mask]
    return x


def _sketch(seed, core, a, n, b):
    count = a * n * b
    ctr = np.zeros((count, 4), dtype=np.uint64)
    ctr[:, 0] = np.arange(count, dtype=np.uint64)
    ctr[:, 1] = core
    x = [(v >> np.uint64(6)).astype(np.float64) for v in _philox(ctr, seed & 0xFFFFFFFF, seed >> 32)]
    u1, u2 = (x[0] * 67108864.0 + x[1] + 0.5) * 2.0 ** -52, (x[2] * 67108864.0 + x[3] + 0.5) * 2.0 ** -52
    g = np.sqrt(-2.0 * np.log(u1)) * np.cos(2.0 * np.pi * u2)
    return (g / math.sqrt(count)).reshape(a, n, b)


def _recompress(Y, Z, want, seed):
    """The left-orthogonal recompression of Y * Z (HaTT-1, no truncation) in 64-bit numpy."""
    d = len(Y)
    n = [c.shape[1] for c in Y]
    r = [1] + [c.shape[2] for c in Y]
    s = [1] + [c.shape[2] for c in Z]
    ell = _sketch_ranks(n, r, s, want)
    W = [None] * d + [np.ones((1, 1))]
    for k in range(d - 1, 0, -1):
        R = _sketch(seed, k, ell[k], n[k], ell[k + 1])
        T = W[k + 1] @ R.transpose(1, 2, 0)                                   # (i, a'b', l)
        T = T.reshape(n[k], r[k + 1], s[k + 1], ell[k])
        T = Z[k].transpose(1, 0, 2)[:, None] @ T                              # (i, a', b, l)
        w = Y[k].reshape(r[k], -1) @ T.reshape(n[k] * r[k + 1], s[k] * ell[k])
        w = w.reshape(r[k] * s[k], ell[k])
        W[k] = w / np.linalg.norm(w)
    C = (Y[0][0][:, :, None] * Z[0][0][:, None, :]).reshape(n[0], -1)
    X = []
    for k in range(d - 1):
        Q, U = np.linalg.qr(C @ W[k + 1])
        Q = Q * np.where(np.diag(U) < 0, -1.0, 1.0)
        X.append(Q.reshape(ell[k], n[k], ell[k + 1]))
        M = (Q.T @ C).reshape(ell[k + 1] * r[k + 1], s[k + 1])
        U1 = (M @ Z[k + 1].reshape(s[k + 1], -1)).reshape(ell[k + 1], r[k + 1], n[k + 1], s[k + 2])
        C = Y[k + 1].transpose(1, 2, 0) @ U1.transpose(0, 2, 1, 3)            # (g, i, a', b')
        C = C.reshape(ell[k + 1] * n[k + 1], -1)
    X.append(C.reshape(ell[d - 1], n[d - 1], 1))
    return X


def _numpy(cores):
    return [c.cpu().numpy() for c in cores]


def exact(case, seed):
    kind = case["kind"]
    if kind == "dot":
        A, B = (_numpy(v) for v in _inputs(case, seed))
        G = np.ones((1, 1))
        for a, b in zip(A, B):
            T = (G @ b.reshape(b.shape[0], -1)).reshape(-1, b.shape[2])
            G = a.reshape(-1, a.shape[2]).T @ T
        return G.reshape(1)
    if kind == "product" and case["variant"] == 1 and case["precision"] in ("fp64", "fp64_tc") and \
            case["tol"] == 0 and not 0 < case["max_rank"] < case["sketch"]:
        Y, Z = (_numpy(v) for v in _inputs(case, seed))
        return _recompress(Y, Z, case["sketch"], seed % 100003)
    if kind == "batch" and case["precision"] == "fp64":
        gen = _generator(seed)
        out = []
        for j, (n, r, s, want) in enumerate(_batch_shapes(case)):
            Y, Z = _numpy(_gaussian(n, r, gen)), _numpy(_gaussian(n, s, gen))
            out.append(np.concatenate([c.reshape(-1) for c in _recompress(Y, Z, want, (seed + j) % 100003)]))
        return out
    return None
