"""Performance cases: inversions as a program that uses this package calls them.

Orders, families and mixes are those of the repository's workloads: the plain
FP64 method on one matrix, the mixed form with refinement on one matrix,
batches of uneven orders, a burst of served requests, and the FP64-class
product of callers who compose the recursion by themselves.

Families:
  sdd  a_ij ~ U(-1, 1), n added to the diagonal (strictly diagonally dominant);
  spd  G G^T / n + alpha I, g_ij ~ N(0, 1), alpha ~ U(0.1, 1).
"""
import math

import numpy as np
import torch

import paper_1801_04723_gb300 as spin

DEVICE = "cuda:0"


def listed():
    return [
        # one small request, the smallest order of the serving mix: a single leaf, latency only
        {"name": "plain_64", "kind": "invert", "precision": "fp64", "family": "spd", "n": 64, "leaf": 0},
        # an order that is no multiple of anything, ragged at every level
        {"name": "plain_777", "kind": "invert", "precision": "fp64", "family": "spd", "n": 777, "leaf": 0},
        # the plain method's first workload: order 1024, leaf 128
        {"name": "plain_1024", "kind": "invert", "precision": "fp64", "family": "sdd", "n": 1024, "leaf": 128},
        # an ordinary plain inversion of a few thousand rows, ragged
        {"name": "plain_3000", "kind": "invert", "precision": "fp64", "family": "spd", "n": 3000, "leaf": 0},
        # the largest order the server takes and the leaf sweep's order, plain
        {"name": "plain_8192", "kind": "invert", "precision": "fp64", "family": "spd", "n": 8192, "leaf": 0},
        # mixed precision with refinement: a small ragged request
        {"name": "mixed_1000", "kind": "invert", "precision": "bf16x3", "family": "spd", "n": 1000, "leaf": 0},
        # mixed precision at an ordinary serving order
        {"name": "mixed_4096", "kind": "invert", "precision": "bf16x3", "family": "spd", "n": 4096, "leaf": 0},
        # mixed precision on a large matrix, as at n = 32768, which takes too long for a repeated case
        {"name": "mixed_16384", "kind": "invert", "precision": "bf16x3", "family": "spd", "n": 16384, "leaf": 0},
        # many small matrices of uneven order in one call: the batching workload's mix, plain and mixed
        {"name": "batch_fp64", "kind": "batch", "precision": "fp64", "count": 256, "lo": 32, "hi": 1024},
        {"name": "batch_mixed", "kind": "batch", "precision": "bf16x3", "count": 256, "lo": 32, "hi": 1024},
        # a burst of requests at the server, half plain and half mixed, collected as they finish
        {"name": "serve_burst", "kind": "serve", "count": 48, "lo": 64, "hi": 2048},
        # an FP64-class product by itself, the Schur complement C - A B of callers that compose the recursion
        {"name": "schur_2048", "kind": "schur", "n": 2048, "slices": 7},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plain", "plain", "mixed", "mixed", "batch", "serve", "schur"])
    if kind == "plain":
        return {"kind": "invert", "precision": "fp64", "family": rng.choice(["sdd", "spd"]),
                "n": _log_int(rng, 64, 8192), "leaf": rng.choice([0, 0, 64, 128, 256])}
    if kind == "mixed":
        return {"kind": "invert", "precision": "bf16x3", "family": "spd", "n": _log_int(rng, 64, 16384),
                "leaf": rng.choice([0, 0, 64, 128])}
    if kind == "batch":
        return {"kind": "batch", "precision": rng.choice(["fp64", "bf16x3"]), "count": _log_int(rng, 16, 256),
                "lo": 32, "hi": rng.choice([256, 512, 1024])}
    if kind == "serve":
        return {"kind": "serve", "count": rng.randint(8, 48), "lo": 64, "hi": _log_int(rng, 512, 2048)}
    return {"kind": "schur", "n": _log_int(rng, 256, 4096), "slices": rng.choice([5, 6, 7])}


def _generator(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)
    return g


def _sdd(n, g):
    A = torch.rand((n, n), generator=g, dtype=torch.float64, device=DEVICE).mul_(2.0).sub_(1.0)
    A.diagonal().add_(float(n))
    return A


def _spd(n, g):
    alpha = 0.1 + 0.9 * float(torch.rand((), generator=g, dtype=torch.float64, device=DEVICE))
    G = torch.randn((n, n), generator=g, dtype=torch.float32, device=DEVICE)
    A = (G @ G.T).double().div_(float(n))
    del G
    A = (A + A.T).mul_(0.5)
    A.diagonal().add_(alpha)
    return A.contiguous()


def _orders(case, seed):
    """Orders log-uniform in [lo, hi]: multiples of 32 in a batch, any integer in a burst.  The mix is the
    case's own (as the workload's trace is), the matrices are the seed's."""
    rng = np.random.default_rng(1801 + 7 * case["count"] + case["hi"])
    x = np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]), case["count"]))
    if case["kind"] == "batch":
        return [int(v) for v in np.clip(np.rint(x / 32).astype(int) * 32, case["lo"], case["hi"])]
    return [int(v) for v in np.rint(x).astype(int)]


def _matrices(case, seed):
    g = _generator(seed)
    if case["kind"] == "batch":
        return [_sdd(n, g) for n in _orders(case, seed)]
    return [_spd(n, g) for n in _orders(case, seed)]


def _flat_outputs(orders):
    """One buffer for all results, and each result's view of it (every one 256-byte aligned)."""
    starts, total = [], 0
    for n in orders:
        starts.append(total)
        total += -(-n * n // 32) * 32
    flat = torch.zeros(total, dtype=torch.float64, device=DEVICE)
    return flat, [flat[s:s + n * n].view(n, n) for s, n in zip(starts, orders)]


def _schur_operands(case, seed):
    """C - A B as at the top level of a recursion: off-diagonal blocks of an spd matrix, and its trailing block."""
    n = case["n"]
    g = _generator(seed)
    A = torch.randn((n, n), generator=g, dtype=torch.float64, device=DEVICE).div_(math.sqrt(2.0 * n))
    B = torch.randn((n, n), generator=g, dtype=torch.float64, device=DEVICE).div_(math.sqrt(2.0 * n))
    return A, B, _spd(n, g)


def prepare(case, seed):
    kind = case["kind"]
    state = {"case": case}
    if kind == "invert":
        g = _generator(seed)
        state["A"] = (_sdd if case["family"] == "sdd" else _spd)(case["n"], g)
        state["X"] = torch.empty_like(state["A"])
    elif kind == "batch":
        state["A"] = _matrices(case, seed)
        state["flat"], state["X"] = _flat_outputs(_orders(case, seed))
    elif kind == "serve":
        state["A"] = _matrices(case, seed)
        state["flat"], state["X"] = _flat_outputs(_orders(case, seed))
        state["server"] = spin.Server(hbm_budget_bytes=32 << 30, max_slots=8, priority_order=1024)
        torch.cuda.synchronize()  # the server's streams read A
    else:
        state["A"], state["B"], state["C"] = _schur_operands(case, seed)
        state["D"] = torch.empty_like(state["C"])
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "invert":
        X, _ = spin.invert(state["A"], out=state["X"], leaf=case["leaf"], precision=case["precision"])
        return X
    if kind == "batch":
        _, status = spin.invert_batched(state["A"], outs=state["X"], precision=case["precision"])
        return [state["flat"], status]
    if kind == "serve":
        server, mats, outs = state["server"], state["A"], state["X"]
        waiting = []
        for i, a in enumerate(mats):
            precision, tol = (("fp64", 1e-13), ("bf16x3", 1e-10))[i % 2]
            waiting.append((server.submit(a, precision=precision, tol=tol), i))
        status = [0] * len(mats)
        while waiting:
            left = []
            for ticket, i in waiting:
                got = server.poll(ticket, out=outs[i])
                if got is None:
                    left.append((ticket, i))
                else:
                    status[i] = got[1]["status"]
            waiting = left
        return [state["flat"], np.array(status, dtype=np.int64)]
    return spin.gemm_ozaki(state["A"], state["B"], slices=case["slices"], alpha=-1.0, beta=1.0, C=state["C"],
                           out=state["D"])


def work(case):
    """The method's 2 n^3 operations per inversion (and per product), operands read once, results written once."""
    if case["kind"] in ("invert", "schur"):
        orders, passes = [case["n"]], 2 if case["kind"] == "invert" else 4
    else:
        orders, passes = _orders(case, 0), 2
    return {"bytes": float(sum(8 * passes * n * n for n in orders)), "flops": float(sum(2 * n ** 3 for n in orders))}


def exact(case, seed):
    kind = case["kind"]
    if kind == "invert":
        g = _generator(seed)
        return torch.linalg.inv((_sdd if case["family"] == "sdd" else _spd)(case["n"], g))
    if kind in ("batch", "serve"):
        flat, views = _flat_outputs(_orders(case, seed))
        for v, a in zip(views, _matrices(case, seed)):
            v.copy_(torch.linalg.inv(a))
        return [flat, None]
    A, B, C = _schur_operands(case, seed)
    return C - A @ B
