"""Performance cases: the work that users of this library have it do, through its public entry points.

Every case is a dict of plain values; `kind` selects the entry point:

  perm   Plan(...)(x): one permutation of an array on the device
  grad   autograd.bmmc_permute and its backward on rows of a tensor
  parm   combinators.parm on rows of a tensor (a permutation, the user's function, the inverse permutation)
  batch  batch.Batch: many arrays of mixed sizes, each with its own matrix
  serve  serving.Server: a burst of requests, submitted as they come, waited for at the end
  sort   sorting.SortingNetwork: rows of keys

Matrices: `dense` (uniform invertible, any complement), `bp` (a random permutation of the index bits), `rev` (bit reversal),
`swap` (the two halves of the index bits exchanged, a matrix transpose). flags: 0 is the default strategy, 1 is BMMC_PLAN_SINGLE_PASS.
Everything moves or orders whole keys, so that every result is exact.
"""
import math
import random

import torch

import paper_2306_07795_gb300 as bm
from paper_2306_07795_gb300 import combinators, serving, sorting
from paper_2306_07795_gb300.autograd import bmmc_permute
from paper_2306_07795_gb300.batch import Batch

DEV = "cuda"
KEYS = {"int32": torch.int32, "float32": torch.float32, "int64": torch.int64, "float64": torch.float64}


def listed():
    return [
        # one small array, as a program with many little tables permutes them one by one: latency and launches
        {"name": "perm_n10_e4", "kind": "perm", "n": 10, "e": 4, "mat": "dense", "flags": 0},
        # the benchmark's 2^20-element int32 configuration: a general matrix on an array that stays in L2
        {"name": "perm_n20_e4", "kind": "perm", "n": 20, "e": 4, "mat": "dense", "flags": 0},
        # a permutation of index bits (a transpose of many axes) of 16-byte structures
        {"name": "perm_bp_n24_e16", "kind": "perm", "n": 24, "e": 16, "mat": "bp", "flags": 0},
        # bit reversal of 2^28 int32, the paper's own headline permutation
        {"name": "perm_rev_n28_e4", "kind": "perm", "n": 28, "e": 4, "mat": "rev", "flags": 0},
        # the largest array of the serving configuration, a general matrix on 8-byte elements
        {"name": "perm_n27_e8", "kind": "perm", "n": 27, "e": 8, "mat": "dense", "flags": 0},
        # the differentiable configuration: [64, 2^20] float32 along its last dimension, forward and backward
        {"name": "grad_64_n20", "kind": "grad", "rows": 64, "n": 20, "mat": "dense", "flags": 0},
        # parm on a tensor whose count of rows is no power of two
        {"name": "parm_24_n16", "kind": "parm", "rows": 24, "n": 16, "flags": 0},
        # many arrays of log-uniform sizes, as the batched configuration has them, in one Batch kept by the program
        {"name": "batch_1024", "kind": "batch", "count": 1024, "lo": 10, "hi": 20, "e": 4, "flags": 0},
        # a burst of requests of mixed sizes and element sizes, one in five a bit permutation, as the serving configuration draws them
        {"name": "serve_40", "kind": "serve", "count": 40, "lo": 12, "hi": 24, "flags": 0},
        # one large sort of float32 keys
        {"name": "sort_f32_n24", "kind": "sort", "rows": 1, "n": 24, "key": "float32"},
        # rows of float64 keys
        {"name": "sort_f64_16_n16", "kind": "sort", "rows": 16, "n": 16, "key": "float64"},
        # one short list of int32 keys
        {"name": "sort_i32_n11", "kind": "sort", "rows": 1, "n": 11, "key": "int32"},
    ]


def draw(rng):
    kind = rng.choice(["perm"] * 4 + ["grad", "parm", "batch", "serve"] + ["sort"] * 3)
    if kind == "perm":
        e = rng.choice([4, 8, 16])
        n = rng.randint(8, 28 - int(math.log2(e // 4)))
        return {"kind": kind, "n": n, "e": e, "mat": rng.choice(["dense", "dense", "bp", "rev", "swap"]), "flags": rng.choice([0, 0, 1])}
    if kind == "grad":
        n = rng.randint(10, 20)
        rows = _log_int(rng, 1, 40)
        return {"kind": kind, "rows": rows, "n": n, "mat": rng.choice(["dense", "bp"]), "flags": rng.choice([0, 1])}
    if kind == "parm":
        n = rng.randint(10, 20)
        return {"kind": kind, "rows": _log_int(rng, 1, min(40, 1 << (24 - n))), "n": n, "flags": rng.choice([0, 1])}
    if kind == "batch":
        lo = rng.randint(8, 14)
        return {"kind": kind, "count": _log_int(rng, 8, 1024), "lo": lo, "hi": rng.randint(lo, 20), "e": rng.choice([4, 8]), "flags": rng.choice([0, 0, 1])}
    if kind == "serve":
        return {"kind": kind, "count": rng.randint(5, 50), "lo": 12, "hi": rng.randint(14, 24), "flags": rng.choice([0, 0, 1])}
    key = rng.choice(sorted(KEYS))
    total = rng.randint(8, 24 if KEYS[key].itemsize == 4 else 21)
    b = rng.randint(0, min(6, total - 5))
    return {"kind": kind, "rows": 1 << b, "n": total - b, "key": key}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# -- matrices: row masks, bit j of rows[i] is a_ij ---------------------------------------------------------------------

def _invertible(rows):
    basis = {}
    for r in rows:
        while r:
            top = r.bit_length()
            if top not in basis:
                basis[top] = r
                break
            r ^= basis[top]
        if not r:
            return False
    return True


def _matrix(mat, n, r):
    """(rows, c) of the class `mat` on n bits."""
    if mat == "dense":
        while True:
            rows = [r.getrandbits(n) for _ in range(n)]
            if _invertible(rows):
                return rows, r.getrandbits(n)
    to = list(range(n))
    if mat == "bp":
        r.shuffle(to)
    elif mat == "rev":
        to.reverse()
    else:
        to = [(b + n // 2) % n for b in range(n)]
    rows = [0] * n
    for b, y in enumerate(to):
        rows[y] = 1 << b
    return rows, 0


def _words(n, e, g):
    """An array of 2^n elements of e bytes: random words, as 16-byte structures for e = 16."""
    if e == 8:
        return torch.randint(-2**62, 2**62, (1 << n,), dtype=torch.int64, device=DEV, generator=g)
    return torch.randint(-2**31, 2**31 - 1, (1 << n,) if e == 4 else (1 << n, 4), dtype=torch.int32, device=DEV, generator=g)


def _sizes(case):
    """(n, e) of each array of a batch and of each request of a burst: drawn for the case, the same for every seed."""
    r = random.Random("%(kind)s %(count)d %(lo)d %(hi)d" % case)
    return [(r.randint(case["lo"], case["hi"]), case.get("e") or r.choice([4, 8])) for _ in range(case["count"])]


def _requests(case, r):
    """(n, e, rows, c) of each request, in order of arrival."""
    return [(n, e, *_matrix("bp" if r.random() < 0.2 else "dense", n, r)) for n, e in _sizes(case)]


def _arrays(case, r):
    """(n, rows, c) of each array of a batch."""
    return [(n, *_matrix("dense", n, r)) for n, _ in _sizes(case)]


def _inputs(case, seed):
    """The matrices and input tensors of a case, the same for prepare and exact."""
    r = random.Random("%d %s" % (seed, sorted((k, v) for k, v in case.items() if k != "name")))
    g = torch.Generator(device=DEV).manual_seed(r.getrandbits(40))
    kind = case["kind"]
    if kind == "perm":
        return _matrix(case["mat"], case["n"], r), _words(case["n"], case["e"], g)
    if kind == "grad":
        shape = (case["rows"], 1 << case["n"])
        return _matrix(case["mat"], case["n"], r), [torch.randn(shape, device=DEV, generator=g) for _ in range(2)]
    if kind == "parm":
        return r.randrange(1, 1 << case["n"]), torch.randn((case["rows"], 1 << case["n"]), device=DEV, generator=g)
    if kind == "batch":
        arrays = _arrays(case, r)
        words = sum(case["e"] // 4 << n for n, _, _ in arrays)
        return arrays, torch.randint(-2**31, 2**31 - 1, (words,), dtype=torch.int32, device=DEV, generator=g)
    if kind == "serve":
        reqs = _requests(case, r)
        return reqs, [_words(n, e, g) for n, e, _, _ in reqs]
    shape, dtype = (case["rows"], 1 << case["n"]), KEYS[case["key"]]
    if dtype.is_floating_point:
        return None, torch.randn(shape, dtype=dtype, device=DEV, generator=g)
    half = 2**31 - 1 if dtype == torch.int32 else 2**62
    return None, torch.randint(-half, half, shape, dtype=dtype, device=DEV, generator=g)


def _parts(case, arrays, flat):
    """The arrays of a batch as slices of one buffer."""
    w, at, out = case["e"] // 4, 0, []
    for n, _, _ in arrays:
        out.append(flat[at:at + (w << n)])
        at += w << n
    return out


# -- the program ------------------------------------------------------------------------------------------------------

def _reverse_each(z):
    """parm's function: each of the two sub-arrays in reverse order."""
    return z.flip(-1)


class _Raw:
    """A kept output as an array that torch can view; it keeps the server, whose arena holds it, alive."""

    def __init__(self, server, ptr, n, e):
        self.server = server
        self.__cuda_array_interface__ = {"shape": (1 << n,), "typestr": "<i%d" % e, "data": (ptr, False), "version": 3}


def prepare(case, seed):
    kind = case["kind"]
    m, x = _inputs(case, seed)
    if kind == "perm":
        return {"kind": kind, "plan": bm.Plan(case["n"], *m, elem_bytes=case["e"], flags=case["flags"]), "x": x}
    if kind == "grad":
        return {"kind": kind, "plan": bm.Plan(case["n"], *m, flags=case["flags"]), "x": x[0].requires_grad_(), "w": x[1]}
    if kind == "parm":
        return {"kind": kind, "mask": m, "x": x, "flags": case["flags"]}
    if kind == "batch":
        plans = [bm.Plan(n, rows, c, elem_bytes=case["e"], flags=case["flags"]) for n, rows, c in m]
        out = torch.empty_like(x)
        return {"kind": kind, "batch": Batch(plans, _parts(case, m, x), _parts(case, m, out)), "out": out}
    if kind == "serve":
        room = 4 * sum(e << n for n, e, _, _ in m) + (64 << 20)
        return {"kind": kind, "server": serving.Server(DEV, budget_bytes=room, flags=case["flags"], keep_outputs=True),
                "reqs": [serving.Request(i, 0.0, n, e, rows, c, t) for i, ((n, e, rows, c), t) in enumerate(zip(m, x))], "kept": []}
    return {"kind": kind, "net": sorting.SortingNetwork(case["n"]), "x": x}


def run(state):
    kind = state["kind"]
    if kind == "perm":
        return state["plan"](state["x"])
    if kind == "grad":
        y = bmmc_permute(state["x"], state["plan"])
        return y.detach(), torch.autograd.grad(y, state["x"], state["w"])[0]
    if kind == "parm":
        return combinators.parm(state["mask"], _reverse_each, state["x"], flags=state["flags"])
    if kind == "batch":
        state["batch"]()
        return state["out"]
    if kind == "serve":
        srv = state["server"]
        for ptr in state["kept"]:
            srv.release(ptr)
        for q in state["reqs"]:
            code = srv.submit(q.rid, q.n, q.rows_c, q.c, q.e, q.x)
            if code != bm.BMMC_OK:
                raise bm.BmmcError(code, "submit")
        srv.drain()
        done = sorted(srv.results())
        state["kept"] = [out for _, _, _, _, out in done]
        bad = [status for _, status, _, _, _ in done if status != bm.BMMC_OK]
        if bad or len(done) != len(state["reqs"]):
            raise bm.BmmcError(bad[0] if bad else bm.BMMC_ERR_CUDA, "serve")
        return [torch.as_tensor(_Raw(srv, ptr, q.n, q.e), device=DEV) for ptr, q in zip(state["kept"], state["reqs"])]
    return state["net"](state["x"])


# -- what a pass cannot do without -------------------------------------------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind == "perm":
        return {"bytes": 2 * case["e"] << case["n"], "flops": 0}
    if kind == "grad":  # x to y, and w to the gradient
        return {"bytes": 4 * 4 * case["rows"] << case["n"], "flops": 0}
    if kind == "parm":  # the sub-arrays are materialised for the user's function, which reads and writes them once
        return {"bytes": 6 * 4 * case["rows"] << case["n"], "flops": 0}
    if kind in ("batch", "serve"):
        return {"bytes": sum(2 * e << n for n, e in _sizes(case)), "flops": 0}
    # one operation for each comparator of the network
    keys = case["rows"] << case["n"]
    return {"bytes": 2 * keys * KEYS[case["key"]].itemsize, "flops": keys * case["n"] * (case["n"] + 1) / 4}


def tolerance(case):
    return "exact"


# -- the same results in plain torch -----------------------------------------------------------------------------------

def _places(n, rows, c):
    """A x + c for every x of n bits."""
    x = torch.arange(1 << n, device=DEV)
    y = torch.full_like(x, c)
    for j in range(n):
        col = sum(((rows[i] >> j) & 1) << i for i in range(n))
        y ^= ((x >> j) & 1) * col
    return y


def _scatter(x, places):
    """out[..., places[i]] = x[..., i] along dimension `places` indexes."""
    out = torch.empty_like(x)
    out[places] = x
    return out


def exact(case, seed):
    kind = case["kind"]
    m, x = _inputs(case, seed)
    if kind == "perm":
        return _scatter(x, _places(case["n"], *m))
    if kind == "grad":
        at = _places(case["n"], *m)
        y = torch.empty_like(x[0])
        y[:, at] = x[0]
        return y, x[1][:, at]
    if kind == "parm":
        i = torch.arange(1 << case["n"], device=DEV)
        side = torch.zeros_like(i)
        for b in range(case["n"]):
            if (m >> b) & 1:
                side ^= (i >> b) & 1
        out = torch.empty_like(x)
        for s in (0, 1):
            at = i[side == s]
            out[:, at] = x[:, at].flip(-1)
        return out
    if kind == "batch":
        out = torch.empty_like(x)
        for (n, rows, c), a, b in zip(m, _parts(case, m, x), _parts(case, m, out)):
            b.view(1 << n, -1)[_places(n, rows, c)] = a.view(1 << n, -1)
        return out
    if kind == "serve":
        return [_scatter(t, _places(n, rows, c)) for (n, e, rows, c), t in zip(m, x)]
    return torch.sort(x, dim=-1).values
