"""The workloads this library is timed on: what a program that uses it calls, over the sizes it meets.

Every case is one call sequence through the public Python entry points
(:mod:`paper_2606_20855_gb300.spgemm`): a sparse product C = A*B, row-wise or
as an outer product, an elementwise operation C = A + B or C = A .* B, or a
sparse matrix - sparse vector product y = A x.  Inputs are drawn on the GPU
from a seed; the 64-bit results they are compared with are plain torch
(products expanded, keys sorted, equal keys summed).

Fields of a case:
  op       "spgemm", "outer" (with parts), "ewise" (with how: "add" or "mul"), "spmspv" (with density)
  input    "uniform"   A is m x k with ra entries in every row, B is k x n with rb (columns uniform)
           "ragged"    the same with row lengths uniform in 0..2*ra and 0..2*rb
           "stencil"   A = B is the 5-point stencil of a g x h grid with varying coefficients
           "rmat"      A = B is an R-MAT graph on n vertices, ef edges drawn per vertex
           "rmat_x"    A is such a graph, B is n x n with rb entries in every row
           "rmat_perm" elementwise: B is the graph A with its vertices relabelled at random
           "rmat_same" elementwise: B has A's pattern and other values
  dtype    "f32" or "f64", the value type
  plan     True: the operation's object (handles, row plan, scratch) is kept between calls, as a program
           that multiplies again and again keeps it; False: the one-shot function
  validate one-shot product: check the inputs' CSR invariants on the device first
"""
from __future__ import annotations

import functools
import math

import torch

from paper_2606_20855_gb300.spgemm import DeviceCSR, Ewise, SpGEMM, SpGEMMOuter, SpMSpV, ewise, spgemm, spgemm_outer, spmspv

_DT = {"f32": torch.float32, "f64": torch.float64}
_RMAT = (0.57, 0.19, 0.19, 0.05)
_BLOCK = 1 << 25  # products expanded at once by the 64-bit reference


def listed():
    return [
        # the smallest call: two small matrices multiplied once, inputs checked (a unit test, a script, a coarse level)
        {"name": "small_checked", "op": "spgemm", "input": "uniform", "m": 300, "k": 500, "n": 400, "ra": 7, "rb": 9,
         "dtype": "f64", "plan": False, "validate": True},
        # a small product repeated with a kept plan: launches and read-backs count
        {"name": "uniform_2k", "op": "spgemm", "input": "uniform", "m": 2048, "k": 2048, "n": 2048, "ra": 8, "rb": 8,
         "dtype": "f64", "plan": True, "validate": False},
        # a discretised operator squared (multigrid setup): short rows, narrow column ranges
        {"name": "stencil_512", "op": "spgemm", "input": "stencil", "g": 512, "h": 512, "dtype": "f64", "plan": True,
         "validate": False},
        # rows of any length, odd sizes, more columns than 65,536, single precision
        {"name": "ragged_200k", "op": "spgemm", "input": "ragged", "m": 100003, "k": 30011, "n": 200003, "ra": 12,
         "rb": 20, "dtype": "f32", "plan": True, "validate": False},
        # two-hop neighbourhoods of a middle-sized graph, called once
        {"name": "rmat_16k_once", "op": "spgemm", "input": "rmat", "n": 16384, "ef": 8, "dtype": "f32", "plan": False,
         "validate": False},
        # a power-law graph squared: hub rows, 400 million products
        {"name": "rmat_64k", "op": "spgemm", "input": "rmat", "n": 65536, "ef": 16, "dtype": "f64", "plan": True,
         "validate": False},
        # the uniform product of the throughput benchmark: 537 million products, 4.3 GB of output
        {"name": "uniform_rect_1m", "op": "spgemm", "input": "uniform", "m": 1 << 20, "k": 1 << 16, "n": 1 << 16,
         "ra": 16, "rb": 32, "dtype": "f32", "plan": True, "validate": False},
        # a large power-law graph times a uniform sparse matrix: rows of every size over a million columns
        {"name": "rmat_1m_x_uniform", "op": "spgemm", "input": "rmat_x", "n": 1 << 20, "ef": 8, "rb": 4, "dtype": "f64",
         "plan": True, "validate": False},
        # two large graphs added
        {"name": "add_rmat_1m", "op": "ewise", "how": "add", "input": "rmat_perm", "n": 1 << 20, "ef": 8,
         "dtype": "f64", "plan": True, "validate": False},
        # a middle-sized graph weighted by another one on the same edges, called once
        {"name": "mul_rmat_200k_once", "op": "ewise", "how": "mul", "input": "rmat_same", "n": 200003, "ef": 8,
         "dtype": "f32", "plan": False, "validate": False},
        # one step of a graph traversal with a tenth of the vertices active
        {"name": "spmspv_rmat_1m", "op": "spmspv", "input": "rmat", "n": 1 << 20, "ef": 16, "density": 0.1,
         "dtype": "f64", "plan": True, "validate": False},
        # the k-parallel product: four partial products, merged by additions
        {"name": "outer_64k", "op": "outer", "parts": 4, "input": "uniform", "m": 65539, "k": 16384, "n": 16411,
         "ra": 16, "rb": 32, "dtype": "f64", "plan": True, "validate": False},
    ]


def _log(rng, lo, hi):
    """A whole number between lo and hi, uniform in its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    case = {"dtype": rng.choice(["f32", "f64"]), "plan": rng.random() < 0.6, "validate": False}
    kind = rng.choice(["uniform", "uniform", "ragged", "stencil", "rmat", "rmat_x", "ewise", "ewise", "spmspv", "outer"])
    if kind in ("uniform", "ragged", "outer"):
        ra, rb = _log(rng, 2, 40), _log(rng, 2, 48)
        n, k = _log(rng, 3000, 1 << 20), _log(rng, 3000, 1 << 18)
        most = (20_000_000 if kind == "outer" else 80_000_000) // (ra * rb)
        m = min(_log(rng, 200, 1 << 20), most)
        case.update(op="spgemm", input="uniform" if kind == "outer" else kind, m=m, k=k, n=n, ra=ra, rb=rb)
        if kind == "outer":
            case.update(op="outer", parts=rng.randint(2, 6))
    elif kind == "stencil":
        case.update(op="spgemm", input="stencil", g=_log(rng, 20, 900), h=_log(rng, 20, 900))
    elif kind == "rmat":
        case.update(op="spgemm", input="rmat", n=_log(rng, 1000, 50_000), ef=rng.randint(3, 16))
    elif kind == "rmat_x":
        case.update(op="spgemm", input="rmat_x", n=_log(rng, 4000, 1 << 20), ef=rng.randint(3, 8), rb=rng.randint(2, 6))
    elif kind == "ewise":
        case.update(op="ewise", how=rng.choice(["add", "mul"]), input=rng.choice(["rmat_perm", "rmat_same"]),
                    n=_log(rng, 1000, 1 << 20), ef=rng.randint(3, 16))
    else:
        case.update(op="spmspv", input="rmat", n=_log(rng, 1000, 1 << 20), ef=rng.randint(3, 16),
                    density=round(math.exp(rng.uniform(math.log(0.001), math.log(0.5))), 5))
    if case["op"] == "spgemm" and not case["plan"]:
        case["validate"] = rng.random() < 0.3
    return case


# ------------------------------------------------------------------ inputs
#
# The pattern of a case is drawn once (generator seed 0) and its rows, inner
# indices and columns are relabelled by permutations of the given seed, so that
# every seed gives other matrices with as many stored entries in operands and
# result.  Uniform patterns are relabelled over their whole range; graphs
# within blocks of 16 neighbouring vertices, which keeps their hubs together
# as R-MAT places them; a stencil keeps its grid numbering.  Values are drawn
# from the given seed.


def _gen(seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return gen


def _values(count, dt, gen, low, high):
    return torch.rand(count, generator=gen, device="cuda", dtype=dt) * (high - low) + low


def _csr(m, n, key, vals):
    """CSR of the sorted distinct keys row * n + column."""
    rows = torch.div(key, n, rounding_mode="floor")
    rowptr = torch.searchsorted(rows, torch.arange(m + 1, device=key.device))
    return DeviceCSR(m, n, rowptr, (key - rows * n).to(torch.int32), vals)


def _keys(M):
    rows = torch.repeat_interleave(torch.arange(M.nrows, device="cuda"), M.rowptr[1:] - M.rowptr[:-1])
    return rows * M.ncols + M.colidx


def _uniform(m, n, r, gen):
    """Keys of r distinct columns in every row, every choice equally likely."""
    cols = torch.randint(0, n, (m, r), generator=gen, device="cuda", dtype=torch.int32).sort(1).values
    while True:
        bad = (cols[:, 1:] == cols[:, :-1]).any(1).nonzero().flatten()
        if bad.numel() == 0:
            break
        cols[bad] = torch.randint(0, n, (bad.numel(), r), generator=gen, device="cuda", dtype=torch.int32).sort(1).values
    return (torch.arange(m, device="cuda")[:, None] * n + cols).flatten()


def _ragged(m, n, r, gen):
    """Keys of rows of 0..2r entries (columns drawn twice in a row are merged)."""
    lens = torch.randint(0, 2 * r + 1, (m,), generator=gen, device="cuda")
    rows = torch.repeat_interleave(torch.arange(m, device="cuda"), lens)
    return torch.unique(rows * n + torch.randint(0, n, rows.shape, generator=gen, device="cuda"))


def _rmat(n, ef, gen):
    """Keys of R-MAT edges among n vertices (quadrants picked level by level, repeated edges merged)."""
    scale, ne = max(1, (n - 1).bit_length()), ef * n
    rows = torch.zeros(ne, dtype=torch.int64, device="cuda")
    cols = torch.zeros(ne, dtype=torch.int64, device="cuda")
    a, b, c, _ = _RMAT
    for level in range(scale):
        u = torch.rand(ne, generator=gen, device="cuda")
        rows |= (u >= a + b).to(torch.int64) << (scale - 1 - level)
        cols |= (((u >= a) & (u < a + b)) | (u >= a + b + c)).to(torch.int64) << (scale - 1 - level)
    return torch.unique((rows * n + cols)[(rows < n) & (cols < n)])


def _stencil(g, h):
    """Keys of the 5-point stencil of a g x h grid."""
    v = torch.arange(g * h, device="cuda")
    r, c = v // h, v % h
    return torch.cat([(v * (g * h) + v + off)[ok] for off, ok in
                      ((-h, r > 0), (-1, c > 0), (0, c >= 0), (1, c < h - 1), (h, r < g - 1))]).sort().values


def _shuffle(n, block, gen):
    """A permutation of 0..n-1 that moves indices only within blocks of `block` neighbours."""
    at = torch.arange(n, device="cuda")
    place = torch.rand(n, generator=gen, device="cuda", dtype=torch.float64) + torch.div(at, block, rounding_mode="floor")
    return torch.argsort(place)


def _relabelled(key, n, rows, cols):
    return (rows[torch.div(key, n, rounding_mode="floor")] * n + cols[key % n]).sort().values


def _inputs(case, seed):
    """(A, B), for "spmspv" (A by columns, x's indices, x's values)."""
    base, gen = _gen(0), _gen(seed + 1)
    dt, kind = _DT[case["dtype"]], case["input"]
    if kind in ("uniform", "ragged"):
        make, (m, k, n) = _uniform if kind == "uniform" else _ragged, (case["m"], case["k"], case["n"])
        rows, inner, cols = (_shuffle(size, size, gen) for size in (m, k, n))
        ka = _relabelled(make(m, k, case["ra"], base), k, rows, inner)
        kb = _relabelled(make(k, n, case["rb"], base), n, inner, cols)
        return (_csr(m, k, ka, _values(ka.numel(), dt, gen, -1, 1)), _csr(k, n, kb, _values(kb.numel(), dt, gen, -1, 1)))
    if kind == "stencil":  # 4 on the diagonal, -(0.5 .. 1.5) for each neighbour
        n = case["g"] * case["h"]
        key = _stencil(case["g"], case["h"])
        vals = _values(key.numel(), dt, gen, -1.5, -0.5)
        vals[key % n == torch.div(key, n, rounding_mode="floor")] = 4.0
        A = _csr(n, n, key, vals)
        return A, A
    n = case["n"]
    key = _rmat(n, case["ef"], base)
    p, q = _shuffle(n, 16, gen), _shuffle(n, 16, gen)
    if kind == "rmat_perm":
        other = torch.randperm(n, generator=base, device="cuda")
        kb = _relabelled(_relabelled(key, n, other, other), n, p, q)
    ka = _relabelled(key, n, p, p if case["op"] in ("spgemm", "outer") else q)
    A = _csr(n, n, ka, _values(ka.numel(), dt, gen, 1, 0))
    if case["op"] == "spmspv":
        count = max(1, int(round(case["density"] * n)))
        idx = p[torch.randperm(n, generator=base, device="cuda")[:count]].sort().values.to(torch.int32)
        return A, idx, _values(count, dt, gen, 1, 0)
    if kind == "rmat":
        return A, A
    if kind == "rmat_x":
        kb = _relabelled(_uniform(n, n, case["rb"], base), n, p, _shuffle(n, n, gen))
    elif kind == "rmat_same":
        kb = ka.clone()
    return A, _csr(n, n, kb, _values(kb.numel(), dt, gen, 1, 0))


def prepare(case, seed):
    ops, state = _inputs(case, seed), {"case": case}
    if case["op"] == "spmspv":
        state.update(At=ops[0], x=ops[1:], plan=SpMSpV(ops[0]) if case["plan"] else None)
        return state
    state.update(A=ops[0], B=ops[1], plan=None)
    if case["plan"]:
        if case["op"] == "spgemm":
            state["plan"] = SpGEMM(*ops)
        elif case["op"] == "outer":
            state["plan"] = SpGEMMOuter(*ops, parts=case["parts"])
        else:
            state["plan"] = Ewise(*ops, op=case["how"])
    return state


def run(state):
    case, plan = state["case"], state["plan"]
    if case["op"] == "spmspv":
        return plan(*state["x"]) if plan is not None else spmspv(state["At"], *state["x"])
    if plan is not None:
        plan.symbolic()
        C = plan.numeric()
        plan.wait()
    elif case["op"] == "spgemm":
        C = spgemm(state["A"], state["B"], validate=case["validate"])
    elif case["op"] == "outer":
        C = spgemm_outer(state["A"], state["B"], case["parts"])
    else:
        C = ewise(state["A"], state["B"], op=case["how"])
    return C.rowptr, C.colidx, C.vals


# ------------------------------------------------- the same results in 64 bits


def _blocks(A, B):
    """Row ranges of A with about _BLOCK products each, and the products before every entry of A."""
    lens = B.rowptr[1:] - B.rowptr[:-1]
    ub = torch.zeros(A.nnz + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens[A.colidx.long()], 0, out=ub[1:])
    row_end = ub[A.rowptr[1:]]
    total = int(ub[-1])
    cuts = torch.searchsorted(row_end, torch.arange(_BLOCK, total + _BLOCK, _BLOCK, device="cuda"))
    cuts = sorted({0, A.nrows, *(min(A.nrows, int(c) + 1) for c in cuts)})
    return list(zip(cuts[:-1], cuts[1:])), ub


def _expand(A, B, r0, r1, ub):
    """Keys row * ncols + column and 64-bit values of all products of A's rows r0..r1."""
    e0, e1 = int(A.rowptr[r0]), int(A.rowptr[r1])
    count = ub[e0 + 1:e1 + 1] - ub[e0:e1]
    entry = torch.repeat_interleave(torch.arange(e0, e1, device="cuda"), count)
    at = torch.arange(entry.numel(), device="cuda") - (ub[entry] - ub[e0]) + B.rowptr[A.colidx[entry].long()]
    row = torch.repeat_interleave(torch.arange(r0, r1, device="cuda"), A.rowptr[r0 + 1:r1 + 1] - A.rowptr[r0:r1])
    return row[entry - e0] * B.ncols + B.colidx[at], A.vals[entry].double() * B.vals[at].double()


def _summed(key, val):
    key, inverse = torch.unique(key, return_inverse=True)
    return key, torch.zeros(key.numel(), dtype=torch.float64, device="cuda").index_add_(0, inverse, val)


def exact(case, seed):
    ops = _inputs(case, seed)
    if case["op"] == "spmspv":
        At, idx, xv = ops
        X = DeviceCSR(1, At.nrows, torch.tensor([0, idx.numel()], device="cuda"), idx, xv)
        ranges, ub = _blocks(X, At)
        key, val = _summed(*_expand(X, At, 0, 1, ub))
        return key.to(torch.int32), val
    A, B = ops
    if case["op"] == "ewise":
        ka, kb = _keys(A), _keys(B)
        if case["how"] == "add":
            key, val = _summed(torch.cat([ka, kb]), torch.cat([A.vals.double(), B.vals.double()]))
        else:
            both = torch.isin(ka, kb, assume_unique=True)
            key = ka[both]
            val = A.vals[both].double() * B.vals[torch.searchsorted(kb, key)].double()
        C = _csr(A.nrows, A.ncols, key, val)
        return C.rowptr, C.colidx, C.vals
    keys, vals = [], []
    ranges, ub = _blocks(A, B)
    for r0, r1 in ranges:
        key, val = _summed(*_expand(A, B, r0, r1, ub))
        keys.append(key)
        vals.append(val)
    C = _csr(A.nrows, B.ncols, torch.cat(keys), torch.cat(vals))
    return C.rowptr, C.colidx, C.vals


# ------------------------------------------------------------- what a pass needs


@functools.lru_cache(maxsize=None)
def _counts(items):
    """(stored entries of the operands, of the result, products or merged entries) of the inputs of seed 0."""
    case = dict(items)
    ops = _inputs(case, 0)
    if case["op"] == "spmspv":
        At, idx, _ = ops
        key = At.colidx[_spans(At.rowptr[idx.long()], At.rowptr[idx.long() + 1])]
        return idx.numel(), int(torch.unique(key).numel()), int(key.numel())
    A, B = ops
    if case["op"] == "ewise":
        union = int(torch.unique(torch.cat([_keys(A), _keys(B)])).numel())
        return A.nnz + B.nnz, union if case["how"] == "add" else A.nnz + B.nnz - union, A.nnz + B.nnz
    ranges, ub = _blocks(A, B)
    out = 0
    for r0, r1 in ranges:
        out += int(torch.unique(_expand(A, B, r0, r1, ub)[0]).numel())
    return A.nnz + (B.nnz if B is not A else 0), out, int(ub[-1])


def _spans(begin, end):
    """All positions of the ranges begin[i]..end[i]."""
    lens = end - begin
    first = torch.cumsum(lens, 0) - lens
    return torch.repeat_interleave(begin - first, lens) + torch.arange(int(lens.sum()), device="cuda")


def work(case):
    """Operands read once (row pointers, columns, values), the result written once."""
    entry = 4 + (4 if case["dtype"] == "f32" else 8)
    read, out, products = _counts(tuple(sorted((k, v) for k, v in case.items() if k != "name")))
    if case["op"] == "spmspv":  # x, the selected columns' bounds and entries, y
        return {"bytes": entry * (read + products + out) + 16 * read, "flops": 2 * products}
    if "m" in case:
        rows = case["m"] + 1 + case["k"] + 1
        m = case["m"]
    else:
        m = case["n"] if "n" in case else case["g"] * case["h"]
        rows = (m + 1) * (1 if case["input"] in ("stencil", "rmat") else 2)
    flops = 2 * products if case["op"] in ("spgemm", "outer") else out
    return {"bytes": entry * (read + out) + 8 * (rows + m + 1), "flops": flops}


def tolerance(case):
    # sums of a row's products in any order, one rounding each (seen: up to 1e-7 and 8e-16 against 64-bit sums
    # in another order); indices and row pointers are exact
    return {"rel": 1e-6 if case["dtype"] == "f32" else 4e-15}
