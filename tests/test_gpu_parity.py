"""GPU parity against the CPU oracle on small and adversarial inputs (through the C ABI).

Structure (rowptr, colidx) must be bit-exact; values within max relative
error 1e-12 (float64) or 1e-5 (float32) of the summation-order bound.
"""
from __future__ import annotations

import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from paper_2606_20855_gb300 import _abi
from synth import HostCSR, random_csr, rmat_pattern, uniform_csr
from tests._gpu import assert_matches_oracle, run_gpu, tuning
from tests._helpers import TOL

pytestmark = pytest.mark.gpu

DTYPES = [np.float64, np.float32]


def _csr(m, n, rows_cols, vals=None, dtype=np.float64):
    rowptr = np.zeros(m + 1, dtype=np.int64)
    cols = []
    for i in range(m):
        c = sorted(set(rows_cols.get(i, [])))
        cols.extend(c)
        rowptr[i + 1] = len(cols)
    colidx = np.array(cols, dtype=np.int32)
    v = np.ones(colidx.size, dtype=dtype) if vals is None else np.asarray(vals, dtype=dtype)
    return HostCSR(m, n, rowptr, colidx, v)


PATHS = {"bitmap": {}, "bitmap_generic": {"register_rows_max_a": 0}, "hash": {"bitmap_span": 0}}


@pytest.mark.parametrize("path", list(PATHS))
@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("seed", range(12))
def test_random_shapes(seed, dtype, path):
    rng = np.random.default_rng(500 + seed)
    m, k, n = (int(x) for x in rng.integers(1, 400, size=3))
    A = random_csr(m, k, float(rng.choice([0.005, 0.02, 0.08])), rng, dtype, "sym", empty_rows=0.1)
    B = random_csr(k, n, float(rng.choice([0.01, 0.05, 0.2])), rng, dtype, "sym", empty_rows=0.1)
    with tuning(**PATHS[path]):
        rowptr, colidx, vals, _ = run_gpu(A, B, validate=True)
    assert_matches_oracle(A, B, rowptr, colidx, vals)


@pytest.mark.parametrize("path", list(PATHS))
@pytest.mark.parametrize("dtype", DTYPES)
def test_uniform_several_tiles(dtype, path):
    # enough rows for many CTAs and a ragged last tile of every kernel
    rng = np.random.default_rng(7)
    A = uniform_csr(40_003, 3_001, 9, rng, dtype, "sym")
    B = uniform_csr(3_001, 5_003, 17, rng, dtype, "sym")
    with tuning(**PATHS[path]):
        rowptr, colidx, vals, info = run_gpu(A, B)
    assert info[f"{path.split('_')[0]}_rows"] == 40_003
    assert_matches_oracle(A, B, rowptr, colidx, vals)


def _banded(m, n, lens, halfwidth, rng, dtype, centre):
    """Rows of the given lengths with distinct columns within halfwidth of centre(i)."""
    rows = {}
    for i, L in enumerate(lens):
        c = int(centre(i))
        lo, hi = max(0, c - halfwidth), min(n, c + halfwidth + 1)
        L = min(L, hi - lo)
        rows[i] = (lo + rng.choice(hi - lo, size=L, replace=False)).tolist()
    M = _csr(m, n, rows, dtype=dtype)
    M.vals = (2 * rng.random(M.nnz) - 1).astype(dtype)
    return M


@pytest.mark.parametrize("b_len", [4, 8])
@pytest.mark.parametrize("dtype", DTYPES)
def test_grouped_register_rows(dtype, b_len):
    """Banded products over more than 65,536 columns whose B rows fit 4 or 8
    lanes: rows of at most 4096 columns are ranked by groups of lanes, several
    rows per warp, with stored-entry counts 0..16 mixed inside every warp,
    repeated columns, a ragged last warp, and wider rows (other bins) between
    them."""
    rng = np.random.default_rng(40 + b_len)
    k = n = 100_000
    B = _banded(k, n, [b_len] * k, 600, rng, dtype, lambda j: j)
    m = 20_011
    lens = rng.integers(0, 17, size=m)
    A = _banded(m, k, lens, 700, rng, dtype, lambda i: i * (k // m))
    wide = rng.choice(m, size=200, replace=False)  # rows spread over a wider range
    rows = {i: A.colidx[A.rowptr[i]:A.rowptr[i + 1]].tolist() for i in range(m)}
    for i in wide:
        L = int(rng.integers(2, 17))
        rows[int(i)] = rng.choice(k, size=L, replace=False).tolist()
    A = _csr(m, k, rows, dtype=dtype)
    A.vals = (2 * rng.random(A.nnz) - 1).astype(dtype)
    rowptr, colidx, vals, info = run_gpu(A, B, validate=True)
    assert_matches_oracle(A, B, rowptr, colidx, vals)


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("n", [2_000, 16_000, 60_000])
def test_bitmap_bins(dtype, n):
    """Rows of every bitmap bin: narrow and wide column ranges, small and large rows."""
    rng = np.random.default_rng(n)
    k = 2500
    B = uniform_csr(k, n, 24, rng, dtype, "sym")
    lens = [2, 3, 6, 11, 20, 40, 90, 200, 330]
    rows = {i: rng.choice(k, size=L, replace=False).tolist() for i, L in enumerate(lens * 20)}
    A = _csr(len(lens) * 20, k, rows, dtype=dtype)
    A.vals = (2 * rng.random(A.nnz) - 1).astype(dtype)
    rowptr, colidx, vals, info = run_gpu(A, B)
    assert info["bitmap_rows"] > 0
    assert_matches_oracle(A, B, rowptr, colidx, vals)


@pytest.mark.parametrize("n", [60_000, 70_000])
@pytest.mark.parametrize("dtype", DTYPES)
def test_every_row_class(dtype, n):
    """Rows of every class: empty, direct, register bitmap, bitmap, hash, dense window.

    With n <= 65,536 the planning pass counts the short rows and leaves the
    others (empty, single-entry, long) to the analysis kernel."""
    rng = np.random.default_rng(11)
    k = 3000
    B = uniform_csr(k, n, 40, rng, dtype, "sym")
    lens = [0, 1, 1, 2, 3, 5, 9, 17, 33, 65, 100, 150, 200, 400, 1000, 2000, 3000]
    rows = {}
    for i, L in enumerate(lens * 3):
        rows[i] = rng.choice(k, size=L, replace=False).tolist()
    A = _csr(len(lens) * 3, k, rows, dtype=dtype)
    A.vals = (2 * rng.random(A.nnz) - 1).astype(dtype)
    rowptr, colidx, vals, info = run_gpu(A, B, validate=True)
    assert info["direct_rows"] == 6 and info["empty_rows"] == 3
    assert info["dense_rows"] + info["rcd_rows"] + info["wb_rows"] > 0
    assert_matches_oracle(A, B, rowptr, colidx, vals)


@pytest.mark.parametrize("dtype", DTYPES)
def test_dense_window_path_everywhere(dtype):
    rng = np.random.default_rng(12)
    A = uniform_csr(3000, 800, 6, rng, dtype, "sym")
    B = uniform_csr(800, 9000, 12, rng, dtype, "sym")
    with tuning(hash_max_products=0, dense_width=1024, bitmap_span=0, wide_bitmap_span=0):
        rowptr, colidx, vals, info = run_gpu(A, B)
    assert info["hash_rows"] == 0 and info["dense_rows"] == 3000 and info["dense_slices"] > 3000
    assert_matches_oracle(A, B, rowptr, colidx, vals)


@pytest.mark.parametrize("dtype", DTYPES)
def test_sort_path_everywhere(dtype):
    rng = np.random.default_rng(13)
    A = uniform_csr(2000, 900, 8, rng, dtype, "sym")
    B = uniform_csr(900, 4000, 20, rng, dtype, "sym")
    with tuning(run_limit=1, bitmap_span=0):
        rowptr, colidx, vals, info = run_gpu(A, B)
    assert info["sorted_rows"] > 0
    assert_matches_oracle(A, B, rowptr, colidx, vals)


HEAVY = {"default": {}, "no_dense_rows": {"dense_rows_max_a": 0}, "wide_bitmap_only": {"dense_rows_max_a": 0, "bitmap_span": 0},
         "sliced_only": {"dense_rows_max_a": 0, "bitmap_span": 0, "wide_bitmap_span": 0, "hash_max_products": 0},
         "dense_rows_few_a": {"dense_rows_max_a": 64}}


@pytest.mark.parametrize("heavy", list(HEAVY))
@pytest.mark.parametrize("dtype", DTYPES)
def test_heavy_rows(heavy, dtype):
    """Hub rows of a skewed product (few stored A entries, long B rows) and
    wide rows with many short B rows, on every heavy-row path."""
    rng = np.random.default_rng(31)
    rp, ci, _ = rmat_pattern(13, 16, (0.57, 0.19, 0.19, 0.05), rng)
    A = HostCSR(8192, 8192, rp, ci, (1.0 - rng.random(ci.size)).astype(dtype))
    from synth import row_subset
    from tests._helpers import products_per_row
    lens, ub = np.diff(rp), products_per_row(A, A)
    hubs = np.argsort(lens)[-100:]                               # many stored entries
    fed = np.flatnonzero((ub > 4096) & (lens <= 64))[:300]      # few entries, long (hub) B rows
    light = rng.choice(8192, size=100, replace=False)
    H = row_subset(A, np.unique(np.concatenate([hubs, fed, light])))
    with tuning(**HEAVY[heavy]):
        rowptr, colidx, vals, info = run_gpu(H, A)
    if heavy == "default":
        assert info["rcd_rows"] > 0
    if heavy == "wide_bitmap_only":
        assert info["wb_rows"] > 0
    if heavy == "sliced_only":
        assert info["dense_rows"] > 0
    assert_matches_oracle(H, A, rowptr, colidx, vals)


@pytest.mark.parametrize("dtype", DTYPES)
def test_direct_rows_long_and_short(dtype):
    """Rows of A with one stored entry copy a scaled B row: B rows of 0 to
    5000 entries around the length where a whole warp takes over (512), among
    many short ones so the lane groups stay small."""
    rng = np.random.default_rng(34)
    n = 20_000
    lens = [0, 1, 3, 31, 32, 33, 511, 512, 513, 1000, 5000]
    rows = {i: rng.choice(n, size=L, replace=False).tolist() for i, L in enumerate(lens)}
    k = 3000
    for i in range(len(lens), k):
        rows[i] = rng.choice(n, size=int(rng.integers(1, 6)), replace=False).tolist()
    B = _csr(k, n, rows, dtype=dtype)
    B.vals = (2 * rng.random(B.nnz) - 1).astype(dtype)
    picks = list(range(len(lens))) * 3 + rng.choice(k, size=400).tolist()
    A = _csr(len(picks), k, {i: [c] for i, c in enumerate(picks)}, dtype=dtype)
    A.vals = (2 * rng.random(A.nnz) - 1).astype(dtype)
    rowptr, colidx, vals, info = run_gpu(A, B)
    blen = np.diff(B.rowptr)
    assert info["direct_rows"] == int(np.count_nonzero(blen[picks]))  # an empty B row gives an empty row
    assert_matches_oracle(A, B, rowptr, colidx, vals)


@pytest.mark.parametrize("dtype", DTYPES)
def test_dense_rows_slice_parts(dtype):
    """Dense heavy rows whose B rows give every kind of part inside a value
    window slice: empty, one entry, just below / at / just above the short-part
    limit (32) and the piece size (128), many pieces, a B row covering all
    65,536 columns, columns on the slice starts and just before them, a B row
    inside one slice; one row with more than 256 stored entries; and rows
    whose output is below, exactly at and one above the value window's size
    (the compact window takes the first two)."""
    rng = np.random.default_rng(33)
    n = 1 << 16
    slice_w = 8192 if dtype == np.float64 else 16384
    lens = [0, 1, 2, 31, 32, 33, 127, 128, 129, 257, 1000, 4000, 20000]
    rows = {i: rng.choice(n, size=L, replace=False).tolist() for i, L in enumerate(lens)}
    rows[len(lens)] = list(range(n))                                       # every column
    rows[len(lens) + 1] = [s * slice_w + d for s in range(n // slice_w) for d in (-1, 0) if 0 <= s * slice_w + d < n]
    rows[len(lens) + 2] = (3 * slice_w + rng.choice(slice_w, size=300, replace=False)).tolist()  # one slice
    x = rng.permutation(n)[:slice_w]                      # exactly one window of distinct columns
    rows[len(lens) + 3] = x.tolist()
    rows[len(lens) + 4] = rng.choice(x, size=500, replace=False).tolist()            # inside x
    outside = np.setdiff1d(np.arange(n), x)
    rows[len(lens) + 5] = rng.choice(x, size=100, replace=False).tolist() + [int(outside[7])]  # one column more
    k = 400
    for i in range(len(lens) + 6, k):
        rows[i] = rng.choice(n, size=int(rng.integers(0, 300)), replace=False).tolist()
    B = _csr(k, n, rows, dtype=dtype)
    B.vals = (2 * rng.random(B.nnz) - 1).astype(dtype)
    special = list(range(len(lens) + 3))
    X = len(lens) + 3
    arows = {0: special, 1: special[:5] + [len(lens)], 2: [len(lens) + 1, len(lens) + 2, 12],
             3: rng.choice(k, size=300, replace=False).tolist(),                 # 300 > 256 entries
             4: [6, 7, 8, 9, 10, 11],                 # output fits one value window
             5: [X, X + 1],                           # output exactly one window wide
             6: [X, X + 2]}                           # one column more than a window
    for i in range(7, 40):
        arows[i] = rng.choice(k, size=int(rng.integers(2, 200)), replace=False).tolist() + [12]
    A = _csr(40, k, arows, dtype=dtype)
    A.vals = (2 * rng.random(A.nnz) - 1).astype(dtype)
    rowptr, colidx, vals, info = run_gpu(A, B)
    assert info["rcd_rows"] >= 38
    assert np.diff(rowptr)[5] == slice_w and np.diff(rowptr)[6] == slice_w + 1
    assert_matches_oracle(A, B, rowptr, colidx, vals)


@pytest.mark.parametrize("dtype", DTYPES)
def test_dense_rows_many_products_few_columns(dtype):
    """Dense heavy rows with far more products than output entries: 200
    stored entries whose B rows (1000 entries each) share a pool of 6000
    columns, so 200,000 products fall on at most 6000 outputs.  The output fits
    one value window, but the products are too many for the per-piece first
    flags, so the column indices come from the bitmap walk instead."""
    rng = np.random.default_rng(36)
    n = 1 << 16
    pool = rng.choice(n, size=6000, replace=False)
    k = 260
    rows = {i: rng.choice(pool, size=1000, replace=False).tolist() for i in range(k)}
    B = _csr(k, n, rows, dtype=dtype)
    B.vals = (2 * rng.random(B.nnz) - 1).astype(dtype)
    arows = {i: rng.choice(k, size=200, replace=False).tolist() for i in range(6)}
    A = _csr(6, k, arows, dtype=dtype)
    A.vals = (2 * rng.random(A.nnz) - 1).astype(dtype)
    rowptr, colidx, vals, info = run_gpu(A, B)
    assert info["rcd_rows"] == 6
    assert assert_matches_oracle(A, B, rowptr, colidx, vals) <= TOL[np.dtype(dtype)]


@pytest.mark.parametrize("dtype", DTYPES)
def test_dense_rows_windows_and_rounds(dtype):
    """Dense heavy rows at the edges of their output windows (49,152 bytes of
    values: one entry less than a window, exactly one, one more, exactly two)
    and of the parts of B rows inside a window: around the short-part limit
    (96), around one and two rounds (512, 1024), more rounds than are
    described at a time (128), and 255, 256 and 257 stored entries (256 are
    cached at a time; the symbolic pass caches 1024)."""
    rng = np.random.default_rng(37)
    n = 1 << 16
    window = 49152 // np.dtype(dtype).itemsize
    perm = rng.permutation(n)
    blocks = [perm[:window - 1], perm[:window], perm[:window + 1], perm[:2 * window]]
    rows = {i: c.tolist() for i, c in enumerate(blocks)}
    lens = [1, 32, 33, 95, 96, 97, 511, 512, 513, 1023, 1024, 1025, 3000]
    first_len = len(rows)
    for L in lens:
        rows[len(rows)] = rng.choice(n, size=L, replace=False).tolist()
    inside = len(rows)                                    # subsets of the smallest block
    for _ in range(20):
        rows[len(rows)] = rng.choice(blocks[0], size=600, replace=False).tolist()
    k = 1400
    many = len(rows)
    while len(rows) < k:
        rows[len(rows)] = rng.choice(n, size=int(rng.integers(0, 120)), replace=False).tolist()
    B = _csr(k, n, rows, dtype=dtype)
    B.vals = (2 * rng.random(B.nnz) - 1).astype(dtype)
    sub = list(range(inside, inside + 20))
    arows = {i: [i] + sub for i in range(4)}              # windows
    arows[4] = list(range(first_len, first_len + len(lens)))
    arows[5] = list(range(k - 200, k)) + list(range(4)) + sub          # more than 128 rounds
    for i, na in enumerate((255, 256, 257, 1030)):
        arows[6 + i] = rng.choice(np.arange(many, k), size=na - 1, replace=False).tolist() + [0]
    A = _csr(10, k, arows, dtype=dtype)
    A.vals = (2 * rng.random(A.nnz) - 1).astype(dtype)
    rowptr, colidx, vals, info = run_gpu(A, B)
    assert info["rcd_rows"] == 10
    assert np.diff(rowptr)[:4].tolist() == [window - 1, window, window + 1, 2 * window]
    assert_matches_oracle(A, B, rowptr, colidx, vals)


def _hash_edge_case(dtype):
    """Rows of every hash bin at its edges (one product less, exactly, one more
    than a power of two), over 3,000,000 columns: B rows of 0, 1 and 40
    entries, rows of many one-entry B rows, repeated columns, and rows whose
    columns crowd at one end."""
    rng = np.random.default_rng(38)
    n = 3_000_000
    rows = {0: [0], 1: [n - 1]}
    rows[2] = []                                                     # an empty B row
    ones = list(range(3, 4500))                                      # one entry each
    for r in ones:
        rows[r] = [int(rng.integers(1, n - 1))]
    forty = list(range(4500, 4650))
    for r in forty:
        rows[r] = rng.choice(n - 2, size=40, replace=False).tolist()
    shared = list(range(4650, 4750))                                 # 40 of 100 columns: repeats
    pool = rng.choice(n - 2, size=100, replace=False)
    for r in shared:
        rows[r] = rng.choice(pool, size=40, replace=False).tolist()
    crowd = list(range(4750, 4850))                                  # 40 of the first 3000 columns
    for r in crowd:
        rows[r] = rng.choice(np.arange(1, 3000), size=40, replace=False).tolist()
    B = _csr(4850, n, rows, dtype=dtype)
    B.vals = (2 * rng.random(B.nnz) - 1).astype(dtype)
    lens = np.diff(B.rowptr)
    arows = {}
    sizes = sorted({s + d for s in (32, 64, 128, 256, 512, 1024, 2048) for d in (-1, 0, 1)} | {2, 3, 4095, 4096})
    for u in sizes:
        for kind in range(4):
            pick = [0, 1, 2]                                         # both ends, and the empty row
            left = u - 2
            group = (forty, shared, crowd, [])[kind]
            for r in rng.permutation(group)[:left // 40]:
                pick.append(int(r))
                left -= int(lens[r])
            pick += [int(r) for r in rng.choice(ones, size=left, replace=False)]
            arows[len(arows)] = pick
    A = _csr(len(arows), 4850, arows, dtype=dtype)
    A.vals = (2 * rng.random(A.nnz) - 1).astype(dtype)
    return A, B


@pytest.mark.parametrize("run_limit", [64, 2])
@pytest.mark.parametrize("dtype", DTYPES)
def test_hash_rows_bin_edges(dtype, run_limit):
    """Every hash bin at its edges, with and without the sort of crowded rows."""
    A, B = _hash_edge_case(dtype)
    with tuning(run_limit=run_limit):
        rowptr, colidx, vals, info = run_gpu(A, B)
    assert info["hash_rows"] == A.nrows
    assert 0 < info["sorted_rows"] < A.nrows
    assert_matches_oracle(A, B, rowptr, colidx, vals)


@pytest.mark.parametrize("dtype", DTYPES)
def test_hash_rows_without_kept_ranks(dtype):
    """The numeric pass works the ranks of every hash bin out itself."""
    A, B = _hash_edge_case(dtype)
    with tuning(kept_bytes=0):
        rowptr, colidx, vals, info = run_gpu(A, B)
    assert info["hash_rows"] == A.nrows
    assert_matches_oracle(A, B, rowptr, colidx, vals)


# A product twice in a process of its own (an earlier test's freed scratch would
# serve): op2 with all the room it wants, then op1 whose symbolic pass finds less
# than 56 MB of device memory left.  `setup` makes A and B, `check` looks at the
# operations and at C as (rp, ci, v) of both.
_SHORT_OF_MEMORY = """
import numpy as np, torch
from tests._gpu import assert_matches_oracle
from paper_2606_20855_gb300.spgemm import DeviceCSR, SpGEMM
%s
dA, dB = DeviceCSR.from_host(A), DeviceCSR.from_host(B)
def product(short):
    op = SpGEMM(dA, dB)
    held = []
    if short:
        size = 1 << 30
        while size >= 1 << 24:
            if torch.cuda.mem_get_info()[0] - size > 40 << 20:
                held.append(torch.empty(size, dtype=torch.uint8, device="cuda"))
            else:
                size >>= 1
    op.symbolic()
    del held
    torch.cuda.empty_cache()
    C = op.numeric()
    op.wait()
    return op, C.to_host()
op2, (rp2, ci2, v2) = product(False)  # its scratch stays taken
op1, (rp1, ci1, v1) = product(True)
assert np.array_equal(rp1, rp2) and np.array_equal(ci1, ci2)
%s
"""


def _run_short_of_memory(setup, check):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    res = subprocess.run([sys.executable, "-c", _SHORT_OF_MEMORY % (setup, check)], cwd=root, capture_output=True,
                         text=True, timeout=300)
    assert res.returncode == 0, res.stderr[-2000:]


def test_dense_rows_without_room_for_bitmaps():
    """With almost all device memory taken the bitmaps of the dense heavy rows
    do not fit: the rows are taken in batches, and the numeric pass makes the
    bitmaps again (more launches, the same C).  (A process of its own: an
    earlier test's freed scratch would serve.)"""
    _run_short_of_memory("""
from synth import HostCSR
rng = np.random.default_rng(39)
k, n, m = 1400, 1 << 16, 12001  # 98 MB of bitmaps, an odd last batch
lens = rng.integers(0, 140, size=k)
brp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
bci = np.concatenate([np.sort(rng.choice(n, size=x, replace=False)) for x in lens]).astype(np.int32)
B = HostCSR(k, n, brp, bci, 2 * rng.random(bci.size) - 1)
aci = np.sort(rng.random((m, k)).argsort(axis=1)[:, :100], axis=1).astype(np.int32).ravel()
A = HostCSR(m, k, np.arange(m + 1, dtype=np.int64) * 100, aci, 2 * rng.random(aci.size) - 1)
""", """
i1, i2 = op1.plan_info(), op2.plan_info()
assert i1["rcd_rows"] == i2["rcd_rows"] > 11900
assert i1["numeric_launches"] > i2["numeric_launches"]
assert_matches_oracle(A, B, rp1, ci1, v1, rows=np.concatenate([np.arange(0, m, 101), [m - 1]]))
""")


def test_hash_rows_without_room_for_ranks():
    """With almost all device memory taken the symbolic pass cannot keep the
    ranks of the hash rows and the numeric pass works them out: the same C.
    (A process of its own: an earlier test's freed scratch would serve.)"""
    _run_short_of_memory("""
from tests.test_gpu_parity import _hash_edge_case
from synth import HostCSR
A, B = _hash_edge_case(np.float64)
reps = 400  # 100 rows, 400 times: the ranks take about 88 MB
rp = np.concatenate([[0], np.cumsum(np.tile(np.diff(A.rowptr), reps))]).astype(np.int64)
A = HostCSR(A.nrows * reps, A.ncols, rp, np.tile(A.colidx, reps), np.tile(A.vals, reps))
""", """
assert op1.plan_info()["hash_rows"] == A.nrows
assert_matches_oracle(A, B, rp1, ci1, v1, rows=np.arange(100))
assert_matches_oracle(A, B, rp1, ci1, v1, rows=np.arange(A.nrows - 100, A.nrows))
""")


@pytest.mark.parametrize("dtype", DTYPES)
def test_wide_heavy_rows(dtype):
    """Rows with thousands of stored A entries over short B rows spanning ~2^20 columns."""
    rng = np.random.default_rng(32)
    k, n = 20_000, 1 << 20
    B = uniform_csr(k, n, 4, rng, dtype, "pos")
    rows = {i: rng.choice(k, size=int(L), replace=False).tolist() for i, L in enumerate([1500, 3000, 6000, 2, 40])}
    A = _csr(5, k, rows, dtype=dtype)
    A.vals = (1.0 - rng.random(A.nnz)).astype(dtype)
    rowptr, colidx, vals, info = run_gpu(A, B)
    assert info["wb_rows"] == 3
    assert_matches_oracle(A, B, rowptr, colidx, vals)


@pytest.mark.parametrize("dtype", DTYPES)
def test_wide_rows_cluster_split(dtype):
    """Wide-bitmap rows whose column ranges sit at the edges of the split of a
    row's bitmap over a cluster of CTAs (runs of a power of two of 128-column
    chunks): one chunk (spans 1 and 128), one chunk past a power of two,
    ranges that leave some CTAs of the cluster without a chunk, the full
    2^20 columns, and one row of many stored entries in the same kernel."""
    rng = np.random.default_rng(33)
    n = 1 << 20
    spans = [1, 127, 128, 129, 1024, 1025, 65537, (1 << 19) + 1, (1 << 20) - 5, 1 << 20]
    b_rows, a_rows = [], {}
    for i, s in enumerate(spans):
        c0 = int(rng.integers(0, n - s + 1))
        first = len(b_rows)
        for j in range(40):
            cols = set(int(c) for c in c0 + rng.integers(0, s, size=int(rng.integers(1, 9))))
            if j == 0:
                cols.add(c0)            # the row's range is exactly [c0, c0 + s)
            if j == 39:
                cols.add(c0 + s - 1)
            b_rows.append(sorted(cols))
        a_rows[i] = list(range(first, first + 40))
    hub = len(spans)  # many stored entries over rows spanning all columns
    first = len(b_rows)
    for j in range(3000):
        b_rows.append(sorted(set(int(c) for c in rng.integers(0, n, size=5))))
    a_rows[hub] = list(range(first, first + 3000))
    B = _csr(len(b_rows), n, dict(enumerate(b_rows)), dtype=dtype)
    B.vals = (1.0 - rng.random(B.nnz)).astype(dtype)
    A = _csr(len(spans) + 1, B.nrows, a_rows, dtype=dtype)
    A.vals = (2 * rng.random(A.nnz) - 1).astype(dtype)
    with tuning(hash_max_products=0, bitmap_span=0, dense_rows_max_a=0, register_rows_max_a=0):
        rowptr, colidx, vals, info = run_gpu(A, B)
    assert info["wb_rows"] == len(spans) + 1
    assert_matches_oracle(A, B, rowptr, colidx, vals)
    assert rowptr[1] == 1  # span 1: forty products, one column


@pytest.mark.parametrize("path", list(PATHS))
def test_skewed_rmat_square(path):
    rng = np.random.default_rng(14)
    rp, ci, _ = rmat_pattern(12, 16, (0.57, 0.19, 0.19, 0.05), rng)
    A = HostCSR(4096, 4096, rp, ci, (1.0 - rng.random(ci.size)))
    with tuning(**PATHS[path]):
        rowptr, colidx, vals, info = run_gpu(A, A)
    if path == "hash":
        assert info["dense_rows"] + info["rcd_rows"] + info["wb_rows"] > 0 and info["bitmap_rows"] == 0
    else:
        assert info["bitmap_rows"] > 0
    assert_matches_oracle(A, A, rowptr, colidx, vals)


def test_rmat_unit_values_exact():
    rng = np.random.default_rng(15)
    rp, ci, _ = rmat_pattern(11, 16, (0.57, 0.19, 0.19, 0.05), rng)
    A = HostCSR(2048, 2048, rp, ci, np.ones(ci.size))
    rowptr, colidx, vals, _ = run_gpu(A, A)
    err = assert_matches_oracle(A, A, rowptr, colidx, vals)
    assert err == 0.0  # path counts are exact integers in any summation order


@pytest.mark.parametrize("m,k,n", [(0, 5, 3), (4, 0, 3), (4, 5, 0), (1, 1, 1), (7, 3, 1)])
def test_degenerate_shapes(m, k, n):
    rng = np.random.default_rng(m * 100 + k * 10 + n)
    A = random_csr(m, k, 0.6, rng)
    B = random_csr(k, n, 0.6, rng)
    rowptr, colidx, vals, _ = run_gpu(A, B, validate=True)
    assert_matches_oracle(A, B, rowptr, colidx, vals)


def test_all_rows_empty_and_empty_b_rows():
    A = _csr(50, 20, {i: [i % 20] for i in range(0, 50, 2)})
    B = _csr(20, 30, {j: [j, j + 1] for j in range(1, 20, 2)})  # even rows of B empty
    rowptr, colidx, vals, info = run_gpu(A, B)
    assert rowptr[-1] == 0 and info["empty_rows"] == 50


def test_direct_rows_scaled_copy():
    rng = np.random.default_rng(16)
    perm = rng.permutation(500)
    A = HostCSR(500, 500, np.arange(501, dtype=np.int64), perm.astype(np.int32), 2 * rng.random(500) - 1)
    B = uniform_csr(500, 2000, 37, rng)
    rowptr, colidx, vals, info = run_gpu(A, B)
    assert info["direct_rows"] == 500
    assert_matches_oracle(A, B, rowptr, colidx, vals)


def test_single_dense_row_and_wide_output():
    rng = np.random.default_rng(17)
    k, n = 600, 1 << 20
    A = _csr(3, k, {0: list(range(k)), 2: [5, 7]}, dtype=np.float64)
    A.vals = 2 * rng.random(A.nnz) - 1
    B = uniform_csr(k, n, 30, rng)
    rowptr, colidx, vals, info = run_gpu(A, B)
    assert info["wb_rows"] == 1
    assert_matches_oracle(A, B, rowptr, colidx, vals)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_wide_rows_in_parts(dtype):
    """Wide-bitmap rows around the 16,384 products of a numeric item: one, two
    and four items, and a hub row of short and long B rows."""
    rng = np.random.default_rng(40)
    k, n = 9000, 1 << 20
    rows = {i: np.unique(rng.integers(0, n, size=8)).tolist() for i in range(k - 40)}
    for i in range(k - 40, k):
        rows[i] = np.unique(rng.integers(0, n, size=700)).tolist()
    rows[0] = [0, 1, 2, 3, 4, 5, 6, n - 1]
    B = _csr(k, n, rows, dtype=dtype)
    B.vals = (2 * rng.random(B.nnz) - 1).astype(dtype)
    eight = np.flatnonzero(np.diff(B.rowptr[:k - 39]) == 8)
    arows = {i: [0] + eight[1:na].tolist() for i, na in enumerate((2047, 2048, 2049, 4096, 4097, 8193))}
    arows[6] = list(range(k - 1500, k))
    A = _csr(7, k, arows, dtype=dtype)
    A.vals = (2 * rng.random(A.nnz) - 1).astype(dtype)
    rowptr, colidx, vals, info = run_gpu(A, B)
    assert info["wb_rows"] == 7
    assert_matches_oracle(A, B, rowptr, colidx, vals)


def _drawn_csr(m, n, r, rng):
    """r distinct columns per row, for any r <= n."""
    cols = np.concatenate([np.sort(rng.choice(n, size=r, replace=False)) for _ in range(m)]).astype(np.int32)
    return HostCSR(m, n, np.arange(m + 1, dtype=np.int64) * r, cols, 2 * rng.random(cols.size) - 1)


@pytest.mark.parametrize("rows,entries,length", [(310, 900, 40), (5, 3, 20_000), (2, 2, 9000)])
def test_wide_rows_in_parts(rows, entries, length):
    """Many wide rows of 36,000 products (larger parts), and rows of more parts by products than stored entries."""
    rng = np.random.default_rng(63)
    A = _drawn_csr(rows, 3000 if length < 100 else 8, entries, rng)
    B = _drawn_csr(A.ncols, 1 << 20, length, rng)
    rowptr, colidx, vals, info = run_gpu(A, B)
    assert info["wb_rows"] == rows
    assert_matches_oracle(A, B, rowptr, colidx, vals, rows=np.arange(0, rows, 1 if rows < 10 else 31))


def test_wide_rows_without_room_for_bitmaps():
    """With almost all device memory taken the bitmaps of the wide rows are not
    kept and the numeric pass makes them again: the same C.  (A process of its
    own: an earlier test's freed scratch would serve.)"""
    _run_short_of_memory("""
from synth import HostCSR, uniform_csr
rng = np.random.default_rng(41)
B = uniform_csr(5000, 1 << 20, 20, rng)
aci = np.sort(rng.random((601, 5000)).argsort(axis=1)[:, :900], axis=1).astype(np.int32).ravel()
A = HostCSR(601, 5000, np.arange(602, dtype=np.int64) * 900, aci, 2 * rng.random(aci.size) - 1)  # 79 MB of bitmaps
""", """
i1, i2 = op1.plan_info(), op2.plan_info()
assert i1["wb_rows"] == i2["wb_rows"] == 601
assert i1["numeric_launches"] < i2["numeric_launches"]  # no launch to zero the values
assert_matches_oracle(A, B, rp1, ci1, v1, rows=np.arange(0, 601, 10))
assert_matches_oracle(A, B, rp2, ci2, v2, rows=np.arange(0, 601, 10))
""")


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("ncols", [1100, 6144, 6145, 12_288, 12_289])
def test_dense_rows_around_the_window(ncols, dtype):
    """Enough dense heavy rows for whole windows, B as wide as a window has places (6,144 in float64, 12,288 in
    float32) and one column wider; rows over all columns and over the last ones only."""
    rng = np.random.default_rng(65)
    whole, last = _drawn_csr(60, ncols, 400, rng), _drawn_csr(60, 1030, 400, rng)
    B = HostCSR(120, ncols, np.arange(121, dtype=np.int64) * 400,
                np.concatenate([whole.colidx, last.colidx + (ncols - 1030)]).astype(np.int32),
                np.concatenate([whole.vals, last.vals]).astype(dtype))
    rows = [np.sort(rng.choice(60, size=25, replace=False)) + 60 * (i % 2) for i in range(200)]
    A = HostCSR(200, 120, np.arange(201, dtype=np.int64) * 25, np.concatenate(rows).astype(np.int32),
                (2 * rng.random(5000) - 1).astype(dtype))
    rowptr, colidx, vals, info = run_gpu(A, B)
    assert info["rcd_rows"] >= 100
    assert_matches_oracle(A, B, rowptr, colidx, vals)


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("length", [513, 1024, 1025, 2049])
def test_dense_rows_of_long_b_rows(length, dtype):
    """Rounds of 1024 entries (float32) and of 512 at their edges, with short B rows among the long ones."""
    rng = np.random.default_rng(66)
    long_rows, short = _drawn_csr(80, 3000, length, rng), _drawn_csr(20, 3000, 40, rng)
    B = HostCSR(100, 3000, np.concatenate([long_rows.rowptr, long_rows.rowptr[-1] + short.rowptr[1:]]),
                np.concatenate([long_rows.colidx, short.colidx]),
                np.concatenate([long_rows.vals, short.vals]).astype(dtype))
    A = _drawn_csr(180, 100, 30, rng)
    A = HostCSR(A.nrows, A.ncols, A.rowptr, A.colidx, A.vals.astype(dtype))
    rowptr, colidx, vals, info = run_gpu(A, B)
    assert info["rcd_rows"] == A.nrows
    assert_matches_oracle(A, B, rowptr, colidx, vals)


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("rows,ncols", [(1, 1100), (3, 1536), (2, 1537), (40, 3000), (7, 30_000)])
def test_few_dense_rows_in_small_windows(rows, ncols, dtype):
    """Too few dense heavy rows for the GPU: windows of 512 entries and more, full and ragged ones."""
    rng = np.random.default_rng(64)
    B = _drawn_csr(400, ncols, min(900, ncols), rng)
    A = _drawn_csr(rows, 400, 130, rng)
    A, B = (HostCSR(x.nrows, x.ncols, x.rowptr, x.colidx, x.vals.astype(dtype)) for x in (A, B))
    rowptr, colidx, vals, info = run_gpu(A, B)
    assert info["rcd_rows"] == rows
    assert_matches_oracle(A, B, rowptr, colidx, vals)


def _box_stencil(dims, dof, rng, dtype):
    """All neighbours of a grid point in a box of three per dimension, dof x dof blocks."""
    at = np.arange(np.prod(dims)).reshape(dims)
    pad = np.full([d + 2 for d in dims], -1)
    pad[tuple(slice(1, -1) for _ in dims)] = at
    near = np.stack([pad[tuple(slice(o, o + d) for o, d in zip(off, dims))].ravel()
                     for off in np.ndindex(*[3] * len(dims))], axis=1)
    cols = np.where(near[:, :, None] < 0, -1, near[:, :, None] * dof + np.arange(dof)).reshape(near.shape[0], -1)
    cols = np.repeat(cols, dof, axis=0)
    lens = (cols >= 0).sum(axis=1)
    rowptr = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    vals = (2 * rng.random(rowptr[-1]) - 1).astype(dtype)
    return HostCSR(cols.shape[0], cols.shape[0], rowptr, cols[cols >= 0].astype(np.int32), vals)


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("dims,dof", [((5, 40, 40), 1), ((7, 90), 3)])
def test_rows_of_neighbouring_columns_take_bitmaps(dims, dof, dtype):
    """Box stencils: wide rows whose columns come in runs would fill a hash bucket with every run."""
    A = _box_stencil(dims, dof, np.random.default_rng(61), dtype)
    rowptr, colidx, vals, info = run_gpu(A, A)
    assert info["hash_rows"] <= 0.02 * A.nrows  # some rows at the edges of the grid
    assert_matches_oracle(A, A, rowptr, colidx, vals, rows=np.arange(0, A.nrows, 5))


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("ra,rb,n,rows_key", [
    (24, 12, 4000, "bitmap_rows"), (42, 12, 16_000, "bitmap_rows"),  # 288 and 504 products of B rows of one length
    (43, 12, 16_000, "hash_rows"), (24, 12, 60_000, "hash_rows"),    # more products, wider than 16,384 columns
    (21, 12, 4000, "hash_rows"), (40, 40, 30_000, "hash_rows"),
    (60, 40, 16_000, "rcd_rows"), (150, 16, 16_000, "rcd_rows"),     # 2400 products of long B rows
    (160, 15, 16_000, "hash_rows"),                                  # and of shorter ones
])
def test_route_of_spread_rows(ra, rb, n, rows_key, dtype):
    rng = np.random.default_rng(ra * rb)
    A, B = uniform_csr(120, 2000, ra, rng), uniform_csr(2000, n, rb, rng)
    A = HostCSR(A.nrows, A.ncols, A.rowptr, A.colidx, A.vals.astype(dtype))
    B = HostCSR(B.nrows, B.ncols, B.rowptr, B.colidx, B.vals.astype(dtype))
    rowptr, colidx, vals, info = run_gpu(A, B)
    assert info[rows_key] >= 0.9 * A.nrows  # a few rows cover a narrower range
    assert_matches_oracle(A, B, rowptr, colidx, vals)


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("ncols", [1100, 40_000])
def test_dense_rows_of_short_b_rows(ncols, dtype):
    """Dense heavy rows over B rows of 0 to 99 entries: every length around the lane groups of the numeric pass, in
    one window and in several."""
    rng = np.random.default_rng(62)
    k = 2600
    rows = {i: rng.choice(ncols, size=min(i % 20 if i % 5 else i % 100, ncols), replace=False) for i in range(k)}
    B = _csr(k, ncols, rows, dtype=dtype)
    B.vals = (2 * rng.random(B.nnz) - 1).astype(dtype)
    A = _csr(12, k, {i: rng.choice(k, size=(600, 257, 256, 2000)[i % 4], replace=False) for i in range(12)}, dtype=dtype)
    A.vals = (2 * rng.random(A.nnz) - 1).astype(dtype)
    rowptr, colidx, vals, info = run_gpu(A, B)
    assert info["rcd_rows"] >= 6
    assert_matches_oracle(A, B, rowptr, colidx, vals)


def _changed_columns_case(kind):
    """(A, B, other columns of B that are valid but leave the range of the rows of A*B)."""
    rng = np.random.default_rng(52)
    if kind == "bitmap":  # 20 entries of 20 over 400 columns: crowded rows; a shift would keep the counts
        A, B, ncols = uniform_csr(200, 300, 20, rng), uniform_csr(300, 400, 20, rng), 70_000
        other = rng.permutation(ncols)[B.colidx]
    elif kind == "dense":  # 5000 products over 30,000 columns, rows for three batches
        A, B, ncols = _drawn_csr(2100, 3000, 250, rng), uniform_csr(3000, 30_000, 20, rng), 200_000
        other = B.colidx + 150_000
    else:  # "wide": 5000 products over 100,000 columns
        A, B, ncols = _drawn_csr(40, 3000, 250, rng), uniform_csr(3000, 100_000, 20, rng), 1 << 21
        other = B.colidx + 1_500_000
    return A, HostCSR(B.nrows, ncols, B.rowptr, B.colidx, B.vals), other.astype(np.int32)


def _check_changed_columns(kind, rows_key):
    from paper_2606_20855_gb300.spgemm import DeviceCSR, SpGEMM
    A, B, other = _changed_columns_case(kind)
    dB = DeviceCSR.from_host(B)
    with SpGEMM(DeviceCSR.from_host(A), dB) as op:
        op.symbolic()
        assert op.plan_info()[rows_key] == A.nrows
        dB.colidx.copy_(torch.from_numpy(other))
        op.numeric()
        with pytest.raises(_abi.WsError, match="WS_ERR_DEVICE"):
            op.wait()
        dB.colidx.copy_(torch.from_numpy(B.colidx))
        op.symbolic()
        C = op.numeric()
        op.wait()
        assert_matches_oracle(A, B, *C.to_host(), rows=np.arange(0, A.nrows, 7))


@pytest.mark.parametrize("kind,rows_key", [("wide", "wb_rows"), ("dense", "rcd_rows")])
def test_columns_changed_before_bitmaps_are_made_again(kind, rows_key):
    with tuning(kept_bytes=0):
        _check_changed_columns(kind, rows_key)


@pytest.mark.parametrize("kind,rows_key", [("bitmap", "bitmap_rows"), ("wide", "wb_rows")])
def test_columns_changed_between_the_passes(kind, rows_key):
    """Columns that leave a row's range after the symbolic pass touch nothing outside its workspace; the error is
    reported and the handle stays usable."""
    _check_changed_columns(kind, rows_key)


def test_cancellation_keeps_structural_zero():
    A = _csr(1, 2, {0: [0, 1]}, vals=[1.0, -1.0])
    B = _csr(2, 3, {0: [0, 2], 1: [0, 1]}, vals=[2.0, 5.0, 2.0, 3.0])
    rowptr, colidx, vals, _ = run_gpu(A, B)
    assert rowptr.tolist() == [0, 3]
    assert colidx.tolist() == [0, 1, 2]
    assert vals.tolist() == [0.0, -3.0, 5.0]


def test_handle_reuse_and_growth():
    """One SpGEMM object re-run, then a second, larger product: scratch grows, results stay exact."""
    from paper_2606_20855_gb300.spgemm import DeviceCSR, SpGEMM
    rng = np.random.default_rng(18)
    A = uniform_csr(1000, 700, 5, rng)
    B = uniform_csr(700, 900, 7, rng)
    dA, dB = DeviceCSR.from_host(A), DeviceCSR.from_host(B)
    with SpGEMM(dA, dB) as op:
        outs = []
        for _ in range(3):
            op.symbolic()
            C = op.numeric()
            op.wait()
            outs.append(C.to_host())
    for o in outs[1:]:
        for a, b in zip(outs[0][:2], o[:2]):
            np.testing.assert_array_equal(a, b)
    assert_matches_oracle(A, B, *outs[-1])
    A2 = uniform_csr(30_000, 700, 9, rng)
    rowptr, colidx, vals, _ = run_gpu(A2, B)
    assert_matches_oracle(A2, B, rowptr, colidx, vals)


@pytest.mark.parametrize("dtype", DTYPES)
@pytest.mark.parametrize("shift", [0, 1, 3])
def test_output_arrays_at_any_alignment(dtype, shift):
    """C's column and value arrays given at an offset of `shift` elements (not
    16-byte aligned unless shift is 0): the register-bitmap rows, copied out
    in 16-byte groups when both arrays are aligned, must give the same C."""
    from paper_2606_20855_gb300.spgemm import DeviceCSR, SpGEMM
    rng = np.random.default_rng(35)
    A = uniform_csr(5000, 3000, 12, rng, dtype, "sym")   # 12 entries per row
    B = uniform_csr(3000, 40_000, 30, rng, dtype, "sym")  # 30 per row: 32-lane groups, ~360 entries per C row
    dA, dB = DeviceCSR.from_host(A), DeviceCSR.from_host(B)
    tdt = torch.float32 if dtype == np.float32 else torch.float64
    with SpGEMM(dA, dB) as op:
        nnz = op.symbolic()
        ci = torch.empty(nnz + shift, dtype=torch.int32, device="cuda")[shift:]
        cv = torch.empty(nnz + shift, dtype=tdt, device="cuda")[shift:]
        C = op.numeric(out=DeviceCSR(A.nrows, B.ncols, op.c_rowptr, ci, cv))
        op.wait()
        info = op.plan_info()
        rowptr, colidx, vals = C.to_host()
    assert info["bitmap_rows"] == A.nrows
    assert_matches_oracle(A, B, rowptr, colidx, vals)


def test_many_live_handles():
    """More live products than one block of recycled pinned summaries (64):
    each of 150 open SpGEMM objects keeps its own summary and result, and
    closing them returns the blocks for the next 150."""
    from paper_2606_20855_gb300.spgemm import DeviceCSR, SpGEMM
    rng = np.random.default_rng(19)
    A = uniform_csr(300, 200, 4, rng)
    B = uniform_csr(200, 250, 5, rng)
    dA, dB = DeviceCSR.from_host(A), DeviceCSR.from_host(B)
    ref = None
    for _ in range(2):
        ops = [SpGEMM(dA, dB) for _ in range(150)]
        nnzs = [op.symbolic() for op in ops]
        outs = [op.numeric() for op in ops]
        for op in ops:
            op.wait()
        assert len(set(nnzs)) == 1
        hosts = [C.to_host() for C in outs]
        for op in ops:
            op.close()
        for h in hosts[1:]:  # structure is unique; values may differ in rounding (atomic order)
            for a, b in zip(hosts[0][:2], h[:2]):
                np.testing.assert_array_equal(a, b)
        assert_matches_oracle(A, B, *hosts[-1])
        if ref is None:
            ref = hosts[0]
        for a, b in zip(ref[:2], hosts[0][:2]):
            np.testing.assert_array_equal(a, b)


def _mixed_rows(seed):
    """A product with rows of many classes: several kernels per pass."""
    rng = np.random.default_rng(seed)
    k, n = 3000, 70_000
    B = uniform_csr(k, n, 40, rng, np.float64, "sym")
    lens = [0, 1, 2, 3, 5, 9, 17, 33, 65, 100, 150, 400, 1000, 2000]
    rows = {i: rng.choice(k, size=L, replace=False).tolist() for i, L in enumerate(lens * 6)}
    A = _csr(len(lens) * 6, k, rows)
    A.vals = 2 * rng.random(A.nnz) - 1
    return A, B


def test_products_on_threads_and_streams():
    """Four threads, each with its own stream, handles and inputs, twenty
    products each: the kernels of a pass spread over recycled side streams and
    every product still sees its own order of work."""
    import threading
    from paper_2606_20855_gb300.spgemm import DeviceCSR, SpGEMM
    cases = [_mixed_rows(s) for s in range(4)]
    results, errors = [None] * 4, []

    def work(i):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                dA, dB = DeviceCSR.from_host(cases[i][0]), DeviceCSR.from_host(cases[i][1])
                with SpGEMM(dA, dB) as op:
                    for _ in range(20):
                        op.symbolic()
                        C = op.numeric()
                        op.wait()
                        results[i] = C.to_host()
        except Exception as e:  # reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for (A, B), (rowptr, colidx, vals) in zip(cases, results):
        assert_matches_oracle(A, B, rowptr, colidx, vals)


def test_numeric_pass_under_capture():
    """The numeric pass of a product with several row classes captured in a
    graph and replayed with other values (captured work stays on the caller's
    stream)."""
    from paper_2606_20855_gb300.spgemm import DeviceCSR, SpGEMM
    A, B = _mixed_rows(9)
    dA, dB = DeviceCSR.from_host(A), DeviceCSR.from_host(B)
    with SpGEMM(dA, dB) as op:
        op.symbolic()
        C = op.numeric()
        op.wait()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            op.numeric(out=C)
        A.vals *= -0.5
        dA.vals.copy_(torch.from_numpy(A.vals))
        C.vals.zero_()
        graph.replay()
        op.wait()
        rowptr, colidx, vals = C.to_host()
    assert_matches_oracle(A, B, rowptr, colidx, vals)


def test_one_shot_calls_reuse_scratch_of_any_kind():
    """One-shot products, elementwise operations, extractions and SpMSpV in
    turn, on two streams: the scratch of a destroyed handle serves the next
    handle, whatever its operation, and leaves no trace in results or counts."""
    from oracle import oracle_ewise, oracle_spmspv
    from paper_2606_20855_gb300.spgemm import DeviceCSR, SpGEMM, ewise, spgemm, spmspv, submatrix
    from synth import sparse_vector, transpose_csr
    rng = np.random.default_rng(51)
    M, N = _mixed_rows(3)
    A = random_csr(300, 280, 0.05, rng, np.float64, "sym")
    B = random_csr(300, 280, 0.06, rng, np.float64, "sym")
    S = uniform_csr(200, 280, 6, rng)
    xi, xv = sparse_vector(280, 0.2, rng, np.float64, "sym")
    ref_y, ref_add = oracle_spmspv(A, xi, xv), oracle_ewise(A, B, "add")
    put = DeviceCSR.from_host
    dM, dN, dA, dB, dS, dT = put(M), put(N), put(A), put(B), put(S), put(transpose_csr(S))
    dAt = put(transpose_csr(A))
    dxi, dxv = torch.from_numpy(xi).cuda(), torch.from_numpy(xv).cuda()
    for stream in [torch.cuda.current_stream(), torch.cuda.Stream()] * 2:
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            C = spgemm(dM, dN)
            y, yv = spmspv(dAt, dxi, dxv)
            D = ewise(dA, dB, "add")
            E = submatrix(dA, 10, 200, 5, 250)
            F = spgemm(dS, dT, validate=True)
            with SpGEMM(dS, dT) as op:
                op.symbolic()
                info = op.plan_info()
            stream.synchronize()
        assert_matches_oracle(M, N, *C.to_host())
        assert_matches_oracle(S, transpose_csr(S), *F.to_host())
        np.testing.assert_array_equal(y.cpu().numpy(), ref_y.idx)
        np.testing.assert_allclose(yv.cpu().numpy(), ref_y.vals, rtol=0, atol=1e-12)
        for got, want in zip(D.to_host(), (ref_add.rowptr, ref_add.colidx, ref_add.vals)):
            np.testing.assert_array_equal(got, want)
        lens = np.diff(A.rowptr)
        keep = (A.colidx >= 5) & (A.colidx < 250) & (np.repeat(np.arange(300), lens) >= 10) & (np.repeat(np.arange(300), lens) < 200)
        np.testing.assert_array_equal(E.to_host()[1], A.colidx[keep] - 5)
        np.testing.assert_array_equal(E.to_host()[2], A.vals[keep])
        assert info["bitmap_rows"] + info["hash_rows"] + info["direct_rows"] + info["empty_rows"] == 200
        assert info["rcd_rows"] == info["wb_rows"] == info["dense_rows"] == 0


def test_device_count_check_reports_error():
    """A row pointer altered between the passes is caught by the numeric pass's count check."""
    from paper_2606_20855_gb300 import _abi
    from paper_2606_20855_gb300.spgemm import DeviceCSR, SpGEMM
    rng = np.random.default_rng(19)
    A = uniform_csr(256, 300, 6, rng)
    B = uniform_csr(300, 5000, 8, rng)
    with SpGEMM(DeviceCSR.from_host(A), DeviceCSR.from_host(B)) as op:
        nnz = op.symbolic()
        # move one entry from row 10 to row 11: every write stays inside [0, nnz)
        op.c_rowptr[11] -= 1
        C = op.numeric()
        with pytest.raises(_abi.WsError) as ei:
            op.wait()
        assert ei.value.status_name == "WS_ERR_DEVICE"
        assert C.nnz == nnz
        # the handle stays usable
        op.symbolic()
        C = op.numeric()
        op.wait()
        rowptr, colidx, vals = C.to_host()
    assert_matches_oracle(A, B, rowptr, colidx, vals)


def test_host_side_errors():
    from paper_2606_20855_gb300 import _abi
    from paper_2606_20855_gb300.spgemm import DeviceCSR, SpGEMM
    rng = np.random.default_rng(20)
    A = uniform_csr(10, 8, 3, rng)
    B = uniform_csr(9, 8, 3, rng)
    with pytest.raises(_abi.WsError) as ei:
        with SpGEMM(DeviceCSR.from_host(A), DeviceCSR.from_host(B)) as op:
            op.symbolic()
    assert ei.value.status_name == "WS_ERR_SHAPE"
    B32 = uniform_csr(8, 8, 3, rng, np.float32)
    with pytest.raises(TypeError):
        SpGEMM(DeviceCSR.from_host(A), DeviceCSR.from_host(B32))
    # invalid CSR: unsorted columns, duplicate, out of range, non-monotone rowptr
    good = uniform_csr(6, 10, 3, rng)
    bads = []
    b = HostCSR(6, 10, good.rowptr.copy(), good.colidx.copy(), good.vals.copy())
    b.colidx[0], b.colidx[1] = b.colidx[1], b.colidx[0]
    bads.append(b)
    b = HostCSR(6, 10, good.rowptr.copy(), good.colidx.copy(), good.vals.copy())
    b.colidx[4] = b.colidx[3]
    bads.append(b)
    b = HostCSR(6, 10, good.rowptr.copy(), good.colidx.copy(), good.vals.copy())
    b.colidx[-1] = 10
    bads.append(b)
    b = HostCSR(6, 10, good.rowptr.copy(), good.colidx.copy(), good.vals.copy())
    b.rowptr[2], b.rowptr[3] = b.rowptr[3], b.rowptr[2]
    bads.append(b)
    for bad in bads:
        with pytest.raises(_abi.WsError) as ei:
            SpGEMM(DeviceCSR.from_host(bad), DeviceCSR.from_host(uniform_csr(10, 4, 2, rng)), validate=True)
        assert ei.value.status_name == "WS_ERR_INVALID_CSR"
    # numeric before symbolic
    with SpGEMM(DeviceCSR.from_host(good), DeviceCSR.from_host(uniform_csr(10, 4, 2, rng))) as op:
        with pytest.raises(RuntimeError):
            op.numeric()
        h = op._hC
        with pytest.raises(_abi.WsError) as ei:
            _abi.ws_spgemm_numeric(op._hA, op._hB, h, 0, 0, torch.cuda.current_stream().cuda_stream)
        assert ei.value.status_name == "WS_ERR_STATE"
