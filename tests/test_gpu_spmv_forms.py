"""The default FP32 / BF16 products of matrices from 2^20 entries on, over the forms that
rows, row lengths and the neighbourhood of a row's columns choose (32-bit columns, 16-bit
offsets, resident blocks) and the bases the offsets count from (blocks of 64 entries, units
of 8): the column format is worked out here from the stored layout, every product must have
the bits of the 32-bit path (a slice of the rows, too small for the others), and the
products that several right-hand sides share the bits of the single ones."""
import functools

import numpy as np
import pytest
import scipy.sparse as sp

from paper_2409_05239_gb300 import build, lslu

pytestmark = pytest.mark.gpu

MIN_ENTRIES = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def built():
    build.build()


FEW, MANY = 4400, 46_000  # rows: below and above three waves of 912 blocks of 16


@functools.lru_cache(maxsize=1)
def matrix(kind, mean, rows, longest=0):
    """CSR with rows of mean/2 .. 3 mean/2 sorted columns: neighbours in pairs (2 columns,
    then a gap), evenly spread, or anywhere; one row of `longest` entries."""
    rng = np.random.default_rng(1)
    lens = rng.integers(mean // 2, mean + mean // 2 + 1, rows)
    lens[:3] = lens[-3:] = 0
    lens[rows // 3] = longest or mean
    ptr = np.zeros(rows + 1, np.int64)
    np.cumsum(lens, out=ptr[1:])
    row = np.repeat(np.arange(rows), lens)
    e = np.arange(ptr[-1]) - ptr[row]
    spacing, n = {"pairs": (16, 60_000), "pairs wide": (2400, 1_000_000), "even": (8, 60_000),
                  "even wide": (1200, 1_000_000), "anywhere": (None, 60_000),
                  "anywhere wide": (None, 6_000_000)}[kind]
    if spacing is None:
        cols = rng.integers(0, n, ptr[-1])
        cols = cols[np.lexsort((cols, row))]
    else:
        step = e // 2 * spacing + e % 2 if kind.startswith("pairs") else e * spacing
        room = n - 1 - (lens // 2 + 1) * spacing * (1 if kind.startswith("pairs") else 2)
        cols = step + (8 * (rng.random(rows) * np.maximum(room, 8) // 8).astype(int))[row]
    assert 0 <= cols.min() and cols.max() < n
    return rows, n, ptr, cols.astype(np.int32), rng.uniform(-1, 1, ptr[-1])


def spans(ptr, cols):
    """Largest column span of a stored 64-entry block and of a stored 8-entry unit (rows
    padded to 8 entries with their last column, full blocks stored transposed, 4 x 16)."""
    lens = np.diff(ptr)
    padded = (lens + 7) // 8 * 8
    at = np.concatenate([[0], np.cumsum(padded)])
    row = np.repeat(np.arange(len(lens)), padded)
    q = np.arange(at[-1]) - at[row]
    w = q % 64
    e = np.where(q // 64 < padded[row] // 64, q - w + 16 * (w % 4) + w // 4, q)
    stored = cols[ptr[row] + np.minimum(e, lens[row] - 1)].astype(np.int64)

    def widest(starts):
        return int((np.maximum.reduceat(stored, starts) - np.minimum.reduceat(stored, starts)).max())

    return widest(np.flatnonzero(q % 64 == 0)), widest(np.flatnonzero(q % 8 == 0))


CASES = [("pairs", 40, MANY, 0, "block"), ("anywhere", 40, MANY, 0, "block"),   # 32-bit columns
         ("pairs", 40, MANY, 3000, "block"),                                    # a long row
         ("pairs", 80, MANY, 0, "block"), ("pairs wide", 80, MANY, 0, "unit"),  # offsets
         ("even", 110, MANY, 0, "block"), ("even wide", 110, MANY, 0, "unit"),  # scattered
         ("anywhere", 110, MANY, 0, "block"),
         ("pairs", 110, MANY, 0, "block"), ("pairs wide", 110, MANY, 0, "unit"),  # resident
         ("pairs", 300, FEW, 0, "block"), ("even wide", 300, FEW, 0, "unit"),
         ("anywhere", 300, FEW, 0, "block"),
         ("anywhere wide", 110, MANY, 0, "none"), ("anywhere wide", 300, FEW, 0, "none")]


@pytest.mark.parametrize("kind,mean,rows,longest,fmt", CASES)
@pytest.mark.parametrize("vt", ["f32", "bf16"])
def test_products(vt, kind, mean, rows, longest, fmt):
    import torch

    m, n, ptr, cols, vals = matrix(kind, mean, rows, longest)
    assert ptr[-1] >= MIN_ENTRIES
    block, unit = spans(ptr, cols)
    assert (fmt == "block") == (block < 65536) and (fmt == "none") == (unit >= 65536)
    rng = np.random.default_rng(2)
    x = rng.standard_normal(n).astype(np.float32)
    d = rng.standard_normal(m).astype(np.float32)

    def products(ptr, cols, vals, d):
        rows = len(ptr) - 1
        u = torch.full((rows,), 7.0, device="cuda")
        q = torch.full((n,), 7.0, device="cuda")
        with lslu.Solver(rows, n, ptr, cols, vals, vt, 1) as s:
            s.spmv(0, torch.from_numpy(x).cuda(), u)
            s.spmv(1, torch.from_numpy(d).cuda(), q)
            return u.cpu().numpy(), q.cpu().numpy(), s.spmv_config()["compressed_A"]

    u, q, compressed = products(ptr, cols, vals, d)
    assert compressed == (fmt != "none")
    part = int(np.searchsorted(ptr, MIN_ENTRIES // 2))
    up, _, _ = products(ptr[:part + 1], cols[:ptr[part]], vals[:ptr[part]], d[:part])
    assert np.array_equal(u[:part], up)
    stored = torch.from_numpy(vals).float()
    if vt == "bf16":
        stored = stored.bfloat16().float()
    stored = stored.double().numpy()
    # (scipy's abs() would add up a row's repeated columns first)
    A, size = (sp.csr_matrix((a, cols, ptr), shape=(m, n)) for a in (stored, np.abs(stored)))
    for M, S, v, y in ((A, size, x, u), (A.T.tocsr(), size.T.tocsr(), d, q)):
        v = v.astype(np.float64)
        bound = (np.diff(M.indptr) + 2) * 2.0 ** -24 * (S @ np.abs(v))
        assert np.all(np.abs(y - M @ v) <= bound)


@pytest.mark.parametrize("nrhs", [3, 7, 16])
@pytest.mark.parametrize("kind,mean,rows", [("pairs", 300, FEW), ("pairs wide", 300, FEW),
                                            ("even wide", 80, MANY), ("anywhere wide", 300, FEW)])
def test_shared_products(kind, mean, rows, nrhs):
    """Four, eight and sixteen interleaved right-hand sides on large matrices: each solve has
    the bits of its own."""
    m, n, ptr, cols, vals = matrix(kind, mean, rows)
    K = 3
    b = np.random.default_rng(nrhs).standard_normal((nrhs, m))
    with lslu.BatchedSolver((m, n, ptr, cols, vals), "f32", K, nrhs=nrhs) as s:
        r = s.solve(b.ravel(), K, "fixed", 0.5)
    with lslu.Solver(m, n, ptr, cols, vals, "f32", K) as s:
        for p in range(nrhs):
            one = s.solve(b[p], K, "fixed", 0.5)
            assert r["status"][p] == one["status"] == lslu.OK
            assert np.array_equal(r["gp"][p], one["gp"]) and np.array_equal(r["tp"][p], one["tp"])
            assert np.array_equal(r["x"][p], one["x"]), p
