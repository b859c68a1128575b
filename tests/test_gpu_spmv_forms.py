"""The default FP32 / BF16 products of matrices from 2^20 entries on, over the forms that
the mean row length and the neighbourhood of a row's columns choose (32-bit columns, 16-bit
offsets, resident blocks) and the bases the offsets count from (blocks of 64 entries, units
of 8): the column format is worked out here from the stored layout, every product must have
the bits of the 32-bit path (a slice of the rows, too small for the others), and the
products that several right-hand sides share the bits of the single ones."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2409_05239_gb300 import build, lslu

pytestmark = pytest.mark.gpu

MIN_ENTRIES = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def built():
    build.build()


def matrix(kind, mean, seed=1):
    """CSR with rows of mean/2 .. 3 mean/2 sorted, distinct columns: neighbours in pairs
    (2 columns, then a gap), evenly spread, or anywhere."""
    rng = np.random.default_rng(seed)
    m = 1_300_000 // mean
    lens = rng.integers(mean // 2, mean + mean // 2 + 1, m)
    lens[:3] = lens[-3:] = 0
    spacing, n = {"pairs": (16, 20_000), "pairs wide": (2400, 1_000_000), "even": (8, 20_000),
                  "even wide": (1200, 1_000_000), "anywhere": (None, 60_000),
                  "anywhere wide": (None, 6_000_000)}[kind]
    rows = []
    for L in lens:
        if spacing is None:
            rows.append(np.sort(rng.choice(n, L, replace=False)) if L else np.zeros(0, int))
            continue
        e = np.arange(L)
        c = e // 2 * spacing + e % 2 if kind.startswith("pairs") else e * spacing
        rows.append(c + 8 * rng.integers(0, max(1, (n - 1 - (c[-1] if L else 0)) // 8)))
    ptr = np.zeros(m + 1, np.int64)
    np.cumsum(lens, out=ptr[1:])
    cols = np.concatenate(rows).astype(np.int32)
    assert cols.max() < n
    return m, n, ptr, cols, rng.uniform(-1, 1, ptr[-1])


def spans(ptr, cols):
    """Largest column span of a stored 64-entry block and of a stored 8-entry unit (full
    blocks are stored transposed, 4 x 16)."""
    block = unit = 0
    for a, b in zip(ptr[:-1], ptr[1:]):
        if a == b:
            continue
        c = np.concatenate([cols[a:b], np.full(-(b - a) % 8, cols[b - 1])]).astype(np.int64)
        full = len(c) // 64 * 64
        if full:
            c[:full] = c[:full].reshape(-1, 4, 16).transpose(0, 2, 1).ravel()
            block = max(block, int(np.ptp(c[:full].reshape(-1, 64), axis=1).max()))
        if len(c) > full:
            block = max(block, int(np.ptp(c[full:])))
        unit = max(unit, int(np.ptp(c.reshape(-1, 8), axis=1).max()))
    return block, unit


CASES = [(kind, mean, fmt) for mean in (40, 80, 300) for kind, fmt in
         (("pairs", "block"), ("pairs wide", "unit"), ("even", "block"), ("even wide", "unit"),
          ("anywhere", "block"), ("anywhere wide", "none"))
         # (a short row of a wide matrix fits in one block)
         if not (mean == 40 and fmt == "unit")]


@pytest.mark.parametrize("vt", ["f32", "bf16"])
@pytest.mark.parametrize("kind,mean,fmt", CASES)
def test_products(vt, kind, mean, fmt):
    import torch

    m, n, ptr, cols, vals = matrix(kind, mean)
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
    A = sp.csr_matrix((stored.double().numpy(), cols, ptr), shape=(m, n))
    for M, v, y in ((A, x, u), (A.T.tocsr(), d, q)):
        v = v.astype(np.float64)
        bound = (np.diff(M.indptr) + 2) * 2.0 ** -24 * (abs(M) @ np.abs(v))
        assert np.all(np.abs(y - M @ v) <= bound)


@pytest.mark.parametrize("nrhs", [3, 7, 16])
@pytest.mark.parametrize("kind,mean", [("pairs", 300), ("pairs wide", 300), ("even wide", 80),
                                       ("anywhere wide", 300)])
def test_shared_products(kind, mean, nrhs):
    """Four, eight and sixteen interleaved right-hand sides on large matrices: each solve has
    the bits of its own."""
    m, n, ptr, cols, vals = matrix(kind, mean)
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
