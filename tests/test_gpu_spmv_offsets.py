"""The default FP32 / BF16 products on large matrices (one MiB of entries up) read 16-bit
column offsets from block or unit bases where the columns allow, in the chunks of the
32-bit format.  Spreading the columns of one matrix keeps the order of every row, so all
three formats, and the small matrices' 32-bit path on a slice of the rows, must give the
same bits; the sums are checked against scipy within the rounding bound of a recursive
sum."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2409_05239_gb300 import lslu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2409_05239_gb300 import build

    build.build()


def rows_of(lens, n, rng):
    """Sorted columns per row, in runs of neighbours with gaps between them."""
    ptr = np.zeros(len(lens) + 1, np.int64)
    np.cumsum(lens, out=ptr[1:])
    cols = np.concatenate([np.sort(rng.choice(n, L, replace=False)) for L in lens if L])
    return ptr, cols.astype(np.int32)


def products(ptr, cols, vals, n, vt, x, d):
    import torch

    s = lslu.Solver(len(ptr) - 1, n, ptr, cols, vals, vt, 4)
    try:
        u = torch.full((len(ptr) - 1,), 7.0, dtype=torch.float32, device="cuda")
        q = torch.full((n,), 7.0, dtype=torch.float32, device="cuda")
        s.spmv(0, torch.from_numpy(x).cuda(), u)
        s.spmv(1, torch.from_numpy(d).cuda(), q)
        torch.cuda.synchronize()
        return u.cpu().numpy(), q.cpu().numpy(), s.spmv_config()
    finally:
        s.close()


@pytest.mark.parametrize("vt", ["f32", "bf16"])
@pytest.mark.parametrize("rows,mean", [(19999, 60), (4099, 300)])
def test_formats_give_the_same_bits(vt, rows, mean):
    rng = np.random.default_rng(rows)
    n = 3001
    lens = rng.integers(0, 2 * mean, size=rows)
    lens[rng.random(rows) < 0.05] = 0
    lens[:3] = lens[-5:] = 0
    ptr, cols = rows_of(lens, n, rng)
    assert ptr[-1] >= 1 << 20
    vals = rng.uniform(-1.0, 1.0, ptr[-1])
    x = rng.standard_normal(n).astype(np.float32)
    d = rng.standard_normal(rows).astype(np.float32)
    u, q, cfg = products(ptr, cols, vals, n, vt, x, d)
    assert cfg["shape_A"] == "16x2" and cfg["compressed_A"]
    # the same rows with their columns spread: blocks, then units, span 2^16 columns or more
    for spread in (80, 8000):
        ns = (n - 1) * spread + 1
        xs = np.zeros(ns, np.float32)
        xs[::spread] = x
        us, qs, _ = products(ptr, cols * spread, vals, ns, vt, xs, d)
        assert np.array_equal(u, us) and np.array_equal(q, qs[::spread])
    # the first rows alone: a small matrix, on 32-bit columns
    part = int(np.searchsorted(ptr, 1 << 19))
    up, _, _ = products(ptr[:part + 1], cols[:ptr[part]], vals[:ptr[part]], n, vt, x, d[:part])
    assert np.array_equal(u[:part], up)
    stored = vals.astype(np.float32)
    if vt == "bf16":
        import torch

        stored = torch.from_numpy(stored).to(torch.bfloat16).float().numpy()
    A = sp.csr_matrix((stored.astype(np.float64), cols, ptr), shape=(rows, n))
    for M, v, y in ((A, x, u), (A.T.tocsr(), d, q)):
        bound = (np.diff(M.indptr) + 2) * 2.0 ** -24 * (abs(M) @ np.abs(v.astype(np.float64)))
        assert np.all(np.abs(y - M @ v.astype(np.float64)) <= bound)
