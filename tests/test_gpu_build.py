"""The stored matrices built on the device from host and device CSRs: products of A and A^T
against scipy on rows with unsorted and repeated columns, empty rows and columns, one dense
row and one dense column longer than a block sorts (kSortMax = 8192: the host's sort), the
same bits for host and device arrays, renumbered handles against natural ones, and the
refusals of invalid device arrays."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2409_05239_gb300 import lslu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2409_05239_gb300 import build

    build.build()


def matrix(m, n, mean, dense_row, dense_col, seed):
    """CSR arrays with unsorted, repeated columns."""
    rng = np.random.default_rng(seed)
    lens = rng.integers(0, 2 * mean + 1, m)
    lens[rng.random(m) < 0.1] = 0
    rows = [rng.integers(0, n, L) for L in lens]
    if dense_row:
        rows[m // 2] = rng.permutation(n)
    if dense_col:
        rows = [np.append(r, n // 3) for r in rows]
    ptr = np.zeros(m + 1, np.int64)
    np.cumsum([len(r) for r in rows], out=ptr[1:])
    cols = np.concatenate(rows).astype(np.int32)
    return ptr, cols, rng.uniform(-1.0, 1.0, ptr[-1])


SHAPES = [(300, 257, 20, False, False), (9001, 700, 3, False, True), (500, 9001, 6, True, False),
          (9003, 8999, 2, True, True), (64, 4096, 150, True, False), (1, 1, 1, True, False)]


@pytest.mark.parametrize("vt", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("m,n,mean,dense_row,dense_col", SHAPES)
def test_products(vt, m, n, mean, dense_row, dense_col):
    import torch

    ptr, cols, vals = matrix(m, n, mean, dense_row, dense_col, seed=m)
    dt = torch.float64 if vt == "f64" else torch.float32
    stored = torch.from_numpy(vals)
    if vt != "f64":
        stored = stored.float().to(torch.float32 if vt == "f32" else torch.bfloat16).double()
    A = sp.csr_matrix((stored.numpy(), cols, ptr), shape=(m, n))  # repeats stay repeats
    rng = np.random.default_rng(1)
    x = torch.from_numpy(rng.standard_normal(n)).to(dt)
    d = torch.from_numpy(rng.standard_normal(m)).to(dt)
    got = []
    for device in (False, True):
        arrays = [torch.from_numpy(a).cuda() for a in (ptr, cols, vals)] if device else (
            ptr, cols, vals)
        s = lslu.Solver(m, n, *arrays, value_type=vt, max_iter=2)
        u = torch.full((m,), 3.0, dtype=dt, device="cuda")
        q = torch.full((n,), 3.0, dtype=dt, device="cuda")
        s.spmv(0, x.cuda(), u)
        s.spmv(1, d.cuda(), q)
        torch.cuda.synchronize()
        s.close()
        got.append((u.cpu().double().numpy(), q.cpu().double().numpy()))
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
    eps = 2.0 ** -53 if vt == "f64" else 2.0 ** -24
    for M, v, y in ((A, x, got[0][0]), (A.T.tocsr(), d, got[0][1])):
        v = v.double().numpy()
        bound = (np.diff(M.indptr) + 2) * eps * (abs(M) @ np.abs(v))
        assert np.all(np.abs(y - M @ v) <= bound)


@pytest.mark.parametrize("dense", [False, True])
def test_renumbered_handle(dense):
    """Renumbered handles of host and device arrays solve as the natural one does
    (FP64, a few iterations; the dense row and column take the host's sorts)."""
    import torch

    m, n, K = (9003, 8999, 3) if dense else (700, 400, 4)
    ptr, cols, vals = matrix(m, n, 6, dense, dense, seed=5)
    rng = np.random.default_rng(2)
    b = rng.standard_normal(m)
    ro, co = rng.permutation(m).astype(np.int32), rng.permutation(n).astype(np.int32)
    with lslu.Solver(m, n, ptr, cols, vals, "f64", K) as s:
        ref = s.solve(b, K, "fixed", 0.1)
    for device in (False, True):
        arrays = (ptr, cols, vals, ro, co)
        if device:
            arrays = [torch.from_numpy(a).cuda() for a in arrays]
        with lslu.Solver(m, n, *arrays[:3], value_type="f64", max_iter=K, row_order=arrays[3],
                         col_order=arrays[4]) as s:
            r = s.solve(b, K, "fixed", 0.1)
        assert np.array_equal(r["gp"], ref["gp"]) and np.array_equal(r["tp"], ref["tp"])
        assert np.linalg.norm(r["x"] - ref["x"]) <= 1e-10 * np.linalg.norm(ref["x"])


def test_invalid_device_arrays_are_refused():
    import torch

    ptr, cols, vals = matrix(50, 40, 5, False, False, seed=3)
    for at, column, value, what in ((7, 40, 1.0, "column index"), (11, -1, 1.0, "column index"),
                                    (3, 0, np.inf, "non-finite"), (9, 1, np.nan, "non-finite")):
        c, v = cols.copy(), vals.copy()
        c[at], v[at] = column, value
        with pytest.raises(lslu.LsluError, match=what):
            lslu.Solver(50, 40, *[torch.from_numpy(a).cuda() for a in (ptr, c, v)], "f32", 4)
