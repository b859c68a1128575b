"""Creation where device memory is short: a handle needs little more than what it stores.
Device memory is taken until what is left holds the handle and a few bytes per entry, less
than the construction on the device wants for itself (8 bytes per entry, 20 from host
arrays), so the host's construction has to serve; the handle gives the same bits.  A handle
that does not fit at all is refused and leaves the library usable."""
import contextlib
import ctypes

import numpy as np
import pytest

from paper_2409_05239_gb300 import build, lslu

pytestmark = pytest.mark.gpu

M, N, K = 100_000, 70_000, 2


@pytest.fixture(scope="module")
def matrix():
    build.build()
    rng = np.random.default_rng(3)
    lens = rng.integers(0, 121, M)
    ptr = np.zeros(M + 1, np.int64)
    np.cumsum(lens, out=ptr[1:])
    cols = rng.integers(0, N, ptr[-1]).astype(np.int32)
    return ptr, cols, rng.uniform(-1, 1, ptr[-1])


@contextlib.contextmanager
def only_left(nbytes):
    """Hold all device memory but nbytes."""
    import torch

    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    lib, p = lslu.load(), ctypes.c_void_p()
    take = torch.cuda.mem_get_info()[0] - nbytes
    assert lib.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(take)) == 0
    try:
        yield
    finally:
        lib.cudaFree(p)


def products(s):
    import torch

    x = torch.linspace(-1, 1, N, dtype=torch.float32, device="cuda")
    d = torch.linspace(-2, 1, M, dtype=torch.float32, device="cuda")
    u, q = torch.empty(M, device="cuda"), torch.empty(N, device="cuda")
    s.spmv(0, x, u)
    s.spmv(1, d, q)
    return u.cpu().numpy(), q.cpu().numpy()


@pytest.mark.parametrize("device", [False, True])
def test_creation_beside_other_memory(matrix, device):
    import torch

    arrays = [torch.from_numpy(a).cuda() for a in matrix] if device else matrix
    nnz = int(matrix[0][-1])
    # the kernels loaded, the caching allocator's blocks given back, then the handle's size
    lslu.Solver(M, N, *arrays, value_type="f32", max_iter=K).close()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    with lslu.Solver(M, N, *arrays, value_type="f32", max_iter=K) as s:
        stored = free - torch.cuda.mem_get_info()[0]
        ref = products(s)
    assert stored >= 2 * 8 * nnz  # columns and values of both matrices
    for spare in (24 * nnz, 4 * nnz):
        with only_left(stored + spare):
            s = lslu.Solver(M, N, *arrays, value_type="f32", max_iter=K)
        with s:
            got = products(s)
        assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])


def test_handle_that_does_not_fit(matrix):
    nnz = int(matrix[0][-1])
    with lslu.Solver(M, N, *matrix, value_type="f32", max_iter=K) as s:
        ref = products(s)
        with only_left(10 * nnz):
            with pytest.raises(lslu.LsluError) as e:
                lslu.Solver(M, N, *matrix, value_type="f32", max_iter=K)
        assert e.value.status == lslu.ERR_OOM
        got = products(s)
    assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])
