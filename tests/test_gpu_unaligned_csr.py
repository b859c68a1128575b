"""Device CSR arrays that do not start on a multiple of their element size: a copy takes
them from any address, a kernel does not, so such a handle is built from host copies and
must give the bits of one built from aligned arrays."""
import ctypes

import numpy as np
import pytest

from paper_2409_05239_gb300 import build, lslu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    build.build()


def on_gpu(a, shift):
    """(keep-alive, address) of a's bytes on the GPU, `shift` bytes off an aligned address."""
    import torch

    raw = torch.empty(a.nbytes + 16, dtype=torch.uint8, device="cuda")
    raw[shift:shift + a.nbytes] = torch.from_numpy(a.view(np.uint8)).cuda()
    return raw, raw.data_ptr() + shift


def csr(m, n, seed):
    rng = np.random.default_rng(seed)
    lens = rng.integers(0, 30, m)
    ptr = np.zeros(m + 1, np.int64)
    np.cumsum(lens, out=ptr[1:])
    return ptr, rng.integers(0, n, ptr[-1]).astype(np.int32), rng.uniform(-1, 1, ptr[-1])


def create(m, n, arrays, shifts, ordered):
    lib, held = lslu.load(), [on_gpu(a, s) for a, s in zip(arrays, shifts)]
    nnz, h = int(arrays[0][-1]), ctypes.c_void_p()
    p = [ctypes.c_void_p(a) for _, a in held]
    if ordered:
        st = lib.lslu_create_ordered(m, n, nnz, p[0], p[1], p[2], lslu.VALUE_TYPES["f64"], 6, p[3],
                                     p[4], lslu.DEVICE, None, ctypes.byref(h))
    else:
        st = lib.lslu_create(m, n, nnz, p[0], p[1], p[2], lslu.VALUE_TYPES["f64"], 6, lslu.DEVICE,
                             None, ctypes.byref(h))
    return lib, st, h


@pytest.mark.parametrize("ordered", [False, True])
@pytest.mark.parametrize("shifts", [(0, 2, 0, 0, 0), (0, 0, 4, 0, 0), (8, 1, 1, 2, 3)])
def test_unaligned_device_arrays(shifts, ordered):
    m, n, K = 700, 500, 5
    rng = np.random.default_rng(9)
    orders = [rng.permutation(m).astype(np.int32), rng.permutation(n).astype(np.int32)]
    arrays = (*csr(m, n, 4), *orders)
    b = rng.standard_normal(m)
    out = []
    for sh in ((0,) * 5, shifts):
        lib, st, h = create(m, n, arrays, sh, ordered)
        assert st == lslu.OK
        x, kd = np.zeros(n), ctypes.c_int32()
        st = lib.lslu_solve(h, b.ctypes.data, None, K, lslu.RULES["fixed"], 0.1, lslu.HOST,
                            x.ctypes.data, None, None, None, None, ctypes.addressof(kd))
        lib.lslu_destroy(h)
        assert st == lslu.OK and kd.value == K
        out.append(x)
    assert np.array_equal(out[0], out[1]) and np.any(out[0])


def test_unaligned_invalid_arrays_are_refused():
    m, n = 700, 500
    ptr, cols, vals = csr(m, n, 4)
    for at, column, value in ((7, n, 1.0), (11, -1, 1.0), (3, 0, np.inf), (9, 1, np.nan)):
        c, v = cols.copy(), vals.copy()
        c[at], v[at] = column, value
        _, st, _ = create(m, n, (ptr, c, v), (0, 1, 1), False)
        assert st == lslu.ERR_INVALID_ARG
