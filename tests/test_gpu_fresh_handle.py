"""A handle's results do not depend on what its device memory held before: device memory
comes back from cudaMalloc as its last owner left it, and the projected solve reads the
entries of H below the subdiagonal, which no basis loop writes."""
import ctypes

import numpy as np
import pytest

import oracle.lslu_oracle as O
from paper_2409_05239_gb300 import lslu, tomo

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2409_05239_gb300 import build

    build.build()


def dirty_free_memory():
    """Fill freed device memory, in blocks of every size the driver carves out of its
    pools, with bytes 0x40 (doubles of about 32.5)."""
    lib, held = lslu.load(), []
    for log2_size, count in ((21, 16), (20, 32), (18, 32), (16, 64), (14, 64), (12, 128), (9, 256)):
        for _ in range(count):
            p = ctypes.c_void_p()
            if lib.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(1 << log2_size)) == 0:
                lib.cudaMemset(p, 0x40, ctypes.c_size_t(1 << log2_size))
                held.append(p)
    for p in held:
        assert lib.cudaFree(p) == 0


@pytest.mark.parametrize("loop", ["graph", "persistent", "cluster"])
def test_solve_on_dirty_memory(loop):
    P = tomo.make_config("ct32")
    K = 12
    ref = O.hybrid_lslu(P.scipy(), P.b, None, K, "gcv")
    dirty_free_memory()
    with lslu.from_problem(P, "f64", max_iter=K) as s:
        s.set_loop(loop)
        r = s.solve(P.b, K, "gcv")
        H = s.state(K)["H"]
    assert np.array_equal(r["gp"], ref.gp)
    assert np.linalg.norm(r["x"] - ref.x) <= 1e-10 * np.linalg.norm(ref.x)
    assert not np.any(np.tril(H, -2))


def test_batch_on_dirty_memory():
    Ps = [tomo.make_problem(24, 36, 34, 3, 0.01, 11), tomo.make_problem(20, 30, 29, 3, 0.01, 12)]
    K = 8
    dirty_free_memory()
    with lslu.from_problems(Ps, "f32", max_iter=K) as s:
        r = s.solve(np.concatenate([P.b for P in Ps]), K, "gcv")
    for P, x in zip(Ps, r["x"]):
        A = P.scipy(tomo.round_values(P.vals, "f32"))
        ref = O.hybrid_lslu(A, P.b, None, K, "gcv")
        assert np.linalg.norm(x - ref.x) <= 2e-4 * np.linalg.norm(ref.x)
