"""The cluster loop while other work holds most of the GPU: its CTAs then start at uneven
times, and the first thing they do is to store pivot keys into each other's shared memory.
The order of every sum is fixed, so each solve must give the bits of one on an idle GPU."""
import numpy as np
import pytest

from paper_2409_05239_gb300 import build, lslu, tomo

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vt", ["f64", "f32"])
def test_cluster_solves_beside_other_kernels(vt):
    import torch

    build.build()
    P = tomo.make_config("ct32")
    K = 8
    a = torch.randn(4096, 4096, device="cuda")
    side = torch.cuda.Stream()
    with lslu.from_problem(P, vt, K) as s:
        s.set_loop("cluster")
        torch.cuda.synchronize()
        ref = s.solve(P.b, K, "gcv")
        for _ in range(20):
            with torch.cuda.stream(side):
                for _ in range(4):
                    a @ a
            r = s.solve(P.b, K, "gcv")
            assert np.array_equal(r["gp"], ref["gp"]) and np.array_equal(r["tp"], ref["tp"])
            assert np.array_equal(r["x"], ref["x"])
    torch.cuda.synchronize()
