"""A handle on a stream that does not wait for the legacy default stream, created, solved
and differentiated while that one is busy: everything a handle zeroes is zeroed on its own
stream, so its results are those of a handle on the default stream."""
import numpy as np
import pytest

from paper_2409_05239_gb300 import build, lslu, tomo

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("loop", ["graph", "persistent"])
def test_handle_beside_a_busy_default_stream(loop):
    import torch

    build.build()
    P = tomo.make_config("ct32")
    K = 10

    def run(stream):
        with lslu.Solver(P.m, P.n, P.row_ptr, P.col_idx, P.vals, "f64", K, stream=stream) as s:
            s.set_loop(loop)
            r = s.solve(P.b, K, "fixed", 0.5, histories=True)
            st = s.state(K)
            s.set_loop("graph")
            s.solve(P.b, K, "fixed", 0.5)
            return r, st, s.adjoint(np.ones(P.n))

    ref, ref_state, ref_adjoint = run(None)
    side = torch.cuda.Stream()
    for _ in range(3):
        torch.cuda.synchronize()
        torch.cuda._sleep(50_000_000)
        r, st, ad = run(side.cuda_stream)
        torch.cuda.synchronize()
        assert np.array_equal(r["gp"], ref["gp"]) and np.array_equal(r["x"], ref["x"])
        assert np.array_equal(r["res_hist"], ref["res_hist"])
        for k in ("H", "W", "L", "D"):
            assert np.array_equal(st[k], ref_state[k]), k
        for k in ref_adjoint:
            assert np.array_equal(ad[k], ref_adjoint[k]), k
