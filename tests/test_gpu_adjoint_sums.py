"""The adjoint's sums over the blocks' partials, taken by threads or by warps depending on
the number of blocks and of sums: with the pivots fixed, x(b) is linear in b at a fixed
lambda, so b_bar . b = x_bar . x.  FP64 sums of a few hundred terms through triangular
factors with entries up to one keep eight digits of the vectors' sizes with room to spare."""
import numpy as np
import pytest

from paper_2409_05239_gb300 import build, lslu, tomo

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side,angles,rays", [(12, 10, 17), (24, 30, 34), (64, 90, 90)])
@pytest.mark.parametrize("K", [1, 2, 8, 9, 33, 60])
def test_linear_in_b(side, angles, rays, K):
    build.build()
    P = tomo.make_problem(side, angles, rays, 3, 0.01, 5)
    with lslu.from_problem(P, "f64", K) as s:
        r = s.solve(P.b, K, "fixed", 0.5)
        assert r["status"] == lslu.OK
        x_bar = np.random.default_rng(K).standard_normal(P.n)
        b_bar = s.adjoint(x_bar)["b_bar"]
    assert np.any(b_bar)
    assert abs(b_bar @ P.b - x_bar @ r["x"]) <= 1e-8 * np.linalg.norm(b_bar) * np.linalg.norm(P.b)
