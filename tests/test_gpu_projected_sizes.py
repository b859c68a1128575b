"""The projected problem (lslu_projected) at the sizes where its kernels change their
split: groups of four right reflectors and 128 threads over y, 32 lanes over the Givens
sweep, 32 x 8 Sturm steps; against the oracle's SVD solution on H with a prescribed
spectrum (condition number 1e3), where a backward stable solve has y within about
10 k eps cond = 1e-9 at k = 513 and sigma within 10 k eps sigma_1."""
import numpy as np
import pytest

from oracle import lslu_oracle as O
from paper_2409_05239_gb300 import lslu, tomo
from tests.test_gpu_lambda_refine import synthetic_H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def handle():
    from paper_2409_05239_gb300 import build

    build.build()
    with lslu.from_problem(tomo.make_config("ct32"), "f64", 520) as s:
        yield s


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 31, 32, 33, 64, 127, 128, 129, 256, 257, 385, 513])
@pytest.mark.parametrize("rule,lam", [("none", 0.0), ("fixed", 1e-2), ("fixed", 2.0)])
def test_solution_at_size_edges(handle, k, rule, lam):
    rng = np.random.default_rng(k)
    sigma = 10.0 ** (-3.0 * np.arange(k) / max(k - 1, 1))
    c = rng.choice([-1.0, 1.0], k + 1) * rng.uniform(0.5, 1.0, k + 1)
    H, beta = synthetic_H(sigma, c, seed=k)
    s_ref, c_ref, V = O.projected_svd(H, beta)
    y_ref = O.tikhonov_y(s_ref, c_ref, V, lam)
    r_ref = O.projected_residual(s_ref, c_ref, lam)
    out = handle.projected(H, beta, rule, lam)
    tol = 10 * max(k, 10) * np.finfo(float).eps
    assert np.max(np.abs(out["sigma"] - s_ref)) <= tol * s_ref[0]
    assert np.linalg.norm(out["y"] - y_ref) <= tol * 1e3 * np.linalg.norm(y_ref)
    assert abs(out["resid"] - r_ref) <= tol * 1e3 * r_ref
