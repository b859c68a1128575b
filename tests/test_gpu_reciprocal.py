"""The reflectors' FP64 reciprocal against exact values and CUDA's division, over the
arguments that a reflector hands it (2^-480 .. 2^482) and beyond: one step of Chebyshev's method from an
approximation of 2^-20 leaves at most 0.51 units of the last place, so a value differs from
the correctly rounded one by a unit at most.  And the projected solve on H scaled by powers
of two, up to and past the squares from which the reflectors divide instead (2^-959 and
2^960): sigma scales, y stays, within the bound of tests/test_gpu_projected_sizes.py."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2409_05239_gb300 import build, lslu, tomo
from tests.test_gpu_lambda_refine import synthetic_H

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "lslu_reciprocal.cuh"
__global__ void k(const double* d, double* own, double* cuda, long n) {
  const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  own[i] = lslu::reciprocal(d[i]);
  cuda[i] = 1.0 / d[i];
}
extern "C" int run(const double* d, double* own, double* cuda, long n) {
  k<<<(unsigned)((n + 255) / 256), 256>>>(d, own, cuda, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def reciprocals(tmp_path_factory):
    import torch

    build.build()
    d = tmp_path_factory.mktemp("reciprocal")
    (d / "r.cu").write_text(SOURCE)
    subprocess.run([build.nvcc_path(), *build.ARCH, "-O3", "-shared", "-Xcompiler", "-fPIC", "-I",
                    os.path.join(os.path.dirname(build.__file__), "csrc"), "-o", str(d / "r.so"),
                    str(d / "r.cu")], check=True)
    lib = ctypes.CDLL(str(d / "r.so"))

    def run(x):
        v = torch.from_numpy(x).cuda()
        own, cuda = torch.empty_like(v), torch.empty_like(v)
        torch.cuda.synchronize()
        assert lib.run(*[ctypes.c_void_p(t.data_ptr()) for t in (v, own, cuda)],
                       ctypes.c_long(len(x))) == 0
        return own.cpu().numpy(), cuda.cpu().numpy()

    return run


@pytest.mark.parametrize("lo,hi", [(-1, 1), (-60, 60), (-480, 482), (-1000, 1000)])
def test_reciprocal(reciprocals, lo, hi):
    rng = np.random.default_rng(hi)
    n = 1 << 20
    m = rng.integers(1 << 52, 1 << 53, n)
    m[:4096] = (1 << 52) + np.arange(4096)  # mantissas next to powers of two, on both sides
    m[4096:8192] = (1 << 53) - 1 - np.arange(4096)
    d = np.ldexp(m.astype(np.float64), rng.integers(lo, hi, n) - 52)
    own, cuda = reciprocals(d)
    exact = np.longdouble(1) / d.astype(np.longdouble)
    assert np.finfo(np.longdouble).nmant >= 63
    unit = np.spacing(cuda).astype(np.longdouble)
    assert np.max(np.abs(own - exact) / unit) <= 0.51
    assert np.max(np.abs(own - cuda) / np.spacing(cuda)) <= 1.0
    assert np.mean(own != cuda) <= 0.01


@pytest.mark.parametrize("k", [1, 5, 62, 63, 64, 90])
def test_scaled_projected_problem(k):
    rng = np.random.default_rng(k)
    sigma = 10.0 ** (-3.0 * np.arange(k) / max(k - 1, 1))
    c = rng.choice([-1.0, 1.0], k + 1) * rng.uniform(0.5, 1.0, k + 1)
    H, beta = synthetic_H(sigma, c, seed=k)
    tol = 10 * max(k, 10) * np.finfo(float).eps
    build.build()
    with lslu.from_problem(tomo.make_config("ct32"), "f64", 90) as s:
        ref = s.projected(H, beta, "fixed", 1e-2)
        assert np.max(np.abs(ref["sigma"] - sigma)) <= tol * sigma[0]
        # the squares of H's entries stay above 2^-1000 and below 2^1000
        for p in (-480, -100, -31, 31, 100, 480):
            f = 2.0 ** p
            out = s.projected(H * f, beta * f, "fixed", 1e-2 * f)
            assert np.max(np.abs(out["sigma"] / f - sigma)) <= tol * sigma[0], p
            assert np.linalg.norm(out["y"] - ref["y"]) <= tol * 1e3 * np.linalg.norm(ref["y"]), p
