"""The tensor-core digit-splitting kernel over FP32 stores
against the CUDA-core kernels on the same handle.

Tolerance: the CUDA-core kernel rounds densities to FP32 and each 64-term brick
sum up to 64 times, the split kernel five times per sum: 70 * 2^-24 = 4.2e-6 of
the sum of the absolute terms, which for these normal densities is below ten
times the result: 4e-5.
"""
import numpy as np
import pytest

from paper_2002_00322_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = 4e-5


def build(fb, D):
    import torch
    got = [x.cpu().numpy() for x in fb.build(torch.from_numpy(np.ascontiguousarray(D)).cuda(), want_F=True)]
    assert fb.device_error() == 0
    return got


def close(got, ref, tol):
    for k in range(len(got[0])):
        for x, r in zip(got[:3], ref[:3]):
            assert np.linalg.norm(x[k] - r[k]) <= tol * np.linalg.norm(r[k])


@pytest.mark.parametrize("n,m,tol", [(1, 1, 0.0), (7, 8, 0.0), (8, 9, 0.0), (9, 16, 0.0), (16, 17, 0.0), (33, 3, 1e-8),
                                     (41, 25, 1e-10), (78, 40, 1e-10)])
def test_sizes(esmf, n, m, tol):
    w = W.small_random(n + n % 2, 1, 11 + n, tol=tol)
    w.basis = w.basis.subset(np.arange(n))
    D = np.random.default_rng(n).standard_normal((m, n, n))
    with esmf.FockBuilder(w.basis, w.tol, "stored", "fp32") as fb:
        got = build(fb, D)
        fb.set_path("cuda_core")
        ref = build(fb, D)
    close(got, ref, TOL)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_density(esmf, bad):
    """A NaN or infinity reaches exactly the outputs that it reaches on CUDA cores."""
    w = W.small_random(26, 2, 7)
    D = np.random.default_rng(3).standard_normal((18, 26, 26))
    D[17, 3, 19] = bad
    with esmf.FockBuilder(w.basis, w.tol, "stored", "fp32") as fb:
        got = build(fb, D)
        fb.set_path("cuda_core")
        ref = build(fb, D)
    for x, r in zip(got, ref):
        assert np.array_equal(np.isnan(x), np.isnan(r)) and np.array_equal(np.isinf(x), np.isinf(r))
        f = np.isfinite(r)
        assert np.linalg.norm(x[f] - r[f]) <= TOL * np.linalg.norm(r[f])
