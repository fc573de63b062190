"""Integral-direct FP64 builds through records in a scratch buffer and the
tensor-core digit-splitting kernel, against the CUDA-core kernel that evaluates
its integrals in place.

Tolerance: either path rounds each 64-term brick sum and each of at most nb^2
accumulator additions in FP64; with nb <= 12 and the cancellation of these
densities (below 100) that is (64 + 144) 2^-53 100 = 2.3e-12.
"""
import numpy as np
import pytest

from paper_2002_00322_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = 2.3e-12


def build(fb, D):
    import torch
    got = [x.cpu().numpy() for x in fb.build(torch.from_numpy(np.ascontiguousarray(D)).cuda(), want_F=True)]
    assert fb.device_error() == 0
    return got


def close(got, ref):
    for k in range(len(got[0])):
        for x, r in zip(got[:3], ref[:3]):
            assert np.linalg.norm(x[k] - r[k]) <= TOL * np.linalg.norm(r[k])


@pytest.mark.parametrize("n,m,tol,budget,chunked", [(1, 1, 0.0, 0, True), (9, 17, 0.0, 0, True), (41, 8, 1e-10, 0, True),
                                                    (96, 9, 1e-10, 64 << 20, True), (96, 9, 1e-10, 1 << 20, False)])
def test_scratch_and_in_place(esmf, n, m, tol, budget, chunked):
    """Whole lists, several chunks (a quarter of the budget holds 16 MB of records
    at a time) and a budget without room for them."""
    w = W.small_random(n + n % 2, 1, 21 + n, tol=tol)
    w.basis = w.basis.subset(np.arange(n))
    D = np.random.default_rng(n).standard_normal((m, n, n))
    with esmf.FockBuilder(w.basis, w.tol, "direct", "fp64", budget_bytes=budget) as fb:
        scratch = fb.stats()["scratch_bytes"]
        assert (scratch > 0) == chunked and (budget == 0 or scratch <= budget // 4)
        got = build(fb, D)
        fb.set_path("cuda_core")
        close(got, build(fb, D))
