"""The tensor-core kernel of FP64 and double-FP32 stores (exact digit
splitting) against the CUDA-core kernels on the same handle.

Tolerance: either path rounds each 64-term brick sum and each of at most nb^2
accumulator additions in FP64, so the two differ by at most about
(64 + nb^2) 2^-53 of the sum of the absolute terms; with nb <= 10 and the
cancellation of these densities (below 100) that is 2e-12.  The double-FP32
CUDA-core kernel keeps 2^-44 per brick sum: 1e-11.
"""
import numpy as np
import pytest

from paper_2002_00322_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = {"fp64": 2e-12, "f32x2": 1e-11}


def both(esmf, w, D, prec):
    import torch
    Dt = torch.from_numpy(np.ascontiguousarray(D)).cuda()
    with esmf.FockBuilder(w.basis, w.tol, "stored", prec) as fb:
        got = [x.cpu().numpy() for x in fb.build(Dt, want_F=True)]
        assert fb.device_error() == 0
        fb.set_path("cuda_core")
        ref = [x.cpu().numpy() for x in fb.build(Dt, want_F=True)]
    return got, ref


def close(got, ref, tol):
    for x, r in zip(got, ref):
        top = max(np.abs(r).max(), 1e-300)           # so that squares stay in range
        assert np.linalg.norm((x - r) / top) <= tol * np.linalg.norm(r / top)


@pytest.mark.parametrize("prec", ["fp64", "f32x2"])
@pytest.mark.parametrize("n,m,tol", [(1, 1, 0.0), (7, 8, 0.0), (8, 9, 0.0), (9, 16, 0.0), (16, 17, 0.0), (33, 3, 1e-8),
                                     (41, 25, 1e-10), (78, 40, 1e-10)])
def test_sizes(esmf, prec, n, m, tol):
    w = W.small_random(n + n % 2, 1, 11 + n, tol=tol)
    w.basis = w.basis.subset(np.arange(n))
    D = np.random.default_rng(n).standard_normal((m, n, n))
    got, ref = both(esmf, w, D, prec)
    for k in range(m):
        close([x[k] for x in got[:3]], [x[k] for x in ref[:3]], TOL[prec])


@pytest.mark.parametrize("scale", [1e-150, 1e-30, 1e120, 1e200])
def test_scaled_densities(esmf, scale):
    """One density of ordinary size beside one far from it (above 2^500 the
    kernel takes its plain loop)."""
    w = W.small_random(24, 2, 3)
    D = np.random.default_rng(1).standard_normal((2, 24, 24))
    D[1] *= scale
    got, ref = both(esmf, w, D, "fp64")
    for k in range(2):
        close([x[k] for x in got[:3]], [x[k] for x in ref[:3]], TOL["fp64"])


def test_zero_density_and_wide_range(esmf):
    """Zero blocks and a density whose elements span 24 decades."""
    w = W.small_random(40, 2, 5)
    rng = np.random.default_rng(2)
    D = np.zeros((3, 40, 40))
    D[1] = rng.standard_normal((40, 40)) * 10.0 ** rng.uniform(-24, 0, (40, 40))
    D[2, 8:16, 24:32] = rng.standard_normal((8, 8))
    got, ref = both(esmf, w, D, "fp64")
    assert not got[0][0].any() and not got[1][0].any() and not got[3][0].any()
    for k in (1, 2):
        close([x[k] for x in got[:3]], [x[k] for x in ref[:3]], TOL["fp64"])


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_density(esmf, bad):
    """A NaN or infinity reaches exactly the outputs that it reaches on CUDA cores."""
    w = W.small_random(26, 2, 7)
    D = np.random.default_rng(3).standard_normal((18, 26, 26))
    D[17, 3, 19] = bad
    got, ref = both(esmf, w, D, "fp64")
    for x, r in zip(got, ref):
        assert np.array_equal(np.isnan(x), np.isnan(r)) and np.array_equal(np.isinf(x), np.isinf(r))
        f = np.isfinite(r)
        assert np.linalg.norm(x[f] - r[f]) <= TOL["fp64"] * np.linalg.norm(r[f])
