"""FP64 and double-FP32 builds at the ends of the exponent range, where the
digit-splitting kernel hands over to FP64 arithmetic: densities and molecules
of any size, infinities and NaN.  Tolerances: those of test_gpu_split.py.
"""
import numpy as np
import pytest

from paper_2002_00322_gb300 import workloads as W

from test_gpu_split import TOL, both, close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "f32x2"])
@pytest.mark.parametrize("e", [-960, -700, -641, -560, -501, -499, -191, -189, 499, 501, 900])
def test_scaled_densities(esmf, prec, e):
    """A density scaled by 2^e in a pass with one of ordinary size; the
    reference is the CUDA-core build of the unscaled densities."""
    w = W.small_random(24, 2, 3)
    D = np.random.default_rng(1).standard_normal((2, 24, 24))
    ref = both(esmf, w, D, prec)[1]
    scaled = D.copy()
    scaled[1] = np.ldexp(D[1], e)
    got = both(esmf, w, scaled, prec)[0]
    close([x[0] for x in got[:3]], [x[0] for x in ref[:3]], TOL[prec])
    close([np.ldexp(x[1], -e) for x in got[:3]], [x[1] for x in ref[:3]], TOL[prec])


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("mode,prec", [("stored", "f32x2"), ("direct", "fp64")])
def test_non_finite_density(esmf, mode, prec, bad):
    """A NaN or infinity reaches the outputs that it reaches in an FP64 store on CUDA cores."""
    import torch
    w = W.small_random(26, 2, 7)
    D = np.random.default_rng(3).standard_normal((18, 26, 26))
    D[17, 3, 19] = bad
    ref = both(esmf, w, D, "fp64")[1]
    with esmf.FockBuilder(w.basis, w.tol, mode, prec) as fb:
        got = [x.cpu().numpy() for x in fb.build(torch.from_numpy(D).cuda(), want_F=True)]
        assert fb.device_error() == 0
    for x, r in zip(got, ref):
        assert np.array_equal(np.isnan(x), np.isnan(r)) and np.array_equal(np.isinf(x), np.isinf(r))
        f = np.isfinite(r)
        assert np.linalg.norm(x[f] - r[f]) <= TOL["f32x2"] * np.linalg.norm(r[f])
