"""The autotuner on handles whose builds do not take a choice of densities per pass."""
import numpy as np
import pytest

from paper_2002_00322_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,prec", [("stored", "fp64"), ("stored", "f32x2"), ("direct", "fp64")])
@pytest.mark.parametrize("m", [3, 24])
def test_reports_the_pass_of_the_splitting_kernel(esmf, mode, prec, m):
    """FP64 and double-FP32 builds pass over 16 densities at a time; on the
    CUDA-core path, which takes 4 or 8, the choice is timed as before."""
    import torch
    w = W.small_random(26, m, 5)
    D = torch.from_numpy(np.random.default_rng(m).standard_normal((m, 26, 26))).cuda()
    with esmf.FockBuilder(w.basis, w.tol, mode, prec) as fb:
        for _ in range(3):
            assert fb.autotune(D, reps=1) == 16
        J, K = torch.empty_like(D), torch.empty_like(D)
        esmf.esmf_fock_autotune(fb.h, m, D, J, K, 1)
        torch.cuda.synchronize()
        assert torch.allclose(J, fb.build(D)[0], rtol=1e-10) and torch.allclose(K, fb.build(D)[1], rtol=1e-10)
        fb.set_path("cuda_core")
        assert fb.autotune(D, reps=1) in (4, 8)
        fb.set_path("auto")
        fb.set_density_screening(1e-12)
        assert fb.autotune(D, reps=1) in (4, 8)
