"""Double-FP32 stores where the low FP32 part is subnormal, one function each."""
import math

import numpy as np
import pytest

from paper_2002_00322_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def coulomb(esmf, a):
    """J and K of one s Gaussian of exponent a for a unit density."""
    import torch
    b = W.Basis(np.zeros((1, 3)), np.ones(1, dtype=np.int32), np.array([a]), np.ones(1))
    with esmf.FockBuilder(b, 0.0, "stored", "f32x2") as fb:
        J, K = fb.build(torch.ones((1, 1, 1), dtype=torch.float64, device="cuda"))[:2]
        return float(J.cpu()), float(K.cpu())


@pytest.mark.parametrize("e", [-104, -110, -118])
def test_subnormal_low_part(esmf, e):
    """The low FP32 part of a value near 2^e is a multiple of 2^-149: what is
    lost is half of that, beside some thirty FP64 roundings."""
    worst = 0.0
    for f in (1.1, 1.3, 1.7):
        ref = math.ldexp(f, e)
        J, K = coulomb(esmf, math.pi * ref * ref / 4.0)        # (pp|pp) = 2 sqrt(a / pi)
        worst = max(worst, abs(J - ref) / ref, abs(K - ref) / ref)
    assert worst <= 2.0 ** (-150 - e) + 4e-15
