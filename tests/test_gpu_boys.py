"""F0 of the FP64 integrals (table, seeded reciprocal square root and their
fallbacks) against closed forms, through one- and two-function handles.

(pp|pp) = 2 sqrt(a / pi) for one s Gaussian of exponent a, and (pp|qq) =
erf(sqrt(rho) R) / R for two, rho = 2 a b / (a + b).  Tolerance: the integral is
about thirty FP64 roundings of at most 2^-53 each: 32 * 2^-53 = 4e-15.
"""
import math

import numpy as np
import pytest

from paper_2002_00322_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = 4e-15


def coulomb(esmf, centers, exps):
    """J_00 for the density concentrated on the last function."""
    import torch
    n = len(exps)
    b = W.Basis(np.asarray(centers, dtype=float), np.ones(n, dtype=np.int32), np.asarray(exps, dtype=float), np.ones(n))
    D = torch.zeros((1, n, n), dtype=torch.float64, device="cuda")
    D[0, n - 1, n - 1] = 1.0
    with esmf.FockBuilder(b, 0.0, "stored", "fp64") as fb:
        return float(fb.build(D)[0][0, 0, 0].cpu())


@pytest.mark.parametrize("a", [1e-45, 1e-33, 0.3, 17.0, 1e33, 1e45])
def test_self_repulsion(esmf, a):
    ref = 2.0 * math.sqrt(a / math.pi)
    assert abs(coulomb(esmf, [[0.1, 0.2, 0.3]], [a]) - ref) <= TOL * ref


@pytest.mark.parametrize("T", [1e-12, 1e-4, 1 / 64, 3 / 64, 0.5, 1.0, 7.77, 20.015, 35.98, 35.99999, 36.0, 36.00001, 41.0, 1e3, 1e6])
def test_two_centres(esmf, T):
    a, b = 1.3, 0.4
    R = math.sqrt(T * (a + b) / (2.0 * a * b))
    x = math.sqrt(2.0 * a * b / (a + b)) * R
    ref = math.erf(x) / R
    assert abs(coulomb(esmf, [[0.0, 0.0, 0.0], [R, 0.0, 0.0]], [a, b]) - ref) <= TOL * ref
