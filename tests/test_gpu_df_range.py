"""Density-fitted FP64 exchange over the whole range of FP64 densities.

Tolerance: either arithmetic rounds each of the n_aux (n + n^2) terms of an
element at most at 2^-53; with the sizes below and a cancellation below 10 that
is 20 * 40 * (40 + 1600) * 2^-53 = 1.5e-10 at worst, and 1e-12 allows for the
sums' random signs (a thousandth of the terms' number).
"""
import numpy as np
import pytest

from paper_2002_00322_gb300 import workloads as W

from test_gpu_df_split import build, molecule

pytestmark = pytest.mark.gpu
TOL = 1e-12


@pytest.mark.parametrize("e", [-1000, -650, -590, -560, -545, -501, -499, 499, 501, 700, 950])
def test_scaled_density(esmf, e):
    """K of a density scaled by 2^e beside ordinary ones, against K of the unscaled density."""
    basis = molecule(40, 11)
    aux = W.even_tempered_aux(basis, count=2)
    D = np.random.default_rng(4).standard_normal((3, 40, 40))
    D[1] = np.ldexp(D[0], e)
    J, K, F, _ = build(esmf, basis, aux, D)
    for x in (J, K, F):
        assert np.linalg.norm(np.ldexp(x[1], -e) - x[0]) <= TOL * np.linalg.norm(x[0])


def test_columns_far_apart(esmf):
    """A column 2^-300 of the others keeps its own digits; the others theirs."""
    basis = molecule(33, 12)
    aux = W.even_tempered_aux(basis, count=2)
    D = np.zeros((2, 33, 33))
    D[0] = np.random.default_rng(5).standard_normal((33, 33))
    D[0, :, 9] = np.ldexp(D[0, :, 9], -300)
    D[1] = D[0]
    D[1, :, 9] = 0.0
    _, K, _, _ = build(esmf, basis, aux, D)
    assert np.linalg.norm(K[0] - K[1]) <= 1e-15 * np.linalg.norm(K[1])


def test_infinities_follow_ieee_rules(esmf):
    """K = B inf B of one function is infinite, not NaN; of many, no element is finite."""
    one = molecule(1, 3)
    _, K, _, _ = build(esmf, one, W.even_tempered_aux(one, count=1), np.array([[[np.inf]], [[2.0]]]))
    assert np.isposinf(K[0, 0, 0]) and np.isfinite(K[1, 0, 0])
    basis = molecule(20, 9)
    D = np.random.default_rng(1).standard_normal((2, 20, 20))
    D[1, 4, 7] = -np.inf
    _, K, _, _ = build(esmf, basis, W.even_tempered_aux(basis, count=2), D)
    assert not np.isfinite(K[1]).any() and np.isfinite(K[0]).all()
