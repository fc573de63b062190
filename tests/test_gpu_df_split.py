"""Density-fitted exchange in FP64 by digit splitting (df_split.cu) against the
same fit in NumPy, at the edges of its 64- and 128-element tiles.

Tolerance: B of the handle and of the reference come from the same metric by two
Cholesky factorisations; the fit's conditioning bounds their difference (the
existing FP64 tests of these sizes use 1e-10); the exchange itself is exact to
about 2^-53 of the sum of absolute terms.
"""
import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2002_00322_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-10


def molecule(n, seed):
    w = W.small_random(n + n % 2, 1, seed, edge=4.0 + 0.1 * n, min_dist=1.0)
    return w.basis.subset(np.arange(n))


def build(esmf, basis, aux, D):
    import torch
    with esmf.FockBuilder(basis, 0.0, "df", "fp64", aux=aux) as fb:
        J, K, F, t = fb.build(torch.from_numpy(np.ascontiguousarray(D)).cuda(), want_F=True)
        out = [x.cpu().numpy() for x in (J, K, F, t)]
        assert fb.device_error() == 0
    return out


@pytest.mark.parametrize("n,m,count", [(1, 1, 1), (15, 2, 3), (16, 33, 2), (17, 1, 2), (63, 2, 1), (64, 3, 1), (65, 2, 1)])
def test_against_the_oracle_fit(esmf, n, m, count):
    basis = molecule(n, 3 + n)
    aux = W.even_tempered_aux(basis, count=count)
    D = np.random.default_rng(n).standard_normal((m, n, n))
    J, K, F, _ = build(esmf, basis, aux, D)
    Jr, Kr = Oracle(basis).jk_df(D, *aux)[:2]
    for k in range(m):
        for x, r in ((J[k], Jr[k]), (K[k], Kr[k])):
            assert np.linalg.norm(x - r) <= TOL * np.linalg.norm(r)


@pytest.mark.parametrize("n", [128, 130, 200])
def test_linear_and_transposed(esmf, n):
    """Larger sizes: K[D^T] = K[D]^T, K of a scaled density, zero, and densities of very different size in one build."""
    basis = molecule(n, 5)
    aux = W.even_tempered_aux(basis, count=2)
    D = np.zeros((5, n, n))
    D[0] = np.random.default_rng(n).standard_normal((n, n))
    D[1], D[2], D[3] = D[0].T, 2.0 ** -70 * D[0], 2.0 ** 300 * D[0]
    _, K, _, _ = build(esmf, basis, aux, D)
    top = np.linalg.norm(K[0])
    assert np.linalg.norm(K[1] - K[0].T) <= 1e-13 * top
    assert np.linalg.norm(K[2] * 2.0 ** 70 - K[0]) <= 1e-15 * top
    assert np.linalg.norm(K[3] * 2.0 ** -300 - K[0]) <= 1e-15 * top
    assert not K[4].any()


def test_non_finite_density(esmf):
    """A density with a NaN gives no finite K, the others of the build are untouched."""
    basis = molecule(20, 9)
    aux = W.even_tempered_aux(basis, count=2)
    D = np.random.default_rng(1).standard_normal((3, 20, 20))
    _, ref, _, _ = build(esmf, basis, aux, D)
    D[1, 4, 7] = np.nan
    _, K, _, _ = build(esmf, basis, aux, D)
    assert np.isnan(K[1]).all()
    assert np.allclose(K[[0, 2]], ref[[0, 2]], rtol=1e-13, atol=0)
