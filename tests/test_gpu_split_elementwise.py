"""Single outputs of FP64 builds against long sums over the handle's integrals.

The integrals come from the CUDA-core kernel with unit densities (products with
one and sums with zeros are exact); J and K are then summed in long double.

Tolerance, the bound of the digit-splitting kernel, with u = 2^-53, Vb the largest
integral of a term's brick and Db the largest density of its 8 x 8 block (for J of
either triangle): a density is rounded to at most u Db, an integral to 2^-62 Vb, and
the digit pairs left out are below 6 * 2^-61 Vb Db, together below u |V| Db +
2^-58 Vb Db a term.  An output is a sum of nb^2 brick sums and their additions, each
rounded once, and J's densities are sums of two: nb^2 + 5 times u of its absolute
terms.  In the compact molecule, whose integrals span a factor of four, that is
what FP64 arithmetic gives; a digit or a group of digit pairs less would not pass.
In the scattered one it is a normwise bound: J of distant functions, far below the
largest of its bricks, may have no correct digit.
"""
import numpy as np
import pytest

from paper_2002_00322_gb300 import workloads as W

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def compact(n):
    rng = W.rng_for(17)
    return W.s_basis(rng, W.cube_centers(rng, (n + 1) // 2, 0.5), 2, 3, 0.5, 2.0).subset(np.arange(n))


def scattered(n):
    rng = W.rng_for(17)
    return W.s_basis(rng, W.cube_centers(rng, (n + 1) // 2, 14.0), 2, 3, 0.1, 1.0).subset(np.arange(n))


def integrals(esmf, basis, mode):
    import torch
    n = basis.n
    D = torch.zeros((n * n, n, n), dtype=torch.float64, device="cuda")
    r, s = np.divmod(np.arange(n * n), n)
    D[np.arange(n * n), r, s] = 1.0
    with esmf.FockBuilder(basis, 0.0, mode, "fp64") as fb:
        fb.set_path("cuda_core")
        V = np.concatenate([fb.build(D[i:i + 512])[0].cpu().numpy() for i in range(0, n * n, 512)])
    return V.reshape(n, n, n, n).transpose(2, 3, 0, 1)            # (pq|rs)


def long_sums(V, D):
    V, D = V.astype(np.longdouble), D.astype(np.longdouble)
    return np.einsum("pqrs,krs->kpq", V, D), np.einsum("prqs,krs->kpq", V, D)


def block_max(x, axes):
    """The largest magnitude of each block of eight along the axes, in every place of the block."""
    for a in axes:
        n = x.shape[a]
        top = np.maximum.reduceat(np.abs(x), np.arange(0, n, 8), axis=a)
        x = np.repeat(top, 8, axis=a).take(np.arange(n), axis=a)
    return x


def densities(n, m):
    """Random ones, then ones with a single element in each 8 x 8 block (one product per brick and output)."""
    rng = np.random.default_rng(n)
    D = rng.standard_normal((m, n, n))
    for k in range(m // 2, m):
        keep = np.zeros((n, n))
        for x in range(0, n, 8):
            for y in range(0, n, 8):
                keep[rng.integers(x, min(x + 8, n)), rng.integers(y, min(y + 8, n))] = 1.0
        D[k] *= keep
    return D


@pytest.mark.parametrize("mode", ["stored", "direct"])
@pytest.mark.parametrize("molecule,n,m", [(compact, 8, 4), (compact, 23, 6), (compact, 24, 18), (scattered, 30, 6)])
def test_each_output(esmf, mode, molecule, n, m):
    import torch
    basis = molecule(n)
    V = integrals(esmf, basis, mode)
    assert molecule is scattered or V.max() <= 4.0 * V.min()
    D = densities(n, m)
    with esmf.FockBuilder(basis, 0.0, mode, "fp64") as fb:
        J, K, F, _ = [x.cpu().numpy() for x in fb.build(torch.from_numpy(D).cuda(), want_F=True)]
        assert fb.device_error() == 0
    Jr, Kr = long_sums(V, D)
    SJ, SK = long_sums(V, np.abs(D))
    Vb, Db = block_max(V, (0, 1, 2, 3)), block_max(D, (1, 2))
    Dj = np.maximum(Db, Db.transpose(0, 2, 1))
    nb2 = ((n + 7) // 8) ** 2
    eJ = (nb2 + 5) * U * SJ + U * long_sums(V, Dj)[0] + 2.0 ** -58 * long_sums(Vb, Dj)[0]
    eK = (nb2 + 5) * U * SK + U * long_sums(V, Db)[1] + 2.0 ** -58 * long_sums(Vb, Db)[1]
    assert (np.abs(J - Jr) <= eJ).all()
    assert (np.abs(K - Kr) <= eK).all()
    assert (np.abs(F - (2 * Jr - Kr)) <= 2 * eJ + eK + U * (2 * SJ + SK)).all()
