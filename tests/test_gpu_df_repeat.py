"""A density-fitted FP64 build gives the same bits each time."""
import numpy as np
import pytest

from paper_2002_00322_gb300 import workloads as W

from test_gpu_df_split import molecule

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [(40, 1), (130, 3), (200, 5)])
def test_bitwise_repeatable(esmf, n, m):
    import torch
    basis = molecule(n, 21)
    D = torch.from_numpy(np.random.default_rng(n).standard_normal((m, n, n))).cuda()
    with esmf.FockBuilder(basis, 0.0, "df", "fp64", aux=W.even_tempered_aux(basis, count=3)) as fb:
        first = fb.build(D)[1].cpu()
        for _ in range(4):
            assert torch.equal(fb.build(D)[1].cpu(), first)
