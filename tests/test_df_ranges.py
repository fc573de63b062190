"""Lengths of the summed ranges of the density-fitted exchange: the integer
sums of k_df_gemm hold 2^11 blocks of 64 summed elements whatever the digits
are (a block adds less than 2^51 + 2^44 to the low sum, 2^41 to the high one).
"""
import pytest

BLOCKS = 2048


@pytest.mark.parametrize("n,naux,group", [(200, 700, 4), (400, 8192, 1), (704, 2464, 1), (800, 2800, 1), (1000, 3500, 1),
                                          (1, 1, 16), (64, 8192, 16), (65, 8191, 2), (1100, 8192, 1)])
@pytest.mark.parametrize("sms", [1, 148, 152])
def test_ranges(n, naux, group, sms):
    from paper_2002_00322_gb300 import build as b
    from paper_2002_00322_gb300 import fock
    b.build()
    splits = fock.load().esmf_df_exchange_ranges(n, naux, group, sms)
    blocks = naux * ((n + 63) // 64)
    cut = [blocks * s // splits for s in range(splits + 1)]
    assert 1 <= splits <= blocks and cut[-1] == blocks
    assert max(y - x for x, y in zip(cut, cut[1:])) <= BLOCKS
    # about four items per SM where the blocks allow it, none of them short
    tiles = group * ((n + 127) // 128) * ((n + 63) // 64)
    assert splits == 1 or blocks // splits >= 4 or blocks <= BLOCKS
    assert splits * tiles >= min(4 * sms, tiles * (blocks // 4))
