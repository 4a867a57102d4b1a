"""Which right-hand sides of an odd-even SAP sweep run two to a thread (no GPU needed).

The rule weighs whole waves of the two forms, so it is checked where one of them would be far slower: an odd one
out beside pairs on a large FP32 operator (2448 against 1808 us, below), and a batch that pairs fit into one wave
and singles do not (599 against 877 us).
"""
import ctypes

import pytest

import paper_1611_01034_gb300 as tm


def paired(L, blk, nrhs, prec):
    """How many of nrhs right-hand sides run in pairs, for the operator's storage prec."""
    f = tm.lib().tmamg_sap_oe_paired
    four = ctypes.c_int * 4
    s16 = prec if prec in (tm.TM_F16, tm.TM_BF16) else 0
    return f(four(*(n // m for n, m in zip(L, blk))), four(*blk), nrhs, s16)


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_1611_01034_gb300 import build
    build.build()


@pytest.mark.parametrize("L,blk,nrhs,prec,expect", [
    ((16, 24, 24, 24), (4, 4, 4, 4), 3, tm.TM_F32, 0), ((48, 24, 24, 24), (4, 4, 4, 4), 5, tm.TM_F32, 0),
    ((16, 24, 24, 24), (4, 4, 4, 4), 4, tm.TM_F32, 4), ((16, 16, 16, 16), (4, 4, 4, 4), 4, tm.TM_F32, 4),
    ((16, 16, 16, 16), (4, 4, 4, 4), 4, tm.TM_F16, 4), ((16, 16, 16, 16), (4, 4, 4, 4), 3, tm.TM_BF16, 0),
    ((48, 24, 24, 24), (4, 4, 4, 4), 6, tm.TM_F16, 6), ((96, 48, 48, 48), (4, 4, 4, 4), 7, tm.TM_F16, 6),
    ((16, 16, 16, 8), (2, 2, 2, 2), 2, tm.TM_F32, 2), ((8, 8, 8, 8), (4, 4, 4, 4), 12, tm.TM_F32, 0)])
def test_pairs_where_they_are_faster(L, blk, nrhs, prec, expect):
    assert paired(L, blk, nrhs, prec) == expect


@pytest.mark.parametrize("prec", [tm.TM_F32, tm.TM_F16])
def test_one_right_hand_side_is_alone_and_pairs_are_whole(prec):
    for n in (8, 16, 32, 64):
        assert paired((n, 16, 16, 16), (4, 4, 4, 4), 1, prec) == 0
        for nrhs in range(2, 30):
            assert paired((n, 16, 16, 16), (4, 4, 4, 4), nrhs, prec) in (0, nrhs & ~1)
