"""Which form of the FP32 transfers a call takes (no GPU needed).

The forms differ most where a small lattice leaves SMs idle, where P stays in L2 and where the count is odd, so the
rules are checked there.
"""
import ctypes

import pytest

import paper_1611_01034_gb300 as tm


def _bytes(prec):
    return 2 if prec in (tm.TM_F16, tm.TM_BF16) else 4


def restrict_pairs(L, agg, nv, nrhs, prec):
    """Pairs of right-hand sides per CTA of the restriction, 0 for one right-hand side per CTA."""
    four = ctypes.c_int * 4
    return tm.lib().tmamg_restrict_pairs(four(*L), four(*agg), nv, nrhs, _bytes(prec))


def prolong_pairs(L, agg, nv, nrhs, accumulate):
    """Whether the prolongation runs pairs."""
    four = ctypes.c_int * 4
    return bool(tm.lib().tmamg_prolong_pairs(four(*L), four(*agg), nv, nrhs, accumulate))


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_1611_01034_gb300 import build
    build.build()


A4 = (4, 4, 4, 4)


@pytest.mark.parametrize("L,agg,nv,nrhs,prec,expect", [
    ((8, 8, 8, 8), A4, 24, 8, tm.TM_F32, 1),       # four CTAs per aggregate and chirality: 14.5 us, 49 in one
    ((8, 8, 8, 8), A4, 24, 7, tm.TM_F32, 0),       # an odd count of a P in L2
    ((24, 16, 24, 8), A4, 8, 3, tm.TM_F16, 0), ((16, 16, 16, 16), A4, 8, 5, tm.TM_F32, 3),
    ((16, 16, 16, 16), A4, 24, 3, tm.TM_F16, 2), ((48, 24, 24, 24), A4, 24, 6, tm.TM_F16, 3),
    ((48, 24, 24, 24), A4, 24, 26, tm.TM_F16, 7), ((32, 16, 16, 16), (2, 2, 2, 2), 24, 6, tm.TM_F32, 0),
    ((16, 16, 16, 16), (4, 4, 4, 8), 8, 4, tm.TM_F32, 0), ((32, 16, 16, 16), (4, 4, 8, 8), 8, 2, tm.TM_F32, 1)])
def test_restriction(L, agg, nv, nrhs, prec, expect):
    assert restrict_pairs(L, agg, nv, nrhs, prec) == expect


@pytest.mark.parametrize("agg", [(4, 4, 4, 4), (2, 2, 2, 4), (4, 4, 8, 8), (4, 4, 4, 6)])
def test_restriction_splits_are_even_and_fit_shared_memory(agg):
    warps = min(16, (agg[0] * agg[1] * agg[2] * agg[3] + 31) // 32)
    for n in (2, 4, 16):
        L = tuple(n * a for a in agg)
        for nrhs in range(1, 80):
            p, pairs = restrict_pairs(L, agg, 28, nrhs, tm.TM_F32), (nrhs + 1) // 2
            if p:
                ctas = -(-pairs // p)
                assert p == -(-pairs // ctas) and 7 * p * warps * 16 * 4 <= 48 * 1024


@pytest.mark.parametrize("L,nv,nrhs,accumulate,expect", [
    ((8, 8, 8, 8), 24, 2, 0, True), ((16, 16, 16, 16), 24, 2, 0, False),  # 29 us in pairs, 21 in lattice order
    ((32, 24, 24, 24), 8, 3, 1, False), ((32, 24, 24, 24), 24, 3, 0, True), ((32, 24, 24, 24), 8, 7, 1, False),
    ((32, 24, 24, 24), 8, 7, 0, True), ((48, 24, 24, 24), 24, 6, 1, True), ((16, 16, 16, 16), 24, 1, 0, False)])
def test_prolongation(L, nv, nrhs, accumulate, expect):
    assert prolong_pairs(L, A4, nv, nrhs, accumulate) == expect
    assert not prolong_pairs(L, (2, 2, 2, 2), nv, nrhs, accumulate)
