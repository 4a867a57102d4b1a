"""SAP on batches of right-hand sides: on enough blocks pairs share a thread and an odd one out runs alone.

Every right-hand side of a batch must get what it gets alone, in every storage of the operator, for
blocks that fill their warps (4^4), leave lanes idle (2^4) and have unequal dims, with and without b;
the last one of a batch is also held against the oracle on the smaller lattices.  Which form the sizes
take is asserted.  Tolerances: the two forms order their FP32 sums differently (4 MR steps amplify 2^-24
to below 5e-6); against the oracle as for one right-hand side (FP32 5e-5, a 16-bit operator 2^-11 or 2^-8
per entry over the same chain).
"""
import functools

import numpy as np
import pytest

import inputs
import paper_1611_01034_gb300 as tm
from oracle.dirac import Operator
from oracle.sap import SAP

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from tests.gpu_helpers import GPU, rel  # noqa: E402
from tests.test_sap_pairs import paired  # noqa: E402

F32 = tm.TM_F32


def _sweeps(g, b, x0, sweeps):
    n = x0.shape[0]
    fx = g.pack(0, F32, x0, n)
    tm.tm_sap(g.h, F32, None if b is None else g.pack(0, F32, b, n), fx, sweeps, n)
    return g.unpack(0, F32, fx, x0.shape, n)


@functools.lru_cache(maxsize=4)
def _oracle(L, blk, nrhs):
    sap = SAP(Operator(inputs.gauge_field(L, 0.5, 17), -0.3, 1.3, 0.05), blk, n_mr=4, block_oe=True)
    b, x0 = inputs.gaussian_spinor(L, 1, nrhs), inputs.gaussian_spinor(L, 2, nrhs)
    return sap.smooth(b[-1], x0[-1], 2), sap.smooth(np.zeros_like(b[0]), x0[0], 1)


# how many run in pairs with the operator in FP32, in 16 bits
@pytest.mark.parametrize("L,blk,nrhs,pairs", [
    ((8, 8, 8, 16), (2, 2, 2, 2), 3, (0, 0)), ((8, 8, 8, 24), (4, 2, 4, 2), 7, (0, 0)),
    ((16, 16, 16, 16), (4, 4, 4, 4), 2, (0, 0)), ((16, 16, 16, 16), (4, 4, 4, 4), 5, (0, 0)),
    ((8, 16, 16, 8), (4, 4, 4, 4), 15, (0, 0)),
    ((16, 16, 16, 8), (4, 4, 4, 4), 8, (8, 8)), ((16, 16, 16, 16), (4, 4, 4, 4), 6, (6, 6)),
    ((16, 16, 24, 32), (4, 4, 4, 4), 7, (0, 6)), ((16, 16, 16, 16), (2, 2, 2, 2), 7, (6, 6)),
    ((16, 16, 16, 16), (4, 2, 4, 4), 4, (4, 4))])
@pytest.mark.parametrize("prec,tol", [(tm.TM_F32, 5e-5), (tm.TM_F16, 5e-3), (tm.TM_BF16, 3e-2)])
def test_odd_even_sap_batches(L, blk, nrhs, pairs, prec, tol):
    assert paired(L, blk, nrhs, prec) == pairs[prec != tm.TM_F32]
    U = inputs.gauge_field(L, 0.5, 17)
    g = GPU(U, m0=-0.3, c_sw=1.3, mu=0.05, nv=2, agg=blk, sap_block=blk, cycle_prec=F32, max_rhs=nrhs, block_oe=1,
            sap_prec=prec)
    b, x0 = inputs.gaussian_spinor(L, 1, nrhs), inputs.gaussian_spinor(L, 2, nrhs)
    tm.tm_profile(g.h, True)
    got, got0 = _sweeps(g, b, x0, 2), _sweeps(g, None, x0, 1)
    two = 0 < paired(L, blk, nrhs, prec) < nrhs  # launches per colour: pairs and an odd one out
    assert tm.tm_profile_read(g.h)["sap"]["launches"] == 3 * 2 * (2 if two else 1)
    tm.tm_profile(g.h, 0)
    for r in range(nrhs):
        assert rel(got[r], _sweeps(g, b[r:r + 1], x0[r:r + 1], 2)[0]) <= 5e-6
        assert rel(got0[r], _sweeps(g, None, x0[r:r + 1], 1)[0]) <= 5e-6
    if np.prod(L) <= 32768 and nrhs in (3, 7, 8):
        want, want0 = _oracle(L, blk, nrhs)
        assert rel(got[-1], want) <= tol
        assert rel(got0[0], want0) <= tol


@pytest.mark.parametrize("prec,tol", [(tm.TM_F32, 1e-4), (tm.TM_F64, 1e-10)])
def test_full_block_sap_batch(prec, tol):
    # 4^4 blocks: FP32 keeps the block's operator on the chip, with and without b, across the T boundary
    L, blk, nrhs = (8, 16, 8, 8), (4, 4, 4, 4), 3
    U = inputs.gauge_field(L, 0.5, 19)
    g = GPU(U, m0=-0.3, c_sw=1.3, mu=0.05, nv=2, agg=blk, sap_block=blk, cycle_prec=prec, max_rhs=nrhs)
    sap = SAP(Operator(U, -0.3, 1.3, 0.05), blk, n_mr=4)
    b, x0 = inputs.gaussian_spinor(L, 1, nrhs), inputs.gaussian_spinor(L, 2, nrhs)
    for bb in (b, None):
        fx = g.pack(0, prec, x0, nrhs)
        tm.tm_sap(g.h, prec, None if bb is None else g.pack(0, prec, bb, nrhs), fx, 2, nrhs)
        got = g.unpack(0, prec, fx, x0.shape, nrhs)
        for r in range(nrhs):
            assert rel(got[r], sap.smooth(np.zeros_like(b[r]) if bb is None else b[r], x0[r], 2)) <= tol


@pytest.mark.parametrize("L,blk,oe,prec,store,tol", [
    ((8, 8, 8, 16), (4, 4, 4, 8), 0, tm.TM_F32, tm.TM_F32, 1e-4), ((8, 8, 8, 16), (4, 4, 4, 8), 1, tm.TM_F32, tm.TM_F32, 1e-4),
    ((8, 8, 16, 16), (4, 4, 8, 8), 0, tm.TM_F64, tm.TM_F32, 1e-10), ((8, 8, 16, 16), (4, 4, 8, 8), 1, tm.TM_F64, tm.TM_F32, 1e-10),
    ((8, 8, 16, 16), (4, 4, 8, 8), 1, tm.TM_F32, tm.TM_F16, 5e-3), ((6, 6, 12, 12), (3, 3, 6, 6), 0, tm.TM_F32, tm.TM_F32, 1e-4)])
def test_blocks_of_more_than_256_sites(L, blk, oe, prec, store, tol):
    # up to the 1024 sites that tm_create takes; two right-hand sides, the second with b = 0
    U = inputs.gauge_field(L, 0.5, 23)
    g = GPU(U, m0=-0.3, c_sw=1.3, mu=0.05, nv=2, agg=(L[0] // 2, L[1] // 2, 2, 2), sap_block=blk, cycle_prec=prec,
            max_rhs=2, block_oe=oe, sap_prec=store)
    sap = SAP(Operator(U, -0.3, 1.3, 0.05), blk, n_mr=4, block_oe=bool(oe))
    b, x0 = inputs.gaussian_spinor(L, 1, 2), inputs.gaussian_spinor(L, 2, 2)
    b[1] = 0
    fx = g.pack(0, prec, x0, 2)
    tm.tm_sap(g.h, prec, g.pack(0, prec, b, 2), fx, 1, 2)
    got = g.unpack(0, prec, fx, x0.shape, 2)
    for r in range(2):
        assert rel(got[r], sap.smooth(b[r], x0[r], 1)) <= tol


@pytest.mark.parametrize("nv,blk,nrhs,pairs", [(5, (2, 2, 2, 2), 5, 1), (28, (2, 2, 2, 2), 3, 2), (28, (2, 2, 2, 2), 5, 3),
                                               (24, (2, 2, 2, 2), 11, 3), (23, (1, 2, 2, 2), 16, 2)])
@pytest.mark.parametrize("prec", [tm.TM_F32, tm.TM_F16, tm.TM_BF16])
def test_level1_sap_batches(nv, blk, nrhs, pairs, prec):
    # 1 to 3 pairs per CTA, each right-hand side as alone (rounding of another order of 4 MR steps: 1e-6)
    L, L1 = (16, 16, 16, 16), (8, 8, 8, 8)
    rows = 2 * nv * int(np.prod(blk))
    assert tm.lib().tmamg_csap_pairs(int(np.prod(L1)) // int(np.prod(blk)) // 2, rows, nrhs) == pairs
    p = dict(m0=-0.3, c_sw=1.4, mu=0.05, delta=3.0, nv=nv, agg=(2, 2, 2, 2), sap_block=(2, 2, 2, 2), cycle_prec=F32,
             max_rhs=nrhs, levels=3, nv2=2, sap1_prec=prec)
    prm = tm.params(L=L, **p)
    prm.agg2[:], prm.sap_block1[:] = (2, 2, 2, 2), blk
    h = tm.tm_create(prm, torch.cuda.current_stream())
    gen = torch.Generator(device="cuda").manual_seed(3)
    draw = lambda n, dtype: torch.randn(n, dtype=dtype, device="cuda", generator=gen)  # noqa: E731
    try:
        tm.tm_load_gauge(h, torch.from_numpy(inputs.gauge_field(L, 0.5, 7)).cuda())
        tm.tm_setup_from_vectors(h, draw(nv * 16 ** 4 * 24 + 2 * 8 ** 4 * 4 * nv, torch.float64))
        one = tm.tm_field_bytes(h, 1, F32, 1) // 4
        b, x0 = draw(nrhs * one, torch.float32), draw(nrhs * one, torch.float32)
        got = x0.clone()
        tm.tm_sap1(h, F32, b, got, 2, nrhs)
        for r in range(nrhs):
            part = slice(r * one, (r + 1) * one)
            x = x0[part].clone()
            tm.tm_sap1(h, F32, b[part].clone(), x, 2, 1)
            assert float((got[part] - x).norm() / x.norm()) <= 1e-6
    finally:
        tm.tm_destroy(h)
