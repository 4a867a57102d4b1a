"""FP32 restriction and prolongation of batches (on many sizes pairs of right-hand sides share a thread).

Every right-hand side against the oracle's P: one alone, whole pairs, an odd one out, and more pairs than
one CTA takes; aggregates below a warp, of one CTA and beyond one CTA; N_v that leaves columns over.
FP32 sums of at most 6144 terms: 1e-5; a 16-bit P rounds every entry by 2^-11 (FP16) or 2^-8 (BF16).
And the FP32 error of P itself.
"""
import numpy as np
import pytest

import inputs
import paper_1611_01034_gb300 as tm
from oracle.coarse import Interpolation

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from tests.gpu_helpers import GPU, rel  # noqa: E402
from tests.test_transfer_pairs import prolong_pairs, restrict_pairs  # noqa: E402

F32 = tm.TM_F32


@pytest.mark.parametrize("L,agg,nv,nrhs", [((4, 4, 8, 8), (2, 2, 2, 2), 5, 1), ((4, 4, 8, 8), (2, 2, 2, 2), 7, 5),
                                           ((8, 8, 8, 8), (4, 4, 4, 4), 9, 1), ((8, 8, 8, 8), (4, 4, 4, 4), 8, 27),
                                           ((8, 8, 16, 12), (4, 4, 4, 6), 6, 3), ((8, 8, 16, 16), (4, 4, 8, 8), 3, 2),
                                           ((4, 4, 4, 8), (2, 1, 1, 4), 5, 6)])
@pytest.mark.parametrize("prec,tol", [(tm.TM_F32, 1e-5), (tm.TM_F16, 5e-3), (tm.TM_BF16, 3e-2)])
def test_transfer_batches(L, agg, nv, nrhs, prec, tol):
    U = inputs.gauge_field(L, 0.3, 3)
    g = GPU(U, m0=0.1, c_sw=1.0, mu=0.1, nv=nv, agg=agg, sap_block=(2, 2, 2, 2),
            cycle_prec=F32, max_rhs=nrhs, transfer_prec=prec)
    tv = inputs.random_test_vectors(L, nv, 4)
    tm.tm_setup_from_vectors(g.h, tv)
    P = Interpolation(tv, agg)
    psi, c = inputs.gaussian_spinor(L, 5, nrhs), inputs.random_coarse_vectors(g.Lc, 2 * nv, nrhs, 6)
    fc, ff = g.field(1, F32, nrhs), g.pack(0, F32, psi, nrhs)
    tm.tm_restrict(g.h, F32, ff, fc, nrhs)
    got = g.unpack(1, F32, fc, c.shape, nrhs)
    tm.tm_prolong(g.h, F32, g.pack(1, F32, c, nrhs), ff, nrhs, 1)  # psi += P c
    acc = g.unpack(0, F32, ff, psi.shape, nrhs)
    fz = g.field(0, F32, nrhs)
    tm.tm_prolong(g.h, F32, g.pack(1, F32, c, nrhs), fz, nrhs, 0)
    new = g.unpack(0, F32, fz, psi.shape, nrhs)
    for r in range(nrhs):
        assert rel(got[r], P.restrict(psi[r])) <= tol
        want = P.prolong(c[r])
        assert rel(new[r], want) <= tol
        assert rel(acc[r], psi[r] + want) <= tol


# restriction in pairs: one CTA for all of them or several, an odd one out, aggregates below a warp's CTA and beyond
# one CTA, and enough pairs to be split by shared memory
@pytest.mark.parametrize("L,agg,nv,nrhs,prec,pairs", [
    ((8, 8, 8, 8), (4, 4, 4, 4), 9, 6, tm.TM_BF16, 1), ((16, 16, 16, 16), (4, 4, 4, 4), 8, 5, tm.TM_F32, 3),
    ((16, 16, 16, 16), (4, 4, 4, 4), 25, 3, tm.TM_F16, 2), ((16, 16, 16, 16), (4, 4, 4, 4), 6, 26, tm.TM_F32, 7),
    ((4, 4, 8, 32), (2, 2, 2, 4), 7, 4, tm.TM_F32, 1), ((16, 16, 16, 32), (4, 4, 8, 8), 9, 4, tm.TM_F32, 2)])
def test_restriction_of_pairs(L, agg, nv, nrhs, prec, pairs):
    assert restrict_pairs(L, agg, nv, nrhs, prec) == pairs
    g = GPU(inputs.gauge_field(L, 0.3, 3), m0=0.1, c_sw=1.0, mu=0.1, nv=nv, agg=agg, sap_block=(2, 2, 2, 2),
            cycle_prec=F32, max_rhs=nrhs, transfer_prec=prec)
    tm.tm_setup_from_vectors(g.h, inputs.random_test_vectors(L, nv, 4))
    psi = inputs.gaussian_spinor(L, 5, nrhs)
    fc, f1 = g.field(1, F32, nrhs), g.field(1, F32, 1)
    tm.tm_restrict(g.h, F32, g.pack(0, F32, psi, nrhs), fc, nrhs)
    got = g.unpack(1, F32, fc, g.coarse_shape(nrhs), nrhs)
    for r in range(nrhs):  # FP32 sums of at most 12288 terms in another order
        tm.tm_restrict(g.h, F32, g.pack(0, F32, psi[r]), f1, 1)
        assert rel(got[r], g.unpack(1, F32, f1, got[r].shape)) <= 1e-6


# prolongation in lattice order beside pairs: both sides of the rule, on more than one CTA's sites
@pytest.mark.parametrize("L,nv,nrhs,acc,pairs", [
    ((16, 12, 12, 12), 5, 2, 0, False), ((16, 12, 12, 12), 5, 3, 1, False), ((16, 12, 12, 12), 5, 4, 0, True),
    ((16, 12, 12, 12), 5, 7, 1, False), ((16, 12, 12, 12), 5, 7, 0, True), ((16, 12, 12, 12), 21, 3, 1, True)])
def test_prolongation_forms(L, nv, nrhs, acc, pairs):
    agg = (4, 6, 6, 6)
    assert prolong_pairs(L, agg, nv, nrhs, acc) == pairs
    g = GPU(inputs.gauge_field(L, 0.3, 3), m0=0.1, c_sw=1.0, mu=0.1, nv=nv, agg=agg, sap_block=(2, 2, 2, 2),
            cycle_prec=F32, max_rhs=nrhs)
    tm.tm_setup_from_vectors(g.h, inputs.random_test_vectors(L, nv, 4))
    psi, c = inputs.gaussian_spinor(L, 5, nrhs), inputs.random_coarse_vectors(g.Lc, 2 * nv, nrhs, 6)
    ff = g.pack(0, F32, psi, nrhs)
    tm.tm_prolong(g.h, F32, g.pack(1, F32, c, nrhs), ff, nrhs, acc)
    got = g.unpack(0, F32, ff, psi.shape, nrhs)
    for r in range(nrhs):
        f1 = g.pack(0, F32, psi[r])
        tm.tm_prolong(g.h, F32, g.pack(1, F32, c[r]), f1, 1, acc)
        assert rel(got[r], g.unpack(0, F32, f1, psi[r].shape)) <= 1e-6


@pytest.mark.parametrize("nrhs", [1, 2])
def test_fp64_transfers_of_the_largest_aggregates(nrhs):
    # 1024 sites, one thread each: orthonormalisation and restriction have 64 registers there
    L, agg, nv = (8, 8, 16, 16), (4, 4, 8, 8), 3
    g = GPU(inputs.gauge_field(L, 0.3, 3), m0=0.1, c_sw=1.0, mu=0.1, nv=nv, agg=agg, sap_block=(2, 2, 2, 2),
            cycle_prec=tm.TM_F64, max_rhs=nrhs)
    tv = inputs.random_test_vectors(L, nv, 4)
    tm.tm_setup_from_vectors(g.h, tv)
    P = Interpolation(tv, agg)
    psi, c = inputs.gaussian_spinor(L, 5, nrhs), inputs.random_coarse_vectors(g.Lc, 2 * nv, nrhs, 6)
    psi, c = psi.reshape((nrhs,) + L + (4, 3)), c.reshape(g.coarse_shape(nrhs))
    fc, ff = g.field(1, tm.TM_F64, nrhs), g.field(0, tm.TM_F64, nrhs)
    tm.tm_restrict(g.h, tm.TM_F64, g.pack(0, tm.TM_F64, psi, nrhs), fc, nrhs)
    tm.tm_prolong(g.h, tm.TM_F64, g.pack(1, tm.TM_F64, c, nrhs), ff, nrhs, 0)
    got, up = g.unpack(1, tm.TM_F64, fc, c.shape, nrhs), g.unpack(0, tm.TM_F64, ff, psi.shape, nrhs)
    for r in range(nrhs):
        assert rel(got[r], P.restrict(psi[r])) <= 1e-12
        assert rel(up[r], P.prolong(c[r])) <= 1e-12


@pytest.mark.parametrize("agg", [(4, 4, 4, 4), (2, 2, 2, 2)])
@pytest.mark.parametrize("nv", [11, 24])
@pytest.mark.parametrize("common", [0, 10])
def test_fp32_error_of_the_orthonormalisation(agg, nv, common):
    # Gram-Schmidt rounds a column once per finished column and pass (nv on average) and once when it is scaled, each
    # time by 2.5e-8 of its size (the root mean square of FP32); a common part of the vectors ten times the rest
    # leaves roundings of ten times that size.  The vectors are exact in FP32.
    L = (8, 8, 8, 8)
    U, tv = inputs.gauge_field(L, 0.3, 3), inputs.random_test_vectors(L, nv, 4)
    tv = (tv + common * inputs.random_test_vectors(L, 1, 5)).astype(np.complex64).astype(np.complex128)
    P = []
    for prec in (tm.TM_F32, tm.TM_F64):
        g = GPU(U, m0=0.1, c_sw=1.0, mu=0.1, nv=nv, agg=agg, sap_block=(2, 2, 2, 2), cycle_prec=prec)
        tm.tm_setup_from_vectors(g.h, tv)
        P.append(g.P_columns())
    assert rel(P[0], P[1]) <= 2.5e-8 * (10 if common else (1 + nv) ** 0.5)
