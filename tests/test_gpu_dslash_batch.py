"""FP32 D(mu) of batches: two right-hand sides per thread (even counts on enough sites) or one.

Both forms sum in the same order, so a batch gives every right-hand side what it gets alone, bit for bit; the
lattice's volume leaves a part-filled last CTA.  The FP64 product bounds the error: 2e-7 is two FP32 roundings of
the result's size, above the mean of a site's few hundred.
"""
import numpy as np
import pytest

import inputs
import paper_1611_01034_gb300 as tm

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from tests.gpu_helpers import GPU, rel  # noqa: E402


@pytest.mark.parametrize("nrhs", [1, 2, 9, 10, 12])
def test_batch_equals_single(nrhs):
    L = (14, 18, 6, 10)
    g = GPU(inputs.gauge_field(L, 0.5, 5), m0=-0.4, c_sw=1.5, mu=0.005, delta=5.0, nv=4, agg=(7, 3, 3, 5),
            sap_block=(7, 3, 3, 5), max_rhs=12)
    psi = inputs.gaussian_spinor(L, 3, nrhs=12)[:nrhs].astype(np.complex64).astype(np.complex128)
    got = g.apply_fine(psi, tm.TM_F32, nrhs=nrhs)
    for r in (0, nrhs - 1):
        assert np.array_equal(got[r], np.asarray(g.apply_fine(psi[r], tm.TM_F32)).reshape(got[r].shape))
        assert rel(got[r], np.asarray(g.apply_fine(psi[r], tm.TM_F64)).reshape(got[r].shape)) <= 2e-7
