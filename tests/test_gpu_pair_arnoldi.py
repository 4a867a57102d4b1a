"""Arnoldi steps in FP32-pair arithmetic at the edges of their kernels.

Bases of up to 4 and up to 8 vectors and longer ones take different kernels, so the restart lengths are one at
and one beyond each edge.  The steps agree with FP64 ones to about 1e-13, far below the FP32 rounding of the
preconditioner that the iteration count depends on: both need the same number of iterations up to one, and the
oracle's residual meets the tolerance.  The point source has exact zeros, which take the slow conversion.
"""
import numpy as np
import pytest

import inputs
import paper_1611_01034_gb300 as tm

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from tests.test_gpu_parity import F32, _case  # noqa: E402


@pytest.mark.parametrize("restart", [3, 4, 5, 8, 9])
@pytest.mark.parametrize("name", ["c1_4x4x4x4", "ragged_4x6x4x10"])
def test_restart_lengths(name, restart):
    iters = []
    for oa in (tm.TM_F64, tm.TM_F32X2):
        U, g, op, seed = _case(name, F32, setup_iters=2, outer_apply=oa, restart=restart)
        tm.tm_setup(g.h, inputs.random_test_vectors(g.L, g.nv, seed + 2000))
        b = inputs.gaussian_spinor(g.L, seed + 1000, nrhs=2)
        b[1] = 0
        b[1].flat[5] = 1
        x = np.zeros_like(b)
        st, info = tm.tm_solve(g.h, b, x, 2, 1e-11)
        assert st == tm.TM_OK and info.converged
        for r in range(2):
            assert np.linalg.norm(b[r] - op.apply(x[r])) / np.linalg.norm(b[r]) <= 1.01e-11
        iters.append(info.iters)
    assert abs(iters[0] - iters[1]) <= 1, iters
