"""The coarse solve in one launch (small systems) against the step-by-step solve.

The one-launch forms (a cluster per right-hand side, the whole chip) take restart lengths up to 48; 49 takes the other form, with the same steps until the
first restart.  FP64 to 1e-9 (rounding of 24 Arnoldi steps of another summation order), FP32 to 1e-3; a zero
right-hand side gives zero in no steps; a batch through the K-cycle gives every right-hand side what it gets
alone (FP64).  Short cycles, with the true residual between them, are held against the oracle's GMRES on the
exported D_c, and K-cycles of a batch too large for the clusters against those of one right-hand side alone.
"""
import ctypes
import threading

import numpy as np
import pytest

import inputs
import paper_1611_01034_gb300 as tm

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from oracle.coarse import CoarseOperator, OddEvenCoarse  # noqa: E402
from oracle.krylov import gmres  # noqa: E402
from tests.gpu_helpers import GPU, rel  # noqa: E402


def _gpu(L, agg, nv, prec, **kw):
    g = GPU(inputs.gauge_field(L, 0.5, 5), m0=-0.4, c_sw=1.5, mu=0.005, delta=5.0, nv=nv, agg=agg, sap_block=(2, 2, 2, 2),
            cycle_prec=prec, **kw)
    tm.tm_setup_from_vectors(g.h, inputs.random_test_vectors(L, nv, 2005))
    return g


@pytest.mark.parametrize("L,agg,nv", [((4, 4, 4, 4), (2, 2, 2, 2), 3), ((8, 8, 8, 8), (4, 4, 4, 4), 9),
                                      ((4, 4, 8, 12), (2, 2, 2, 2), 8), ((8, 8, 8, 16), (4, 4, 4, 4), 28),
                                      ((8, 8, 16, 16), (2, 2, 2, 2), 12)])
@pytest.mark.parametrize("prec,tol", [(tm.TM_F64, 1e-9), (tm.TM_F32, 1e-3)])
def test_one_launch_solve(L, agg, nv, prec, tol):
    one, ref = _gpu(L, agg, nv, prec, coarse_restart=48), _gpu(L, agg, nv, prec, coarse_restart=49)
    rng = np.random.default_rng(3)
    b = rng.standard_normal(one.coarse_shape()) + 1j * rng.standard_normal(one.coarse_shape())
    for target, maxit in ((0.0, 24), (1e-4, 200)):
        xs, its, units = [], [], []
        for g in (one, ref):
            fx = g.field(1, prec)
            tm.tm_profile(g.h, True)
            its.append(tm.tm_coarse_solve(g.h, prec, g.pack(1, prec, b), fx, target, maxit))
            units.append(tm.tm_profile_read(g.h)["coarse_oe"]["units"])
            tm.tm_profile(g.h, 0)
            xs.append(g.unpack(1, prec, fx, b.shape))
        assert its[0] == its[1]
        # operator applications; step by step the host may have one more under way when it stops
        assert units[1] - 1 <= units[0] <= units[1], units
        assert rel(xs[0], xs[1]) <= tol
    fx = one.pack(1, prec, b)
    assert tm.tm_coarse_solve(one.h, prec, one.pack(1, prec, 0 * b), fx, 0.0, 24) == 0
    assert not one.unpack(1, prec, fx, b.shape).any()


@pytest.mark.parametrize("L,nv", [((8, 8, 8, 8), 9), ((8, 8, 16, 16), 20)])  # a cluster's size, the whole chip's
@pytest.mark.parametrize("prec,tol,to", [(tm.TM_F64, 1e-9, 1e-8), (tm.TM_F32, 1e-3, 1e-4)])
def test_short_cycles(L, nv, prec, tol, to):
    g = _gpu(L, (4, 4, 4, 4), nv, prec, coarse_restart=2)
    rng = np.random.default_rng(3)
    b = rng.standard_normal(g.coarse_shape()) + 1j * rng.standard_normal(g.coarse_shape())
    oe = OddEvenCoarse(CoarseOperator(g.Dc_blocks(), nv, 5.0 * 0.005))
    for target, maxit in ((0.0, 8), (to, 200)):
        want = gmres(oe.schur, oe.reduced_rhs(b), tol=target, restart=2, maxit=maxit)
        assert want.iters > 2
        fx = g.field(1, prec)
        it = tm.tm_coarse_solve(g.h, prec, g.pack(1, prec, b), fx, target, maxit)
        assert it == want.iters
        assert rel(g.unpack(1, prec, fx, b.shape), oe.reconstruct(b, want.x)) <= tol


# clusters for the batch too; a batch step by step, one alone on the whole chip
@pytest.mark.parametrize("L,nv,tol", [((8, 8, 8, 8), 8, 1e-12), ((8, 8, 16, 16), 20, 1e-9)])
@pytest.mark.parametrize("steps", [0, 5])
def test_one_launch_solve_of_a_batch(L, nv, tol, steps):
    g = _gpu(L, (4, 4, 4, 4), nv, tm.TM_F64, max_rhs=3, coarse_tol=0.0, coarse_maxit=7, coarse_restart=3,
             coarsest_steps=steps)
    v = inputs.gaussian_spinor(L, 11, 3)
    z = g.field(0, tm.TM_F64, 3)
    tm.tm_kcycle(g.h, tm.TM_F64, g.pack(0, tm.TM_F64, v, 3), z, 3)
    got = g.unpack(0, tm.TM_F64, z, v.shape, 3)
    for r in range(3):
        z1 = g.field(0, tm.TM_F64)
        tm.tm_kcycle(g.h, tm.TM_F64, g.pack(0, tm.TM_F64, v[r]), z1, 1)
        assert rel(got[r], g.unpack(0, tm.TM_F64, z1, v[r].shape)) <= tol


@pytest.mark.parametrize("nrhs", [1, 2])
def test_fixed_step_kcycle_does_not_wait(nrhs):
    # with a fixed step count the host has nothing to decide: tm_kcycle returns while the stream is still busy
    L = (8, 8, 8, 8)
    g = _gpu(L, (4, 4, 4, 4), 8, tm.TM_F32, max_rhs=2, coarsest_steps=5)
    v = g.pack(0, tm.TM_F32, inputs.gaussian_spinor(L, 11, nrhs), nrhs)
    z = g.field(0, tm.TM_F32, nrhs)
    tm.tm_kcycle(g.h, tm.TM_F32, v, z, nrhs)  # work buffers are made in the first call
    tm.tm_synchronize(g.h)
    slept = torch.cuda.Event()
    torch.cuda._sleep(400_000_000)  # about 0.2 s of the stream
    slept.record()
    tm.tm_kcycle(g.h, tm.TM_F32, v, z, nrhs)
    assert not slept.query()
    tm.tm_synchronize(g.h)


@pytest.mark.parametrize("steps", [0, 5])
def test_whole_chip_barrier_times_out_cleanly(steps):
    # 64 coarse sites of 40 complex unknowns in FP64 are beyond the cluster's 6 MB: the whole chip, whose barriers
    # may poll once.  The call says so, nothing stays behind on the handle, and a fresh handle solves.
    L = (8, 8, 16, 16)
    kw = dict(L=L, agg=(4, 4, 4, 4), nv=20, prec=tm.TM_F64, coarsest_steps=steps)
    g = _gpu(**kw, tc_spin_limit=1)
    rng = np.random.default_rng(5)
    b = rng.standard_normal(g.coarse_shape()) + 1j * rng.standard_normal(g.coarse_shape())
    fb, fx = g.pack(1, tm.TM_F64, b), g.field(1, tm.TM_F64)
    v, z = g.pack(0, tm.TM_F64, inputs.gaussian_spinor(L, 11)), g.field(0, tm.TM_F64)

    def kcycle():
        tm.tm_kcycle(g.h, tm.TM_F64, v, z, 1)
        tm.tm_synchronize(g.h)

    bd = inputs.gaussian_spinor(L, 12)
    for call in (lambda: tm.tm_coarse_solve(g.h, tm.TM_F64, fb, fx, 1e-8, 200), kcycle,
                 lambda: tm.tm_solve(g.h, bd, np.zeros_like(bd), 1, 1e-6)):
        with pytest.raises(tm.TMError) as e:
            call()
        assert e.value.status == tm.TM_ERR_TIMEOUT
        tm.tm_synchronize(g.h)
    fy = g.field(1, tm.TM_F64)
    tm.tm_apply(g.h, 1, tm.TM_F64, fb, fy, 1)
    g2 = _gpu(**kw)
    f2 = g2.field(1, tm.TM_F64)
    tm.tm_apply(g2.h, 1, tm.TM_F64, fb, f2, 1)
    assert torch.equal(fy, f2)
    assert tm.tm_solve(g2.h, bd, np.zeros_like(bd), 1, 1e-6)[0] == tm.TM_OK


class _Part:
    """A stream on a part of the GPU's SMs (a green context), for the length of a with block."""

    class Res(ctypes.Structure):  # CUdevResource, with room to spare
        _fields_ = [("type", ctypes.c_int), ("pad", ctypes.c_ubyte * 92), ("sm", ctypes.c_uint * 64)]

    def __init__(self, sms, flags):
        cu, ref = ctypes.CDLL("libcuda.so.1"), ctypes.byref
        dev, part, rest, n = self.Res(), self.Res(), self.Res(), ctypes.c_uint(1)
        desc, self.ctx, self.st = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
        torch.cuda.synchronize()
        for r in (cu.cuDeviceGetDevResource(0, ref(dev), 1),
                  cu.cuDevSmResourceSplitByCount(ref(part), ref(n), ref(dev), ref(rest), flags, sms),
                  cu.cuDevResourceGenerateDesc(ref(desc), ref(part), 1), cu.cuGreenCtxCreate(ref(self.ctx), desc, 0, 1),
                  cu.cuGreenCtxStreamCreate(ref(self.st), self.ctx, 1, 0)):
            if r:
                pytest.skip(f"no green context on this driver ({r})")
        self.cu = cu

    def __enter__(self):
        self.on = torch.cuda.stream(torch.cuda.ExternalStream(self.st.value))
        self.on.__enter__()

    def __exit__(self, *exc):
        torch.cuda.synchronize()
        self.on.__exit__(*exc)
        self.cu.cuStreamDestroy_v2(self.st)
        self.cu.cuGreenCtxDestroy(self.ctx)


@pytest.mark.parametrize("sms,flags", [(16, 0), (4, 1)])  # whole clusters of SMs, or SMs from anywhere
@pytest.mark.parametrize("L,nv", [((8, 8, 8, 8), 9), ((8, 8, 16, 16), 20)])  # a cluster's size, the whole chip's
def test_stream_on_part_of_the_chip(L, nv, sms, flags):
    # the one-launch forms need their CTAs resident together: on fewer SMs the step-by-step solve runs
    rng = np.random.default_rng(3)
    shape = tuple(n // 4 for n in L) + (2 * nv,)
    b = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)

    def solves():
        out = []
        for steps in (0, 7):
            g = _gpu(L, (4, 4, 4, 4), nv, tm.TM_F64, coarsest_steps=steps)
            fx = g.field(1, tm.TM_F64)
            it = tm.tm_coarse_solve(g.h, tm.TM_F64, g.pack(1, tm.TM_F64, b), fx, 1e-6, 24)
            out.append((it, g.unpack(1, tm.TM_F64, fx, shape)))
            g.close()
        return out

    whole = solves()
    part = _Part(sms, flags)
    with part:
        got = solves()
    for (i0, x0), (i1, x1) in zip(whole, got):
        assert i0 == i1
        assert rel(x1, x0) <= 1e-9


def test_first_call_of_a_thread_takes_one_launch():
    # on the default stream, before anything has made the device's context current in that thread
    g = _gpu((8, 8, 8, 8), (4, 4, 4, 4), 8, tm.TM_F32)
    fb, fx = g.pack(1, tm.TM_F32, np.ones(g.coarse_shape())), g.field(1, tm.TM_F32)
    tm.tm_profile(g.h, True)
    t = threading.Thread(target=tm.tm_coarse_solve, args=(g.h, tm.TM_F32, fb, fx, 0.0, 7))
    t.start()
    t.join()
    assert tm.tm_profile_read(g.h)["coarse_oe"]["launches"] == 1
