"""The work that users of this library have it do, through the C ABI's Python binding.

A case is a dict of plain values.  ``kind`` says which entry points it calls:

* ``solve``     tm_solve, with the adaptive setup beforehand; with ``whole`` set the pass also loads
                the gauge field and runs the setup (what a first propagator on a new field costs);
* ``apply``     tm_apply of D(mu) on fine fields (FP32, FP64, FP32 pairs);
* ``sap``       tm_sap, the fine smoother (full or odd-even block solves, FP32 or 16-bit operator);
* ``transfer``  tm_restrict and tm_prolong between the fine and the first coarse level;
* ``sap1``      tm_sap1, the smoother of the first coarse level of a three-level handle;
* ``schur``     tm_schur, the coarsest odd-even Schur complement (CUDA cores or TF32 tensor cores);
* ``build``     tm_setup_from_vectors (P orthonormalised, D_c built), then tm_prolong and tm_apply of
                the new coarse operator, which show P and D_c;
* ``nn``        tm_nn_apply and tm_nn_grad, the learned layer's inference and its forward and backward
                pass.

Inputs are synthetic: links exp(i eps H) with Gaussian traceless Hermitian H, Gaussian vectors, all
drawn on the device from the seed.  ``exact`` evaluates the same maps with plain torch in 64 bits.
"""
import math

import numpy as np
import torch

import paper_1611_01034_gb300 as tm

PREC = {"f64": tm.TM_F64, "f32": tm.TM_F32, "f16": tm.TM_F16, "bf16": tm.TM_BF16, "f32x2": tm.TM_F32X2}
# bare masses near the critical mass of fields of the given link strength and clover coefficient
M0 = {0.5: (-0.4176881402499312, 1.5), 0.6: (-0.5948514200964429, 1.57551)}


def _dims(text):
    return tuple(int(v) for v in text.split("x"))


def _volume(dims):
    return math.prod(dims)


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the smallest solve: one source on 8^4, all launches and latency
        dict(name="solve_8x8x8x8_1rhs", kind="solve", lat="8x8x8x8", levels=2, nv=8, nv2=0, nrhs=1, whole=False,
             outer="f64", oe=0, sap="f32", xfer="f32", mma=0, steps=0, delta=5.0, mu=0.005, eps=0.5),
        # an ordinary propagator on a new gauge field: load, adaptive setup and solve, one source
        dict(name="propagator_32x16x16x16_1rhs", kind="solve", lat="32x16x16x16", levels=2, nv=20, nv2=0, nrhs=1,
             whole=True, outer="f64", oe=0, sap="f32", xfer="f32", mma=1, steps=20, delta=5.0, mu=0.003, eps=0.5),
        # production: three levels, six sources at once, the mixed-precision settings of the benchmark
        dict(name="solve_64x32x32x32_3lvl_6rhs", kind="solve", lat="64x32x32x32", levels=3, nv=24, nv2=28, nrhs=6,
             whole=False, outer="f32x2", oe=1, sap="f16", xfer="f16", mma=1, steps=0, delta=5.0, mu=0.0009, eps=0.6),
        # the twelve spin-colour vectors of one point source through D(mu)
        dict(name="apply_f32_48x24x24x24_12rhs", kind="apply", lat="48x24x24x24", prec="f32", nrhs=12),
        # the outer solver's products at FP64 accuracy
        dict(name="apply_f32x2_48x24x24x24_6rhs", kind="apply", lat="48x24x24x24", prec="f32x2", nrhs=6),
        # the default smoother, one right-hand side
        dict(name="sap_f32_32x16x16x16_1rhs", kind="sap", lat="32x16x16x16", block="4x4x4x4", oe=0, sap="f32",
             sweeps=4, nrhs=1),
        # the benchmark's smoother: odd-even block solves on a 16-bit operator copy
        dict(name="sap_oe_f16_48x24x24x24_6rhs", kind="sap", lat="48x24x24x24", block="4x4x4x4", oe=1, sap="f16",
             sweeps=3, nrhs=6),
        # between the fine and the first coarse level with a 16-bit P
        dict(name="transfer_f16_48x24x24x24_6rhs", kind="transfer", lat="48x24x24x24", agg="4x4x4x4", nv=24,
             xfer="f16", nrhs=6),
        # the smoother of the first coarse level
        dict(name="sap1_f16_16x8x8x8_nv24_6rhs", kind="sap1", lat="16x8x8x8", nv=24, sap1="f16", sweeps=2, nrhs=6),
        # one step of the coarsest solve for twelve sources
        dict(name="schur_tf32_12x6x6x6_nv24_12rhs", kind="schur", lat="12x6x6x6", nv=24, mma=1, nrhs=12),
        # rebuilding the hierarchy from given test vectors
        dict(name="build_32x16x16x16_nv20", kind="build", lat="32x16x16x16", agg="4x4x4x4", nv=20, nrhs=4),
        # the learned layer: inference in FP16 and a training step's gradient in FP32
        dict(name="nn_16x16x16x16_16pairs", kind="nn", lat="16x16x16x16", prec="f16", nrhs=16),
    ]


def _lattice(rng, step, most_sites, lo=1):
    """Four extents, multiples of `step`, spread over the logarithm of the volume up to most_sites."""
    least = (lo * step) ** 4
    aim = math.exp(rng.uniform(math.log(least), math.log(most_sites)))
    dims = [lo * step] * 4
    while True:
        d = rng.randrange(4)
        more = [n + (step if k == d else 0) for k, n in enumerate(dims)]
        if _volume(more) > aim or more[d] > 6 * lo * step:
            return "x".join(str(n) for n in dims)
        dims = more


def draw(rng):
    kind = rng.choice(["solve", "apply", "apply", "sap", "sap", "transfer", "sap1", "schur", "build", "nn"])
    nrhs = min(12, int(math.exp(rng.uniform(0.0, math.log(13.0)))))
    if kind == "solve":
        case = dict(kind=kind, lat=_lattice(rng, 8, 150_000), levels=2, nv=rng.randint(8, 24), nv2=0, nrhs=min(nrhs, 6),
                    whole=rng.random() < 0.3, outer="f64", oe=0, sap="f32", xfer="f32", mma=0, steps=0,
                    delta=rng.choice([1.0, 5.0]), mu=rng.choice([0.002, 0.003, 0.005]), eps=0.5)
        if rng.random() < 0.4:
            case.update(lat=_lattice(rng, 16, 600_000), levels=3, nv2=rng.randint(8, 28))
        if rng.random() < 0.6:
            case.update(outer="f32x2", oe=1, sap=rng.choice(["f32", "f16", "bf16"]), mma=rng.choice([0, 1, 3]),
                        xfer=rng.choice(["f32", "f16"]))
        return case
    if kind == "apply":
        return dict(kind=kind, lat=_lattice(rng, 8, 700_000), prec=rng.choice(["f32", "f32", "f64", "f32x2"]),
                    nrhs=min(nrhs, 6))
    if kind == "sap":
        oe = rng.randint(0, 1)
        block = rng.choice(["4x4x4x4", "4x4x4x4", "2x2x2x2", "4x2x4x4"])
        return dict(kind=kind, lat=_lattice(rng, 8, 700_000), block=block, oe=oe,
                    sap=rng.choice(["f32", "f16", "bf16"]) if oe else rng.choice(["f32", "f32", "f64"]),
                    sweeps=rng.randint(1, 4), nrhs=min(nrhs, 7))
    if kind == "transfer":
        return dict(kind=kind, lat=_lattice(rng, 8, 700_000), agg=rng.choice(["4x4x4x4", "2x2x2x2"]),
                    nv=rng.randint(8, 24), xfer=rng.choice(["f32", "f16", "bf16"]), nrhs=min(nrhs, 8))
    if kind == "sap1":
        return dict(kind=kind, lat=_lattice(rng, 4, 8_192), nv=rng.randint(8, 24), sap1=rng.choice(["f32", "f16", "bf16"]),
                    sweeps=rng.randint(1, 3), nrhs=min(nrhs, 7))
    if kind == "schur":
        return dict(kind=kind, lat=_lattice(rng, 2, 3_000), nv=rng.randint(8, 28), mma=rng.choice([0, 1, 3]), nrhs=nrhs)
    if kind == "build":
        return dict(kind=kind, lat=_lattice(rng, 8, 140_000), agg=rng.choice(["4x4x4x4", "4x4x4x4", "2x2x2x2"]),
                    nv=rng.randint(8, 24), nrhs=min(nrhs, 4))
    return dict(kind=kind, lat=_lattice(rng, 8, 70_000), prec=rng.choice(["f32", "f16"]), nrhs=nrhs)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

class _Gen:
    """Random numbers of one seed on the device; every array has a stream of its own."""

    def __init__(self, seed):
        self.seed = int(seed)

    def normal(self, tag, *shape):
        g = torch.Generator(device="cuda")
        g.manual_seed(self.seed * 64 + tag)
        return torch.randn(*shape, dtype=torch.float64, device="cuda", generator=g)

    def cx(self, tag, *shape):
        """Complex Gaussian numbers that are FP32 numbers held in FP64."""
        return torch.view_as_complex(self.normal(tag, *shape, 2).float().double())

    def cx64(self, tag, *shape):
        return torch.view_as_complex(self.normal(tag, *shape, 2))


def _links(gen, dims, eps):
    """exp(i eps H), [T, Z, Y, X, 4, 3, 3]: the Taylor series of exp(i eps H / 16), squared four times."""
    h = gen.normal(1, 8, _volume(dims) * 4)
    s3 = 1.0 / math.sqrt(3.0)
    a = torch.zeros(3, 3, h.shape[1], dtype=torch.complex128, device="cuda")  # links last: 3 x 3 products by element
    a[0, 0] = h[2] + s3 * h[7]
    a[1, 1] = -h[2] + s3 * h[7]
    a[2, 2] = -2 * s3 * h[7]
    for (r, c), (x, y) in {(0, 1): (0, 1), (0, 2): (3, 4), (1, 2): (5, 6)}.items():
        a[r, c] = torch.complex(h[x], -h[y])
        a[c, r] = torch.complex(h[x], h[y])
    a *= 1j * eps / 2 / 16
    times = lambda p, q: sum(p[:, k, None] * q[None, k] for k in range(3))  # noqa: E731
    one = torch.eye(3, dtype=torch.complex128, device="cuda")[..., None]
    u = one + a / 12
    for k in range(11, 0, -1):
        u = one + times(a, u) / k
    for _ in range(4):
        u = times(u, u)
    u = u.permute(2, 0, 1)
    return u.reshape(*dims, 4, 3, 3).contiguous()


class _State:
    """A handle and the buffers that a program keeps beside it; the handle goes with the object."""

    def __init__(self, **params):
        agg2 = {k: params.pop(k) for k in ("agg2", "sap_block1") if k in params}
        p = tm.params(**params)
        for k, v in agg2.items():
            getattr(p, k)[:] = v
        self.h = None
        self.h = tm.tm_create(p, torch.cuda.current_stream())

    def __del__(self):
        if self.h is not None:
            tm.tm_destroy(self.h)
            self.h = None

    def field(self, level, prec, nrhs):
        n = tm.tm_field_bytes(self.h, level, PREC[prec], nrhs)
        return torch.zeros(n // (8 if prec == "f64" else 4), dtype=torch.float64 if prec == "f64" else torch.float32,
                           device="cuda")

    def pack(self, level, prec, natural):
        f = self.field(level, prec, natural.shape[0])
        tm.tm_pack(self.h, level, PREC[prec], natural.contiguous(), f, natural.shape[0])
        return f


def _solve_inputs(case, gen):
    dims = _dims(case["lat"])
    m0, c_sw = M0[case["eps"]]
    u = _links(gen, dims, case["eps"])
    nv = case["nv"]
    parts = [gen.cx64(2, nv * _volume(dims) * 12) * math.sqrt(0.5)]
    if case["levels"] == 3:
        parts.append(gen.cx64(3, case["nv2"] * _volume(dims) // 256 * 2 * nv) * math.sqrt(0.5))
    b = gen.cx64(4, case["nrhs"], *dims, 4, 3)
    return dims, m0, c_sw, u, torch.cat(parts), b


def prepare(case, seed):
    gen, kind, nrhs = _Gen(seed), case["kind"], case["nrhs"]
    if kind == "solve":
        dims, m0, c_sw, u, tv, b = _solve_inputs(case, gen)
        three = case["levels"] == 3
        more = dict(levels=3, nv2=case["nv2"], agg2=(2, 2, 2, 2), sap_block1=(2, 2, 2, 2), restart=4, post_smooth=3,
                    coarse_tol=0.1, sap1_prec=PREC[case["sap"]]) if three else {}
        s = _State(L=dims, m0=m0, c_sw=c_sw, mu=case["mu"], delta=case["delta"], nv=case["nv"], agg=(4, 4, 4, 4),
                   sap_block=(4, 4, 4, 4), setup_iters=3, cycle_prec=tm.TM_F32, max_rhs=nrhs,
                   outer_apply=PREC[case["outer"]], block_oe=case["oe"], sap_prec=PREC[case["sap"]],
                   transfer_prec=PREC[case["xfer"]], coarse_mma=case["mma"], coarsest_steps=case["steps"], **more)
        s.b, s.x = b, torch.zeros_like(b)
        if case["whole"]:
            s.gauge, s.tv = u, tv
        else:
            tm.tm_load_gauge(s.h, u)
            tm.tm_setup(s.h, tv)
    elif kind in ("apply", "sap", "nn"):
        dims = _dims(case["lat"])
        m0, c_sw = M0[0.5]
        oe = case.get("oe", 0)
        f64 = case.get("sap") == "f64"
        s = _State(L=dims, m0=m0, c_sw=c_sw, mu=0.003, delta=5.0, nv=1, agg=(4, 4, 4, 4),
                   sap_block=_dims(case.get("block", "4x4x4x4")), max_rhs=nrhs,
                   cycle_prec=tm.TM_F64 if f64 else tm.TM_F32,
                   outer_apply=tm.TM_F32X2 if case.get("prec") == "f32x2" else tm.TM_F64, block_oe=oe,
                   sap_prec=PREC[case["sap"]] if oe else tm.TM_F32)
        tm.tm_load_gauge(s.h, _links(gen, dims, 0.5))
        v = gen.cx(5, nrhs, *dims, 4, 3)
        if kind == "apply":
            s.x = s.pack(0, "f64" if case["prec"] == "f64" else "f32", v)
            s.y = s.field(0, "f32" if case["prec"] == "f32" else "f64", nrhs)
        elif kind == "sap":
            s.prec = "f64" if f64 else "f32"
            s.b, s.x0 = s.pack(0, s.prec, v), s.pack(0, s.prec, gen.cx(6, nrhs, *dims, 4, 3))
            s.x = torch.empty_like(s.x0)
        else:
            tm.tm_nn_set_weights(s.h, _weights(gen).cpu().numpy())
            s.r, s.e = s.pack(0, "f32", v), s.pack(0, "f32", gen.cx(6, nrhs, *dims, 4, 3))
            s.y = s.field(0, "f32", nrhs)
    else:
        s = _coarse_state(case, gen)
    s.case = dict(case)
    return s


def _weights(gen):
    return gen.cx(7, 2304) * 0.05


def _coarse_geometry(case):
    """(fine extents, aggregate) of the kinds that work on a coarse level."""
    if case["kind"] in ("transfer", "build"):
        return _dims(case["lat"]), _dims(case["agg"])
    return tuple(2 * n for n in _dims(case["lat"])), (2, 2, 2, 2)


def _coarse_state(case, gen):
    kind, nrhs, nv = case["kind"], case["nrhs"], case["nv"]
    dims, agg = _coarse_geometry(case)
    vc = _volume(dims) // _volume(agg)
    more = {}
    if kind == "sap1":
        more = dict(levels=3, nv2=1, agg2=(2, 2, 2, 2), sap_block1=(2, 2, 2, 2), sap1_prec=PREC[case["sap1"]])
    elif kind == "schur":
        more = dict(coarse_mma=case["mma"])
    elif kind == "transfer":
        more = dict(transfer_prec=PREC[case["xfer"]])
    m0, c_sw = M0[0.5]
    s = _State(L=dims, m0=m0, c_sw=c_sw, mu=0.003, delta=5.0, nv=nv, agg=agg, sap_block=(2, 2, 2, 2), max_rhs=nrhs,
               cycle_prec=tm.TM_F32, **more)
    tm.tm_load_gauge(s.h, _links(gen, dims, 0.5))
    tv = gen.cx(2, nv * _volume(dims) * 12)
    if kind == "sap1":
        tv = torch.cat([tv, gen.cx(3, vc * 2 * nv)])
    v = gen.cx(5, nrhs, vc, 2 * nv)
    if kind != "build":
        tm.tm_setup_from_vectors(s.h, tv)
    if kind == "transfer":
        s.f, s.fo = s.pack(0, "f32", gen.cx(6, nrhs, *dims, 4, 3)), s.field(0, "f32", nrhs)
        s.c, s.co = s.pack(1, "f32", v), s.field(1, "f32", nrhs)
    elif kind == "build":
        s.tv, s.c, s.co, s.fo = tv, s.pack(1, "f32", v), s.field(1, "f32", nrhs), s.field(0, "f32", nrhs)
    elif kind == "sap1":
        s.b, s.x0 = s.pack(1, "f32", v), s.pack(1, "f32", gen.cx(6, nrhs, vc, 2 * nv))
        s.x = torch.empty_like(s.x0)
    else:
        s.v = torch.view_as_real(gen.cx(6, nrhs, vc // 2, 2 * nv)).float().contiguous()
        s.y = torch.zeros_like(s.v)
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(s):
    case, h = s.case, s.h
    kind, nrhs = case["kind"], case["nrhs"]
    if kind == "solve":
        if case["whole"]:
            tm.tm_load_gauge(h, s.gauge)
            tm.tm_setup(h, s.tv)
        s.x.zero_()
        status, info = tm.tm_solve(h, s.b, s.x, nrhs, 1e-10)
        if status != tm.TM_OK:
            raise RuntimeError("the solve did not converge: %r" % (info.as_dict(),))
        return s.x
    if kind == "apply":
        tm.tm_apply(h, 0, PREC[case["prec"]], s.x, s.y, nrhs)
        return s.y
    if kind == "sap":
        s.x.copy_(s.x0)
        tm.tm_sap(h, PREC[s.prec], s.b, s.x, case["sweeps"], nrhs)
        return s.x
    if kind == "transfer":
        tm.tm_restrict(h, tm.TM_F32, s.f, s.co, nrhs)
        tm.tm_prolong(h, tm.TM_F32, s.c, s.fo, nrhs, 0)
        return s.co, s.fo
    if kind == "sap1":
        s.x.copy_(s.x0)
        tm.tm_sap1(h, tm.TM_F32, s.b, s.x, case["sweeps"], nrhs)
        return s.x
    if kind == "schur":
        tm.tm_schur(h, tm.TM_F32, s.v, s.y, nrhs)
        return s.y
    if kind == "build":
        tm.tm_setup_from_vectors(h, s.tv)
        tm.tm_prolong(h, tm.TM_F32, s.c, s.fo, nrhs, 0)
        tm.tm_apply(h, 1, tm.TM_F32, s.c, s.co, nrhs)
        return s.fo, s.co
    tm.tm_nn_apply(h, PREC[case["prec"]], s.r, s.y, nrhs)
    loss, grad = tm.tm_nn_grad(h, s.r, s.e, nrhs)
    return s.y, loss, grad


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

D_FLOPS = 2232.0           # real operations of D(mu) per site
SAP_OE_FLOPS = 10356.0     # residual and four MR steps of an odd-even 4^4 block solve, per site


def work(case):
    kind, nrhs = case["kind"], case["nrhs"]
    dims = _dims(case["lat"])
    v = _volume(dims)
    if kind == "solve":
        # nominal: ten outer iterations, each a K-cycle with three sweeps and one product with D(mu); the
        # operator and the Krylov vectors once per iteration; an adaptive setup is three such K-cycles on
        # every test vector
        n = 10.0 * nrhs + (3.0 * case["nv"] if case["whole"] else 0.0)
        return {"flops": v * n * (3 * SAP_OE_FLOPS + D_FLOPS + 16 * 24 * case["nv"]),
                "bytes": v * (10.0 * (480 * 3 + 24 * 4 * case["nv"] * 2) + n * (3 * 288 + 10 * 192))}
    if kind == "apply":
        size = 8 if case["prec"] == "f64" else 4
        op, vec = (1152, 96 + 192) if case["prec"] == "f32x2" else (120 * size, 48 * size)
        return {"bytes": v * (op + nrhs * vec), "flops": v * nrhs * D_FLOPS}
    if kind == "sap":
        size = {"f64": 8, "f32": 4}.get(case["sap"], 2)
        vec = 8 if case["sap"] == "f64" else 4
        per = SAP_OE_FLOPS if case["oe"] else 5 * D_FLOPS
        return {"bytes": v * ((120 + (72 if case["oe"] else 0)) * size + nrhs * 72 * vec),
                "flops": v * nrhs * case["sweeps"] * per}
    if kind == "nn":
        return {"bytes": v * (48 * 4 + nrhs * 96 * 3.0), "flops": v * nrhs * 5.0 * 8 * (8 * 9 * 48 + 8 * 36)}
    nv, n = case["nv"], 2 * case["nv"]
    if kind == "transfer":
        size = 4 if case["xfer"] == "f32" else 2
        return {"bytes": v * (2 * 24 * nv * size + nrhs * 192), "flops": v * nrhs * nv * 12 * 8 * 2}
    if kind == "sap1":
        size = 8 if case["sap1"] == "f32" else 4
        return {"bytes": v * (9.0 * n * n * size + nrhs * n * 24), "flops": v * nrhs * case["sweeps"] * 8.0 * n * n * 29}
    if kind == "schur":
        return {"bytes": v / 2 * (17.0 * n * n * 8 + nrhs * n * 16), "flops": v / 2 * nrhs * 8.0 * n * n * 18}
    agg = _volume(_dims(case["agg"]))
    face = sum(agg // a for a in _dims(case["agg"])) * 2
    return {"bytes": v * nv * (192 + 96.0 * 2) + v / agg * 9.0 * n * n * 8,
            "flops": v / agg * 8.0 * (n * n * 6 * (agg + face) + 430.0 * nv * agg)}


def tolerance(case):
    """About four times the distance from `exact` that was measured; a 16-bit operator copy, TF32 products and FP16
    hidden channels are the larger part of it where there are any."""
    kind = case["kind"]
    by = {"f64": 1e-14, "f32": 1e-6, "f16": 1.2e-3, "bf16": 1e-2}
    if kind == "solve":
        return {"rel": 1e-8}  # solutions to residual 1e-10 and 1e-12 differ by up to 7e-10
    if kind == "apply":
        return {"rel": {"f32": 5e-7, "f64": 2e-15, "f32x2": 5e-14}[case["prec"]]}
    if kind == "sap":
        return {"rel": by[case["sap"]]}
    if kind == "transfer":
        return {"rel": by[case["xfer"]]}
    if kind == "sap1":
        return {"rel": by[case["sap1"]]}
    if kind == "schur":
        return {"rel": 1e-3 if case["mma"] in (1, 2) else 4e-6}
    if kind == "nn":
        return {"rel": 1.5e-3 if case["prec"] == "f16" else 2e-6}
    return {"rel": 4e-6}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------

def _gammas():
    s = torch.zeros(3, 2, 2, dtype=torch.complex128)
    s[0, 0, 1] = s[0, 1, 0] = 1
    s[1, 0, 1], s[1, 1, 0] = -1j, 1j
    s[2, 0, 0], s[2, 1, 1] = 1, -1
    upper = [-torch.eye(2, dtype=torch.complex128), -1j * s[2], -1j * s[1], -1j * s[0]]
    g = torch.zeros(4, 4, 4, dtype=torch.complex128)
    for k, a in enumerate(upper):
        g[k, :2, 2:], g[k, 2:, :2] = a, a.conj().T
    return g.cuda()


class _Exact:
    """D(mu), its blocks and its coarse projections in complex128; vectors [R, T, Z, Y, X, 4, 3]."""

    def __init__(self, u, m0, c_sw, mu):
        self.u, self.dims, self.mu = u, tuple(u.shape[:4]), mu
        self.gamma = _gammas()
        self.one = torch.eye(4, dtype=torch.complex128, device="cuda")
        self.g5 = torch.tensor([-1.0, -1.0, 1.0, 1.0], dtype=torch.float64, device="cuda")
        dag = lambda a: a.conj().transpose(-1, -2)  # noqa: E731
        to = lambda a, d, n: torch.roll(a, -n, d)   # noqa: E731  the field at x + n d
        m = torch.zeros(*self.dims, 12, 12, dtype=torch.complex128, device="cuda")
        for a in range(4):
            for b in range(a):
                ua, ub = u[..., a, :, :], u[..., b, :, :]
                # the four plaquettes of the a-b plane that start and end at x
                q = ua @ to(ub, a, 1) @ dag(to(ua, b, 1)) @ dag(ub)
                q = q + ub @ dag(to(to(ua, b, 1), a, -1)) @ dag(to(ub, a, -1)) @ to(ua, a, -1)
                q = q + dag(to(ua, a, -1)) @ dag(to(to(ub, a, -1), b, -1)) @ to(to(ua, a, -1), b, -1) @ to(ub, b, -1)
                q = q + dag(to(ub, b, -1)) @ to(ua, b, -1) @ to(to(ub, b, -1), a, 1) @ dag(ua)
                s = 2 * (self.gamma[a] @ self.gamma[b])  # the a-b and the b-a term are equal
                m += torch.einsum("st,...kl->...sktl", s, q - dag(q)).reshape(*self.dims, 12, 12)
        m *= -c_sw / 32
        m += (m0 + 4) * torch.eye(12, dtype=torch.complex128, device="cuda")
        self.a = m

    def transport(self, psi, d, back):
        """U(x) psi(x + d), or U(x - d)^dagger psi(x - d), antiperiodic in T; psi [..., T, Z, Y, X, 4, 3]."""
        at = psi.dim() - 6 + d
        u = self.u[..., d, :, :]
        if back:
            y = torch.roll(torch.einsum("tzyxba,...tzyxsb->...tzyxsa", u.conj(), psi), 1, at)
        else:
            y = torch.einsum("tzyxab,...tzyxsb->...tzyxsa", u, torch.roll(psi, -1, at))
        if d == 0:
            y.select(at, 0 if back else self.dims[0] - 1).neg_()
        return y

    def hop(self, psi, d, back):
        p = self.one + self.gamma[d] if back else self.one - self.gamma[d]
        return -0.5 * torch.einsum("st,...tc->...sc", p, self.transport(psi, d, back))

    def diag(self, psi, mu=None):
        y = torch.einsum("tzyxij,...tzyxj->...tzyxi", self.a, psi.flatten(-2)).reshape(psi.shape)
        return y + 1j * (self.mu if mu is None else mu) * self.g5[:, None] * psi

    def apply(self, psi, mu=None):
        y = self.diag(psi, mu)
        for d in range(4):
            y = y + self.hop(psi, d, False) + self.hop(psi, d, True)
        return y

    # -- blocks ---------------------------------------------------------------------------------
    def blocks(self, block):
        c = torch.meshgrid(*[torch.arange(n, device="cuda") for n in self.dims], indexing="ij")
        self.block = block
        self.colour = sum(c[d] // block[d] for d in range(4)) % 2
        self.odd = (sum(c) % 2)[..., None, None]
        self.inside = [((c[d] % block[d] < block[d] - 1)[..., None, None], (c[d] % block[d] > 0)[..., None, None])
                       for d in range(4)]

    def block_hops(self, psi):
        y = 0
        for d in range(4):
            y = y + self.inside[d][0] * self.hop(psi, d, False) + self.inside[d][1] * self.hop(psi, d, True)
        return y

    def block_dot(self, a, b):
        p = (a.conj() * b).sum((-2, -1))
        shape = [p.shape[0]]
        for n, k in zip(self.dims, self.block):
            shape += [n // k, k]
        p = p.reshape(shape).sum((2, 4, 6, 8))
        for d in range(4):
            p = p.repeat_interleave(self.block[d], d + 1)
        return p[..., None, None]

    def minimal_residual(self, op, r, steps):
        e = torch.zeros_like(r)
        for _ in range(steps):
            q = op(r)
            qq = self.block_dot(q, q).real
            alpha = torch.where(qq > 0, self.block_dot(q, r) / torch.where(qq > 0, qq, 1.0), 0)
            e = e + alpha * r
            r = r - alpha * q
        return e

    def sap(self, b, x, sweeps, oe):
        if oe:
            m = self.a + 1j * self.mu * torch.diag(self.g5.repeat_interleave(3).to(torch.complex128))
            inv = torch.linalg.inv(m)
            dinv = lambda f: self.odd * torch.einsum("tzyxij,...tzyxj->...tzyxi", inv, f.flatten(-2)).reshape(f.shape)  # noqa: E731
            even = 1 - self.odd
            schur = lambda f: even * (self.diag(f) - self.block_hops(dinv(self.block_hops(f))))  # noqa: E731
        for _ in range(sweeps):
            for colour in (0, 1):
                mask = (self.colour == colour)[..., None, None]
                r = mask * (b - self.apply(x))
                if oe:
                    e = self.minimal_residual(schur, even * (r - self.block_hops(dinv(r))), 4)
                    e = e + dinv(r - self.block_hops(e))
                else:
                    e = self.minimal_residual(lambda f: self.diag(f) + self.block_hops(f), r, 4)
                x = x + mask * e
        return x

    # -- aggregation ----------------------------------------------------------------------------
    def split(self, psi):
        """[R, T, Z, Y, X, 4, 3] as [R, aggregate, chirality, rows]."""
        r, g = psi.shape[0], self.agg
        n = [a // b for a, b in zip(self.dims, g)]
        f = psi.reshape(r, n[0], g[0], n[1], g[1], n[2], g[2], n[3], g[3], 2, 6)
        f = f.permute(0, 1, 3, 5, 7, 9, 2, 4, 6, 8, 10)
        return f.reshape(r, _volume(n), 2, _volume(g) * 6)

    def join(self, f):
        r, g = f.shape[0], self.agg
        n = [a // b for a, b in zip(self.dims, g)]
        f = f.reshape(r, *n, 2, *g, 6).permute(0, 1, 6, 2, 7, 3, 8, 4, 9, 5, 10)
        return f.reshape(r, *self.dims, 4, 3)

    def aggregate(self, tv, agg):
        """P from the test vectors: the orthonormal factor of each aggregate and chirality."""
        self.agg = agg
        self.cdims = tuple(a // b for a, b in zip(self.dims, agg))
        f = self.split(tv).permute(1, 2, 3, 0)
        self.p = torch.empty_like(f)
        for k in range(0, f.shape[0], 512):
            q, r = torch.linalg.qr(f[k:k + 512])
            ph = torch.diagonal(r, dim1=-2, dim2=-1)
            self.p[k:k + 512] = q * (ph / ph.abs())[..., None, :]
        self.nv = self.p.shape[-1]

    def restrict(self, psi):
        return torch.einsum("acij,raci->racj", self.p.conj(), self.split(psi)).flatten(2)

    def prolong(self, c):
        c = c.reshape(c.shape[0], -1, 2, self.nv)
        return self.join(torch.einsum("acij,racj->raci", self.p, c))

    def coarse(self, c, mu):
        g5 = torch.ones(2 * self.nv, dtype=torch.float64, device="cuda")
        g5[:self.nv] = -1
        y = torch.empty_like(c)
        for k in range(c.shape[0]):
            y[k:k + 1] = self.restrict(self.apply(self.prolong(c[k:k + 1]), 0.0))
        return y + 1j * mu * g5 * c

    def coarse_blocks(self, mu):
        """The nine blocks of D_c + i mu Gamma5_c, [site, 9, row, column]."""
        n, vc = 2 * self.nv, _volume(self.cdims)
        out = torch.zeros(vc, 9, n, n, dtype=torch.complex128, device="cuda")
        self.blocks(self.agg)
        for k in range(n):
            unit = torch.zeros(1, vc, n, dtype=torch.complex128, device="cuda")
            unit[..., k] = 1
            f = self.prolong(unit)
            own = self.diag(f, 0.0)
            for d in range(4):
                for back in (False, True):
                    w, inside = self.hop(f, d, back), self.inside[d][int(back)]
                    own = own + inside * w
                    out[:, 1 + 2 * d + int(back), :, k] = self.restrict(~inside * w)[0]
            out[:, 0, :, k] = self.restrict(own)[0]
        i = torch.arange(n, device="cuda")
        out[:, 0, i, i] += 1j * mu * torch.where(i < self.nv, -1.0, 1.0)
        return out

    # -- the learned layer ------------------------------------------------------------------------
    def layer(self, psi, w):
        """psi [Cin, T, Z, Y, X, 4, 3], w [Cout, Cin, 9, 4, 4]."""
        y = torch.einsum("oist,i...tc->o...sc", w[:, :, 0], psi)
        for d in range(4):
            for back in (False, True):
                y = y + torch.einsum("oist,i...tc->o...sc", w[:, :, 1 + 2 * d + int(back)], self.transport(psi, d, back))
        return y


def _chunked(psi, dtype):
    """Natural spinors in the library's field layout: [R][6 chunks][V][4 reals]."""
    f = torch.view_as_real(psi.resolve_conj().contiguous()).reshape(psi.shape[0], -1, 6, 4)
    return f.permute(0, 2, 1, 3).contiguous().reshape(-1).to(dtype)


def _flat(c):
    return torch.view_as_real(c.contiguous()).reshape(-1)


def _coarse_neighbours(dims):
    idx = torch.arange(_volume(dims), device="cuda").reshape(dims)
    nb = [idx]
    for d in range(4):
        nb += [torch.roll(idx, -1, d), torch.roll(idx, 1, d)]
    return [t.reshape(-1) for t in nb]


def exact(case, seed):
    kind, nrhs = case["kind"], case["nrhs"]
    if kind == "solve":
        return None  # a solve to 1e-10 without a preconditioner takes minutes
    gen = _Gen(seed)
    m0, c_sw = M0[0.5]
    if kind in ("apply", "sap", "nn"):
        dims = _dims(case["lat"])
        x = _Exact(_links(gen, dims, 0.5), m0, c_sw, 0.003)
        v = gen.cx(5, nrhs, *dims, 4, 3)
        each = lambda f: torch.cat([f(k) for k in range(nrhs)])  # noqa: E731
        if kind == "apply":
            return _chunked(each(lambda k: x.apply(v[k:k + 1])), torch.float64)
        if kind == "sap":
            x.blocks(_dims(case["block"]))
            x0 = gen.cx(6, nrhs, *dims, 4, 3)
            return _chunked(each(lambda k: x.sap(v[k:k + 1], x0[k:k + 1], case["sweeps"], case["oe"])), torch.float64)
        e = gen.cx(6, nrhs, *dims, 4, 3)
        w = _weights(gen).requires_grad_(True)
        w1, w2 = w[:1152].reshape(8, 1, 9, 4, 4), w[1152:].reshape(1, 8, 9, 4, 4)
        total, loss, ys = float((e.abs() ** 2).sum()), 0.0, []
        for k in range(nrhs):
            y = x.layer(x.layer(v[k:k + 1], w1), w2)
            one = (y - e[k:k + 1]).abs().square().sum() / total
            one.backward()
            loss += float(one.detach())
            ys.append(y.detach())
            w1, w2 = w[:1152].reshape(8, 1, 9, 4, 4), w[1152:].reshape(1, 8, 9, 4, 4)
        # torch's gradient of a real loss is twice the derivative with respect to the conjugate
        return _chunked(torch.cat(ys), torch.float64), loss, (w.grad / 2).cpu().numpy()
    nv = case["nv"]
    dims, agg = _coarse_geometry(case)
    x = _Exact(_links(gen, dims, 0.5), m0, c_sw, 0.003)
    x.aggregate(gen.cx(2, nv * _volume(dims) * 12).reshape(nv, *dims, 4, 3), agg)
    vc, n, mu_c = _volume(x.cdims), 2 * nv, 5.0 * 0.003
    v = gen.cx(5, nrhs, vc, n)
    if kind == "transfer":
        f = gen.cx(6, nrhs, *dims, 4, 3)
        return _flat(x.restrict(f)), _chunked(x.prolong(v), torch.float64)
    if kind == "build":
        return _chunked(x.prolong(v), torch.float64), _flat(x.coarse(v, mu_c))
    nb = _coarse_neighbours(x.cdims)
    if kind == "sap1":
        return _flat(_sap1(x.coarse_blocks(0.003), nb, x.cdims, v, gen.cx(6, nrhs, vc, n), case["sweeps"]))
    blocks = x.coarse_blocks(mu_c)
    c = torch.meshgrid(*[torch.arange(k, device="cuda") for k in x.cdims], indexing="ij")
    odd = (sum(c) % 2).reshape(-1).bool()
    full = torch.zeros(nrhs, vc, n, dtype=torch.complex128, device="cuda")
    full[:, ~odd] = gen.cx(6, nrhs, vc // 2, n)
    hop = lambda f: sum(torch.einsum("vij,rvj->rvi", blocks[:, t], f[:, nb[t]]) for t in range(1, 9))  # noqa: E731
    mid = torch.zeros_like(full)
    mid[:, odd] = torch.einsum("vij,rvj->rvi", torch.linalg.inv(blocks[odd, 0]), hop(full)[:, odd])
    return torch.view_as_real((torch.einsum("vij,rvj->rvi", blocks[:, 0], full) - hop(mid))[:, ~odd].contiguous())


def _sap1(blocks, nb, dims, b, x, sweeps):
    """Red and black sweeps over 2^4 blocks of the coarse lattice, four MR steps per block."""
    c = torch.stack(torch.meshgrid(*[torch.arange(k, device="cuda") for k in dims], indexing="ij")).reshape(4, -1)
    colour = ((c // 2).sum(0) % 2)
    half = [k // 2 for k in dims]
    block = ((c[0] // 2 * half[1] + c[1] // 2) * half[2] + c[2] // 2) * half[3] + c[3] // 2
    inside = [torch.ones_like(colour).bool()] + [m for d in range(4) for m in (c[d] % 2 == 0, c[d] % 2 == 1)]

    def apply(f, within):
        y = 0
        for t in range(9):
            w = torch.einsum("vij,rvj->rvi", blocks[:, t], f[:, nb[t]])
            y = y + (w * inside[t][None, :, None] if within else w)
        return y

    def dot(p, q):
        s = torch.zeros(p.shape[0], _volume(half), dtype=torch.complex128, device="cuda")
        s.index_add_(1, block, (p.conj() * q).sum(-1))
        return s[:, block][..., None]

    for _ in range(sweeps):
        for k in (0, 1):
            mask = (colour == k)[None, :, None]
            r = mask * (b - apply(x, False))
            e = torch.zeros_like(r)
            for _ in range(4):
                q = mask * apply(r, True)
                qq = dot(q, q).real
                alpha = torch.where(qq > 0, dot(q, r) / torch.where(qq > 0, qq, 1.0), 0)
                e = e + alpha * r
                r = r - alpha * q
            x = x + e
    return x
