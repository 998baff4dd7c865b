"""Band kernels and the magnitudes of their inputs, against the fp64 CPU oracle: what the scales of the FP16 parts must not lose."""
import math

import numpy as np
import pytest
import torch

from oracle import sna_oracle as orc
from paper_2505_11157_b200 import sna
from paper_2505_11157_b200.synthetic import make_inputs, small_workload

pytestmark = pytest.mark.gpu

# relative error of a product of split operands (2^-22 each way, see test_gpu_band.py), of single products in reduced precision
TOL = {"fp32": 5e-6, "tf32": 3e-3}
SHAPE, CUTOFF = (16, 32, 16, 32), 0.6


def run(shape, theta, q, k, v, dout, precision="fp32", recompute=False, **plan_args):
    """([out, dq, dk, dv], the oracle's) as float64 arrays."""
    g = orc.geometry(*shape, 0, 0, theta)
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (q, k, v, dout)]
    with sna.Plan(*shape, 0, 0, theta, **plan_args) as plan:
        out, lse = plan.forward(*dev[:3], return_lse=True, precision=precision)
        grads = plan.backward(*dev, precision=precision, **({} if recompute else {"out": out, "lse": lse}))
        torch.cuda.synchronize()
        sna.sna_plan_check(plan.handle)
    refs = [orc.forward(g, q, k, v), *orc.backward(g, q, k, v, dout)]
    return [t.cpu().numpy().astype(np.float64).reshape(r.shape) for t, r in zip((out, *grads), refs)], refs


def rel(x, ref):
    return float(np.linalg.norm(x - ref) / np.linalg.norm(ref))


def rel_points(x, ref):
    """The largest relative error of a grid point's channel vector."""
    return float(np.max(np.linalg.norm(x - ref, axis=-1) / np.maximum(np.linalg.norm(ref, axis=-1), 1e-300)))


@pytest.mark.parametrize("C", [16, 24, 32, 64])
@pytest.mark.parametrize("precision", ["fp32", "tf32"])
@pytest.mark.parametrize("slices", [2, 300])      # streams shared by a block's warps, and private
def test_peaked_softmax(C, precision, slices):
    """Scores that spread over hundreds of nats: the first weights of a stream may be 2^-126 of the later ones."""
    if precision == "tf32" and C == 24:
        pytest.skip("no such width")
    for factor in (4, 10, 15):
        wl = small_workload("peaked", *SHAPE, 0, 0, CUTOFF, 1, slices, C, 91)
        q, k, v, dout = make_inputs(wl)
        q *= np.float32(factor); k *= np.float32(factor)
        if slices > 2:      # the same slice everywhere: the oracle's time
            q, k, v, dout = (np.array(np.broadcast_to(a[:, :1], a.shape)) for a in (q, k, v, dout))
        # a score has an absolute error of 2^-22 (2^-11) of the sum of |q k| and of 2^-23 of itself and of lse
        largest = float(np.abs(q).max() * np.abs(k).max() * math.sqrt(C))
        got, refs = run_slices(q, k, v, dout, precision, slices > 2)
        for name, x, r in zip(("out", "dq", "dk", "dv"), got, refs):
            assert np.isfinite(x).all(), (name, factor)
            if precision == "fp32":
                assert rel(x, r) <= TOL["fp32"] * max(1.0, largest / 5), (name, factor)


def run_slices(q, k, v, dout, precision, same):
    if not same:
        return run(SHAPE, CUTOFF, q, k, v, dout, precision)
    got, refs = run(SHAPE, CUTOFF, *(np.ascontiguousarray(a[:, :1]) for a in (q, k, v, dout)), precision)
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (q, k, v, dout)]
    with sna.Plan(*SHAPE, 0, 0, CUTOFF) as plan:
        out, lse = plan.forward(*dev[:3], return_lse=True, precision=precision)
        grads = plan.backward(*dev, out=out, lse=lse, precision=precision)
    return [t[:, -1:].cpu().numpy().astype(np.float64).reshape(r.shape) for t, r in zip((out, *grads), refs)], refs


@pytest.mark.parametrize("C", [16, 24, 32, 64])
def test_a_gap_between_the_first_scores_and_the_largest(C):
    """Every third ring's keys lie `gap` nats below the others, so that many streams begin with weights of e^-gap."""
    wl = small_workload("gap", *SHAPE, 0, 0, CUTOFF, 1, 2, C, 73)
    q, k, v, dout = make_inputs(wl)
    q, k = q * np.float32(0.1), k * np.float32(0.1)
    q[..., 0] = 1.0
    for gap in range(60, 100, 2):
        k[..., 0] = 0.0
        k[:, :, ::3, :, 0] = -gap * math.sqrt(C)
        for recompute in (False, True):
            got, refs = run(SHAPE, CUTOFF, q, k, v, dout, recompute=recompute)
            for name, x, r in zip(("out", "dq", "dk", "dv"), got, refs):
                assert rel(x, r) <= TOL["fp32"] * 4, (name, gap)       # |s| up to 100 nats in the excluded rings, 20 relative to lse


@pytest.mark.parametrize("shape, C", [((64, 128, 64, 128), 16), ((40, 80, 40, 80), 64)], ids=["64x128", "40x80"])
def test_small_probabilities_of_global_attention(shape, C):
    """Near the poles each of the points gets 2^-20 and less of every output point's attention: dv there is as accurate as elsewhere."""
    wl = small_workload("global", *shape, 0, 0, math.pi, 1, 1, C, 75)
    got, refs = run(shape, math.pi, *make_inputs(wl), global_attention=True)
    for name, x, r in zip(("out", "dq", "dk", "dv"), got, refs):
        assert rel_points(x, r) <= TOL["fp32"], name


@pytest.mark.parametrize("C", [16, 32, 64])
def test_keys_that_little_attention_reaches(C):
    """Pairs of rings whose keys lie `gap` nats below the others: their dk and dv are as small, not lost."""
    wl = small_workload("little", *SHAPE, 0, 0, CUTOFF, 1, 2, C, 76)
    q, k, v, dout = make_inputs(wl)
    q, k = q * np.float32(0.1), k * np.float32(0.1)
    q[..., 0] = 1.0
    for gap in (5, 15, 30, 60):
        k[..., 0] = 0.0
        for h in (4, 5, 10, 11):
            k[:, :, h, :, 0] = -gap * math.sqrt(C)
        got, refs = run(SHAPE, CUTOFF, q, k, v, dout)
        for name, x, r in zip(("dk", "dv"), got[2:], refs[2:]):
            # p = e^(s - lse): relative to the gap s carries 2^-22 from its split operands, 2^-23 from each of three accumulations (the
            # tensor core truncates) and 2^-24 from each of four fp32 roundings (q log2 e, the scaled sum, lse log2 e, the difference)
            assert rel_points(x[:, :, [4, 5, 10, 11]], r[:, :, [4, 5, 10, 11]]) <= TOL["fp32"] + gap * 7 * 2.0 ** -23, (name, gap)


def yardsticks(q, k, v, dout):
    """For out, dq, dk, dv: the sums of the magnitudes of their terms, in which rounding errors are measured (dense, one grid)."""
    with sna.Plan(*SHAPE, 0, 0, CUTOFF, host_only=True) as plan:
        ptr, lat, off = plan.table()
        omega = np.repeat(plan.quad_weights(), SHAPE[1])
    n = SHAPE[0] * SHAPE[1]
    member = np.zeros((n, n), dtype=bool)
    for h in range(SHAPE[0]):
        for w in range(SHAPE[1]):
            e = slice(ptr[h], ptr[h + 1])
            member[h * SHAPE[1] + w, lat[e] * SHAPE[1] + (w + off[e]) % SHAPE[1]] = True
    flat = [a.astype(np.float64).reshape(-1, n, a.shape[-1]) for a in (q, k, v, dout)]
    scale = 1 / math.sqrt(q.shape[-1])
    with np.errstate(all="ignore"):
        s = scale * flat[0] @ flat[1].transpose(0, 2, 1)
        s = np.where(member, s, -np.inf)
        p = np.exp(s - s.max(axis=-1, keepdims=True)) * omega
        p /= p.sum(axis=-1, keepdims=True)
    aq, ak, av, ad = (np.abs(a) for a in flat)
    t = ad @ av.transpose(0, 2, 1)
    ds = scale * p * (t + (p * t).sum(axis=-1, keepdims=True))
    pt, dst = p.transpose(0, 2, 1), ds.transpose(0, 2, 1)
    return [a.reshape(q.shape) for a in (p @ av, ds @ ak, dst @ aq, pt @ ad)]


def spread(which, q, k, v, dout):
    """Inputs of very unequal magnitudes; scores stay of order 1 to 10, but for one point's in point_q and point_k."""
    C, (array, kind) = q.shape[-1], which.split("_")
    factor = {"channel": np.where(np.arange(C) == 0, 5e4, 1e-5), "mild": np.where(np.arange(C) == 0, 100, 1e-6),
              "ramp": np.exp2(-np.linspace(0, 24, 16)).reshape(16, 1, 1), "point": np.ones(1)}[kind].astype(np.float32)
    x = dict(q=q, k=k, v=v, dout=dout)
    other = {"q": "k", "k": "q"}.get(array)
    x[array] = x[array] * factor
    if kind == "channel" and other:
        x[other] = x[other] / factor
    if kind == "point":
        x[array] = x[array].copy()
        x[array][..., 7, 9, :] *= np.float32(1e20 if array in ("v", "dout") else 1e7)
    return x["q"], x["k"], x["v"], x["dout"]


@pytest.mark.parametrize("which", [f"{a}_{kind}" for kind in ("channel", "ramp", "point") for a in ("q", "k", "v", "dout")] + ["v_mild", "dout_mild"])
@pytest.mark.parametrize("C, precision, slices", [(16, "fp32", 1), (24, "fp32", 2), (32, "fp32", 2), (64, "fp32", 60), (32, "tf32", 2), (64, "tf32", 1)])
def test_unequal_magnitudes(which, C, precision, slices):
    """Small channels beside large ones, rows that get smaller along a stream, one large point beside small ones whose windows do not
    hold it: every element keeps its accuracy relative to its own terms.  2^-17 is what the floor of the FP16 parts may take of a
    sum (2^-11 in reduced precision), and the products have 2^-21 (2^-10 each way) besides."""
    wl = small_workload("spread", *SHAPE, 0, 0, CUTOFF, 1, 1, C, 77)
    q, k, v, dout = spread(which, *make_inputs(wl))
    yards = yardsticks(q, k, v, dout)
    same = [np.array(np.broadcast_to(a, (1, slices, *a.shape[2:])), order="C") for a in (q, k, v, dout)]
    g = orc.geometry(*SHAPE, 0, 0, CUTOFF)
    refs = [orc.forward(g, q, k, v), *orc.backward(g, q, k, v, dout)]
    dev = [torch.from_numpy(a).cuda() for a in same]
    with sna.Plan(*SHAPE, 0, 0, CUTOFF) as plan:
        out, lse = plan.forward(*dev[:3], return_lse=True, precision=precision)
        grads = plan.backward(*dev, out=out, lse=lse, precision=precision)
        torch.cuda.synchronize()
    bound = 2e-5 if precision == "fp32" else 1e-2
    for name, x, r, y in zip(("out", "dq", "dk", "dv"), (out, *grads), refs, yards):
        if which in ("q_point", "k_point") and name != "out":
            continue        # (fp32 cannot hold p of scores of 1e7)
        x = x[:, -1:].cpu().numpy().astype(np.float64)
        keep = np.ones(SHAPE[2:], dtype=bool)
        if which == "q_point":
            keep[7, 9] = False
        if which == "k_point":      # the points whose scores it takes part in
            keep = ~attending(7, 9)
        error = np.abs(x - r.reshape(x.shape))[..., keep, :]
        assert np.all(error <= bound * y.reshape(x.shape)[..., keep, :] + 1e-36), (name, np.max(error / y.reshape(x.shape)[..., keep, :]))


def attending(lat, lon):
    """Output points whose window holds the input point (lat, lon)."""
    with sna.Plan(*SHAPE, 0, 0, CUTOFF, host_only=True) as plan:
        ptr, lats, offs = plan.table()
    hit = np.zeros(SHAPE[2:], dtype=bool)
    for h in range(SHAPE[2]):
        for la, off in zip(lats[ptr[h]:ptr[h + 1]], offs[ptr[h]:ptr[h + 1]]):
            if la == lat:
                hit[h, (lon - off) % SHAPE[3]] = True
    return hit


@pytest.mark.parametrize("value", [math.inf, -math.inf, math.nan])
@pytest.mark.parametrize("C", [16, 24, 32, 64])
def test_what_is_not_finite_stays_with_the_points_that_attend_to_it(C, value):
    """A point that is not finite, in q, k or v: the outputs and dq that do not depend on it are what they are without it."""
    wl = small_workload("nonfinite", *SHAPE, 0, 0, CUTOFF, 1, 1, C, 78)
    q, k, v, dout = make_inputs(wl)
    refs = run(SHAPE, CUTOFF, q, k, v, dout)[1]
    hit = attending(7, 9)
    alone = np.zeros_like(hit)
    alone[7, 9] = True
    for name, touched in (("q", alone), ("k", hit), ("v", hit)):
        x = dict(q=q.copy(), k=k.copy(), v=v.copy())
        x[name][..., 7, 9, :] = value
        dev = [torch.from_numpy(x[n]).cuda() for n in "qkv"] + [torch.from_numpy(dout).cuda()]
        with sna.Plan(*SHAPE, 0, 0, CUTOFF) as plan:
            out, lse = plan.forward(*dev[:3], return_lse=True)
            dq = plan.backward(*dev, out=out, lse=lse)[0]
        for got, ref in ((out, refs[0]), (dq, refs[1])):
            got = got.cpu().numpy().astype(np.float64).reshape(ref.shape)
            assert rel_points(got[..., ~touched, :], ref[..., ~touched, :]) <= 4 * TOL["fp32"], name
            if name != "k":     # (a key that is not finite may get a weight of zero)
                assert not np.isfinite(got[..., touched, :]).any(), name


@pytest.mark.parametrize("C, precision", [(16, "fp32"), (32, "fp32"), (64, "fp32"), (32, "tf32")])
def test_channels_and_regions_of_zeros(C, precision):
    """Zeros are not small values: a channel of v, the dout of a region, and all of v."""
    wl = small_workload("zeros", *SHAPE, 0, 0, CUTOFF, 1, 2, C, 79)
    q, k, v, dout = make_inputs(wl)
    v[..., 3] = 0.0
    dout[:, :, 6:, 10:20] = 0.0
    for x in ((q, k, v, dout), (q, k, 0 * v, dout), (q, k, v, 0 * dout)):
        got, refs = run(SHAPE, CUTOFF, *x, precision)
        for name, a, r in zip(("out", "dq", "dk", "dv"), got, refs):
            assert not a[r == 0].any() or name == "dq", name       # (dq of a point whose t is D: zero but for rounding)
            assert np.linalg.norm(a - r) <= 2 * TOL[precision] * np.linalg.norm(r), name
