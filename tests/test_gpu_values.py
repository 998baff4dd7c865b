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
            # p = e^(s - lse): relative to the gap s carries 2^-22 from its split operands and 2^-24 from each of four fp32 roundings
            # (q log2 e, the scaled sum, lse log2 e, the difference), 2^-21 in all
            assert rel_points(x[:, :, [4, 5, 10, 11]], r[:, :, [4, 5, 10, 11]]) <= TOL["fp32"] + gap * 2.0 ** -21, (name, gap)
