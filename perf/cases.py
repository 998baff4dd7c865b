"""Timing cases of the attention operator: what a program that uses the package runs, over the range it runs it in.

A case is one pass through the public entry points.  Its keys:

* ``nlat_in, nlon_in, nlat_out, nlon_out, grid_in, grid_out`` - the two grids (0 equiangular, 1 Gauss-Legendre);
* ``theta`` - the cutoff in radians; 0 stands for global attention (a plan without a cutoff);
* ``B, H, C`` - batch, heads, channels per head;
* ``mode`` - ``train``: forward and backward through the autograd operator, ``train_cf``: the same on channels-first
  tensors, ``train_tf32``: forward and backward in the reduced-precision variant, ``infer``: forward only,
  ``recompute``: backward without saved state (activation checkpointing).
"""
import math

import torch

from paper_2505_11157_b200 import sna
from paper_2505_11157_b200.autograd import spherical_neighborhood_attention, spherical_neighborhood_attention_cf

EQ, GL = sna.SNA_GRID_EQUIANGULAR, sna.SNA_GRID_LEGENDRE_GAUSS


def _case(name, grid_shape, theta, B, H, C, mode, grids=(EQ, EQ)):
    case = dict(zip(("nlat_in", "nlon_in", "nlat_out", "nlon_out"), grid_shape))
    case.update(grid_in=grids[0], grid_out=grids[1], theta=theta, B=B, H=H, C=C, mode=mode)
    return dict(case, name=name) if name else case


def listed():
    return [
        # the smallest training step: a coarse level or a unit test, bound by latency and launches
        _case("coarse_train", (32, 64, 32, 64), 0.3, 1, 1, 16, "train"),
        # ordinary training step of an attention layer on panoramas, embedding 128 in four heads
        _case("pano128_train", (128, 256, 128, 256), 4 * math.pi / 127, 4, 4, 32, "train"),
        # the down-sampling layer of an encoder: 256x512 -> 128x256
        _case("down256_train", (256, 512, 128, 256), 3 * math.pi / 127, 2, 8, 32, "train"),
        # the largest: a quarter-million-point field on a Gaussian grid, odd ring count
        _case("gauss361_train", (361, 720, 361, 720), 5 * math.pi / 360, 1, 8, 32, "train", (GL, GL)),
        # global attention in training, and for inference on a single field
        _case("global64_train", (64, 128, 64, 128), 0.0, 2, 4, 32, "train"),
        _case("global64_infer", (64, 128, 64, 128), 0.0, 1, 4, 32, "infer"),
        # inference on a single panorama
        _case("pano128_infer", (128, 256, 128, 256), 4 * math.pi / 127, 1, 4, 32, "infer"),
        # a layer inside a 2D convolutional network (channels-first feature maps)
        _case("pano128_cf_train", (128, 256, 128, 256), 4 * math.pi / 127, 4, 4, 32, "train_cf"),
        # a head width that is no power of two, on an odd and ragged Gaussian grid
        _case("gauss91_c24_train", (91, 180, 91, 180), 4.5 * math.pi / 90, 2, 4, 24, "train", (GL, GL)),
        # wide heads
        _case("pano128_c64_train", (128, 256, 128, 256), 4 * math.pi / 127, 2, 4, 64, "train"),
        # the reduced-precision variant
        _case("pano128_tf32_train", (128, 256, 128, 256), 4 * math.pi / 127, 4, 4, 32, "train_tf32"),
        # gradients under activation checkpointing: nothing saved from the forward pass
        _case("down256_recompute", (256, 512, 128, 256), 3 * math.pi / 127, 1, 4, 32, "recompute"),
    ]


_pairs = {}     # table entries per grid pair and cutoff: the planner's count, for work()


def _table_entries(case):
    shape = tuple(case[k] for k in ("nlat_in", "nlon_in", "nlat_out", "nlon_out"))
    if case["theta"] == 0.0:
        return shape[0] * shape[1] * shape[2]
    key = shape + (case["grid_in"], case["grid_out"], case["theta"])
    if key not in _pairs:
        with sna.Plan(*shape, case["grid_in"], case["grid_out"], case["theta"], host_only=True) as plan:
            _pairs[key] = plan.nnz
    return _pairs[key]


def _flops(case):
    # score and weighted sum forward (2 FMA per pair and channel); s, t, dq, dk, dv backward (5), 6 if s and out are recomputed
    fma = {"train": 7, "train_cf": 7, "train_tf32": 7, "infer": 2, "recompute": 6}[case["mode"]]
    return 2.0 * fma * _table_entries(case) * case["nlon_out"] * case["B"] * case["H"] * case["C"]


def draw(rng):
    """Grids of 24 to 361 rings (down-sampling by 1 to 4), cutoffs of 2 to 6 grid spacings or none, head widths of 8 to 128."""
    largest = _flops(listed()[3])
    while True:
        mode = rng.choice(["train", "train", "train", "infer", "train_cf", "train_tf32", "recompute"])
        is_global = rng.random() < 0.15
        ps = rng.choice([1, 1, 1, 2, 2, 3, 4])
        nlat_out = round(math.exp(rng.uniform(math.log(16), math.log(96 if is_global else 361 / ps))))
        nlon_out = max(24, 2 * nlat_out + rng.choice([0, 0, 0, -1, 2, 5]))
        nlat_in = nlat_out if ps == 1 else min(361, ps * nlat_out + rng.choice([0, 1]))
        grids = rng.choice([(EQ, EQ), (EQ, EQ), (GL, GL), (GL, EQ)])
        C = rng.choice([16, 32, 32, 32, 32, 64, 8, 24, 48, 128])
        if mode == "train_tf32":
            is_global, C, nlon_out = False, rng.choice([16, 32, 64]), max(32, nlon_out)
        theta = 0.0 if is_global else rng.choice([2, 3, 4, 5, 6, 2.5, 3.7]) * math.pi / (nlat_out - 1)
        B, H = rng.choice([1, 1, 2, 4]), rng.choice([1, 2, 4, 8])
        case = _case(None, (nlat_in, ps * nlon_out, nlat_out, nlon_out), theta, B, H, C, mode, grids)
        try:
            # head widths outside 16, 32, 64 are rarer and are drawn at moderate sizes
            if _flops(case) <= largest * (1.0 if C in (16, 32, 64) else 0.05):
                return case
        except sna.SnaError:
            pass        # a grid point too close to the cutoff to decide: the planner refuses it


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    shape = tuple(case[k] for k in ("nlat_in", "nlon_in", "nlat_out", "nlon_out"))
    plan = sna.Plan(*shape, case["grid_in"], case["grid_out"], case["theta"] or math.pi, global_attention=case["theta"] == 0.0)
    B, H, C = case["B"], case["H"], case["C"]
    cf = case["mode"] == "train_cf"
    dims = lambda nlat, nlon: (B, H * C, nlat, nlon) if cf else (B, H, nlat, nlon, C)
    draw_normal = lambda nlat, nlon: torch.randn(dims(nlat, nlon), generator=gen, device="cuda")
    state = {"plan": plan, "mode": case["mode"], "heads": H, "q": draw_normal(*shape[2:]), "k": draw_normal(*shape[:2]),
             "v": draw_normal(*shape[:2])}
    if case["mode"] != "infer":
        state["dout"] = draw_normal(*shape[2:])
    if case["mode"] in ("train", "train_cf"):
        for name in "qkv":
            state[name].requires_grad_(True)
    return state


def run(state):
    plan, mode, q, k, v = (state[key] for key in ("plan", "mode", "q", "k", "v"))
    if mode == "infer":
        return plan.forward(q, k, v)
    dout = state["dout"]
    if mode == "recompute":
        return plan.backward(q, k, v, dout)
    if mode == "train_tf32":
        out, lse = plan.forward(q, k, v, return_lse=True, precision="tf32")
        return (out, *plan.backward(q, k, v, dout, out=out, lse=lse, precision="tf32"))
    out = spherical_neighborhood_attention(plan, q, k, v) if mode == "train" else \
        spherical_neighborhood_attention_cf(plan, q, k, v, heads=state["heads"])
    return (out, *torch.autograd.grad(out, (q, k, v), dout))


def work(case):
    per_point = 4 * case["B"] * case["H"] * case["C"]
    o, i = case["nlat_out"] * case["nlon_out"] * per_point, case["nlat_in"] * case["nlon_in"] * per_point
    # infer: q, out; k, v.  recompute: q, dout, dq; k, v, dk, dv.  training: both passes (backward reads q, k, v, dout).
    tensors = {"infer": (2, 2), "recompute": (3, 4)}.get(case["mode"], (5, 6))
    return {"bytes": tensors[0] * o + tensors[1] * i, "flops": _flops(case)}


def tolerance(case):
    # four times the 2-norm error measured against 64-bit arithmetic over these ranges: products split into two or three
    # tensor-core terms for C of 16, 32 and 64 (out 2e-6, gradients 7e-6), plain fp32 for the other widths (4e-7), one
    # TF32 product in the reduced-precision variant (1.4e-3)
    if case["mode"] == "train_tf32":
        return {"rel": 6e-3}
    if case["C"] not in (16, 32, 64):
        return {"rel": 1.6e-6}
    return {"rel": 8e-6 if case["mode"] == "infer" else 3e-5}
