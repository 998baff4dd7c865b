"""Band kernels at the edges of their tiles and value ranges, against the fp64 CPU oracle.

Tolerance: every operand of a product is held to 22 significant bits, so a score of magnitude s (log2 domain) carries an error of
about 2^-21 * sum|q k|, which is |s| * sqrt(C) at most; with unit-variance inputs (|s| <= 5, C <= 64) that is 2e-5 for the worst
weight and, as errors are independent, below 2e-6 in the 2-norm over an output.  5e-6 is used; measured 4e-7 to 1.3e-6.
"""
import math

import numpy as np
import pytest
import torch

from oracle import sna_oracle as orc
from paper_2505_11157_b200 import sna
from paper_2505_11157_b200.synthetic import make_inputs, small_workload

pytestmark = pytest.mark.gpu

TOL, TOL_REDUCED = 5e-6, 3e-3        # reduced precision: 2^-11 per operand, 2^10 times the above


def rel(x, ref):
    return float(np.linalg.norm(x.detach().cpu().numpy().reshape(ref.shape).astype(np.float64) - ref) / np.linalg.norm(ref))


def check(wl, q, k, v, dout, tol=TOL, precision="fp32", recompute=False):
    g = orc.geometry(wl.nlat_in, wl.nlon_in, wl.nlat_out, wl.nlon_out, wl.grid_in, wl.grid_out, wl.theta_cutoff)
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (q, k, v, dout)]
    with sna.Plan(wl.nlat_in, wl.nlon_in, wl.nlat_out, wl.nlon_out, wl.grid_in, wl.grid_out, wl.theta_cutoff) as plan:
        out, lse = plan.forward(*dev[:3], return_lse=True, precision=precision)
        state = {} if recompute else {"out": out, "lse": lse}
        grads = plan.backward(*dev, precision=precision, **state)
        torch.cuda.synchronize()
        sna.sna_plan_check(plan.handle)
    ref, ref_lse = orc.forward(g, q, k, v, return_lse=True)
    assert rel(out, ref) <= tol
    assert np.max(np.abs(lse.cpu().numpy().reshape(ref_lse.shape) - ref_lse)) <= 20 * tol
    for name, x, r in zip(("dq", "dk", "dv"), grads, orc.backward(g, q, k, v, dout)):
        assert rel(x, r) <= tol, name


@pytest.mark.parametrize("C", [4, 12, 16, 20, 28, 32, 36, 52, 60, 64])
@pytest.mark.parametrize("shape", [(9, 17, 9, 17, 0.7), (12, 34, 7, 17, 0.6), (13, 96, 7, 32, 0.5)], ids=["odd", "down2", "down3"])
def test_head_widths_and_ragged_tiles(C, shape):
    """Partial pieces of a row, rings that end inside a tile, a last ring without a partner, strides 1 to 3."""
    wl = small_workload("edge", *shape[:4], 0, 0, shape[4], 1, 2, C, 70 + C)
    check(wl, *make_inputs(wl), recompute=C % 8 == 4)


@pytest.mark.parametrize("slices", [1, 5, 300])
def test_shared_and_private_streams(slices):
    """Few slices: the warps of a block share a tile's stream; many: each warp walks its own."""
    wl = small_workload("streams", 24, 48, 24, 48, 0, 1, 0.4, 1, slices, 16, 71)
    check(wl, *make_inputs(wl))


@pytest.mark.parametrize("slices", [1, 24])
def test_dense_kernels_above_a_size(slices):
    """C = 32: whole rings on the dense kernels for many slices, everything on the band kernels for few."""
    wl = small_workload("dense_rule", 40, 160, 40, 160, 0, 0, 0.25, 1, slices, 32, 72)
    check(wl, *make_inputs(wl))


@pytest.mark.parametrize("precision, tol", [("fp32", TOL), ("tf32", TOL_REDUCED)])
@pytest.mark.parametrize("C", [16, 32, 64])
@pytest.mark.parametrize("which", ["k", "v", "dout", "all_tiny"])
def test_value_ranges(which, C, precision, tol):
    """Rows that grow by 2^24 along a stream overflow the scale taken from its first chunk: the tile is computed again.  Rows that
    are zero at first, and inputs far below 1, must find a scale too."""
    wl = small_workload("range", 16, 32, 16, 32, 0, 0, 0.6, 1, 2, C, 73)
    q, k, v, dout = make_inputs(wl)
    grow = np.exp2(np.linspace(0.0, 24.0, 16)).astype(np.float32).reshape(1, 1, 16, 1, 1)
    grow[..., :2, :, :] = 0.0
    if which == "k":
        k, q = k * grow, q * np.float32(2.0 ** -24)
    elif which == "v":
        v = v * grow
    elif which == "dout":
        dout = dout * grow
    else:
        k, v, dout, q = (a * np.float32(s) for a, s in ((k, 2.0 ** -30), (v, 2.0 ** -30), (dout, 2.0 ** -20), (q, 2.0 ** 30)))      # gradients down to 2^-80
    check(wl, q, k, v, dout, tol=tol, precision=precision)


def test_an_infinite_value_reaches_the_outputs_that_attend_to_it():
    wl = small_workload("inf", 16, 32, 16, 32, 0, 0, 0.3, 1, 1, 32, 74)
    q, k, v, _ = make_inputs(wl)
    v = v.copy()
    v[0, 0, 8, 10, :] = math.inf
    with sna.Plan(16, 32, 16, 32, 0, 0, 0.3) as plan:
        out = plan.forward(*(torch.from_numpy(a).cuda() for a in (q, k, v))).cpu()
    assert not torch.isfinite(out[0, 0, 8, 10]).any()
    assert torch.isfinite(out[0, 0, 0]).all()


@pytest.mark.parametrize("shape", [(5, 17, 5, 17), (9, 48, 4, 16), (8, 36, 5, 36), (3, 128, 3, 128)], ids=["odd", "down3", "ragged", "one_tile"])
@pytest.mark.parametrize("C, slices, grid", [(8, 1, 0), (20, 3, 1), (32, 2, 2), (64, 40, 0)])
@pytest.mark.parametrize("recompute", [False, True])
def test_global_attention_on_the_band_kernels(shape, C, slices, grid, recompute):
    """A global plan's single stream: shared by all ring groups, split over a block's warps or not, zero-weight rings left out."""
    wl = small_workload("global_band", *shape, grid, 0, math.pi, 1, slices, C, 75)
    q, k, v, dout = make_inputs(wl)
    g = orc.geometry(*shape, grid, 0, math.pi)
    dev = [torch.from_numpy(a).cuda() for a in (q, k, v, dout)]
    with sna.Plan(*shape, grid, 0, global_attention=True) as plan:
        out, lse = plan.forward(*dev[:3], return_lse=True)
        grads = plan.backward(*dev, **({} if recompute else {"out": out, "lse": lse}))
        torch.cuda.synchronize()
        sna.sna_plan_check(plan.handle)
    assert rel(out, orc.forward(g, q, k, v)) <= TOL
    for name, x, r in zip(("dq", "dk", "dv"), grads, orc.backward(g, q, k, v, dout)):
        assert rel(x, r) <= (TOL if C != 32 else 1e-5), name       # (C = 32: a pass may run on the dense kernels, 2^-21 per operand)
    if grid == 2:
        assert not grads[1][..., 0, :, :].any() and not grads[2][..., 0, :, :].any()


@pytest.mark.parametrize("shape, slices", [((128, 256, 128, 256, 0.1), 8), ((96, 384, 48, 192, 0.15), 12)], ids=["same_grid", "down2"])
def test_band_kernels_that_start_before_the_dense_ones_have_finished(shape, slices):
    """Calls in a row on one stream, on several streams and replayed from a captured graph give the same bits: nothing is read before
    the dense kernels have written it, and the next call waits for both."""
    nlat_in, nlon_in, nlat_out, nlon_out, theta = shape
    with sna.Plan(nlat_in, nlon_in, nlat_out, nlon_out, 0, 0, theta) as plan:
        gen = torch.Generator(device="cuda").manual_seed(76)
        q, dout = (torch.randn(1, slices, nlat_out, nlon_out, 32, generator=gen, device="cuda") for _ in range(2))
        k, v = (torch.randn(1, slices, nlat_in, nlon_in, 32, generator=gen, device="cuda") for _ in range(2))

        def step():
            out, lse = plan.forward(q, k, v, return_lse=True)
            return [out, lse, *plan.backward(q, k, v, dout, out=out, lse=lse)]

        ref = [t.clone() for t in step()]
        for _ in range(10):
            again = [torch.full_like(t, math.nan) for t in ref]
            plan.forward(q, k, v, out=again[0], lse=again[1], return_lse=True)
            plan.backward(q, k, v, dout, out=again[0], lse=again[1], dq=again[2], dk=again[3], dv=again[4])
            assert all(torch.equal(a, b) for a, b in zip(again, ref))
        torch.cuda.synchronize()
        streams, results = [torch.cuda.Stream() for _ in range(3)], []
        for s in streams:
            with torch.cuda.stream(s):
                results.append(step())
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            results.append(step())
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for r in results for a, b in zip(r, ref))
        sna.sna_plan_check(plan.handle)
