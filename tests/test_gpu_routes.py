"""Which kernels a plan's passes run on, at the edges of the rules that choose them, against the fp64 CPU oracle.

Tolerances: 5e-6 per tensor where the band kernels run alone, 1e-5 where the dense kernels take part (their first products keep
19 to 21 bits of an operand); measured 3e-7 to 7e-6.
"""
import math

import numpy as np
import pytest
import torch

from oracle import sna_oracle as orc
from paper_2505_11157_b200 import sna
from paper_2505_11157_b200.synthetic import make_inputs, small_workload

pytestmark = pytest.mark.gpu

TOL_DENSE = 1e-5


def rel(x, ref):
    return float(np.linalg.norm(x.detach().cpu().numpy().reshape(ref.shape).astype(np.float64) - ref) / np.linalg.norm(ref))


def check(wl, tol):
    """Forward with and without lse, backward with and without saved state; the gradients start as NaN."""
    q, k, v, dout = make_inputs(wl)
    g = orc.geometry(wl.nlat_in, wl.nlon_in, wl.nlat_out, wl.nlon_out, wl.grid_in, wl.grid_out, wl.theta_cutoff)
    dev = [torch.from_numpy(a).cuda() for a in (q, k, v, dout)]
    ref, refs = orc.forward(g, q, k, v), orc.backward(g, q, k, v, dout)
    with sna.Plan(wl.nlat_in, wl.nlon_in, wl.nlat_out, wl.nlon_out, wl.grid_in, wl.grid_out, wl.theta_cutoff) as plan:
        out, lse = plan.forward(*dev[:3], return_lse=True)
        assert rel(out, ref) <= tol
        assert rel(plan.forward(*dev[:3]), ref) <= tol
        for state in ({"out": out, "lse": lse}, {}):
            grads = [torch.full_like(dev[i], math.nan) for i in range(3)]
            plan.backward(*dev, dq=grads[0], dk=grads[1], dv=grads[2], **state)
            for name, x, r in zip(("dq", "dk", "dv"), grads, refs):
                assert rel(x, r) <= tol, (name, bool(state))
        torch.cuda.synchronize()
        sna.sna_plan_check(plan.handle)


@pytest.mark.parametrize("slices", [1, 4])
def test_a_few_narrow_windows_beside_whole_rings_are_not_left_out(slices):
    """14x256, cutoff 2.66: all but 26 of the table's entries (0.06 %) lie in whole rings or windows of 128 columns and more."""
    check(small_workload("nearly_global", 14, 256, 14, 256, 0, 0, 2.66, 1, slices, 32, 81), TOL_DENSE)


@pytest.mark.parametrize("slices", [1, 8])
def test_input_rings_that_no_window_reaches_get_zero_gradients(slices):
    """Output rings at the two poles only: every window is a whole ring, and ten of the sixteen input rings are in none."""
    wl = small_workload("poles", 16, 128, 2, 128, 0, 0, 0.5, 1, slices, 32, 82)
    check(wl, TOL_DENSE)


def launches(call):
    """Kernel nodes of a captured call."""
    from cuda.bindings import runtime
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call()
    raw = runtime.cudaGraph_t(graph.raw_cuda_graph())
    _, _, count = runtime.cudaGraphGetNodes(raw)
    _, nodes, _ = runtime.cudaGraphGetNodes(raw, count)
    kernel = runtime.cudaGraphNodeType.cudaGraphNodeTypeKernel
    return sum(runtime.cudaGraphNodeGetType(n)[1] == kernel for n in nodes[:count])


@pytest.mark.parametrize("slices", [1, 24])
@pytest.mark.parametrize("C", [16, 32])
@pytest.mark.parametrize("args", [dict(theta_cutoff=0.25), dict(global_attention=True)], ids=["band", "global"])
def test_kernel_counts(args, C, slices):
    """What the queries say for a problem is what its calls launch; for a plan and a width, what the largest problem would."""
    with sna.Plan(40, 160, 40, 160, 0, 0, **args) as plan:
        q, k, v, dout = (torch.randn(1, slices, 40, 160, C, device="cuda") for _ in range(4))
        out, lse = plan.forward(q, k, v, return_lse=True)
        ws = torch.empty(plan.workspace_bytes(1, slices, C), dtype=torch.uint8, device="cuda")
        grads = [torch.empty_like(t) for t in (q, k, v)]
        counts = [sna.sna_forward_kernel_count_for(plan.handle, 1, slices, C, lse_wanted) for lse_wanted in (False, True)]
        assert counts[0] == launches(lambda: plan.forward(q, k, v, out=out))
        assert counts[1] == launches(lambda: plan.forward(q, k, v, out=out, lse=lse))
        assert sna.sna_backward_kernel_count_for(plan.handle, 1, slices, C) == launches(
            lambda: plan.backward(q, k, v, dout, out=out, lse=lse, dq=grads[0], dk=grads[1], dv=grads[2], workspace=ws))
        limit = [sna.sna_forward_kernel_count(plan.handle, C, lse_wanted) for lse_wanted in (False, True)]
        assert counts[1] <= limit[1] and (slices == 1 or counts == limit)


@pytest.mark.parametrize("slices", [1, 300])
@pytest.mark.parametrize("C", [4, 8])
@pytest.mark.parametrize("shape", [(9, 256, 9, 256), (12, 512, 6, 256)], ids=["same_grid", "down2"])
def test_narrow_heads_in_small_and_large_launches(shape, C, slices):
    """C = 4 and 8: band kernels for few slices; for many, passes on the generic kernels where those are faster."""
    wl = small_workload("narrow", *shape, 0, 0, 0.45, 1, 1, C, 83)
    one = make_inputs(wl)
    g = orc.geometry(*shape, 0, 0, 0.45)
    refs = [orc.forward(g, *one[:3]), *orc.backward(g, *one)]
    dev = [torch.from_numpy(a).cuda().expand(1, slices, -1, -1, -1).contiguous() for a in one]
    with sna.Plan(*shape, 0, 0, 0.45) as plan:
        out, lse = plan.forward(*dev[:3], return_lse=True)
        for state in ({"out": out, "lse": lse}, {}):
            for x, r in zip((out, *plan.backward(*dev, **state)), refs):
                assert rel(x[:, -1:], r) <= 5e-6 and torch.equal(x[:, 0], x[:, -1])
