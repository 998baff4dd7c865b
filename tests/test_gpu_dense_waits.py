"""Waits of the dense (tcgen05) kernels: one that runs out ends for its whole warp, and one for data that another warp stored."""
import math

import numpy as np
import pytest
import torch

from oracle import sna_oracle as orc
from paper_2505_11157_b200 import sna
from paper_2505_11157_b200.synthetic import make_inputs, small_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("polls", [1, 7, 1000])
def test_a_wait_that_runs_out_in_one_lane_ends_for_its_warp(polls):
    """The probe's last lane waits in vain, the others' barrier is complete, and its first lane reports: were the answer each lane's own,
    the warp would go on divided (in the kernels: into instructions that need all of its lanes) and nothing would be reported."""
    with sna.Plan(16, 32, 16, 32, 0, 0, 0.6) as plan:
        sna.sna_plan_check(plan.handle)
        sna.sna_debug_exercise_bounded_wait(plan.handle, polls)
        with pytest.raises(sna.SnaError) as e:
            sna.sna_plan_check(plan.handle)
        assert e.value.status == sna.SNA_ERR_CUDA
        sna.sna_plan_check(plan.handle)


@pytest.mark.parametrize("shape, theta, slices", [((32, 128, 32, 128), None, 16), ((40, 160, 40, 160), 0.25, 24)], ids=["global", "local"])
def test_statistics_of_the_partner_points_are_this_blocks(shape, theta, slices):
    """lse differs by up to four units, and D with it, between a block of 32 points and the one that its stage held before (five blocks
    ago, one ring or two): with that one's it would be far off.  All slices hold the same values: gradients equal bit for bit, over the slices and over repeated passes."""
    wl = small_workload("statistics", *shape, 0, 0, theta or math.pi, 1, 1, 32, 95)
    q, k, v, dout = make_inputs(wl)
    factor = (1 + 0.5 * ((np.arange(shape[2])[:, None] + np.arange(shape[3]) // 32) % 5)).astype(np.float32)[..., None]      # 1 to 3
    q, dout = q * factor, dout * factor
    refs = orc.backward(orc.geometry(*shape, 0, 0, theta or math.pi), q, k, v, dout)
    dev = [torch.from_numpy(a).cuda().expand(1, slices, -1, -1, -1).contiguous() for a in (q, k, v, dout)]
    with sna.Plan(*shape, 0, 0, **({"theta_cutoff": theta} if theta else {"global_attention": True})) as plan:
        out, lse = plan.forward(*dev[:3], return_lse=True)
        first = plan.backward(*dev, out=out, lse=lse)
        for _ in range(10):
            assert all(torch.equal(a, b) for a, b in zip(plan.backward(*dev, out=out, lse=lse), first))
        sna.sna_plan_check(plan.handle)
    for name, x, r in zip(("dq", "dk", "dv"), first, refs):
        assert torch.equal(x, x[:, :1].expand_as(x)), name
        err = np.linalg.norm(x[:, :1].cpu().numpy().reshape(r.shape).astype(np.float64) - r) / np.linalg.norm(r)
        # the first products keep 19 bits of the sum of |q k| (3.6 for unit channels, 3 times that here): a weight is off by 2e-5 of itself
        assert err <= 3e-5, (name, err)
