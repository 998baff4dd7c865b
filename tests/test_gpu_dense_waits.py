"""Waits of the dense (tcgen05) kernels: one that runs out ends for its whole warp, and one for data that another warp stored."""
import pytest

from paper_2505_11157_b200 import sna

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
