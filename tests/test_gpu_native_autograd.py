"""The native autograd function: who owns the plan, and what it says about arguments that the plan does not take."""
import copy
import gc
import threading

import pytest
import torch

from paper_2505_11157_b200 import sna
from paper_2505_11157_b200.autograd import spherical_neighborhood_attention as attention

pytestmark = pytest.mark.gpu


def inputs(C=16, **kw):
    return [torch.randn(1, 2, 12, 24, C, device="cuda", **kw).requires_grad_() for _ in range(3)]


def test_same_values_as_the_plan_calls_also_for_strided_inputs():
    q, k, v = (torch.randn(1, 12, 24, 2, 16, device="cuda").permute(0, 3, 1, 2, 4).requires_grad_() for _ in range(3))
    with sna.Plan(12, 24, 12, 24, 0, 0, 0.6) as plan:
        dout = torch.randn(1, 12, 24, 2, 16, device="cuda").permute(0, 3, 1, 2, 4)
        out = attention(plan, q, k, v)
        grads = torch.autograd.grad(out, (q, k, v), dout, retain_graph=True)
        again = torch.autograd.grad(out, (q, k, v), dout)
        with torch.no_grad():
            dense = [t.contiguous() for t in (q, k, v)]
            ref, lse = plan.forward(*dense, return_lse=True)
            ref_grads = plan.backward(*dense, dout.contiguous(), out=ref, lse=lse)
    assert torch.equal(out, ref)
    for a, b, c in zip(grads, again, ref_grads):
        assert torch.equal(a, c) and torch.equal(b, c)


def test_a_graph_outlives_the_plan_object_but_not_close():
    q, k, v = inputs()
    plan = sna.Plan(12, 24, 12, 24, 0, 0, 0.6)
    out = attention(plan, q, k, v)
    del plan
    gc.collect()
    assert torch.isfinite(torch.autograd.grad(out.sum(), q)[0]).all()
    plan = sna.Plan(12, 24, 12, 24, 0, 0, 0.6)
    out = attention(plan, q, k, v)
    plan.close()
    with pytest.raises(RuntimeError, match="plan is NULL"):
        torch.autograd.grad(out.sum(), q)
    with pytest.raises(sna.SnaError, match="plan is NULL"):
        attention(plan, q, k, v)


def test_wrong_arguments_are_refused_as_by_the_plan():
    q, k, v = inputs()
    with sna.Plan(12, 24, 12, 24, 0, 0, 0.6) as plan:
        with pytest.raises(ValueError, match="computes in float32"):
            attention(plan, q.half(), k, v)
        with pytest.raises(ValueError, match="shapes do not match"):
            attention(plan, q, k[:, :, :6], v)
        with pytest.raises(ValueError, match="v has shape"):
            attention(plan, q, k, v[:, :1])
        with pytest.raises(ValueError, match="CUDA tensor"):
            attention(plan, q, k, v.detach().cpu())
        with pytest.raises(sna.SnaError, match="unsupported"):
            attention(plan, *inputs(C=6))


def test_threads_share_a_plan_from_its_first_use():
    with sna.Plan(12, 24, 12, 24, 0, 0, 0.6) as plan:
        q, k, v = inputs()
        results = [None] * 8

        def work(i):
            results[i] = torch.autograd.grad(attention(plan, q, k, v).sum(), (q, k, v))

        threads = [threading.Thread(target=work, args=(i,)) for i in range(8)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        torch.cuda.synchronize()
    for r in results[1:]:
        assert all(torch.equal(a, b) for a, b in zip(r, results[0]))


@pytest.mark.parametrize("saved", range(5), ids=["q", "k", "v", "out", "lse"])
@pytest.mark.parametrize("change, says", [(lambda t: t.cpu(), "CUDA tensor"), (lambda t: t.half(), "float32"), (lambda t: t[..., :1], "has shape"),
                                          (lambda t: t.transpose(2, 3).contiguous().transpose(2, 3), "contiguous"), (lambda t: t + 0, None)],
                         ids=["host", "half", "shape", "strides", "copy"])
def test_saved_tensors_that_hooks_return_are_checked(saved, change, says):
    q, k, v = inputs()
    seen = []

    def unpack(t):
        seen.append(t)
        return change(t) if len(seen) == saved + 1 else t

    with sna.Plan(12, 24, 12, 24, 0, 0, 0.6) as plan:
        ref = torch.autograd.grad(attention(plan, q, k, v).sum(), (q, k, v))
        with torch.autograd.graph.saved_tensors_hooks(lambda t: t, unpack):
            total = attention(plan, q, k, v).sum()
        if says:
            with pytest.raises(ValueError, match=says):
                torch.autograd.grad(total, (q, k, v))
        else:
            assert all(torch.equal(a, b) for a, b in zip(torch.autograd.grad(total, (q, k, v)), ref))


def test_a_failing_call_raises_the_same_error_in_forward_and_backward():
    q, k, v = inputs()
    plan = sna.Plan(12, 24, 12, 24, 0, 0, 0.6)
    out = attention(plan, q, k, v)
    plan.close()
    for call in (lambda: torch.autograd.grad(out.sum(), q), lambda: attention(plan, q, k, v)):
        with pytest.raises(sna.SnaError, match="plan is NULL") as e:
            call()
        assert e.value.status == sna.SNA_ERR_INVALID_ARG


@pytest.mark.filterwarnings("ignore")
def test_a_trace_and_a_tensor_subclass_run_the_operator():
    class Sub(torch.Tensor):
        pass

    with sna.Plan(12, 24, 12, 24, 0, 0, 0.6) as plan:
        q, k, v = inputs()
        traced = torch.jit.trace(lambda a, b, c: 2 * attention(plan, a, b, c), (q, k, v), check_trace=False)
        q, k, v = inputs()
        ref = attention(plan, q, k, v)
        again = traced(q, k, v)
        assert torch.equal(again, 2 * ref)
        for a, b in zip(torch.autograd.grad(again.sum(), (q, k, v)), torch.autograd.grad(2 * ref.sum(), (q, k, v))):
            assert torch.equal(a, b)
        with torch.no_grad():
            out = attention(plan, q.as_subclass(Sub), k, v)
        assert type(out) is Sub and torch.equal(out.as_subclass(torch.Tensor), ref)


def test_copies_share_the_plan():
    q, k, v = inputs()
    plan = sna.Plan(12, 24, 12, 24, 0, 0, 0.6)
    ref = attention(plan, q, k, v)
    copies = [copy.copy(plan), copy.deepcopy({"plan": plan})["plan"]]
    del plan
    gc.collect()
    assert all(torch.equal(attention(p, q, k, v), ref) for p in copies)
