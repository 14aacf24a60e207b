"""The CTA-pair plan is built when its path is selected and shares the scratch of the single-CTA path: switching back and
forth on one plan, with passes in between, eager or captured, must give what each path gives on a plan of its own."""
import numpy as np
import pytest
import torch

from lr_workloads import make_config, make_random_mid, make_tree
from paper_2506_19830_b200 import binding as B
from paper_2506_19830_b200 import runner as R

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make", [lambda: make_config(2, with_logits=False), lambda: make_random_mid(3), lambda: make_tree(2, 2, with_logits=False)])
def test_switching_paths_on_one_plan(make):
    w = make()
    b, t = w.batch, w.tensors
    ctx = B.Context(b.model, 0)
    x = R.DeviceInputs(b, t, with_logits=False)

    def one(plan, path):
        plan.lr_plan_set_attention_path(path)
        out = torch.full((b.n_q_rows, b.model.n_q_heads, b.model.head_dim), float("nan"), dtype=torch.bfloat16, device="cuda:0")
        plan.lr_verify_attention(x.q, x.k_pool, x.v_pool, out)
        plan.lr_verify_attention(x.q, x.k_pool, x.v_pool, out)
        assert plan.lr_poll_status() == 0
        return R.bf16_bits(out)

    alone = {path: one(B.Plan(ctx, b), path) for path in (B.PATH_TENSOR_CORE, B.PATH_PAIR)}
    plan = B.Plan(ctx, b)
    for path in (B.PATH_PAIR, B.PATH_TENSOR_CORE, B.PATH_PAIR, B.PATH_PAIR, B.PATH_AUTO, B.PATH_PAIR):
        assert np.array_equal(one(plan, path), alone[path or B.PATH_TENSOR_CORE]), path
    ctx.close()


@pytest.mark.parametrize("select_in_capture", [False, True])
@pytest.mark.parametrize("warm", [False, True])
def test_captured_passes_and_other_paths_in_between(select_in_capture, warm):
    """The tables of the CTA-pair path are where its launches look for them from its selection on: before a captured pass
    has been replayed, and after another path has used the scratch."""
    w = make_config(2, with_logits=False)
    b, t = w.batch, w.tensors
    ctx = B.Context(b.model, 0)
    x = R.DeviceInputs(b, t, with_logits=False)
    outs = [torch.full((b.n_q_rows, b.model.n_q_heads, b.model.head_dim), float("nan"), dtype=torch.bfloat16, device="cuda:0") for _ in range(2)]
    want = {}
    for path in (B.PATH_TENSOR_CORE, B.PATH_PAIR):
        plan = B.Plan(ctx, b)
        plan.lr_plan_set_attention_path(path)
        plan.lr_verify_attention(x.q, x.k_pool, x.v_pool, outs[0])
        want[path] = R.bf16_bits(outs[0])
    plan = B.Plan(ctx, b)
    if not select_in_capture:
        plan.lr_plan_set_attention_path(B.PATH_PAIR)
    if warm:
        plan.lr_plan_set_attention_path(B.PATH_PAIR)
        plan.lr_verify_attention(x.q, x.k_pool, x.v_pool, outs[0])
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        if select_in_capture:
            plan.lr_plan_set_attention_path(B.PATH_PAIR)
        plan.lr_verify_attention(x.q, x.k_pool, x.v_pool, outs[0])
    plan.lr_verify_attention(x.q, x.k_pool, x.v_pool, outs[1])  # eager, before the first replay
    assert plan.lr_poll_status() == 0
    assert np.array_equal(R.bf16_bits(outs[1]), want[B.PATH_PAIR])
    for _ in range(2):
        outs[0].fill_(float("nan"))
        graph.replay()
        assert np.array_equal(R.bf16_bits(outs[0]), want[B.PATH_PAIR])
        plan.lr_plan_set_attention_path(B.PATH_TENSOR_CORE)  # fp32 partials into the shared scratch
        plan.lr_verify_attention(x.q, x.k_pool, x.v_pool, outs[1])
        assert np.array_equal(R.bf16_bits(outs[1]), want[B.PATH_TENSOR_CORE])
    assert plan.lr_poll_status() == 0
    del graph
    ctx.close()


def test_plan_made_in_a_capture():
    w = make_config(2, with_logits=False)
    b, t = w.batch, w.tensors
    ctx = B.Context(b.model, 0)
    x = R.DeviceInputs(b, t, with_logits=False)
    want = torch.empty((b.n_q_rows, b.model.n_q_heads, b.model.head_dim), dtype=torch.bfloat16, device="cuda:0")
    plan = B.Plan(ctx, b)
    plan.lr_plan_set_attention_path(B.PATH_PAIR)
    plan.lr_verify_attention(x.q, x.k_pool, x.v_pool, want)
    plan.close()  # its pinned buffer serves the next plan: none can be allocated in a capture
    torch.cuda.synchronize()
    out = torch.full_like(want, float("nan"))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="relaxed"):  # taking the buffer waits for an event
        plan = B.Plan(ctx, b)
        plan.lr_plan_set_attention_path(B.PATH_PAIR)
        plan.lr_verify_attention(x.q, x.k_pool, x.v_pool, out)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    del graph
    plan.close()
    ctx.close()
