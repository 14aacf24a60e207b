"""A small plan serves lr_verify_attention, which has all SMs, and lr_verify_pass, which with head size 64 may leave some to the
acceptance: the former's partition, launches and bits do not hang on the vocabulary, both are right, and both see a page id that is
changed."""
import numpy as np
import pytest
import torch

from gpu_util import REL_LARGE, check_attention, check_commit
from lr_workloads import Model
from lr_workloads.gen import _finish
from oracle import lr_oracle as O
from paper_2506_19830_b200 import binding as B
from paper_2506_19830_b200 import runner as R

pytestmark = pytest.mark.gpu


def _work(heads, head_dim, vocab, n_req, prefix, steps, drafts, with_logits):
    rng = np.random.Generator(np.random.PCG64(n_req + prefix))
    reqs = [{"P": prefix, "segs": [32] * steps, "branches": [(n, drafts, drafts, drafts) for n in range(1, steps + 1)]} for _ in range(n_req)]
    return _finish("plans", 3, Model(*heads, head_dim, vocab), reqs, rng, 0.3, 0.7, with_logits, True, "nan")


@pytest.mark.parametrize("heads,head_dim,vocab,n_req,prefix,steps,drafts,own,form", [
    ((5, 1), 128, 152064, 16, 100, 3, 4, False, 1), ((40, 8), 128, 32000, 4, 500, 3, 16, False, 2), ((40, 8), 128, 152064, 4, 100, 5, 4, False, 2),
    ((40, 8), 128, 152064, 1, 1500, 3, 16, False, 2), ((32, 8), 64, 152064, 1, 1500, 3, 16, True, 1), ((32, 8), 64, 152064, 4, 100, 5, 4, True, 1)])
def test_two_partitions(heads, head_dim, vocab, n_req, prefix, steps, drafts, own, form):
    w = _work(heads, head_dim, 8, n_req, prefix, steps, drafts, False)
    b, t = w.batch, w.tensors
    got = []
    for v in (8, vocab):
        ctx = B.Context(Model(*heads, head_dim, v), 0)
        plan, x, y = B.Plan(ctx, b), R.DeviceInputs(b, t, with_logits=False), R.PassOutputs(b)
        n = ctx.launch_count
        plan.lr_verify_attention(x.q, x.k_pool, x.v_pool, y.out, y.lse)
        got.append((plan.lr_plan_describe(), ctx.launch_count - n, y.out, y.lse))
        assert plan.lr_poll_status() == 0
        plan.close()
        ctx.close()
    assert got[0][:2] == got[1][:2] and all(torch.equal(p, q) for p, q in zip(got[0][2:], got[1][2:]))
    assert got[0][1] == (2 if got[0][0]["n_merge_targets"] else 1)
    o_ref, l_ref = O.verify_attention(b, t.q, t.k_pool, t.v_pool)
    check_attention(got[0][2], got[0][3], o_ref, l_ref, rel_large=REL_LARGE)
    # the pass of the large vocabulary: with head size 128 the same bits, whatever the acceptance needs
    ctx = B.Context(Model(*heads, head_dim, vocab), 0)
    attention, of_pass, small = B.lr_debug_partitions(ctx.model, b, torch.cuda.get_device_properties(0).multi_processor_count)
    assert attention["n_cta"] == got[0][0]["n_cta"] and (of_pass != attention) == own and small == form
    plan, x, y = B.Plan(ctx, b), R.DeviceInputs(b, t, with_logits=False), R.PassOutputs(b)
    x.logits = torch.randn((b.n_logit_rows, vocab), device="cuda:0", dtype=torch.bfloat16)
    x.draft_ids = torch.zeros(max(1, int(b.cu_draft[-1])), dtype=torch.int32, device="cuda:0")
    n = ctx.launch_count
    R.run_pass(ctx, plan, x, y)
    assert ctx.launch_count - n == 2
    assert plan.lr_poll_status() == 0
    check_attention(y.out, y.lse, o_ref, l_ref, rel_large=REL_LARGE)
    assert own or (torch.equal(y.out, got[0][2]) and torch.equal(y.lse, got[0][3]))
    logits = x.logits.float()
    top = torch.where(logits == logits.max(1, keepdim=True).values, torch.arange(vocab, device="cuda:0"), vocab).min(1).values
    assert torch.equal(y.row_argmax, top.int()) and int(y.scratch.abs().sum().item()) == 0
    # an id outside the pool, in every table of the plan
    for k in range(2):
        call = (lambda: R.run_pass(ctx, plan, x, y)) if k == 0 else (lambda: plan.lr_verify_attention(x.q, x.k_pool, x.v_pool, y.out, y.lse))
        slot = int(b.span_slot[0])
        plan.lr_plan_debug_set_page(slot, b.n_pool_pages + 7)
        call()
        with pytest.raises(B.LrError):
            plan.lr_poll_status()
        plan.lr_plan_debug_set_page(slot, int(b.page_ids[slot]))
        call()
        assert plan.lr_poll_status() == 0
        check_attention(y.out, y.lse, o_ref, l_ref, rel_large=REL_LARGE)
    plan.close()
    ctx.close()


@pytest.mark.parametrize("heads,head_dim,vocab,form", [((40, 8), 128, 5000, 1), ((40, 8), 128, 152064, 2), ((32, 8), 64, 152064, 1)])
def test_a_second_stream(heads, head_dim, vocab, form):
    """Launched, the pass is attention on all SMs with acceptance and commit as two kernels beside it; in a graph they are one where
    attention leaves SMs for it, and a pass on one stream forks where it does not."""
    w = _work(heads, head_dim, vocab, 1, 1500, 3, 16, True)
    b, t = w.batch, w.tensors
    ctx = B.Context(b.model, 0)
    assert B.lr_debug_partitions(b.model, b, torch.cuda.get_device_properties(0).multi_processor_count)[2] == form
    plan, x, y, side = B.Plan(ctx, b), R.DeviceInputs(b, t), R.PassOutputs(b), torch.cuda.Stream()
    plan.lr_verify_attention(x.q, x.k_pool, x.v_pool, y.out)
    want = y.out.clone()
    n_ref, bonus_ref, _ = O.accept_greedy(t.logits, t.draft_ids, b.cu_draft)
    o_ref, _ = O.verify_attention(b, t.q, t.k_pool, t.v_pool)
    for _ in range(3):
        n = ctx.launch_count
        R.run_pass_overlapped(ctx, plan, x, y, side)
        assert ctx.launch_count - n == 4
        assert plan.lr_poll_status() == 0 and torch.equal(y.out, want)
        assert np.array_equal(y.n_accept.cpu().numpy(), n_ref) and np.array_equal(y.bonus_id.cpu().numpy(), bonus_ref)
        check_commit(y.commit_dict(), O.commit(b, t.verdict, n_ref))
        y.n_accept.zero_(), y.keep_pages.zero_(), y.out.zero_()
    for call, n_launches in ((lambda: R.run_pass_overlapped(ctx, plan, x, y, side), 3 if form == 1 else 4),
                             (lambda: R.run_pass(ctx, plan, x, y), 2 if form == 1 else 4)):
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            n = ctx.launch_count
            call()
            assert ctx.launch_count - n == n_launches
        for _ in range(2):
            y.n_accept.zero_(), y.keep_pages.zero_(), y.out.zero_()
            graph.replay()
            assert plan.lr_poll_status() == 0
            check_attention(y.out, None, o_ref, None, rel_large=REL_LARGE)
            assert head_dim == 64 or torch.equal(y.out, want)
            assert np.array_equal(y.n_accept.cpu().numpy(), n_ref) and np.array_equal(y.bonus_id.cpu().numpy(), bonus_ref)
            check_commit(y.commit_dict(), O.commit(b, t.verdict, n_ref))
        del graph
    plan.close()
    ctx.close()


@pytest.mark.parametrize("n_req,vocab,n", [(8, 5748, 2), (8, 152064, 3)])
def test_a_second_stream_without_a_merge(n_req, vocab, n):
    """Few logits and no merge: acceptance and commit are one kernel, which fits the SMs that attention leaves; many: two."""
    w = _work((32, 8), 64, vocab, n_req, 60, 1, 4, True)
    b, t = w.batch, w.tensors
    ctx = B.Context(b.model, 0)
    plan, x, y, side = B.Plan(ctx, b), R.DeviceInputs(b, t), R.PassOutputs(b), torch.cuda.Stream()
    n_ref, bonus_ref, _ = O.accept_greedy(t.logits, t.draft_ids, b.cu_draft)
    o_ref, _ = O.verify_attention(b, t.q, t.k_pool, t.v_pool)
    assert plan.lr_plan_describe()["n_merge_targets"] == 0
    for _ in range(3):
        before = ctx.launch_count
        R.run_pass_overlapped(ctx, plan, x, y, side)
        assert ctx.launch_count - before == n
        assert plan.lr_poll_status() == 0
        check_attention(y.out, None, o_ref, None, rel_large=REL_LARGE)
        assert np.array_equal(y.n_accept.cpu().numpy(), n_ref) and np.array_equal(y.bonus_id.cpu().numpy(), bonus_ref)
        check_commit(y.commit_dict(), O.commit(b, t.verdict, n_ref))
        assert int(y.scratch.abs().sum().item()) == 0
        y.n_accept.zero_(), y.keep_pages.zero_(), y.out.zero_()
    plan.close()
    ctx.close()
