"""A small pass in two kernels (attention; acceptance, commit and merge beside and behind it): both sides of the lines that
decide whether a pass goes that way, vocabularies around a unit of logits, chains and trees, both head sizes, a second
stream, a graph, scratch that is shared with the acceptance alone, and a wait that runs out."""
import numpy as np
import pytest
import torch

from gpu_util import REL_LARGE, check_attention, check_commit, run_and_check_pass
from lr_workloads import Model, make_tree
from lr_workloads.gen import _finish
from oracle import lr_oracle as O
from paper_2506_19830_b200 import binding as B
from paper_2506_19830_b200 import runner as R

pytestmark = pytest.mark.gpu
UNIT = 6 * 32 * 8  # logits


def _work(seed, vocab, n_req, prefix, heads=(4, 1), head_dim=128, segs=2, most_seg=15, drafts=4, branches=None):
    rng = np.random.Generator(np.random.PCG64(seed))
    reqs = []
    for _ in range(n_req):
        sg = [int(x) for x in rng.integers(1, most_seg + 1, size=segs)]
        depths = sorted(int(x) for x in rng.integers(0, segs + 1, size=branches or 1 + seed % 3))
        reqs.append({"P": prefix, "segs": sg, "branches": [(g, drafts, drafts, drafts) for g in depths]})
    return _finish("small", seed, Model(*heads, head_dim, vocab), reqs, rng, 0.3, 0.7, True, True, "nan")


def _launches(w):
    b, t = w.batch, w.tensors
    ctx = B.Context(b.model, 0)
    plan, x, y = B.Plan(ctx, b), R.DeviceInputs(b, t), R.PassOutputs(b)
    n = ctx.launch_count
    R.run_pass(ctx, plan, x, y)
    n = ctx.launch_count - n
    assert plan.lr_poll_status() == 0
    ctx.close()
    return n


@pytest.mark.parametrize("vocab", [1, 7, 9, UNIT - 1, UNIT, UNIT + 1, 2 * UNIT + 5, 40_003])
@pytest.mark.parametrize("head_dim", [64, 128])
def test_vocabularies(vocab, head_dim):
    w = _work(vocab % 97, vocab, 3, 300, heads=(8, 2), head_dim=head_dim)
    assert _launches(w) == 2
    run_and_check_pass(w, rel_large=REL_LARGE)


# requests up to 512, page slots up to 2048; past them the four kernels
@pytest.mark.parametrize("n_req,prefix,two", [(255, 5, True), (257, 5, True), (512, 5, True), (513, 5, False), (2, 16_000, True), (2, 16_400, False)])
def test_lines_of_the_dispatch(n_req, prefix, two):
    w = _work(n_req, 70, n_req, prefix, segs=1, drafts=2, branches=1)
    assert (_launches(w) == 2) == two
    run_and_check_pass(w, rel_large=REL_LARGE)


@pytest.mark.parametrize("args", [(2, 2, "tiny"), (4, 2, "tiny"), (2, 3, "layer")])
def test_trees(args):
    w = make_tree(args[0], args[1], size=args[2])
    run_and_check_pass(w)


@pytest.mark.parametrize("slots", [3, 6, 17])  # partial results an M-tile: both forms of the merge, and more than it has in flight
def test_streams_graphs_and_shared_scratch(slots):
    w = _work(slots, 5000, 1, {3: 700, 6: 3000, 17: 9000}[slots], heads=(40, 8), drafts=16, segs=3, most_seg=40)
    b, t = w.batch, w.tensors
    ctx = B.Context(b.model, 0)
    plan, x, y, side = B.Plan(ctx, b), R.DeviceInputs(b, t), R.PassOutputs(b), torch.cuda.Stream()
    n_ref, bonus_ref, _ = O.accept_greedy(t.logits, t.draft_ids, b.cu_draft)
    c_ref = O.commit(b, t.verdict, n_ref)
    o_ref, _ = O.verify_attention(b, t.q, t.k_pool, t.v_pool)

    def check():
        assert plan.lr_poll_status() == 0
        assert np.array_equal(y.n_accept.cpu().numpy(), n_ref) and np.array_equal(y.bonus_id.cpu().numpy(), bonus_ref)
        check_commit(y.commit_dict(), c_ref)
        check_attention(y.out, None, o_ref, None, rel_large=REL_LARGE)
        assert int(y.scratch.abs().sum().item()) == 0
        for name in ("n_accept", "bonus_id", "keep_off", "keep_pages", "free_pages", "out"):
            getattr(y, name).zero_()

    for _ in range(3):
        R.run_pass(ctx, plan, x, y)
        ctx.lr_accept_greedy(x.logits, x.draft_ids, x.cu_draft, y.n_accept, y.bonus_id, y.scratch)
        check()
        R.run_pass_overlapped(ctx, plan, x, y, side)
        check()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        R.run_pass(ctx, plan, x, y)
        R.run_pass(ctx, plan, x, y)
    for _ in range(3):
        graph.replay()
        check()
    del graph
    ctx.close()


def test_a_wait_that_runs_out():
    w = _work(5, 20_000, 4, 200, drafts=16)
    assert _launches(w) == 2
    b, t = w.batch, w.tensors
    ctx = B.Context(b.model, 0)
    plan, x, y = B.Plan(ctx, b), R.DeviceInputs(b, t), R.PassOutputs(b)
    R.run_pass(ctx, plan, x, y)
    assert plan.lr_poll_status() == 0
    want = [v.clone() for v in (y.out, y.n_accept, y.keep_off)]
    # scratch that was not zeroed: the count of finished units never is what the commit waits for
    y.scratch[0] = 900_000
    plan.lr_plan_debug_set_wait_limit(100)
    R.run_pass(ctx, plan, x, y)
    with pytest.raises(B.LrError) as e:
        plan.lr_poll_status()
    assert e.value.status == -4, e.value  # LR_ETIMEOUT
    assert int(y.scratch.abs().sum().item()) == 0
    plan.lr_plan_debug_set_wait_limit(1_000_000)
    for _ in range(2):
        R.run_pass(ctx, plan, x, y)
        assert plan.lr_poll_status() == 0
        for got, v in zip((y.out, y.n_accept, y.keep_off), want):
            assert torch.equal(got, v)
    ctx.close()
