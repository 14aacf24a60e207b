"""A whole pass in one call, whose acceptance and commit run on a second stream: its results are ready in the order of the
stream the caller gave (work queued behind it sees them, work queued before it is seen), passes of two plans on two streams
do not disturb one another, and a capture as the very first use works."""
import numpy as np
import pytest
import torch
from cuda.bindings import runtime as cudart

from lr_workloads import make_config, make_random_small
from oracle import lr_oracle as O
from paper_2506_19830_b200 import binding as B
from paper_2506_19830_b200 import runner as R

pytestmark = pytest.mark.gpu


def _expect(w):
    n, bonus, _ = O.accept_greedy(w.tensors.logits, w.tensors.draft_ids, w.batch.cu_draft)
    return n, bonus, O.commit(w.batch, w.tensors.verdict, n)["committed_len"]


def _same(got, want):
    assert all(np.array_equal(g.cpu().numpy(), w) for g, w in zip(got, want))


@pytest.mark.parametrize("given_side", [False, True])
def test_order_of_the_callers_streams(given_side):
    works = [make_config(1), make_random_small(31)]
    ctxs = [B.Context(w.batch.model, 0) for w in works]
    plans = [B.Plan(c, w.batch) for c, w in zip(ctxs, works)]
    xs, ys = [R.DeviceInputs(w.batch, w.tensors) for w in works], [R.PassOutputs(w.batch) for w in works]
    streams, sides = [torch.cuda.Stream() for _ in works], [torch.cuda.Stream() for _ in works]
    inputs = [x.logits.clone() for x in xs]
    torch.cuda.synchronize()
    copies = [[] for _ in works]
    for _ in range(10):
        for i in range(2):
            with torch.cuda.stream(streams[i]):
                xs[i].logits.zero_()
                torch.cuda._sleep(100_000)  # the pass must wait for this and for the copy behind it
                xs[i].logits.copy_(inputs[i])
                if given_side:
                    R.run_pass_overlapped(ctxs[i], plans[i], xs[i], ys[i], sides[i])
                else:
                    R.run_pass(ctxs[i], plans[i], xs[i], ys[i])
                copies[i].append([t.clone() for t in (ys[i].n_accept, ys[i].bonus_id, ys[i].committed_len)])
    torch.cuda.synchronize()
    for w, plan, got in zip(works, plans, copies):
        assert plan.lr_poll_status() == 0
        want = _expect(w)
        for g in got:
            _same(g, want)
    for c in ctxs:
        c.close()


@pytest.mark.parametrize("warm", [False, True])
def test_capture(warm):
    w = make_config(1)
    ctx = B.Context(w.batch.model, 0)
    plan, x, y = B.Plan(ctx, w.batch), R.DeviceInputs(w.batch, w.tensors), R.PassOutputs(w.batch)
    if warm:
        R.run_pass(ctx, plan, x, y)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        R.run_pass(ctx, plan, x, y)
    for t in (y.n_accept, y.bonus_id, y.committed_len, y.out):
        t.zero_()
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    assert plan.lr_poll_status() == 0
    _same((y.n_accept, y.bonus_id, y.committed_len), _expect(w))
    captured = y.out.clone()
    R.run_pass(ctx, plan, x, y)
    assert torch.equal(captured, y.out)
    del graph
    ctx.close()


@pytest.mark.parametrize("given_side", [False, True])
@pytest.mark.parametrize("n_plans", [1, 3])  # the context has a stream for the first one, the others need new ones
def test_a_capture_as_first_use_forks(n_plans, given_side):
    w = make_config(1)
    ctx = B.Context(w.batch.model, 0)
    plans, x = [B.Plan(ctx, w.batch) for _ in range(n_plans)], R.DeviceInputs(w.batch, w.tensors)
    for plan in plans:
        y = R.PassOutputs(w.batch)
        torch.cuda.synchronize()
        graph, side = torch.cuda.CUDAGraph(keep_graph=True), torch.cuda.Stream()
        with torch.cuda.graph(graph):
            if given_side:
                R.run_pass_overlapped(ctx, plan, x, y, side)
            else:
                R.run_pass(ctx, plan, x, y)
        err, _, n_roots = cudart.cudaGraphGetRootNodes(graph.raw_cuda_graph(), 0)
        assert int(err) == 0 and n_roots == 2  # attention and acceptance, neither behind the other
        graph.replay()
        torch.cuda.synchronize()
        assert plan.lr_poll_status() == 0
        _same((y.n_accept, y.bonus_id, y.committed_len), _expect(w))
        del graph
    ctx.close()
