"""The forms of a small pass, each shown to be the one that ran: the merge with four, with up to eight and with more partial
results an M-tile, on one stream, on two and in a graph, trees; rows of logits that several warps share, with ties, signed zeros,
NaN and infinities, and a row stride above the vocabulary; a wait for the row keys that runs out."""
import ctypes as C

import numpy as np
import pytest
import torch

from gpu_util import REL_LARGE, check_attention, check_commit
from lr_workloads import Model, bf16_round, build_batch, make_tree
from lr_workloads.gen import _finish
from oracle import lr_oracle as O
from paper_2506_19830_b200 import binding as B
from paper_2506_19830_b200 import runner as R

pytestmark = pytest.mark.gpu
UNIT = 6 * 32 * 8  # logits a warp reduces at a time


def _n_sm():
    return torch.cuda.get_device_properties(0).multi_processor_count


def _launches(ctx, call):
    n = ctx.launch_count
    call()
    return ctx.launch_count - n


@pytest.mark.parametrize("prefix,slots", [(300, 4), (700, 7), (3000, 9)])
@pytest.mark.parametrize("heads,head_dim", [((40, 8), 128), ((32, 8), 64)])
def test_merge(prefix, slots, heads, head_dim):
    rng = np.random.Generator(np.random.PCG64(prefix))
    w = _finish("forms", 3, Model(*heads, head_dim, 5000), [{"P": prefix, "segs": [32] * 3, "branches": [(n, 16, 16, 16) for n in (1, 2, 3)]}], rng, 0.3,
                0.7, True, True, "nan")
    b, t = w.batch, w.tensors
    _, part, small = B.lr_debug_partitions(b.model, b, _n_sm())
    assert small and part["n_merge_targets"] > 0
    if _n_sm() == 148:
        assert part["n_partial_slots"] == slots * part["n_merge_targets"]
    ctx = B.Context(b.model, 0)
    plan, x, y, side = B.Plan(ctx, b), R.DeviceInputs(b, t), R.PassOutputs(b), torch.cuda.Stream()
    n_ref, bonus_ref, arg_ref = O.accept_greedy(t.logits, t.draft_ids, b.cu_draft)
    c_ref = O.commit(b, t.verdict, n_ref)
    o_ref, l_ref = O.verify_attention(b, t.q, t.k_pool, t.v_pool)

    def check(lse):
        assert plan.lr_poll_status() == 0
        assert np.array_equal(y.n_accept.cpu().numpy(), n_ref) and np.array_equal(y.bonus_id.cpu().numpy(), bonus_ref)
        check_commit(y.commit_dict(), c_ref)
        check_attention(y.out, y.lse if lse else None, o_ref, l_ref, rel_large=REL_LARGE)
        assert int(y.scratch.abs().sum().item()) == 0
        for name in ("n_accept", "bonus_id", "keep_off", "keep_pages", "free_pages", "out", "lse"):
            getattr(y, name).zero_()

    one, two = (lambda: R.run_pass(ctx, plan, x, y)), (lambda: R.run_pass_overlapped(ctx, plan, x, y, side))
    assert _launches(ctx, one) == 2
    assert np.array_equal(y.row_argmax.cpu().numpy(), arg_ref)
    check(True)
    assert _launches(ctx, two) == 4  # attention and its merge, acceptance, commit
    check(False)
    for call, n in ((one, 3 if 2 * part["n_cta"] <= _n_sm() else 2), (two, 3)):  # 3: attention and its merge, the rest a root of its own
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            assert _launches(ctx, call) == n
        for _ in range(2):
            graph.replay()
            check(call is one)
        del graph
    plan.close()
    ctx.close()


@pytest.mark.parametrize("args", [(2, 2, "tiny"), (4, 2, "tiny")])
def test_trees(args):
    w = make_tree(args[0], args[1], size=args[2])
    b, t = w.batch, w.tensors
    ctx = B.Context(b.model, 0)
    plan, x, y = B.Plan(ctx, b), R.DeviceInputs(b, t), R.PassOutputs(b)
    assert _launches(ctx, lambda: R.run_pass(ctx, plan, x, y)) == 2
    n_ref, _, _ = O.accept_greedy(t.logits, t.draft_ids, b.cu_draft)
    assert plan.lr_poll_status() == 0
    check_commit(y.commit_dict(), O.commit(b, t.verdict, n_ref))
    plan.close()
    ctx.close()


# 152003: a warp has five units, so most rows are shared by many warps and several warps end inside a row
@pytest.mark.parametrize("vocab,stride", [(5, 8), (1003, 1008), (1003, 1600), (2 * UNIT + 24, 2 * UNIT + 24), (152_003, 152_008), (152_003, 153_600)])
def test_special_rows_and_ties(vocab, stride):
    rng = np.random.default_rng(vocab)
    model = Model(40, 8, 128, vocab)
    b = build_batch(model, [{"P": 700, "segs": [20, 30, 10], "branches": [(n, 16, 16, 16) for n in (1, 2, 3)]}], rng)
    n_rows = b.n_logit_rows
    x = np.round(rng.standard_normal((n_rows, stride)).astype(np.float32) * 2) / 2  # coarse: many ties
    x[0, :] = -np.inf
    x[1, :] = np.nan
    x[2, :] = -0.0
    x[2, vocab - 1] = 0.0
    x[3, :] = np.nan
    x[3, vocab - 1] = -np.inf
    x[4, :] = 1.0
    x[5, :] = -1.0
    x[5, vocab - 1] = 4.0  # in the ragged end
    x[6, :] = np.inf
    x[7, :] = np.nan
    x[7, vocab // 2] = -7.0
    x[8, :] = -np.inf
    x[8, vocab - 1] = np.nan
    x[9, :] = -1.0
    x[9, 0] = x[9, vocab - 1] = 9.0  # the two ends
    row = 10
    for k in range(1, 9):  # across units: some of these are ends of a warp's run
        if k * UNIT < vocab:
            x[row, :] = -1.0
            x[row, k * UNIT - 1] = x[row, k * UNIT] = 9.0
            x[row + 1, :] = -np.inf
            x[row + 1, k * UNIT] = -3.0
            row += 2
    x[:, vocab:] = 99.0  # behind the vocabulary
    bits = bf16_round(x)
    bits[2, : vocab - 1] = 0x8000
    ref = O.row_argmax(bits[:, :vocab])
    drafts = ref.reshape(3, 17)[:, :16].copy()
    drafts[1, 9] = vocab  # never matches
    drafts[2, 0] = -1
    drafts = drafts.reshape(-1).astype(np.int32)
    n_ref, bonus_ref, _ = O.accept_greedy(bits[:, :vocab], drafts, b.cu_draft)
    verdict = np.ones(max(1, int(b.cu_verdict[-1])), dtype=np.uint8)
    ctx = B.Context(model, 0)
    plan, y = B.Plan(ctx, b), R.PassOutputs(b)
    zeros = type("T", (), dict(q=np.zeros((b.n_q_rows, 40, 128), np.uint16), k_pool=np.zeros((b.n_pool_pages, 8, 16, 128), np.uint16),
                               v_pool=np.zeros((b.n_pool_pages, 8, 16, 128), np.uint16), logits=None, draft_ids=drafts, verdict=verdict))
    dev = R.DeviceInputs(b, zeros, with_logits=False)
    dev.logits = R.bf16_tensor(bits, "cuda:0")[:, :vocab]
    for _ in range(2):  # the scratch comes back zeroed
        assert _launches(ctx, lambda: R.run_pass(ctx, plan, dev, y)) == 2
        assert plan.lr_poll_status() == 0
        assert np.array_equal(y.row_argmax.cpu().numpy(), ref)
        assert np.array_equal(y.n_accept.cpu().numpy(), n_ref) and np.array_equal(y.bonus_id.cpu().numpy(), bonus_ref)
        check_commit(y.commit_dict(), O.commit(b, verdict, n_ref))
    plan.close()
    ctx.close()


def test_the_wait_for_the_keys_runs_out():
    """The count of finished units never is what the commit waits for: the status says which wait it was; attention and the
    merge do not hang on it."""
    rng = np.random.Generator(np.random.PCG64(9))
    w = _finish("late", 3, Model(4, 1, 128, 20_000), [{"P": 600, "segs": [9, 20], "branches": [(n, 16, 16, 16) for n in (0, 1, 2)]} for _ in range(4)], rng,
                0.3, 0.7, True, True, "nan")
    b, t = w.batch, w.tensors
    ctx = B.Context(b.model, 0)
    plan, x, y = B.Plan(ctx, b), R.DeviceInputs(b, t), R.PassOutputs(b)
    assert _launches(ctx, lambda: R.run_pass(ctx, plan, x, y)) == 2
    assert plan.lr_poll_status() == 0
    want = [v.clone() for v in (y.out, y.lse)]
    y.out.zero_()
    y.scratch[0] = 900_000
    plan.lr_plan_debug_set_wait_limit(50_000)  # long enough for attention; this wait has twenty times as long
    R.run_pass(ctx, plan, x, y)
    detail = C.c_int32()
    assert B.lib().lr_poll_status(plan.handle, torch.cuda.current_stream().cuda_stream, C.byref(detail)) == -4  # LR_ETIMEOUT
    assert detail.value == 400
    assert all(torch.equal(v, u) for v, u in zip((y.out, y.lse), want))
    assert int(y.scratch.abs().sum().item()) == 0
    plan.close()
    ctx.close()
