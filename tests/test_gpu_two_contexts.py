"""A pass whose context is not the plan's: the acceptance goes by the given context's vocabulary, on both sides of the lines that
decide how a pass is launched, on one stream and on two.  The buffers are large enough for either vocabulary."""
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
SMALL, LARGE = 1000, 5008


@pytest.mark.parametrize("n_req,two", [(2, True), (513, False)])  # requests: 512 at most in two kernels
@pytest.mark.parametrize("plan_vocab,given_vocab", [(LARGE, SMALL), (SMALL, LARGE)])
@pytest.mark.parametrize("second_stream", [False, True])
def test_the_given_vocabulary_counts(n_req, two, plan_vocab, given_vocab, second_stream):
    rng = np.random.Generator(np.random.PCG64(n_req))
    reqs = [{"P": 40, "segs": [3, 5], "branches": [(g, 3, 3, 3) for g in (0, 1, 2)]} for _ in range(n_req)]
    w = _finish("two", 7, Model(4, 1, 128, SMALL), reqs, rng, 0.6, 0.8, True, True, "nan")
    b, t = w.batch, w.tensors
    padded = np.full((t.logits.shape[0], LARGE), 0x4700, dtype=np.uint16)  # 32768 behind the smaller vocabulary
    padded[:, :SMALL] = t.logits
    padded[:, LARGE - 8] = 0x4780  # twice that
    ctx, given = B.Context(Model(4, 1, 128, plan_vocab), 0), B.Context(Model(4, 1, 128, given_vocab), 0)
    plan, x, y = B.Plan(ctx, b), R.DeviceInputs(b, t, with_logits=False), R.PassOutputs(b)
    x.logits = R.bf16_tensor(padded, "cuda:0")
    before = ctx.launch_count + given.launch_count
    if second_stream:
        R.run_pass_overlapped(given, plan, x, y, torch.cuda.Stream())
    else:
        R.run_pass(given, plan, x, y)
        assert (ctx.launch_count + given.launch_count - before == 2) == two
    assert plan.lr_poll_status() == 0
    n_ref, bonus_ref, _ = O.accept_greedy(padded[:, :given_vocab], t.draft_ids, b.cu_draft)
    assert np.array_equal(y.n_accept.cpu().numpy(), n_ref) and np.array_equal(y.bonus_id.cpu().numpy(), bonus_ref)
    check_commit(y.commit_dict(), O.commit(b, t.verdict, n_ref))
    assert int(y.scratch.abs().sum().item()) == 0
    out_ref, _ = O.verify_attention(b, t.q, t.k_pool, t.v_pool)
    check_attention(y.out, None, out_ref, None, rel_large=REL_LARGE)
    plan.close()
    given.close()
    ctx.close()
