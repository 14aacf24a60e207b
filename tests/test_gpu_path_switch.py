"""The CTA-pair plan is built when its path is selected and lies over the scratch of the single-CTA path: switching back and
forth on one plan, with passes in between, must give what each path gives on a plan of its own."""
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
