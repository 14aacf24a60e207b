"""The tensor-core attention kernel at head size 64, named explicitly, against the fp64 oracle: one partial tile up to
plans whose pieces hold two query tiles, chains and trees, split keys and unsplit ones."""
import numpy as np
import pytest
import torch

from gpu_util import REL_LARGE, run_and_check_pass
from lr_workloads import Model, make_config, make_random_small, make_random_tree
from lr_workloads.gen import _finish
from oracle import lr_oracle as O
from paper_2506_19830_b200 import binding as B
from paper_2506_19830_b200 import runner as R

pytestmark = pytest.mark.gpu


def _chain(seed, hq, hkv, P, gamma, L, n_req=1):
    rng = np.random.Generator(np.random.PCG64(seed))
    reqs = [{"P": P + 37 * r, "segs": [int(v) for v in rng.integers(5, 70, size=gamma)], "branches": [(j, L, L, L) for j in range(gamma + 1)]}
            for r in range(n_req)]
    return _finish(f"chain64_{seed}", seed, Model(hq, hkv, 64, 1000), reqs, rng, 0.3, 0.6, True, True, "nan")


@pytest.mark.parametrize("make", [lambda: make_config(1)] + [lambda s=s: make_random_small(4200 + s, head_dim=64) for s in range(6)]
                         + [lambda s=s: make_random_tree(4300 + s, head_dim=64) for s in range(4)])
def test_small(make):
    run_and_check_pass(make(), path=B.PATH_TENSOR_CORE, rel_large=REL_LARGE)


@pytest.mark.parametrize("args", [(1, 16, 4, 2500, 3, 16), (2, 5, 1, 6000, 4, 9), (3, 8, 8, 1111, 2, 7, 3), (4, 32, 8, 9000, 3, 16, 2)])
def test_split_keys(args):
    w = _chain(*args)
    n = w.batch.n_branch
    run_and_check_pass(w, path=B.PATH_TENSOR_CORE, check_rows_of_branches=sorted({0, n // 2, n - 1}))


def test_weights_are_not_rounded_to_bf16():
    """Several bf16 terms per weight leave at most 2^-17 of it, so the output's own rounding (at most 2^-9 of every value) is
    all that is left to see in the 2-norm; bf16 weights alone would add 1.6e-3 to it."""
    w = _chain(5, 16, 4, 1500, 3, 16)
    b, t = w.batch, w.tensors
    ctx = B.Context(b.model, 0)
    plan = B.Plan(ctx, b)
    assert plan.lr_plan_describe()["uses_tensor_core"] == 1  # the automatic choice
    x, y = R.DeviceInputs(b, t), R.PassOutputs(b)
    plan.lr_verify_attention(x.q, x.k_pool, x.v_pool, y.out)
    assert plan.lr_poll_status() == 0
    ref, _ = O.verify_attention(b, t.q, t.k_pool, t.v_pool)
    got = y.out.to(torch.float64).cpu().numpy()
    assert np.linalg.norm(got - ref) <= (2.0 ** -9 + 2.0 ** -15) * np.linalg.norm(ref)
    ctx.close()


def test_weights_keep_their_fp32_bits():
    """The weights go to the tensor core as three bf16 terms that add up to the fp32 weight, so the kernel's only errors are
    those of fp32 sums (some 2^-21 of a value) and the rounding of the output.  An output is not the closest bf16 when
    the former carry it over the middle between two neighbours: twice 2^-21 / 2^-9, 5e-4 of them.  Two terms would leave
    2^-17 of a weight and 2e-3 of the outputs."""
    off, total = 0, 0
    for args in [(1, 16, 4, 2500, 3, 16), (2, 5, 1, 600, 4, 9), (3, 8, 8, 111, 2, 7, 3), (4, 32, 8, 256, 3, 16, 2)]:
        w = _chain(*args)
        b, t = w.batch, w.tensors
        ctx = B.Context(b.model, 0)
        plan = B.Plan(ctx, b)
        assert plan.lr_plan_describe()["uses_tensor_core"] == 1  # the automatic choice
        x, y = R.DeviceInputs(b, t), R.PassOutputs(b)
        plan.lr_verify_attention(x.q, x.k_pool, x.v_pool, y.out)
        assert plan.lr_poll_status() == 0
        ref, _ = O.verify_attention(b, t.q, t.k_pool, t.v_pool)
        got = y.out.to(torch.float64).cpu().numpy()
        closest = torch.from_numpy(ref).to(torch.bfloat16).to(torch.float64).numpy()
        off, total = off + int((closest != got).sum()), total + got.size
        ctx.close()
    assert off <= 1e-3 * total, off / total


def test_a_wait_that_runs_out():
    """As in test_gpu_errors, at this head size: the issuers' drain commits from the lane that issued the products."""
    w = _chain(6, 16, 4, 1500, 3, 16)
    b, t = w.batch, w.tensors
    ctx = B.Context(b.model, 0)
    plan = B.Plan(ctx, b)
    x, y = R.DeviceInputs(b, t), R.PassOutputs(b)
    plan.lr_verify_attention(x.q, x.k_pool, x.v_pool, y.out)
    want = y.out.clone()
    plan.lr_plan_debug_set_wait_limit(3000)
    plan.lr_plan_debug_set_phantom_bytes(4096)
    plan.lr_verify_attention(x.q, x.k_pool, x.v_pool, y.out)
    with pytest.raises(B.LrError) as e:
        plan.lr_poll_status()
    assert e.value.status == -4, e.value  # LR_ETIMEOUT
    plan.lr_plan_debug_set_phantom_bytes(0)
    plan.lr_plan_debug_set_wait_limit(1_000_000)
    for _ in range(2):
        plan.lr_verify_attention(x.q, x.k_pool, x.v_pool, y.out)
        assert plan.lr_poll_status() == 0
        assert torch.equal(y.out, want)
    ctx.close()


@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("args", [(7, 16, 4, 300, 2, 6), (8, 16, 4, 4000, 3, 16), (9, 32, 8, 2000, 3, 16, 12)])
def test_values_a_row_does_not_see_do_not_reach_it(args, value):
    """One branch's tail and the deepest step hold values that are not finite: rows that do not see them come out as
    without them, a row that does shows it in the channels concerned."""
    w = _chain(*args)
    b, t = w.batch, w.tensors
    ctx = B.Context(b.model, 0)
    plan = B.Plan(ctx, b)
    x, clean, got = R.DeviceInputs(b, t), R.PassOutputs(b), R.PassOutputs(b)
    plan.lr_verify_attention(x.q, x.k_pool, x.v_pool, clean.out, clean.lse)
    rows = np.zeros(b.n_q_rows, dtype=bool)
    page = int(b.page_ids[int(b.br_own_slot[1])])  # the second branch of the first request, from its third tail token on
    x.v_pool[page, :, 2, 5:9] = value
    rows[int(b.cu_q[1]) + max(0, 2 - int(b.br_own_len[1] - (b.cu_q[2] - b.cu_q[1]))): int(b.cu_q[2])] = True
    deepest = int(b.req_span_off[1]) - 1  # the last step of the first request
    x.v_pool[int(b.page_ids[int(b.span_slot[deepest])]), :, 1, 5:9] = value
    bad = [i for i in range(b.n_branch) if b.br_req[i] == 0 and b.br_depth[i] == deepest]
    for i in bad:
        rows[int(b.cu_q[i]): int(b.cu_q[i + 1])] = True
    for _ in range(2):
        plan.lr_verify_attention(x.q, x.k_pool, x.v_pool, got.out, got.lse)
        assert plan.lr_poll_status() == 0
        g, c = got.out.float().cpu().numpy(), clean.out.float().cpu().numpy()
        assert np.isfinite(g[~rows]).all() and np.abs(g[~rows] - c[~rows]).max() <= 2.0 ** -7 * np.abs(c).max()
        assert not np.isfinite(g[rows][:, :, 5:9]).any() and np.isfinite(np.delete(g[rows], np.s_[5:9], axis=2)).all()
        assert torch.equal(got.lse, clean.lse)
    ctx.close()
