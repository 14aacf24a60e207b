"""A plan made in two steps is the plan made in one: the same size, the same results; a draft may also be dropped."""
import ctypes as C

import numpy as np
import pytest
import torch

from lr_workloads import make_config, make_random_tree
from paper_2506_19830_b200 import binding as B
from paper_2506_19830_b200 import runner as R

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make", [lambda: make_config(1), lambda: make_random_tree(77, head_dim=128)])
def test_one_step_and_two(make):
    w = make()
    b, t = w.batch, w.tensors
    ctx = B.Context(b.model, 0)
    two = B.Plan(ctx, b)
    lib, host, n, draft, handle = B.lib(), B.HostBatch(b), C.c_size_t(), C.c_void_p(), C.c_void_p()
    assert lib.lr_plan_begin(ctx.handle, C.byref(host.c), C.byref(n), C.byref(draft)) == 0 and lib.lr_plan_drop(draft) == 0
    assert n.value == two.workspace_bytes
    n = C.c_size_t()
    assert lib.lr_plan_bytes(ctx.handle, C.byref(host.c), C.byref(n)) == 0 and n.value == two.workspace_bytes
    one = B.Plan(ctx, b)  # its handle is replaced by the one-step plan's
    lib.lr_plan_destroy(one.handle)
    assert lib.lr_plan_create(ctx.handle, C.byref(host.c), one._ws_ptr, n.value, B._stream_ptr(None), C.byref(handle)) == 0
    one.handle = handle
    x, outs = R.DeviceInputs(b, t), []
    for plan in (two, one):
        y = R.PassOutputs(b)
        R.run_pass(ctx, plan, x, y)
        assert plan.lr_poll_status() == 0
        outs.append((y.out.view(torch.int16).cpu().numpy(), y.commit_dict()))
    assert np.array_equal(outs[0][0], outs[1][0])
    assert all(np.array_equal(outs[0][1][k], outs[1][1][k]) for k in outs[0][1])
    ctx.close()


def test_too_small_a_workspace_ends_the_draft():
    b = make_config(1).batch
    ctx = B.Context(b.model, 0)
    lib, host, n, draft, handle = B.lib(), B.HostBatch(b), C.c_size_t(), C.c_void_p(), C.c_void_p()
    assert lib.lr_plan_begin(ctx.handle, C.byref(host.c), C.byref(n), C.byref(draft)) == 0
    ws = torch.empty(n.value, dtype=torch.uint8, device="cuda:0")
    assert lib.lr_plan_finish(draft, ws.data_ptr(), n.value - 1, None, C.byref(handle)) != 0 and not handle.value
    ctx.close()
