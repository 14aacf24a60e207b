"""Attention set up while the kernel before it still runs: queries and cache hold other values until a kernel that lets its
successor start at once writes the real ones some 50 us later.  Group sizes that leave rows of an M-tile without a query, and
fewer pages, or more, than a CTA's record carries (32)."""
import numpy as np
import pytest
import torch

from gpu_util import REL_LARGE, check_attention
from lr_workloads import Model
from lr_workloads.gen import _finish
from oracle import lr_oracle as O
from paper_2506_19830_b200 import binding as B
from paper_2506_19830_b200 import runner as R
from test_gpu_early_reads import write_late  # noqa: F401 (a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("group,head_dim,prefix,n_req", [(1, 128, 40, 1), (3, 64, 500, 2), (5, 128, 530, 2), (7, 64, 17, 3), (9, 128, 1500, 1), (16, 128, 700, 2)])
def test_inputs_written_late(write_late, group, head_dim, prefix, n_req):  # noqa: F811
    rng = np.random.Generator(np.random.PCG64(group))
    reqs = [{"P": prefix + 3 * r, "segs": [20, 33], "branches": [(0, 9, 4, 4), (1, 30, 30, 3), (2, 5, 5, 5)]} for r in range(n_req)]
    w = _finish("start", group, Model(2 * group, 2, head_dim, 64), reqs, rng, 0.4, 0.8, True, True, "nan")
    b, t = w.batch, w.tensors
    ctx = B.Context(b.model, 0)
    plan, x, y = B.Plan(ctx, b), R.DeviceInputs(b, t), R.PassOutputs(b)
    o_ref, l_ref = O.verify_attention(b, t.q, t.k_pool, t.v_pool)
    for name in ("q", "k_pool", "v_pool"):
        now, real = getattr(x, name), getattr(x, name).clone()
        for _ in range(3):
            now.zero_()
            y.out.fill_(float("nan"))
            write_late(now.view(torch.uint8).flatten(), real.view(torch.uint8).flatten())
            plan.lr_verify_attention(x.q, x.k_pool, x.v_pool, y.out, y.lse)
            assert plan.lr_poll_status() == 0
            check_attention(y.out, y.lse, o_ref, l_ref, rel_large=REL_LARGE)
    ctx.close()
