"""A plan is destroyed once and before its context, in whatever order the two Python objects go."""
import gc

import numpy as np
import pytest
import torch

from lr_workloads import Model, build_batch
from paper_2506_19830_b200 import binding as B


class _Lib:
    """Hands out handles and writes down what is destroyed."""

    def __init__(self):
        self.gone, self.n = [], 100

    def _new(self, out):
        self.n += 8
        out._obj.value = self.n
        return 0

    def lr_create(self, out, model, device):
        return self._new(out)

    def lr_plan_begin(self, ctx, batch, n_bytes, draft):
        n_bytes._obj.value = 1024
        return self._new(draft)

    def lr_plan_finish(self, draft, ws, n_bytes, stream, out):
        return self._new(out)

    def lr_plan_destroy(self, plan):
        self.gone.append(("plan", getattr(plan, "value", plan)))
        return 0

    def lr_destroy(self, ctx):
        self.gone.append(("ctx", ctx.value))
        return 0


def _make(monkeypatch):
    fake = _Lib()
    monkeypatch.setattr(B, "lib", lambda: fake)
    monkeypatch.setattr(B, "_stream_ptr", lambda stream: 0)
    monkeypatch.setattr(torch, "empty", lambda n, dtype=None, device=None: torch.zeros(n, dtype=dtype))
    model = Model(2, 1, 64, 16)
    b = build_batch(model, [{"P": 5, "segs": [3], "branches": [(1, 2, 2, 2)]}], np.random.default_rng(0))
    ctx = B.Context(model, 0)
    return fake, ctx, [B.Plan(ctx, b) for _ in range(2)]


def _expect(fake, ctx, plans):
    kinds = [k for k, _ in fake.gone]
    assert kinds == ["plan"] * len(plans) + ["ctx"] and {v for k, v in fake.gone if k == "plan"} == set(plans) and fake.gone[-1] == ("ctx", ctx)


@pytest.mark.parametrize("how", ["cycle", "context first", "plans first", "one closed"])
def test_order(monkeypatch, how):
    fake, ctx, plans = _make(monkeypatch)
    c, ps = ctx.handle.value, [p.handle.value for p in plans]
    if how == "cycle":
        everything = [ctx, *plans]
        everything.append(everything)
        del ctx, plans, everything
        gc.collect()
    elif how == "context first":
        ctx.close()
        for p in plans:
            p.close()
    else:
        for p in plans[: 1 if how == "one closed" else 2]:
            p.close()
            p.close()
        ctx.close()
    _expect(fake, c, ps)
