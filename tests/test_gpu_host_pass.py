"""A pass from host buffers whose logits lie below and above the size from which the acceptance runs in two parts: every
result equals the oracle's (acceptance, lists) or, bit for bit, the same attention from device buffers."""
import numpy as np
import pytest
import torch

from lr_workloads import Model
from lr_workloads.gen import _finish
from oracle import lr_oracle as O
from paper_2506_19830_b200 import binding as B
from paper_2506_19830_b200 import runner as R

pytestmark = pytest.mark.gpu

PARTS_BYTES = 64 << 20


# (draft lengths of the branches, vocabulary): one branch only (nothing to part), one row under the line, at it, a last
# branch longer than a sixteenth of the rows, branches of one row
@pytest.mark.parametrize("drafts,vocab", [([40], 900_000), ([3] * 8, 1_048_568), ([3] * 8, 1_048_576), ([2] * 9 + [30], 600_000), ([0] * 40, 840_000)])
@pytest.mark.parametrize("pinned", [True, False])
def test_host_pass(drafts, vocab, pinned):
    rng = np.random.Generator(np.random.PCG64(len(drafts) * 7 + drafts[-1]))
    reqs = [{"P": 40 + 9 * (i % 5), "segs": [7], "branches": [(1, max(n, 1), max(n, 1), n)]} for i, n in enumerate(drafts)]
    w = _finish("host", 3, Model(4, 1, 128, vocab), reqs, rng, 0.5, 0.6, True, True, "nan")
    b, t = w.batch, w.tensors
    n_rows = sum(drafts) + len(drafts)
    assert (n_rows * vocab * 2 >= PARTS_BYTES) == (vocab != 1_048_568)
    ctx = B.Context(b.model, 0)
    plan = B.Plan(ctx, b)
    x, y = R.DeviceInputs(b, t), R.PassOutputs(b)
    plan.lr_verify_attention(x.q, x.k_pool, x.v_pool, y.out)
    assert plan.lr_poll_status() == 0
    keep = (lambda a: a.pin_memory()) if pinned else (lambda a: a)
    host = {"q_h": keep(torch.from_numpy(t.q.view(np.int16))), "logits_h": keep(torch.from_numpy(t.logits.view(np.int16))),
            "draft_ids_h": keep(torch.from_numpy(t.draft_ids)), "verdict_h": keep(torch.from_numpy(t.verdict)),
            "out_h": keep(torch.zeros((b.n_q_rows, b.model.n_q_heads, b.model.head_dim), dtype=torch.int16))}
    for name, n in (("n_accept_h", b.n_branch), ("bonus_id_h", b.n_branch), ("n_steps_accepted_h", b.n_req), ("survivor_h", b.n_req),
                    ("committed_len_h", b.n_req), ("keep_off_h", b.n_req + 1), ("free_off_h", b.n_req + 1), ("keep_pages_h", b.n_page_slots),
                    ("keep_valid_h", b.n_page_slots), ("free_pages_h", b.n_page_slots)):
        host[name] = keep(torch.zeros(n, dtype=torch.int32))
    io, staging = B.lr_pass_host_io(**{k: v.data_ptr() for k, v in host.items()}), plan.pass_staging()
    n_ref, bonus_ref, _ = O.accept_greedy(t.logits, t.draft_ids, b.cu_draft)
    c = O.commit(b, t.verdict, n_ref)
    nk, nf = int(c["keep_off"][-1]), int(c["free_off"][-1])
    for _ in range(2):
        assert plan.lr_verify_pass_host(io, x.k_pool, x.v_pool, staging) in (0, None)
        assert torch.equal(host["out_h"], y.out.view(torch.int16).cpu().view(host["out_h"].shape))
        assert np.array_equal(host["n_accept_h"].numpy(), n_ref) and np.array_equal(host["bonus_id_h"].numpy(), bonus_ref)
        for name, n in (("keep_off", None), ("free_off", None), ("committed_len", None), ("keep_pages", nk), ("keep_valid", nk), ("free_pages", nf)):
            assert np.array_equal(host[name + "_h"].numpy()[:n], c[name][:n]), name
        for k in ("out_h", "n_accept_h", "bonus_id_h", "keep_pages_h"):
            host[k].zero_()
    plan.close()
    ctx.close()
