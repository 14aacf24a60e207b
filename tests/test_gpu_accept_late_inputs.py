"""lr_accept_greedy by itself behind a kernel that lets its successor start at once and writes drafts, their ranges and the logits
some 50 us later."""
import numpy as np
import pytest
import torch

from lr_workloads import Model, bf16_round
from oracle import lr_oracle as O
from paper_2506_19830_b200 import binding as B
from paper_2506_19830_b200 import runner as R
from test_gpu_early_reads import DEV, ROUNDS, Packed, write_late  # noqa: F401  (write_late is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vocab,n_branch", [(64, 5), (4000, 5), (64, 400)])
def test_greedy_acceptance(write_late, vocab, n_branch):  # noqa: F811
    rng = np.random.default_rng(vocab + n_branch)
    n_draft = 6 * n_branch
    n_rows = n_branch + n_draft
    ctx = B.Context(Model(1, 1, 64, vocab), 0)
    versions, want = [], []
    for _ in range(3):
        bits = bf16_round((rng.standard_normal((n_rows, vocab)) * 3).astype(np.float32))
        cu = np.concatenate([[0], np.sort(rng.integers(0, n_draft + 1, n_branch - 1)), [n_draft]]).astype(np.int32)
        top = O.row_argmax(bits)
        likely = np.concatenate([top[cu[i] + i:cu[i + 1] + i] for i in range(n_branch)])
        drafts = np.where(rng.random(n_draft) < 0.8, likely, rng.integers(0, vocab, n_draft)).astype(np.int32)
        versions.append({"logits": bits.reshape(-1).view(np.int16), "n_accept": np.zeros(n_branch, np.int32), "drafts": drafts, "cu": cu,
                         "bonus": np.zeros(n_branch, np.int32)})
        want.append(O.accept_greedy(bits, drafts, cu)[:2])
    mem, scratch = Packed(versions), B.Context.accept_scratch(n_rows, DEV)
    mem.buf[:mem.n].copy_(mem.versions[2])
    logits = mem["logits"].view(torch.bfloat16).view(n_rows, vocab)
    got = []
    torch.cuda.synchronize()
    for i in range(ROUNDS):
        write_late(mem.buf, mem.versions[i % 3])
        ctx.lr_accept_greedy(logits, mem["drafts"], mem["cu"], mem["n_accept"], mem["bonus"], scratch)
        got.append([mem[k].clone() for k in ("n_accept", "bonus")])
    torch.cuda.synchronize()
    for i, g in enumerate(got):
        assert all(np.array_equal(a.cpu().numpy(), r) for a, r in zip(g, want[i % 3])), i
    assert int(scratch.abs().sum().item()) == 0
    ctx.close()
