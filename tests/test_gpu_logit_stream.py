"""The streaming part of the acceptance kernels at the sizes where its bookkeeping can go wrong: rows shorter than one
16-byte vector, rows that end inside a step, shares of a CTA that hold many rows or a sliver of one, chunks that grow
with the vocabulary.  Greedy results are exact; the sampled ones follow the rule of test_gpu_accept_sample."""
import numpy as np
import pytest
import torch

from lr_workloads import Model, bf16_round
from oracle import lr_oracle as O
from paper_2506_19830_b200 import binding as B
from paper_2506_19830_b200 import runner as R
from test_gpu_accept_sample import _check, _run

pytestmark = pytest.mark.gpu

# vocabulary, branches, drafts per branch
SIZES = [(1, 1, 0), (3, 40, 9), (7, 3, 1), (8, 5, 2), (9, 700, 3), (1023, 17, 4), (2047, 6, 3), (2048, 6, 3), (2049, 130, 5), (8193, 61, 8),
         (65543, 40, 6), (327680, 3, 2), (327681, 3, 2), (700001, 2, 1)]


def _make(vocab, nb, L, seed):
    rng = np.random.default_rng(seed)
    n_rows = nb * (L + 1)
    bits = bf16_round((rng.standard_normal((n_rows, vocab), dtype=np.float32) * 2))
    bits[::5, vocab // 2:] = 0xFF80  # -inf
    bits[1::7, : min(vocab, 6) - 1] = 0x7FC0  # NaN counts as -inf
    ref = O.row_argmax(bits)
    cu = (np.arange(nb + 1) * L).astype(np.int32)
    drafts = ref.reshape(nb, L + 1)[:, :L].reshape(-1).astype(np.int32).copy()
    flip = rng.random(len(drafts)) < 0.15
    drafts[flip] = (drafts[flip] + 1) % vocab
    return rng, bits, ref, cu, drafts


@pytest.mark.parametrize("vocab,nb,L", SIZES)
def test_greedy(vocab, nb, L):
    _, bits, ref, cu, drafts = _make(vocab, nb, L, vocab)
    n_ref, b_ref, _ = O.accept_greedy(bits, drafts, cu)
    stride = (vocab + 7) // 8 * 8
    padded = np.full((len(bits), stride), 0x7F80, dtype=np.uint16)
    padded[:, :vocab] = bits
    ctx = B.Context(Model(1, 1, 64, vocab), 0)
    i32 = dict(dtype=torch.int32, device="cuda:0")
    n_acc, bonus, arg = torch.empty(nb, **i32), torch.empty(nb, **i32), torch.empty(len(bits), **i32)
    d = torch.from_numpy(drafts if len(drafts) else np.zeros(1, np.int32)).to("cuda:0")
    ctx.lr_accept_greedy(R.bf16_tensor(padded, "cuda:0")[:, :vocab], d, torch.from_numpy(cu).to("cuda:0"), n_acc, bonus,
                         B.Context.accept_scratch(len(bits), "cuda:0"), arg)
    assert np.array_equal(arg.cpu().numpy(), ref) and np.array_equal(n_acc.cpu().numpy(), n_ref) and np.array_equal(bonus.cpu().numpy(), b_ref)
    ctx.close()


@pytest.mark.parametrize("vocab,nb,L", [s for s in SIZES if s[0] >= 8])
def test_sample(vocab, nb, L):
    rng, bits, _, cu, drafts = _make(vocab, nb, L, vocab + 1)
    bits[:, vocab // 2] = 0x3F80  # a row without a finite logit has no distribution
    ua, uf = rng.uniform(0, 1, max(1, len(drafts))), rng.uniform(0, 1, nb)
    ua[::2] = 0.0
    if not len(drafts):
        drafts = np.zeros(1, np.int32)
    got = _run(Model(1, 1, 64, vocab), bits, drafts, cu, 0.7, ua, uf)
    _check(bits, drafts, cu, 0.7, ua, uf, got)


@pytest.mark.parametrize("static", [False, True])
@pytest.mark.parametrize("b0", [0, 1, 20])
def test_greedy_on_the_later_branches_of_a_batch(b0, static):
    """Branch b's rows start at cu_draft[b] + b, also where cu_draft does not start at 0."""
    vocab, nb, L = 2049, 30, 5
    _, bits, ref, cu, drafts = _make(vocab, nb, L, 7)
    n_ref, b_ref, _ = O.accept_greedy(bits, drafts, cu)
    padded = np.full((len(bits), 2056), 0x7F80, dtype=np.uint16)
    padded[:, :vocab] = bits
    ctx = B.Context(Model(1, 1, 64, vocab), 0)
    i32 = dict(dtype=torch.int32, device="cuda:0")
    n, rows = nb - b0, len(bits) - b0
    n_acc, bonus, arg = torch.empty(n, **i32), torch.empty(n, **i32), torch.empty(rows, **i32)
    lg, d, c = R.bf16_tensor(padded, "cuda:0")[b0:, :vocab], torch.from_numpy(drafts).to("cuda:0"), torch.from_numpy(cu[b0:].copy()).to("cuda:0")
    if static:
        ctx.lr_accept_greedy_static(lg, d, c, n_acc, bonus, arg)
    else:
        ctx.lr_accept_greedy(lg, d, c, n_acc, bonus, B.Context.accept_scratch(rows, "cuda:0"), arg)
    assert np.array_equal(arg.cpu().numpy(), ref[b0:]) and np.array_equal(n_acc.cpu().numpy(), n_ref[b0:]) and np.array_equal(bonus.cpu().numpy(), b_ref[b0:])
    ctx.close()
