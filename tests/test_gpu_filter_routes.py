"""lr_accept_sample_filtered on both sides of every line its dispatch draws -- group sizes, candidates or windows, rows
left over by the candidates, cluster sizes, rows in and out of shared memory -- by the rule of test_gpu_accept_filtered."""
import numpy as np
import pytest
import torch

from lr_workloads import Model, bf16_round
from paper_2506_19830_b200 import binding as B
from paper_2506_19830_b200 import runner as R
from test_gpu_accept_filtered import _check, _run

pytestmark = pytest.mark.gpu

# vocabulary, branches, drafts per branch, top_k, top_p (not a multiple of 1 / top_k: with tokens of equal
# mass the cut would lie on a step)
ROUTES = [
    (5, 3, 2, 2, 0.9), (300, 4, 3, 20, 0.93), (1023, 4, 3, 0, 0.9), (1025, 170, 2, 0, 0.9),  # fewer groups than leading tokens
    (5119, 5, 3, 20, 0.93), (5120, 5, 3, 20, 0.93), (5121, 5, 3, 20, 1.0),                     # groups of 8, of 64
    (4100, 5, 3, 256, 0.97), (65600, 5, 2, 256, 1.0), (65600, 5, 2, 257, 1.0),                 # the longest list of kept tokens
    (65600, 3, 2, 1024, 1.0), (65600, 3, 2, 1025, 0.9), (5000, 40, 2, 1024, 0.97),             # the largest top_k of the candidates
    (20011, 150, 2, 3000, 0.9131), (160011, 60, 1, 2000, 0.9131), (160011, 150, 1, 2000, 0.9131),       # single CTAs, pairs, fours, eights
    (90001, 4, 1, 2000, 0.9131), (600, 130, 1, 500, 0.9131),
    (32771, 12, 2, 0, 0.95), (32771, 160, 2, 0, 0.95), (40009, 30, 4, 0, 0.6),                 # few rows by windows, many by candidates
    (100003, 150, 1, 500, 0.9131), (100003, 300, 1, 800, 0.9131),                              # groups of 32 and of 16, sorted candidates
    (655361, 2, 1, 20, 0.93), (1700003, 1, 1, 0, 0.9), (9000, 2, 1, 0, 1.0),                   # too many groups; shares beyond shared memory
]


@pytest.mark.parametrize("vocab,nb,L,top_k,top_p", ROUTES)
def test_routes(vocab, nb, L, top_k, top_p):
    rng = np.random.default_rng(vocab + nb)
    n_rows = nb * (L + 1)
    x = (rng.standard_normal((n_rows, vocab), dtype=np.float32) * 1.5)
    lead = rng.integers(0, vocab, (n_rows, 3))
    for r in range(n_rows):  # peaked, flat, coarse (many ties), and rows with values outside the usual octaves
        if r % 4 != 1:
            x[r, lead[r]] = rng.uniform(6, 20, 3)
        if r % 4 == 2:
            x[r] = np.round(x[r] * 2) / 2
        if r % 4 == 3:
            x[r, : max(1, vocab // 100)] = 1e-9
            x[r, vocab // 2] = -7000.0
    x[::5, vocab // 3: vocab // 2] = -np.inf
    x[::6, vocab // 5: vocab // 4] = 1e-8  # with the ties of 0 in the coarse rows: the cut in, above and below the middle group
    x[::9] = np.minimum(x[::9], -1.0)
    bits = bf16_round(x)
    bits[::3, -1] = 0x7FC0  # NaN counts as -inf
    cu = (np.arange(nb + 1) * L).astype(np.int32)
    drafts = lead.reshape(nb, L + 1, 3)[:, :L, 0].reshape(-1).astype(np.int32).copy()
    ua, uf = rng.uniform(0, 1, len(drafts)), rng.uniform(0, 1, nb)
    ua[::3] = 0.0
    got = _run(Model(1, 1, 64, vocab), bits, drafts, cu, 0.8, top_k, top_p, ua, uf)
    rows = None if n_rows * vocab < 3e6 else sorted(set(rng.integers(0, n_rows, 12).tolist()))
    # A flat row of 40009 tokens keeps some 2000 at top_p 0.6, the last with 1.5e-4 of their mass: above HEAVY, and within
    # the rule's 4e-5 of the step in one row of four.  A branch looks at two rows or so, one in four of them flat, and
    # draws differ on a few more: 0.4 of the branches leaves room for twice the expected number.
    _check(bits, drafts, cu, 0.8, top_k, top_p, ua, uf, got, max_ambiguous_frac=0.4, rows_to_check=rows)


# Top-p alone over many rows: the candidates are tried on 16 of them first.  Which rows are flat -- none, all, those tried
# only, those behind only -- decides whether the rest is tried and by which windows the open rows go.
@pytest.mark.parametrize("flat", ["none", "all", "first", "rest", "mixed"])
def test_probe(flat):
    vocab, nb, L = 40009, 150, 3
    n_rows = nb * (L + 1)
    rng = np.random.default_rng(len(flat))
    x = rng.standard_normal((n_rows, vocab), dtype=np.float32)
    lead = rng.integers(0, vocab, n_rows)
    r = np.arange(n_rows)
    peaked = {"none": r >= 0, "all": r < 0, "first": r >= 16, "rest": r < 16, "mixed": r % 2 == 0}[flat]
    x[r[peaked], lead[peaked]] = 18.0
    bits = bf16_round(x)
    cu = (np.arange(nb + 1) * L).astype(np.int32)
    drafts = lead.reshape(nb, L + 1)[:, :L].reshape(-1).astype(np.int32).copy()
    ua, uf = rng.uniform(0, 1, len(drafts)), rng.uniform(0, 1, nb)
    ua[::3] = 0.0
    got = _run(Model(1, 1, 64, vocab), bits, drafts, cu, 0.8, 0, 0.93, ua, uf)
    rows = sorted({0, 15, 16, 17, n_rows - 1} | set(rng.integers(0, n_rows, 12).tolist()))
    # A flat row keeps some 25000 tokens, the last one with 1e-5 of their mass: nearly every draw from one lies within the
    # rule's 4e-5 of a step, so that all branches that reach one may be undecided by it; the kept counts and masses are
    # checked all the same.  Four of the 150 branches have the first 16 rows; without flat rows no branch is undecided.
    undecided = {"none": 0.0, "first": 4 / 150}.get(flat, 1.0)
    _check(bits, drafts, cu, 0.8, 0, 0.93, ua, uf, got, max_ambiguous_frac=undecided, rows_to_check=rows)


def _same_in_parts(bits, L, T, top_k, top_p, drafts, ua, uf, part=3):
    """One call on all rows, and calls on a few branches at a time that go through the windows alone: every output equal."""
    n_rows, vocab = bits.shape
    nb = n_rows // (L + 1)
    cu = (np.arange(nb + 1) * L).astype(np.int32)
    lg = R.bf16_tensor(bits, "cuda:0")
    ctx = B.Context(Model(1, 1, 64, vocab), 0)

    def call(b0, b1):
        r, d = slice(b0 * (L + 1), b1 * (L + 1)), slice(b0 * L, b1 * L)
        t = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a, dtype=dt)).to("cuda:0")  # noqa: E731
        out = [torch.full((n,), -7, dtype=dt, device="cuda:0") for n, dt in ((b1 - b0, torch.int32), (b1 - b0, torch.int32), ((b1 - b0) * L, torch.float32),
                                                                           ((b1 - b0) * (L + 1), torch.int32))]
        before = ctx.launch_count
        ctx.lr_accept_sample_filtered(lg[r], t(drafts[d], np.int32), t(cu[: b1 - b0 + 1], np.int32), T, top_k, top_p, t(ua[d], np.float32),
                                      t(uf[b0:b1], np.float32), out[0], out[1], ctx.accept_sample_filtered_scratch((b1 - b0) * (L + 1)), out[2], out[3])
        return [o.cpu().numpy() for o in out], ctx.launch_count - before

    many, n_many = call(0, nb)
    for b in range(0, nb, part):
        few, n_few = call(b, b + part)
        assert n_few < n_many  # windows alone
        for name, a, e, size in zip(("n_accept", "final_id", "p_draft", "n_kept"), many, few, (1, 1, L, L + 1)):
            assert np.array_equal(a[b * size: (b + part) * size], e), (name, b)
    ctx.close()


# Which route a row takes depends on how many rows the call has; what comes out must not.  Low temperatures and offsets make
# the scaled logits large, equal leaders put top_p next to a step of the cumulative mass (0.94999 of 20 equal tokens: 19
# are kept, by a margin of 1e-5).
@pytest.mark.parametrize("T,offset,top_p", [(0.05, 0.0, 0.94999), (0.1, 0.0, 0.94999), (0.1, 0.0, 0.9), (0.6, 0.0, 0.94999), (0.6, 250.0, 0.94999),
                                            (0.6, -1000.0, 0.94999), (1.0, 1000.0, 0.94999)])
def test_routes_agree(T, offset, top_p):
    vocab, nb, L = 152064, 102, 3
    n_rows = nb * (L + 1)
    rng = np.random.default_rng(int(abs(offset) + 100 * T))
    x = rng.standard_normal((n_rows, vocab), dtype=np.float32) * np.float32(1.5 * min(T, 0.6) / 0.6)
    lead = rng.integers(0, vocab // 20, n_rows)
    for r in range(n_rows):
        n = (20, 1, 20, 4, 20, 19)[r % 6]
        x[r, lead[r] + vocab // 20 * np.arange(n)] = rng.uniform(18, 60)
    drafts = lead.reshape(nb, L + 1)[:, :L].reshape(-1).astype(np.int32).copy()
    ua, uf = rng.uniform(0, 1, len(drafts)), rng.uniform(0, 1, nb)
    ua[::3] = 0.0
    _same_in_parts(bf16_round(x + np.float32(offset)), L, T, 0, top_p, drafts, ua, uf)


# The same for a top-k of several hundred (candidates read many at a time, in groups of 64 and of 32, ranked by counting and
# by sorting, among them many of equal value), and for flat rows, on which the candidates are given up.
@pytest.mark.parametrize("flat,top_k,top_p", [(0, 130, 0.9131), (0, 200, 1.0), (0, 400, 0.9131), (0, 800, 0.9131), (0, 1000, 1.0), (1, 400, 0.9131), (1, 0, 0.95), (2, 0, 0.95)])
def test_routes_agree_on_large_kept_sets(flat, top_k, top_p):
    vocab, nb, L = 152064, 102, 3
    n_rows = nb * (L + 1)
    rng = np.random.default_rng(flat + top_k)
    x = rng.standard_normal((n_rows, vocab), dtype=np.float32) * np.float32(1.5)
    lead = rng.integers(0, vocab, n_rows)
    rows = np.arange(n_rows)[{0: slice(None), 1: slice(0, 0), 2: slice(16, None)}[flat]]
    x[rows, lead[rows]] = rng.uniform(4, 22, len(rows))
    x[::7] = np.round(x[::7] * 4) / 4  # thousands of equal values
    x[::5, : vocab // 3] = -np.inf
    drafts = lead.reshape(nb, L + 1)[:, :L].reshape(-1).astype(np.int32).copy()
    ua, uf = rng.uniform(0, 1, len(drafts)), rng.uniform(0, 1, nb)
    ua[::3] = 0.0
    _same_in_parts(bf16_round(x), L, 0.6, top_k, top_p, drafts, ua, uf)


def test_scratch_does_not_grow_with_groups_nobody_uses():
    """Per row: the list (2 KB), 32 bytes for the cut, a pair per 2048 tokens and the group maxima, of which there are at most
    8192 (twice the four times 1024 a top-k can ask for), or one per 64 tokens where that is more, two bytes each."""
    for vocab in (1000, 32768, 50000, 65536, 65537, 152064, 400003):
        ctx = B.Context(Model(1, 1, 64, vocab), 0)
        n_chunks = (vocab + 2047) // 2048
        groups = min(256 * n_chunks, max(8192 + 256, 32 * n_chunks))
        assert ctx.accept_sample_filtered_scratch(1000).numel() * 8 <= 1000 * (2048 + 32 + 8 * n_chunks + 2 * groups + 4) + 128, vocab
        ctx.close()
