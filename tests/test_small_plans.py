"""How the attention work of a batch is split (host side of the planner): lr_verify_attention's partition knows nothing of the
logits, a small pass with head size 64 that has one of its own keeps to its bounds, and one with head size 128, whose results hang
on the split of the keys, has attention's."""
import numpy as np
import pytest

from lr_workloads import Model, build_batch
from paper_2506_19830_b200 import binding as B

GEOMETRIES = [(40, 8, 128), (32, 8, 128), (16, 4, 128), (8, 8, 128), (5, 1, 128), (32, 8, 64), (4, 1, 64)]


def _batch(geometry, vocab, n_req, prefix, steps, drafts, seed=0):
    rng = np.random.default_rng(seed)
    reqs = [{"P": prefix, "segs": [32] * steps, "branches": [(n, drafts, drafts, drafts) for n in range(1, steps + 1)]} for _ in range(n_req)]
    return build_batch(Model(*geometry, vocab), reqs, rng)


def _time(part):  # microseconds, as the planner counts them
    return 4.1 + part["longest_load"] / 50.0


@pytest.mark.parametrize("geometry", GEOMETRIES)
@pytest.mark.parametrize("n_sm", [148, 132])
def test_bounds(geometry, n_sm):
    narrow = 0
    for n_req in (1, 2, 4, 8, 16, 32):
        for prefix in (100, 500, 1000, 4000, 8000, 32000):
            for steps, drafts in ((3, 4), (5, 4), (3, 16)):
                seen = set()
                for vocab in (8, 8000, 32000, 152064):
                    b = _batch(geometry, vocab, n_req, prefix, steps, drafts)
                    attention, own, small = B.lr_debug_partitions(b.model, b, n_sm)
                    seen.add(tuple(attention.values()))
                    assert 1 <= own["n_cta"] <= attention["n_cta"] <= n_sm
                    assert small != 2 or (own == attention and attention["n_merge_targets"] > 0)
                    if own != attention:
                        narrow += 1
                        assert geometry[2] == 64 and small == 1 and own["n_cta"] < attention["n_cta"]
                        assert _time(own) <= 1.25 * _time(attention)
                        assert attention["n_merge_targets"] > 0 or own["n_merge_targets"] == 0
                assert len(seen) == 1  # whatever the vocabulary
    assert geometry != (32, 8, 64) or narrow > 0


# (geometry, vocabulary, requests, prefix, steps, drafts): the CTAs of attention, and its merge targets
@pytest.mark.parametrize("args,n_cta,merges", [(((32, 8, 128), 32000, 16, 500, 3, 4), 128, 0), (((32, 8, 128), 32000, 16, 100, 3, 4), 128, 0),
                                               (((40, 8, 128), 32000, 4, 500, 3, 16), 128, 64), (((40, 8, 128), 152064, 4, 100, 5, 4), 96, 32),
                                               (((5, 1, 128), 152064, 16, 100, 3, 4), 16, 0), (((40, 8, 128), 152064, 1, 4096, 3, 16), 144, 16)])
def test_attention_has_all_sms(args, n_cta, merges):
    b = _batch(*args)
    attention, _, _ = B.lr_debug_partitions(b.model, b, 148)
    assert (attention["n_cta"], attention["n_merge_targets"]) == (n_cta, merges)
