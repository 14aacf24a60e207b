"""The work that users of this package have it do, as cases that can be timed and compared.

A case describes one call sequence of a serving program on one batch: ``step`` names the sequence (see ``run``), the
head geometry and the vocabulary describe the model, and the rest the batch -- how many requests, the range their
prefix lengths, draft steps, step lengths and token drafts are drawn from, a chain of draft steps (``tree_width`` 0)
or a full tree.  ``lengths`` seeds those lengths, so the work of a case is fixed; ``prepare``'s seed gives the values
and the page table.

Sequences:
  pass    attention, greedy acceptance, commit, one after another on the caller's stream (the README's example)
  overlap the same with acceptance and commit on a second stream
  sample  what follows the last layer when the target samples: stochastic acceptance, commit
  filter  the same with the top-k / top-p filters on the target distribution
  cycle   a whole serving cycle: the K/V of the newly drafted tokens go into their pages, a plan is made for the batch,
          attention runs on every layer, then acceptance, commit, compaction of every layer and the status
  host    one pass from pinned host buffers
"""
from __future__ import annotations

import math

import numpy as np
import torch

from lr_workloads import Model, build_batch
from paper_2506_19830_b200 import binding as B
from paper_2506_19830_b200 import runner as R

DEV = "cuda:0"

BASE = {
    "step": "pass", "q_heads": 40, "kv_heads": 8, "head_dim": 128, "vocab": 152064, "requests": 1, "prefix_min": 4096, "prefix_max": 4096,
    "steps_min": 3, "steps_max": 3, "seg_min": 32, "seg_max": 32, "drafts_min": 16, "drafts_max": 16, "tree_width": 0, "carry_in": False,
    "layers": 1, "temperature": 0.0, "top_k": 0, "top_p": 1.0, "lengths": 1,
}
SERVING = {"requests": 16, "prefix_min": 1024, "prefix_max": 16384, "steps_min": 2, "steps_max": 6, "seg_min": 16, "seg_max": 64,
           "drafts_min": 4, "drafts_max": 16, "lengths": 5}


def listed():
    def case(name, **kw):
        return dict(BASE, name=name, **kw)

    return [
        # a very small model early in its answer: the smallest call there is, latency and launches only (head size 64)
        case("tiny_chain", q_heads=4, kv_heads=1, head_dim=64, vocab=1024, prefix_min=256, prefix_max=256, steps_min=2, steps_max=2, seg_min=24,
             seg_max=24, drafts_min=8, drafts_max=8),
        # one request of a 32B-class model, 4 K tokens in: a single user waiting for an answer
        case("layer_chain"),
        # the same for a smaller model, whose heads are 64 wide
        case("layer_head64", q_heads=32, head_dim=64),
        # a few requests far into long reasoning traces
        case("long_context", requests=4, prefix_min=16384, prefix_max=16384, steps_min=4, steps_max=4, seg_min=48, seg_max=48, drafts_min=8,
             drafts_max=8),
        # one request at 32 K tokens with deep speculation: many query rows for one cache
        case("long_request", q_heads=32, prefix_min=32768, prefix_max=32768, steps_min=6, steps_max=6, seg_min=40, seg_max=40),
        # a serving batch: ragged lengths everywhere, acceptance beside attention
        case("ragged_serving", **dict(SERVING, step="overlap")),
        # multi-branch drafting in a serving batch: four proposals a step, two steps deep, a target branch on every node
        case("tree_serving", **dict(SERVING, requests=8, steps_min=2, steps_max=2, tree_width=4)),
        # sampling at the paper's temperature, no filters, over a serving batch
        case("sample_serving", **dict(SERVING, step="sample", temperature=0.6)),
        # the paper's two sampling settings: top-k 20 with top-p 0.95 over a serving batch ...
        case("topk_topp_serving", **dict(SERVING, step="filter", temperature=0.6, top_k=20, top_p=0.95)),
        # ... and top-p 0.95 alone, for a single request
        case("topp_layer", step="filter", temperature=0.6, top_p=0.95),
        # a whole cycle of a serving engine, over a few layers, with the carried-in token as a query (the plan is made
        # once a cycle, attention runs once a layer)
        case("cycle_serving", **dict(SERVING, step="cycle", requests=8, layers=4, carry_in=True)),
        # a program whose logits and queries are in host memory: the whole pass from pinned buffers
        case("host_serving", **dict(SERVING, step="host")),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    # a drawn case has no more work than the largest listed one of its sequence (or, with a head size of 64, of that size)
    kind = lambda c: (c["step"] in ("sample", "filter"), c["head_dim"]) if c["step"] in ("sample", "filter") or c["head_dim"] == 64 else c["step"]  # noqa: E731
    most = {}
    for c in listed():
        w, m = work(c), most.setdefault(kind(c), {"bytes": 0.0, "flops": 0.0})
        most[kind(c)] = {k: max(w[k], m[k]) for k in m}
    most[(True, 64)] = most[(True, 128)]
    while True:
        step = rng.choices(["pass", "overlap", "sample", "filter", "cycle", "host"], [30, 20, 12, 24, 8, 6])[0]
        hq, hkv, hd = rng.choice([(40, 8, 128)] * 3 + [(32, 8, 128)] * 2 + [(16, 4, 128), (8, 8, 128), (5, 1, 128), (32, 8, 64), (4, 1, 64)])
        pmax = _log_int(rng, 100, 32768)
        tree = rng.choice([0, 0, 0, 2, 3, 4])
        gmax = rng.randint(1, 2) if tree else rng.randint(1, 6)
        smax, dmax = _log_int(rng, 8, 80), rng.randint(1, 20)
        vocab = _log_int(rng, 1000, 152064)
        c = dict(BASE, step=step, q_heads=hq, kv_heads=hkv, head_dim=hd, vocab=vocab // 8 * 8 if step == "host" else vocab,
                 requests=_log_int(rng, 1, 32), prefix_min=int(pmax * rng.uniform(0.1, 1.0)), prefix_max=pmax,
                 steps_min=rng.randint(1, gmax), steps_max=gmax, seg_min=rng.randint(1, smax), seg_max=smax, drafts_min=rng.randint(1, dmax),
                 drafts_max=dmax, tree_width=tree, carry_in=rng.random() < 0.3, lengths=rng.randrange(1 << 20))
        if step == "cycle":
            c["layers"] = rng.randint(1, 4)
        if step in ("sample", "filter"):
            c["temperature"] = round(rng.uniform(0.4, 1.2), 2)
        if step == "filter":
            c["top_k"] = rng.choice([0, 20, rng.randint(1, 200)])
            c["top_p"] = round(rng.uniform(0.8, 0.99), 3) if c["top_k"] == 0 else rng.choice([0.95, 1.0, round(rng.uniform(0.8, 0.99), 3)])
        top, w = most[kind(c)], work(c)
        if w["bytes"] <= top["bytes"] and w["flops"] <= top["flops"]:
            return c


# ---- the batch of a case --------------------------------------------------------------------------------------------
def _requests(case):
    """Per request: prefix length, step lengths, parents of the steps (tree), token drafts."""
    rng = np.random.default_rng(case["lengths"])
    between = lambda a: int(rng.integers(case[a + "_min"], case[a + "_max"] + 1))  # noqa: E731
    out = []
    for _ in range(case["requests"]):
        prefix, depth, n_draft = between("prefix"), between("steps"), between("drafts")
        parents = None
        n_seg = depth
        if case["tree_width"]:  # a full tree of draft steps, numbered level by level; a branch on every node
            parents, level = [], [0]
            for _ in range(depth):
                nxt = []
                for node in level:
                    for _ in range(case["tree_width"]):
                        parents.append(node)
                        nxt.append(len(parents))
                level = nxt
            n_seg = len(parents)
        q = n_draft + (1 if case["carry_in"] else 0)
        req = {"P": prefix, "segs": [between("seg") for _ in range(n_seg)],
               "branches": [(n, q, q, n_draft) for n in range(0 if parents is not None else 1, n_seg + 1)]}
        if parents is not None:
            req["parents"] = parents
        out.append(req)
    return out


def _sizes(case):
    """(KV tokens, query rows, (row, visible key) pairs, logits rows, branches)"""
    kv = rows = vis = lrows = branches = 0
    for r in _requests(case):
        segs = r["segs"]
        kv += r["P"] + sum(segs)
        for node, own, q, n_draft in r["branches"]:
            seen = r["P"]
            if "parents" in r:
                while node:
                    seen += segs[node - 1]
                    node = r["parents"][node - 1]
            else:
                seen += sum(segs[:node])
            kv += own
            rows += q
            vis += sum(seen + own - q + i + 1 for i in range(q))
            lrows += n_draft + 1
            branches += 1
    return kv, rows, vis, lrows, branches


def work(case):
    kv, rows, vis, lrows, branches = _sizes(case)
    hq, hkv, d = case["q_heads"], case["kv_heads"], case["head_dim"]
    accept = 2.0 * lrows * case["vocab"]
    attn_bytes = 4.0 * kv * hkv * d + 4.0 * rows * hq * d
    attn_flops = 4.0 * hq * d * vis
    lists = 12.0 * kv / 16  # page ids in, page lists out
    if case["step"] in ("sample", "filter"):
        return {"bytes": accept + lists, "flops": 4.0 * lrows * case["vocab"]}
    if case["step"] == "cycle":  # the drafted tokens written to the cache; compaction moves about as many
        new = sum(sum(r["segs"]) + sum(b[1] for b in r["branches"]) for r in _requests(case))
        return {"bytes": case["layers"] * (attn_bytes + 8.0 * new * hkv * d) + accept + lists, "flops": case["layers"] * attn_flops}
    return {"bytes": attn_bytes + accept + lists, "flops": attn_flops}


def tolerance(case):
    if case["step"] == "sample":
        # fp32 sums: P(draft) is within 3e-7 of its 64-bit value (1e-6 at most); a final draw whose uniform lies within
        # rounding of a step of the cumulative sum may go to the neighbouring token
        return {"rel": 2e-6, "max": 2e-5, "differ": 0.01}
    if case["step"] == "filter":
        # the masses are integers, so the kept sets and the draws are the same however they are summed; P(draft) is one
        # fp32 division of two of them
        return {"rel": 2e-6, "max": 2e-5, "differ": 0.0}
    # bf16 output (2^-9 per value) of products whose weights are bf16 too: within 2.4e-3 of the 64-bit result (0.016 at
    # most) over these ranges; the log-sum-exp is fp32
    return {"rel": 1e-2, "max": 0.06, "differ": 0.0}


# ---- inputs ---------------------------------------------------------------------------------------------------------
def _logits(gen, rng, cu_draft, n_branch, vocab):
    """Rows as a language model gives them: a broad background, one leading token and a few alternatives below it; in
    about a quarter of the rows the lead is too small to hold most of the mass.  The drafts follow the leading tokens
    for a geometric number of rows, then go elsewhere.  Row stride: the vocabulary rounded up to 8 values."""
    n_rows, stride = int(cu_draft[-1]) + n_branch, (vocab + 7) // 8 * 8
    logits = torch.empty((n_rows, stride), dtype=torch.bfloat16, device=DEV)
    logits.normal_(0.0, 1.5, generator=gen)
    lead = 8.0 + 12.0 * torch.rand((n_rows, 1), device=DEV, generator=gen)
    gap = torch.empty((n_rows, 20), device=DEV).exponential_(0.4, generator=gen)
    lead_id = torch.randint(0, vocab, (n_rows, 1), device=DEV, generator=gen)
    alt_id = (lead_id + torch.arange(1, 21, device=DEV) * (vocab // 21)) % vocab  # all different
    logits.scatter_(1, alt_id, (lead - gap).to(torch.bfloat16))
    logits.scatter_(1, lead_id, lead.to(torch.bfloat16))
    ids, alts = lead_id.cpu().numpy()[:, 0], alt_id.cpu().numpy()[:, 0]
    drafts = np.zeros(max(1, int(cu_draft[-1])), dtype=np.int32)
    for b in range(n_branch):
        d0, n = int(cu_draft[b]), int(cu_draft[b + 1] - cu_draft[b])
        match = int(rng.geometric(0.25)) - 1
        for i in range(n):
            other = alts[d0 + b + i] if rng.random() < 0.5 else int(rng.integers(0, vocab))
            drafts[d0 + i] = ids[d0 + b + i] if i < match or (i > match and rng.random() < 0.5) else other
    return logits[:, :vocab], torch.from_numpy(drafts[: max(1, int(cu_draft[-1]))]).to(DEV)


def _randn(gen, *shape):
    return torch.empty(shape, dtype=torch.bfloat16, device=DEV).normal_(generator=gen)


class _State:
    pass


def prepare(case, seed):
    rng = np.random.default_rng([seed & 0x7FFFFFFF, case["lengths"]])
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    model = Model(case["q_heads"], case["kv_heads"], case["head_dim"], case["vocab"])
    s = _State()
    s.step, s.case = case["step"], case
    s.batch = b = build_batch(model, _requests(case), rng)
    s.ctx = B.Context(model, 0)
    s.plan = None if s.step == "cycle" else B.Plan(s.ctx, b)
    s.x = x = R.DeviceInputs.__new__(R.DeviceInputs)
    x.cu_draft = torch.from_numpy(np.ascontiguousarray(b.cu_draft, dtype=np.int32)).to(DEV)
    x.logits, x.draft_ids = _logits(gen, rng, b.cu_draft, b.n_branch, model.vocab)
    n_verdict = int(b.cu_verdict[-1])
    x.verdict = torch.from_numpy((rng.random(max(1, n_verdict)) < 0.6).astype(np.uint8)).to(DEV)
    s.y = R.PassOutputs(b)
    if s.step in ("sample", "filter"):
        s.u_accept = torch.rand(x.draft_ids.numel(), device=DEV, generator=gen)
        s.u_final = torch.rand(b.n_branch, device=DEV, generator=gen)
        s.p_draft = torch.zeros(x.draft_ids.numel(), device=DEV)
        s.n_kept = torch.zeros(b.n_logit_rows, dtype=torch.int32, device=DEV)
        s.scratch = (s.ctx.accept_sample_scratch if s.step == "sample" else s.ctx.accept_sample_filtered_scratch)(b.n_logit_rows)
        return s
    pool = (b.n_pool_pages, model.n_kv_heads, model.page_size, model.head_dim)
    q = (b.n_q_rows, model.n_q_heads, model.head_dim)
    if s.step == "cycle":
        # the pages of the draft steps and the branch tails: their content is new in every cycle
        new = np.concatenate([b.page_ids[int(f): int(f) + (int(n) + 15) // 16]
                              for first, length, keep in ((b.span_slot, b.span_len, ~np.isin(np.arange(b.n_span), b.req_span_off[:-1])),
                                                          (b.br_own_slot, b.br_own_len, np.ones(b.n_branch, bool)))
                              for f, n in zip(first[keep], length[keep])])
        s.new_pages = torch.from_numpy(new.astype(np.int64)).to(DEV)
        s.layers = []
        for _ in range(case["layers"]):
            y = torch.empty(q, dtype=torch.bfloat16, device=DEV)
            s.layers.append((_randn(gen, *q), _randn(gen, *pool), _randn(gen, *pool), _randn(gen, len(new), *pool[1:]), _randn(gen, len(new), *pool[1:]), y))
        s.new_len, s.n_kept = (torch.empty(b.n_req, dtype=torch.int32, device=DEV) for _ in range(2))
        return s
    x.q, x.k_pool, x.v_pool = _randn(gen, *q), _randn(gen, *pool), _randn(gen, *pool)
    if s.step == "overlap":
        s.side = torch.cuda.Stream()
    if s.step == "host":
        pin = lambda t: t.cpu().pin_memory()  # noqa: E731
        h = {"q_h": pin(x.q), "logits_h": pin(x.logits), "draft_ids_h": pin(x.draft_ids), "verdict_h": pin(x.verdict),
             "out_h": torch.empty(q, dtype=torch.bfloat16).pin_memory()}
        for name, n in (("n_accept_h", b.n_branch), ("bonus_id_h", b.n_branch), ("n_steps_accepted_h", b.n_req), ("survivor_h", b.n_req),
                        ("committed_len_h", b.n_req), ("keep_off_h", b.n_req + 1), ("free_off_h", b.n_req + 1), ("keep_pages_h", b.n_page_slots),
                        ("keep_valid_h", b.n_page_slots), ("free_pages_h", b.n_page_slots)):
            h[name] = torch.zeros(n, dtype=torch.int32).pin_memory()
        s.host, s.io, s.staging = h, B.lr_pass_host_io(**{k: v.data_ptr() for k, v in h.items()}), s.plan.pass_staging()
        x.q = x.logits = None
    return s


# ---- one pass -------------------------------------------------------------------------------------------------------
def _commit(s, plan, n_accept):
    y = s.y
    plan.lr_commit(s.x.verdict, n_accept, y.n_steps_accepted, y.survivor, y.committed_len, y.keep_off, y.keep_pages, y.keep_valid, y.free_off, y.free_pages)
    return [y.n_steps_accepted, y.survivor, y.committed_len, y.keep_off, y.keep_pages, y.keep_valid, y.free_off, y.free_pages]


def run(s):
    x, y, c = s.x, s.y, s.case
    if s.step == "pass":
        R.run_pass(s.ctx, s.plan, x, y)
        return [y.out, y.lse, y.n_accept, y.bonus_id, y.row_argmax, y.n_steps_accepted, y.survivor, y.committed_len, y.keep_off, y.keep_pages,
                y.keep_valid, y.free_off, y.free_pages]
    if s.step == "overlap":
        R.run_pass_overlapped(s.ctx, s.plan, x, y, s.side)
        return [y.out, y.n_accept, y.bonus_id, y.n_steps_accepted, y.survivor, y.committed_len, y.keep_off, y.keep_pages, y.keep_valid, y.free_off,
                y.free_pages]
    if s.step == "sample":
        s.ctx.lr_accept_sample(x.logits, x.draft_ids, x.cu_draft, c["temperature"], s.u_accept, s.u_final, y.n_accept, y.bonus_id, s.scratch, s.p_draft)
        return [y.n_accept, y.bonus_id, s.p_draft] + _commit(s, s.plan, y.n_accept)
    if s.step == "filter":
        s.ctx.lr_accept_sample_filtered(x.logits, x.draft_ids, x.cu_draft, c["temperature"], c["top_k"], c["top_p"], s.u_accept, s.u_final, y.n_accept,
                                        y.bonus_id, s.scratch, s.p_draft, s.n_kept)
        return [y.n_accept, y.bonus_id, s.p_draft, s.n_kept] + _commit(s, s.plan, y.n_accept)
    if s.step == "cycle":
        for _, k, v, k_new, v_new, _ in s.layers:
            k.index_copy_(0, s.new_pages, k_new)
            v.index_copy_(0, s.new_pages, v_new)
        plan = B.Plan(s.ctx, s.batch)
        for q, k, v, _, _, out in s.layers:
            plan.lr_verify_attention(q, k, v, out)
        s.ctx.lr_accept_greedy(x.logits, x.draft_ids, x.cu_draft, y.n_accept, y.bonus_id, y.scratch)
        lists = _commit(s, plan, y.n_accept)
        scratch = plan.compact_scratch()
        for _, k, v, _, _, _ in s.layers:
            plan.lr_compact(y.keep_off, y.keep_pages, y.keep_valid, k, v, s.new_len, s.n_kept, scratch)
        plan.lr_poll_status()
        plan.close()
        return [y.n_accept, y.bonus_id, s.new_len, s.n_kept] + lists + [t for layer in s.layers for t in (layer[5], layer[1], layer[2])]
    s.plan.lr_verify_pass_host(s.io, x.k_pool, x.v_pool, s.staging)
    return [v for k, v in s.host.items() if k not in ("q_h", "logits_h", "draft_ids_h", "verdict_h")]
