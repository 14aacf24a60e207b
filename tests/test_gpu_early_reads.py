"""Kernels that load some of their inputs while the kernel before them still runs.  The inputs of every call below hold other
valid values until a kernel that lets its successor start at once writes the real ones some 50 us later; inputs and outputs
lie side by side, so that one cache line holds what is read early and what is written late."""
import numpy as np
import pytest
import torch

from gpu_util import check_commit
from lr_workloads import Model, bf16_round, build_batch
from lr_workloads.gen import _finish
from oracle import lr_oracle as O
from paper_2506_19830_b200 import binding as B
from paper_2506_19830_b200 import runner as R

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
ROUNDS = 8

WRITE_LATE = r"""
extern "C" __global__ void write_late(unsigned char *dst, const unsigned char *src, int n, int cycles) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const long long t0 = clock64();
  while (clock64() - t0 < cycles) {}
  for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}
"""


@pytest.fixture(scope="module")
def write_late():
    kernel = torch.cuda._compile_kernel(WRITE_LATE, "write_late")
    return lambda dst, src: kernel(grid=(1, 1, 1), block=(256, 1, 1), args=[dst, src, src.numel(), 100_000])


class Packed:
    """Arrays side by side in one device buffer, in several versions; the buffer ends with ``extra`` bytes of scratch."""

    def __init__(self, versions, extra=0):
        self.at, n = {}, 0
        for name, a in versions[0].items():
            n = -(-n // a.itemsize) * a.itemsize
            self.at[name] = (n, a.nbytes, a.dtype)
            n += a.nbytes
        self.n = -(-n // 8) * 8
        self.buf = torch.zeros(self.n + extra, dtype=torch.uint8, device=DEV)
        self.versions = []
        for v in versions:
            host = np.zeros(self.n, dtype=np.uint8)
            for name, (off, size, _) in self.at.items():
                host[off:off + size] = np.ascontiguousarray(v[name]).view(np.uint8)
            self.versions.append(torch.from_numpy(host).to(DEV))

    def __getitem__(self, name):
        off, size, dtype = self.at[name]
        return self.buf[off:off + size].view(torch.from_numpy(np.zeros(1, dtype)).dtype)

    def scratch(self):
        return self.buf[self.n:].view(torch.int64)


def _requests(n_req, tree, rng):
    reqs = []
    for _ in range(n_req):
        n = int(rng.integers(0, 9 if tree else 12))
        depths = sorted(int(x) for x in rng.integers(0, n + 1, size=int(rng.integers(1, 8))))
        req = {"P": int(rng.integers(0, 60)), "segs": [int(x) for x in rng.integers(1, 20, size=n)], "branches": [(g, 5, 3, 4) for g in depths]}
        if tree:
            req["parents"] = [int(rng.integers(0, c + 1)) for c in range(n)]
        reqs.append(req)
    return reqs


@pytest.mark.parametrize("tree", [False, True])
@pytest.mark.parametrize("n_req", [3, 300])
def test_commit_alone(write_late, n_req, tree):
    rng = np.random.default_rng(n_req)
    b = build_batch(Model(2, 1, 64, 16), _requests(n_req, tree, rng), rng)
    versions = [{"verdict": (rng.random(max(1, int(b.cu_verdict[-1]))) < 0.6).astype(np.uint8),
                 "n_accept": rng.integers(0, b.br_n_draft + 1).astype(np.int32)} for _ in range(3)]
    ctx = B.Context(b.model, 0)
    plan, mem = B.Plan(ctx, b), Packed(versions)
    ys = [R.PassOutputs(b, n_rows=1) for _ in range(ROUNDS)]
    torch.cuda.synchronize()
    for i, y in enumerate(ys):
        write_late(mem.buf, mem.versions[i % 3])
        plan.lr_commit(mem["verdict"], mem["n_accept"], y.n_steps_accepted, y.survivor, y.committed_len, y.keep_off, y.keep_pages, y.keep_valid,
                       y.free_off, y.free_pages)
    assert plan.lr_poll_status() == 0
    for i, y in enumerate(ys):
        v = versions[i % 3]
        check_commit(y.commit_dict(), O.commit(b, v["verdict"], v["n_accept"]))
    ctx.close()


@pytest.mark.parametrize("tree", [False, True])
@pytest.mark.parametrize("n_req", [3, 300])
def test_pass(write_late, n_req, tree):
    rng = np.random.Generator(np.random.PCG64(n_req))
    w = _finish("early", 5, Model(2, 1, 64, 64), _requests(n_req, tree, rng), rng, 0.4, 0.8, True, True, "nan")
    b, t = w.batch, w.tensors
    versions = []
    for _ in range(3):
        drafts = np.where(rng.random(len(t.draft_ids)) < 0.2, rng.integers(0, 64, len(t.draft_ids)), t.draft_ids)
        versions.append({"n_accept": np.zeros(b.n_branch, np.int32), "verdict": (rng.random(max(1, len(t.verdict))) < 0.6).astype(np.uint8),
                         "cu_draft": b.cu_draft.astype(np.int32), "drafts": drafts.astype(np.int32)})
    ctx = B.Context(b.model, 0)
    plan, mem, x = B.Plan(ctx, b), Packed(versions), R.DeviceInputs(b, t)
    x.verdict, x.draft_ids, x.cu_draft = mem["verdict"], mem["drafts"], mem["cu_draft"]
    ys = [R.PassOutputs(b) for _ in range(ROUNDS)]
    late = [torch.empty_like(y.n_accept) for y in ys]
    torch.cuda.synchronize()
    for i, y in enumerate(ys):
        y.n_accept = mem["n_accept"]
        write_late(mem.buf, mem.versions[i % 3])
        R.run_pass(ctx, plan, x, y)
        late[i].copy_(y.n_accept)
    assert plan.lr_poll_status() == 0
    for i, y in enumerate(ys):
        v = versions[i % 3]
        n, bonus, _ = O.accept_greedy(t.logits, v["drafts"], b.cu_draft)
        assert np.array_equal(late[i].cpu().numpy(), n) and np.array_equal(y.bonus_id.cpu().numpy(), bonus)
        check_commit(y.commit_dict(), O.commit(b, v["verdict"], n))
    ctx.close()


@pytest.mark.parametrize("vocab,top_k,top_p", [(20000, None, 1.0), (20000, 20, 1.0), (20000, 300, 0.9), (20000, 0, 0.9), (20000, 5000, 0.7), (4000, 0, 0.9),
                                               (152064, 0, 0.95)])
def test_sampled_acceptance(write_late, vocab, top_k, top_p):
    """Unfiltered (top_k None), through the candidates, through the windows alone, with one and with eight CTAs a branch."""
    rng = np.random.default_rng(vocab + (top_k or 0))
    n_branch, n_draft = 5, 62
    n_rows = n_branch + n_draft
    model = Model(1, 1, 64, vocab)
    ctx = B.Context(model, 0)
    bits = bf16_round((rng.standard_normal((n_rows, vocab)) * 3).astype(np.float32))
    lg, top = R.bf16_tensor(bits, DEV), O.row_argmax(bits)
    versions = []
    for _ in range(3):
        cu = np.concatenate([[0], np.sort(rng.integers(0, n_draft + 1, n_branch - 1)), [n_draft]]).astype(np.int32)
        likely = np.concatenate([top[cu[i] + i:cu[i + 1] + i] for i in range(n_branch)])
        drafts = np.where(rng.random(n_draft) < 0.8, likely, rng.integers(0, vocab, n_draft)).astype(np.int32)
        versions.append({"n_accept": np.zeros(n_branch, np.int32), "final": np.zeros(n_branch, np.int32), "p_draft": np.zeros(n_draft, np.float32),
                         "cu": cu, "drafts": drafts, "u_accept": (rng.random(n_draft) * 0.5).astype(np.float32),
                         "u_final": rng.random(n_branch).astype(np.float32)})

    def call(a, scratch):
        if top_k is None:
            ctx.lr_accept_sample(lg, a["drafts"], a["cu"], 0.8, a["u_accept"], a["u_final"], a["n_accept"], a["final"], scratch, a["p_draft"])
        else:
            ctx.lr_accept_sample_filtered(lg, a["drafts"], a["cu"], 0.8, top_k, top_p, a["u_accept"], a["u_final"], a["n_accept"], a["final"], scratch,
                                          a["p_draft"])

    fresh = (lambda: ctx.accept_sample_scratch(n_rows)) if top_k is None else (lambda: ctx.accept_sample_filtered_scratch(n_rows))
    want = []
    for v in versions:  # the same call on inputs that have been there for long
        a = {k: torch.from_numpy(x.copy()).to(DEV) for k, x in v.items()}
        torch.cuda.synchronize()
        call(a, fresh())
        torch.cuda.synchronize()
        want.append([a[k].cpu() for k in ("n_accept", "final", "p_draft")])
    mem = Packed(versions, extra=fresh().numel() * 8)
    mem.buf[:mem.n].copy_(mem.versions[2])
    got = []
    torch.cuda.synchronize()
    for i in range(ROUNDS):
        write_late(mem.buf, mem.versions[i % 3])
        call(mem, mem.scratch())
        got.append([mem[k].clone() for k in ("n_accept", "final", "p_draft")])
    torch.cuda.synchronize()
    for i, g in enumerate(got):
        assert all(torch.equal(x.cpu(), y) for x, y in zip(g, want[i % 3])), i
    ctx.close()
