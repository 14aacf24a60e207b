// The work of a CTA of the step-level commit, for the kernels that do it (commit.cu, pass_tail.cu).
#pragma once

#include "lr_common.cuh"

namespace lr {

constexpr int kCommitThreads = 256;
// bytes of shared memory per request; a tree's walk takes a byte a move
template <bool kTree>
constexpr int kCommitSmemPerReq = 7 * 4 + (kTree ? kMaxTreeDepth : 0);

__device__ __forceinline__ int pages_of(int n_tok) { return (n_tok + kPage - 1) / kPage; }

// exclusive scan of a[0..n) in shared memory, in place, by one CTA; the total goes to *carry_slot
static __device__ void block_exclusive_scan(int32_t *a, int n, int32_t *carry_slot) {
  __shared__ int32_t warp_sum[kCommitThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (tid == 0) *carry_slot = 0;
  __syncthreads();
  for (int base = 0; base < n; base += kCommitThreads) {
    int i = base + tid;
    int32_t x = (i < n) ? a[i] : 0;
    int32_t inc = x;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      int32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, off);
      if (lane >= off) inc += y;
    }
    if (lane == 31) warp_sum[wid] = inc;
    __syncthreads();
    int32_t wbase = 0;
    for (int w = 0; w < wid; ++w) wbase += warp_sum[w];
    int32_t carry = *carry_slot;
    if (i < n) a[i] = carry + wbase + inc - x;
    __syncthreads();
    if (tid == kCommitThreads - 1) *carry_slot = carry + wbase + inc;
    __syncthreads();
  }
}

// What follows from the plan and the verdicts for a request, whatever the acceptance counts are.
struct Step {
  int a, surv, drafts, own;        // j*, decisive branch (or -1), its drafts and tail tokens
  int kchain, all, tokens;         // pages of the kept chain spans, of the whole request, tokens of the former
};
__device__ __forceinline__ Step decide(const DevBatch &d, const uint8_t *verdict, int r) {
  const int s0 = d.req_span_off[r], s1 = d.req_span_off[r + 1];
  const int b0 = d.req_br_off[r], b1 = d.req_br_off[r + 1];
  const int gamma = s1 - s0 - 1, base = s0 + r;
  const uint8_t *v = verdict + (s0 - r);
  Step st;
  st.a = gamma;  // first rejected step, gamma if none
  for (int c0 = 0; c0 < gamma && st.a == gamma; c0 += 8) {
    uint8_t w[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) w[k] = (c0 + k < gamma) ? v[c0 + k] : (uint8_t)1;
#pragma unroll
    for (int k = 7; k >= 0; --k)
      if (w[k] == 0) st.a = c0 + k;
  }
  st.surv = -1;  // lowest-numbered branch of depth j*
  for (int i0 = b0; i0 < b1 && st.surv < 0; i0 += 8) {
    int dep[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) dep[k] = (i0 + k < b1) ? d.br_depth[i0 + k] : -1;
#pragma unroll
    for (int k = 7; k >= 0; --k)
      if (dep[k] == st.a) st.surv = i0 + k;
  }
  st.drafts = st.surv >= 0 ? d.br_n_draft[st.surv] : 0;
  st.own = st.surv >= 0 ? d.br_own_len[st.surv] : 0;
  st.kchain = d.chain_pg[base + st.a + 1];
  st.all = d.chain_pg[base + gamma + 1] + d.tail_pg[b0 + r + (b1 - b0)];
  st.tokens = d.chain_tok[base + st.a + 1];
  return st;
}

// The same for a tree of steps (Section 3, "Multi-Branch Drafting"): the kept steps are those of a walk from the prefix that
// moves, at every node, to the lowest-numbered child whose verdict is set.  The walked nodes (at most kMaxTreeDepth, local
// indices below 256) go to `walk`.
__device__ __forceinline__ Step decide_tree(const DevBatch &d, const uint8_t *verdict, int r, uint8_t *walk) {
  const int s0 = d.req_span_off[r], s1 = d.req_span_off[r + 1];
  const int b0 = d.req_br_off[r], b1 = d.req_br_off[r + 1];
  const int n_seg = s1 - s0 - 1, base = s0 + r;
  const uint8_t *v = verdict + (s0 - r);  // v[c - 1]: verdict of segment c
  Step st;
  int node = 0;
  st.a = 0;
  st.kchain = d.chain_pg[base + 1];
  st.tokens = d.chain_tok[base + 1];
  while (st.a < kMaxTreeDepth) {
    int next = -1;
    for (int k = d.child_off[s0 + node], k1 = d.child_off[s0 + node + 1]; k < k1 && next < 0; ++k) {
      const int c = d.child_list[k];
      if (v[c - 1] != 0) next = c;
    }
    if (next < 0) break;
    walk[st.a++] = (uint8_t)next;
    node = next;
    st.kchain += d.chain_pg[base + node + 1] - d.chain_pg[base + node];
    st.tokens += d.chain_tok[base + node + 1] - d.chain_tok[base + node];
  }
  st.surv = -1;  // lowest-numbered branch that continues the node where the walk stopped
  for (int i0 = b0; i0 < b1 && st.surv < 0; i0 += 8) {
    int dep[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) dep[k] = (i0 + k < b1) ? d.br_depth[i0 + k] : -1;
#pragma unroll
    for (int k = 7; k >= 0; --k)
      if (dep[k] == node) st.surv = i0 + k;
  }
  st.drafts = st.surv >= 0 ? d.br_n_draft[st.surv] : 0;
  st.own = st.surv >= 0 ? d.br_own_len[st.surv] : 0;
  st.all = d.chain_pg[base + n_seg + 1] + d.tail_pg[b0 + r + (b1 - b0)];
  return st;
}

// What the plan says of a page slot that belongs to a span: its page, its request, the span's number in the request (for a
// tail: ~branch), its place among the pages of that kind, and the tokens of the span from it on (for a tail: its place in the
// tail).  It stays in registers across the wait, hence few words.
struct Slot {
  int pid, r, part, at, rest;
};
__device__ __forceinline__ Slot slot_of(const DevBatch &d, int i) {
  Slot t;
  t.r = -1;  // a slot no span refers to
  const int item = i < d.n_page_slots ? d.slot_item[i] : -1;
  if (item < 0) return t;
  t.pid = d.page_ids[i];
  if (item < d.n_span) {
    t.r = d.span_req[item];
    const int s0 = d.req_span_off[t.r], idx = i - d.span_slot[item];
    t.part = item - s0;
    t.at = d.chain_pg[s0 + t.r + t.part] + idx;
    t.rest = d.span_len[item] - idx * kPage;
  } else {
    const int b = item - d.n_span;
    t.part = ~b;
    t.r = d.br_req[b];
    const int s0 = d.req_span_off[t.r], s1 = d.req_span_off[t.r + 1], b0 = d.req_br_off[t.r];
    t.rest = i - d.br_own_slot[b];
    t.at = d.chain_pg[s0 + t.r + (s1 - s0)] + d.tail_pg[b0 + t.r + (b - b0)] + t.rest;
  }
  return t;
}

// The counts of the acceptance step, for lr_commit: written by the kernel launched just before.
struct CountsGiven {
  const int32_t *n_accept;
  __device__ __forceinline__ void before(int) {}
  __device__ __forceinline__ bool ready() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    return true;
  }
  __device__ __forceinline__ int count(int b) const { return ld_behind_wait(n_accept + b); }
  __device__ __forceinline__ void beside(int, int) {}
  __device__ __forceinline__ void through() {}
  __device__ __forceinline__ void end() {}
};

// One CTA of the commit.  The chain of loads is what it takes, so all of it that does not hang on the kernel just before is gone
// through while that one drains: what the plan says of a thread's first page slot always (its tables come by copies), and -- with
// `early`, whose terms stand at launch_commit -- the decision on a thread's first request too.  Then one trip for the counts, the
// scans and the stores are left.  Behind the sampled acceptance, plan tables only: 50.3 -> 49.3 and 51.2 -> 49.5 us (617 rows without and
// with filters), 36.0 -> 35.1 (51 rows, top-p).  As a kernel of its own behind the greedy one, the decision too: 27.9 -> 24.8 us for a pass over
// one request of 4 K tokens when such passes had it.
// The counts, and without `early` the verdicts, may be written while this kernel is resident: neither is __restrict__.
template <bool kTree, class Counts>
__device__ __forceinline__ void commit_cta(const DevBatch &d, int cta, int n_cta, bool early, const uint8_t *verdict, Counts counts, const CommitOut &o) {
  extern __shared__ int32_t sm[];
  const int R = d.n_req;
  int32_t *s_keep = sm;            // keep count -> keep offset
  int32_t *s_free = sm + R;        // free count -> free offset
  int32_t *s_a = sm + 2 * R;       // j* (tree: moves of the walk)
  int32_t *s_surv = sm + 3 * R;    // decisive branch or -1
  int32_t *s_kp = sm + 4 * R;      // kept tail pages of the decisive branch
  int32_t *s_kt = sm + 5 * R;      // kept tail tokens
  int32_t *s_kchain = sm + 6 * R;  // pages of the kept chain spans (prefix and the kept segments)
  uint8_t *s_walk = reinterpret_cast<uint8_t *>(sm + 7 * R);  // tree: [R][kMaxTreeDepth]
  __shared__ int32_t s_total[2];
  const int tid = threadIdx.x;
  const int slot0 = cta * kCommitThreads + tid;
  Slot first_slot = slot_of(d, slot0);
  auto decision = [&](int r) {
    if constexpr (kTree) return decide_tree(d, verdict, r, s_walk + r * kMaxTreeDepth);
    else return decide(d, verdict, r);
  };
  Step first = {};
  if (early && tid < R) first = decision(tid);
  counts.before(early && tid < R ? first.surv : -1);
  if (!counts.ready()) {
    counts.through();
    counts.end();
    return;
  }

  // ---- per-request decisions --------------------------------------------------
  for (int r = tid; r < R; r += kCommitThreads) {
    const Step st = early && r == tid ? first : decision(r);
    int kept_tail = 0;
    if (st.surv >= 0) {
      int na = counts.count(st.surv);
      if (na < 0 || na > st.drafts) {  // not a value the acceptance step can produce
        na = na < 0 ? 0 : st.drafts;
        d.status[0] = kDevBounds;
        d.status[1] = kTree ? 301 : 300;
      }
      kept_tail = st.own - st.drafts + na;
    }
    const int kp = pages_of(kept_tail);
    s_keep[r] = st.kchain + kp;
    s_free[r] = st.all - st.kchain - kp;
    s_a[r] = st.a;
    s_surv[r] = st.surv;
    s_kp[r] = kp;
    s_kt[r] = kept_tail;
    s_kchain[r] = st.kchain;
    if (cta == 0) {
      o.n_steps[r] = st.a;
      o.survivor[r] = st.surv;
      o.committed[r] = st.tokens + kept_tail;
    }
  }
  counts.beside(cta, n_cta);
  __syncthreads();
  block_exclusive_scan(s_keep, R, &s_total[0]);
  block_exclusive_scan(s_free, R, &s_total[1]);
  if (cta == 0) {
    for (int r = tid; r < R; r += kCommitThreads) {
      o.keep_off[r] = s_keep[r];
      o.free_off[r] = s_free[r];
    }
    if (tid == 0) {
      o.keep_off[R] = s_total[0];
      o.free_off[R] = s_total[1];
    }
  }

  counts.through();
  // ---- page lists: one thread per page slot --------------------------------------
  for (int i = slot0; i < d.n_page_slots; i += n_cta * kCommitThreads) {
    const Slot t = i == slot0 ? first_slot : slot_of(d, i);
    if (t.r < 0) continue;
    const int kchain = s_kchain[t.r];
    if (t.part >= 0) {
      // the span's place: kept or not, and for a tree how many pages of walked segments are numbered below it
      bool kept = t.part <= s_a[t.r];
      int at = t.at, freed = t.at - kchain;
      if constexpr (kTree) {
        const int c = t.part, base = d.req_span_off[t.r] + t.r, a = s_a[t.r];
        int walked_before = 0;
        kept = c == 0;
        for (int k = 0; k < a; ++k) {  // walked indices increase
          const int w = s_walk[t.r * kMaxTreeDepth + k];
          if (w < c) walked_before += d.chain_pg[base + w + 1] - d.chain_pg[base + w];
          kept |= w == c;
        }
        const int prefix = d.chain_pg[base + 1];
        at = c == 0 ? t.at : prefix + walked_before + (t.at - d.chain_pg[base + c]);
        freed = t.at - prefix - walked_before;
      }
      if (kept) {
        const int dst = s_keep[t.r] + at;
        o.keep_pages[dst] = t.pid;
        o.keep_valid[dst] = min(kPage, t.rest);
      } else {
        o.free_pages[s_free[t.r] + freed] = t.pid;
      }
    } else {
      const int b = ~t.part, surv = s_surv[t.r], kp = s_kp[t.r];
      if (b == surv && t.rest < kp) {
        const int dst = s_keep[t.r] + kchain + t.rest;
        o.keep_pages[dst] = t.pid;
        o.keep_valid[dst] = min(kPage, s_kt[t.r] - t.rest * kPage);
      } else {
        const int kept_before = (surv >= 0 && b >= surv) ? kp : 0;  // kept pages precede this one in tail order
        o.free_pages[s_free[t.r] + t.at - kchain - kept_before] = t.pid;
      }
    }
  }
  counts.end();
}

// CTAs of a commit: every one repeats the per-request phase, so few CTAs when there are many requests
inline int commit_ctas(const DevBatch &d) {
  const int cap = d.n_req <= 64 ? 148 : (d.n_req <= 512 ? 32 : 8), grid = (d.n_page_slots + kCommitThreads - 1) / kCommitThreads;
  return grid < 1 ? 1 : (grid > cap ? cap : grid);
}

}  // namespace lr
