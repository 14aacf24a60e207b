// What is left of a small pass beside and behind its attention kernel, in one launch: the acceptance, the commit and the merge of
// the partial results.
//
// A small pass is a chain of latencies: as four kernels on two streams it was attention (13 us for one request of 4 K tokens),
// acceptance behind it because an attention CTA leaves no registers for another on its SM (8), and commit (2), with events at
// both ends.  Here the launch is a programmatic dependent of the attention kernel, and only the CTAs that merge wait for it.  The
// others run on SMs that attention leaves free, or behind it where it leaves too few (plan_small_pass): first the CTAs of the
// commit, which go through their plan tables and then wait for the row keys, then those that stream the logits.
// As four kernels and as two, with the same attention, one after another on the same buffers: 256 tokens 13.6 -> 12.1 us; 4 K tokens with
// head size 64, beside a narrower attention, 22.4 -> 16.9; with head size 128, behind it, 22.5 -> 19.9; 8 K so 27.3 -> 25.4.  Some of that is
// the set-up of the next pass's attention while this one ends: passes that are waited for one by one take 20.0 and 20.5, 32.1 and
// 26.1, 33.2 and 29.5, 38.4 and 34.8.
//
// What streams is warps: an SM's rate grows with them and hardly with the loads a lane has in flight (one SM alone: 8 warps 30
// GB/s, 16 54, 32 80 to 90, with four, eight or sixteen 16-byte loads a lane).  A warp takes consecutive units and publishes once
// a row: handing units out by a counter, or an atomic for each of them, cost more than the reading (one address takes about one
// atomic a nanosecond).
//
// Every wait ends: the CTAs of the commit are the first of the grid and wait for those that stream, which wait for nothing and need only
// places; those that merge are the last and wait for an attention whose CTAs all run by then.  At most two CTAs of a pass hold places
// while they wait for others to get some, and at most 128 grids run on a GPU at a time: 256 of the 444 places and more that it has, so
// passes on other streams cannot take the last ones either.  (Attention CTAs that wait for the kernel before them are launched when all of
// that kernel's streaming CTAs have ended.)  And the wait gives up after a limit.
#include <algorithm>

#include "accept_stream.cuh"
#include "attn_merge.cuh"
#include "commit.cuh"

namespace lr {

namespace {

constexpr int kThreads = 256;
static_assert(kCommitThreads == kThreads, "one block size for all");
constexpr int kVecPerThread = 6;     // eight spill
// CTAs an SM: 64 registers a thread, or 72 where the merge has eight slots in flight.
constexpr int kFewSlots = 4;         // partial slots an M-tile up to which the merge takes the narrower form, as when it is alone
constexpr int tail_ctas(int batch) { return batch <= kFewSlots ? 4 : 3; }
// CTAs of the commit: they wait for others of the grid, so they are few.
constexpr int kCommitCtas = tail_ctas(8) - 1;
constexpr int kCommitSlots = 2048;   // page slots that so few write: four a thread
constexpr int kMostRequests = 512;   // every CTA has shared memory for the decisions of so many, 18 KB
constexpr int kUnitBits = 20;        // of the word that counts finished units; the bits above count CTAs that are through
constexpr uint64_t kPatience = 20;   // of the plan's limit: what is waited for may have to be scheduled first, beside other work on the GPU
constexpr uint32_t kMostUnits = (1u << kUnitBits) - 1u;
// CTAs an SM that stream where attention leaves no SMs for them; the merge's come behind them.  Two, three, four, five an SM: one request of
// 4 K tokens 20.4, 19.8, 19.9, 21.4 us, four of 500 18.1, 18.0, 17.6, 17.6, of 100 19.4, 17.1, 17.1, 16.5.
constexpr int kStreamCtas = 4;

struct PassAccept {
  AcceptWork w;
  const int32_t *draft_ids, *cu_draft;
  int32_t *n_accept, *bonus, *row_argmax;
  int32_t n_branch, n_rows;
  int32_t n_commit, n_stream;  // CTAs
  uint32_t share;              // units a warp streams
  uint64_t wait_limit_ns;
};

__device__ __forceinline__ uint32_t *done_word(const AcceptWork &w) { return reinterpret_cast<uint32_t *>(w.scratch); }

// One thread of a CTA that is through with the scratch, and has finished `units` units: whether it is the last one ...
__device__ __forceinline__ bool leave(const PassAccept &a, uint32_t units) {
  __threadfence();
  const uint32_t add = units + (1u << kUnitBits);
  return (atomicAdd(done_word(a.w), add) + add) >> kUnitBits == (uint32_t)(a.n_commit + a.n_stream);
}
// ... which leaves it zeroed.
__device__ __forceinline__ void clear(const PassAccept &a, bool last) {
  if (__syncthreads_or(last))
    for (int r = threadIdx.x; r <= a.n_rows; r += kThreads) a.w.scratch[r] = 0ull;
}

__device__ __forceinline__ void stream_cta(const PassAccept &a) {
  const int cta = blockIdx.x - a.n_commit;
  const uint32_t first = (uint32_t)(cta * (kThreads / 32) + (threadIdx.x >> 5)) * a.share;
  accept_run<kVecPerThread>(a.w, first, min(first + a.share, a.w.total), threadIdx.x & 31);
  const uint32_t from = (uint32_t)(cta * (kThreads / 32)) * a.share;
  __syncthreads();
  clear(a, threadIdx.x == 0 && leave(a, min(a.w.total - from, a.share * (kThreads / 32))));
}

// Acceptance counts from the row keys.  Every CTA of the commit works out those of its requests' decisive branches; all branches
// and rows are written by one of them or another.
struct CountsFromKeys {
  const PassAccept &a;
  int32_t *status;
  int32_t surv, surv_d0, surv_len;  // the branch that decides the thread's first request, its draft range
  bool last;

  __device__ __forceinline__ void range(int b, int32_t &d0, int32_t &len) const {
    d0 = a.cu_draft[b];
    len = a.cu_draft[b + 1] - d0;
  }
  __device__ __forceinline__ void before(int decisive) {
    surv = decisive;
    if (surv >= 0) range(surv, surv_d0, surv_len);
  }
  __device__ __forceinline__ bool ready() {  // every unit is finished; gives up after the plan's limit
    bool ok = true;
    if (threadIdx.x == 0) {
      uint64_t t0 = 0;
      for (uint32_t i = 0;; ++i) {
        uint32_t state;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(state) : "l"(done_word(a.w)) : "memory");
        if ((state & kMostUnits) == a.w.total) break;
        if ((i & 255u) == 0u) {
          uint64_t t;
          asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
          if (i == 0u) t0 = t;
          else if (t - t0 > a.wait_limit_ns) {
            ok = false;
            break;
          }
        }
      }
      if (!ok) {
        status[0] = kDevTimeout;
        status[1] = 400;
      }
      __threadfence();
    }
    return __syncthreads_and(ok) != 0;
  }
  __device__ __forceinline__ int count(int b) const {
    int32_t d0 = surv_d0, len = surv_len, token;
    if (b != surv) range(b, d0, len);
    return accept_branch(a.w.scratch + 1 + (d0 + b), a.draft_ids, d0, len, token);
  }
  // Beside the decisions, for which the first warp is enough when there are few requests: counted from the last thread.
  __device__ __forceinline__ void beside(int cta, int n_cta) {
    const int first = cta * kThreads + kThreads - 1 - (int)threadIdx.x, step = n_cta * kThreads;
    for (int b = first; b < a.n_branch; b += step) {
      int32_t d0, len, token;
      range(b, d0, len);
      a.n_accept[b] = accept_branch(a.w.scratch + 1 + (d0 + b), a.draft_ids, d0, len, token);
      a.bonus[b] = token;
    }
    if (a.row_argmax != nullptr)
      for (int r = first; r < a.n_rows; r += step) a.row_argmax[r] = (int32_t)(0xFFFFFFFFu - (uint32_t)ld_behind_wait(a.w.scratch + 1 + r));
  }
  // No thread of the CTA reads keys any more; the last warp has no page slots to write where lists are short.
  __device__ __forceinline__ void through() { last = threadIdx.x == kThreads - 1 && leave(a, 0u); }
  __device__ __forceinline__ void end() { clear(a, last); }
};

template <int kD, int kBatch, bool kTree>
__global__ void __launch_bounds__(kThreads, tail_ctas(kBatch))
pass_tail_kernel(DevBatch d, DevTcPlan tc, uint16_t *__restrict__ out, float *__restrict__ lse, PassAccept a, const uint8_t *verdict, CommitOut o) {
  const int cta = blockIdx.x, m = cta - a.n_commit - a.n_stream;
  if (m >= 0) {
    merge_cta<kD, kBatch>(d, tc, m % tc.n_targets, m / tc.n_targets, out, lse);
    return;
  }
  if (cta < a.n_commit) {
    commit_cta<kTree>(d, cta, a.n_commit, true, verdict, CountsFromKeys{a, d.status}, o);
    // what comes next may count on attention too
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  } else {
    stream_cta(a);
  }
}

template <int kD, int kBatch>
auto tail_kernel(bool tree) {
  return tree ? pass_tail_kernel<kD, kBatch, true> : pass_tail_kernel<kD, kBatch, false>;
}

// CTAs of the commit and those that stream; a warp's share is what the places beside attention, or behind it, stream in one go.
struct TailGrid {
  int n_commit, n_stream;
  uint32_t share;
};
TailGrid tail_grid(const lr_plan *p, uint32_t total) {
  const DevTcPlan &tc = p->tc_pass;
  TailGrid g;
  g.n_commit = std::min(commit_ctas(p->dev), kCommitCtas);
  const int n_sm = p->ctx->sm_count, most = p->small == kBehindAttention ? kStreamCtas * n_sm : tail_ctas(tc.most_slots) * (n_sm - tc.n_cta);
  const uint32_t warps = (uint32_t)std::max(1, most - g.n_commit) * (kThreads / 32);
  g.share = (total + warps - 1) / warps;
  g.n_stream = (int)((total + g.share * (kThreads / 32) - 1) / (g.share * (kThreads / 32)));
  return g;
}

}  // namespace

bool pass_tail_apart(const lr_ctx *ctx, const lr_plan *p, int32_t n_rows) {
  const TailGrid g = tail_grid(p, accept_work(ctx, nullptr, 0, n_rows, nullptr, kVecPerThread).total);
  return p->small == kBesideAttention && p->tc_pass.n_targets == 0 && g.n_commit + g.n_stream <= p->ctx->sm_count - p->tc_pass.n_cta;
}

bool pass_tail_fits(const lr_ctx *ctx, const lr_plan *p, int64_t n_rows) {
  const int vecs = ctx->model.vocab >> 3, unit = 32 * kVecPerThread;
  return p->small != kNotSmall && p->dev.n_req <= kMostRequests && p->dev.n_page_slots <= kCommitSlots &&
         n_rows * std::max(1, (vecs + unit - 1) / unit) <= (int64_t)kMostUnits;
}

int launch_pass_tail(lr_ctx *ctx, lr_plan *p, const lr_pass_io *io, bool behind_attention, cudaStream_t s) {
  const DevBatch &d = p->dev;
  PassAccept a = {accept_work(ctx, io->logits_d, io->logits_stride, (int32_t)io->n_rows, io->accept_scratch_d, kVecPerThread),
                  io->draft_ids_d, io->cu_draft_d, io->n_accept_d, io->bonus_id_d, io->row_argmax_d, d.n_branch, (int32_t)io->n_rows};
  const DevTcPlan &tc = p->tc_pass;
  const bool few = tc.most_slots <= kFewSlots;
  const TailGrid grid = tail_grid(p, a.w.total);
  a.n_commit = grid.n_commit;
  a.n_stream = grid.n_stream;
  a.share = grid.share;
  a.wait_limit_ns = 1000ull * kPatience * tc.wait_limit_us;
  const CommitOut o = {io->n_steps_accepted_d, io->survivor_d, io->committed_len_d, io->keep_off_d,
                       io->keep_pages_d, io->keep_valid_d, io->free_off_d, io->free_pages_d};
  const auto kernel = d.head_dim == 128 ? (few ? tail_kernel<128, 4>(d.tree) : tail_kernel<128, 8>(d.tree))
                                        : (few ? tail_kernel<64, 4>(d.tree) : tail_kernel<64, 8>(d.tree));
  const size_t smem = (size_t)d.n_req * (d.tree ? kCommitSmemPerReq<true> : kCommitSmemPerReq<false>);
  uint16_t *out = reinterpret_cast<uint16_t *>(io->out_d);
  ctx->launches++;
  if (!behind_attention) {  // an ordinary launch: most CTAs do not wait for what is just before
    kernel<<<a.n_commit + a.n_stream, kThreads, smem, s>>>(d, tc, out, io->lse_d, a, io->verdict_d, o);
    return cuda_fail(cudaGetLastError(), "pass_tail_kernel launch");
  }
  return cuda_fail(launch_dependent(kernel, dim3((unsigned)(a.n_commit + a.n_stream + tc.n_targets * (d.head_dim / 8))), dim3(kThreads), smem, s, d, tc,
                                    out, io->lse_d, a, io->verdict_d, o),
                   "pass_tail_kernel launch");
}

}  // namespace lr
