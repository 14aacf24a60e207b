// Step-level commit on the paged KV cache (Algorithm 1, last two lines).
//
// Integer work on a few KB of tables: latency-bound, so it is one launch with no
// inter-CTA communication and as few dependent loads as possible.  Every CTA
// recomputes the per-request decisions (j*, decisive branch, kept tail, list
// sizes) -- one thread per request, with the verdict and depth scans unrolled in
// groups of 8 so that their loads are in flight together -- and the exclusive
// scans of the list sizes in shared memory.  The page lists are then written
// one thread per page slot: the plan holds, for every slot, the span or tail
// that owns it and prefix sums of pages per request, so a slot's place in the
// keep or free list is a handful of independent loads and adds.  What a CTA does is in commit.cuh, for a chain of steps and for a tree.
#include "commit.cuh"

namespace lr {

namespace {

constexpr int kMaxReq = LR_COMMIT_MAX_REQUESTS;

template <bool kTree>
__global__ void __launch_bounds__(kCommitThreads)
commit_kernel(DevBatch d, bool after_accept, const uint8_t *verdict, const int32_t *n_accept, CommitOut o) {
  commit_cta<kTree>(d, blockIdx.x, gridDim.x, after_accept, verdict, CountsGiven{n_accept}, o);
}

}  // namespace

int init_commit_kernel() {
  if (int rc = cuda_fail(cudaFuncSetAttribute(commit_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              kMaxReq * kCommitSmemPerReq<true>), "commit_kernel<tree> shared-memory attribute"))
    return rc;
  return cuda_fail(cudaFuncSetAttribute(commit_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxReq * kCommitSmemPerReq<false>),
                   "commit_kernel shared-memory attribute");
}

int launch_commit(lr_plan *p, const uint8_t *verdict, const int32_t *n_accept, const CommitOut &o, bool after_accept, cudaStream_t s) {
  const DevBatch &d = p->dev;
  if (d.n_req > kMaxReq) {
    set_error("lr_commit: more than %d requests in one pass", kMaxReq);
    return LR_EUNSUPPORTED;
  }
  const int per_req = d.tree ? kCommitSmemPerReq<true> : kCommitSmemPerReq<false>;
  p->ctx->launches++;
  return cuda_fail(launch_dependent(d.tree ? commit_kernel<true> : commit_kernel<false>, dim3((unsigned)commit_ctas(d)), dim3(kCommitThreads),
                                    (size_t)d.n_req * per_req, s, d, after_accept, verdict, n_accept, o),
                   "commit_kernel launch");
}

}  // namespace lr
