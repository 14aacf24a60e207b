// Greedy token-level acceptance: one streaming pass over the bf16 logits.
//
// The rows are cut into chunks of 2048 logits, which the warps of a fixed grid take
// in turn; a warp reduces a chunk to (max value, lowest index) and publishes it
// with one 64-bit atomicMax on the row's key.  Warps never wait for one another.
// A CTA then takes a ticket, and the one holding the last ticket turns the row
// keys into n_accept / bonus per branch and zeroes the scratch again.
//
// The work is bound by HBM reads: 2 bytes per logit, read once, 16-byte loads,
// eight independent loads in flight per thread.  The maximum is taken with
// packed bf16x2 max instructions on whole 16-byte vectors (about one
// instruction per logit); the index is resolved only inside the winning vector.
// Small passes are bound by the chain load - atomic - ticket - last CTA
// (inside a whole pass they go another way, pass_tail.cu).
#include <algorithm>

#include "accept_stream.cuh"

namespace lr {

namespace {

constexpr int kThreads = 256;
constexpr int kVecPerThread = 8;                          // 16-byte vectors in flight per thread
constexpr int kCtasPerSm = 4;

// What a CTA that knows all keys to be there makes of them: one thread per branch, so that hundreds of branches cost one pass.
// Branch b's rows start at cu_draft[b] - first_draft + b.  Leaves the keys zeroed.  Drafts and their ranges may have been written while
// this kernel was resident, hence neither is __restrict__ in the kernel, and they are read from L2.
__device__ __forceinline__ void accept_finish(unsigned long long *scratch, const int32_t *draft_ids, const int32_t *cu_draft, int32_t n_branch,
                                              int32_t n_rows, int32_t first_draft, int32_t *n_accept, int32_t *bonus_id, int32_t *row_argmax) {
  unsigned long long *row_key = scratch + 1;
  const int tid = threadIdx.x;
  for (int b = tid; b < n_branch; b += kThreads) {
    const int32_t d0 = ld_behind_wait(cu_draft + b), L = ld_behind_wait(cu_draft + b + 1) - d0;
    int32_t bonus;
    n_accept[b] = accept_branch(row_key + (d0 - first_draft + b), draft_ids, d0, L, bonus);
    bonus_id[b] = bonus;
  }
  if (row_argmax != nullptr)
    for (int r = tid; r < n_rows; r += kThreads) row_argmax[r] = (int32_t)(0xFFFFFFFFu - (uint32_t)ld_behind_wait(row_key + r));
  __syncthreads();
  for (int r = tid; r < n_rows; r += kThreads) row_key[r] = 0ull;
}

__global__ void __launch_bounds__(kThreads)
accept_greedy_kernel(AcceptWork w, const int32_t *draft_ids, const int32_t *cu_draft, int32_t n_branch, int32_t n_rows, int32_t first_draft,
                     int32_t *__restrict__ n_accept, int32_t *__restrict__ bonus_id, int32_t *__restrict__ row_argmax) {
  unsigned int *counter = reinterpret_cast<unsigned int *>(w.scratch);
  const int tid = threadIdx.x, lane = tid & 31;
  __shared__ int s_last;
  // commit_kernel reads the verdicts as soon as this kernel lets it start, so all that is older must have finished by then: that
  // is why the wait comes first.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  for (uint32_t unit = blockIdx.x * (kThreads / 32) + (tid >> 5); unit < w.total; unit += gridDim.x * (kThreads / 32)) {
    uint4 v[kVecPerThread];
    accept_load(w, unit, lane, v);
    accept_publish(w, unit / w.n_chunks, lane, accept_best(w, unit, lane, v));
  }
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    unsigned int t = atomicAdd(counter, 1u);
    s_last = (t == gridDim.x - 1);
  }
  __syncthreads();
  if (!s_last) return;

  __threadfence();
  accept_finish(w.scratch, draft_ids, cu_draft, n_branch, n_rows, first_draft, n_accept, bonus_id, row_argmax);
  if (tid == 0) *counter = 0u;
}

// Scratch of lr_accept_greedy_static: row keys + ticket counter for up to LR_ACCEPT_STATIC_MAX_ROWS rows.
// Lives in every context that loads the library, for the life of the process.
static __device__ __align__(256) unsigned long long g_static_scratch[LR_ACCEPT_STATIC_MAX_ROWS + 1];

}  // namespace

// Device address of g_static_scratch per device ordinal, resolved on the first call for that device.
static void *g_static_scratch_addr[64] = {nullptr};

int launch_accept_static(lr_ctx *ctx, const void *logits, int64_t stride, const int32_t *drafts, const int32_t *cu_draft,
                         int32_t n_branch, int32_t n_rows, int32_t *n_accept, int32_t *bonus, int32_t *row_argmax,
                         cudaStream_t s) {
  if (n_rows > LR_ACCEPT_STATIC_MAX_ROWS) {
    set_error("lr_accept_greedy_static: %d logits rows, the built-in scratch holds at most %d; use lr_accept_greedy",
              n_rows, LR_ACCEPT_STATIC_MAX_ROWS);
    return LR_EINVAL;
  }
  if (ctx->device < 0 || ctx->device >= 64) {
    set_error("lr_accept_greedy_static: device ordinal %d not supported", ctx->device);
    return LR_EUNSUPPORTED;
  }
  // ctx's device is made current for the symbol look-up and the launch; the caller's own choice is put back afterwards
  int prev_device = -1;
  if (int rc = cuda_fail(cudaGetDevice(&prev_device), "cudaGetDevice")) return rc;
  if (prev_device != ctx->device)
    if (int rc = cuda_fail(cudaSetDevice(ctx->device), "cudaSetDevice")) return rc;
  int rc = LR_OK;
  void *ptr = g_static_scratch_addr[ctx->device];
  if (ptr == nullptr) {
    // In host code the array's name is only a handle; the kernel needs the address the symbol has
    // on *this* device.  Done once per device, with that device current.  The cache is written without a
    // lock (every writer stores the same value); the first call per device should still come from one thread.
    rc = cuda_fail(cudaGetSymbolAddress(&ptr, g_static_scratch), "cudaGetSymbolAddress(static scratch)");
    if (rc == LR_OK) g_static_scratch_addr[ctx->device] = ptr;
  }
  // Every call shares the array and it keeps what the last call left: start from zero regardless.
  if (rc == LR_OK) rc = cuda_fail(cudaMemsetAsync(ptr, 0, 8 * ((size_t)n_rows + 1), s), "cudaMemsetAsync(static scratch)");
  if (rc == LR_OK) rc = launch_accept(ctx, logits, stride, drafts, cu_draft, n_branch, n_rows, 0, n_accept, bonus, row_argmax, ptr, s);
  if (prev_device != ctx->device) {
    const cudaError_t e = cudaSetDevice(prev_device);
    if (rc == LR_OK) rc = cuda_fail(e, "cudaSetDevice(restore)");
  }
  return rc;
}

int launch_accept(lr_ctx *ctx, const void *logits, int64_t stride, const int32_t *drafts, const int32_t *cu_draft,
                  int32_t n_branch, int32_t n_rows, int32_t first_draft, int32_t *n_accept, int32_t *bonus, int32_t *row_argmax,
                  void *scratch, cudaStream_t s) {
  const AcceptWork w = accept_work(ctx, logits, stride, n_rows, scratch, kVecPerThread);
  // a chunk per warp at least, at most kCtasPerSm CTAs per SM
  const unsigned grid = std::min((w.total + kThreads / 32 - 1) / (kThreads / 32), (uint32_t)(ctx->sm_count * kCtasPerSm));
  // Set up while whatever is before it drains; see the kernel's first lines.  Behind a fill of 64 values, the attention of one request
  // of 4 K tokens, and that of 4 ragged ones, 51 to 2268 rows of 152064 are ready 0.3 to 2.8 us sooner than with an ordinary launch
  // (411 rows: 32.1 -> 29.8, 44.7 -> 42.5, 59.0 -> 57.0; 2268: 110.5 -> 108.2, 124.9 -> 123.2, 140.3 -> 138.6), in a graph 0.2.  Behind
  // another acceptance of the same size, as a benchmark of the kernel alone has it and no program, an ordinary launch is the faster one
  // from 300 rows on in a graph (411 rows 25.1 and 29.0, 500 28.4 and 31.1, 2268 105.4 and 107.0) and at some sizes without (411 rows
  // 27.9 and 29.4, 500 30.6 and 31.5; 206 17.7 and 17.6, 1000 53.5 and 53.3); starting CTAs or warps apart from one another changes nothing.
  ctx->launches++;
  return cuda_fail(launch_dependent(accept_greedy_kernel, dim3(grid), dim3(kThreads), 0, s, w, drafts, cu_draft, n_branch, n_rows, first_draft, n_accept, bonus,
                                    row_argmax),
                   "accept_greedy_kernel launch");
}

}  // namespace lr
