// Compaction of the committed KV after lr_commit: token k of a request's committed sequence goes to slot
// k % 16 of its kept page number k / 16.
//
// The moves are in place in the caller's pools.  Counted along the keep list (list index x 16 + slot), a token only ever
// moves towards the front, so a CTA that owns some columns of a request (one KV head of K or V, or a slice of its
// channels) can sweep them in order without a staging area: it loads a round of rows into registers, meets at a
// barrier, and stores them; what a round overwrites lies in front of everything a later round still has to read.
// Different CTAs never touch the same bytes.  Every CTA scans its request's valid counts itself (a few hundred to a few
// thousand integers, in L2 after the first reader); tokens in front of the first partly filled page stay where they are.
//
// Bytes moved: 2 (K, V) x H_kv x D x 2 B per displaced token, read and written once.  Bound by the chain of dependent
// reads (list bounds, counts, page ids, data), not by bandwidth.  One launch; as three (scan, gather to a staging area,
// scatter) with the bytes read and written twice, one layer of 8 ragged requests took 16.3 us on a B200, this takes 4.1.
#include <algorithm>

#include "lr_common.cuh"

namespace lr {

namespace {

constexpr int kThreads = 256;
constexpr int kMaxReq = LR_COMPACT_MAX_REQUESTS;
constexpr int kPerThread = 4;                  // pages per thread and step of the scan
constexpr int kScan = kThreads * kPerThread;   // pages per step
constexpr int kRows = 8;                       // 16-byte vectors a thread holds per round

// blockIdx.x: (KV head, K or V, slice of the row); blockIdx.y: request.  1 << shift 16-byte vectors per slice.  sides: 2, or 1
// when K and V are the same pool, whose bytes one CTA has to own as well.
__global__ void __launch_bounds__(kThreads)
compact_kernel(DevBatch d, const int32_t *__restrict__ keep_off, const int32_t *__restrict__ keep_pages,
               const int32_t *__restrict__ keep_valid, int shift, int sides, uint4 *k_pool, uint4 *v_pool, int32_t *__restrict__ new_len,
               int32_t *__restrict__ n_pages_kept) {
  __shared__ int32_t s_off[kScan + 1];  // tokens of the request in front of each page of the step
  __shared__ int32_t warp_sum[kThreads / 32], warp_first[kThreads / 32];
  const int r = blockIdx.y, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int vec_per_row = d.head_dim / 8, slices = vec_per_row >> shift;
  const int slice = blockIdx.x % slices, h = blockIdx.x / slices / sides;
  uint4 *pool = blockIdx.x / slices % sides ? v_pool : k_pool;
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the keep list comes from the kernel launched just before
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // the next layer's grid may be set up meanwhile
  const int i0 = keep_off[r], i1 = keep_off[r + 1];
  if (i0 < 0 || i1 > d.n_page_slots) {  // keep lists that do not come from lr_commit
    if (tid == 0) {
      d.status[0] = kDevBounds;
      d.status[1] = 402;
    }
    return;
  }
  int32_t carry = 0;
  bool moved = false;  // a page of an earlier step was displaced, hence every page of this one
  for (int base = i0; base < i1; base += kScan) {
    const int n_here = min(kScan, i1 - base);
    int32_t x[kPerThread], sum = 0;
#pragma unroll
    for (int j = 0; j < kPerThread; ++j) {
      const int p = tid * kPerThread + j;
      x[j] = p < n_here ? keep_valid[base + p] : 0;
      if ((uint32_t)x[j] > kPage) {  // not from lr_commit
        d.status[0] = kDevBounds;
        d.status[1] = 400;
      }
    }
#pragma unroll
    for (int j = 0; j < kPerThread; ++j) sum += x[j];
    int32_t inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) warp_sum[wid] = inc;
    __syncthreads();
    int32_t off = carry + inc - sum;
    for (int w = 0; w < wid; ++w) off += warp_sum[w];
    int32_t first = kScan;  // first page of the step with a page that is not full somewhere in front of it
#pragma unroll
    for (int j = 0; j < kPerThread; ++j) {
      const int p = tid * kPerThread + j;
      s_off[p] = off;
      if (p < n_here && off != (base + p - i0) * kPage) first = min(first, p);
      off += x[j];
    }
    if (tid == kThreads - 1) s_off[kScan] = off;
    first = __reduce_min_sync(0xFFFFFFFFu, first);
    if (lane == 0) warp_first[wid] = first;
    __syncthreads();
    carry = s_off[kScan];
    if (moved) {
      first = 0;
    } else {
      for (int w = 0; w < kThreads / 32; ++w) first = min(first, warp_first[w]);
    }
    moved = moved || first < n_here;
    // rounds of kThreads * kRows vectors, in token order
    const int total = ((n_here - first) * kPage) << shift;
    for (int at = 0; at < total; at += kThreads * kRows) {
      uint4 v[kRows];
      int64_t to[kRows];
#pragma unroll
      for (int u = 0; u < kRows; ++u) {
        const int item = at + u * kThreads + tid, p = first + (item >> shift) / kPage, t = (item >> shift) % kPage;
        const int c = (slice << shift) + (item & ((1 << shift) - 1));
        to[u] = -1;
        if (item >= total) continue;
        const int32_t k0 = s_off[p], valid = s_off[p + 1] - k0, k = k0 + t;
        if (t >= valid) continue;
        const int32_t dst_entry = k / kPage;
        // never touch memory outside the pools, nor a page behind the token's own
        int code = 0;
        int64_t src_page = 0, dst_page = 0;
        if (valid > kPage || k0 < 0 || dst_entry > base + p - i0) {
          code = 400;
        } else {
          src_page = keep_pages[base + p];
          dst_page = keep_pages[i0 + dst_entry];
          if (src_page < 0 || src_page >= d.n_pool_pages) code = 400;
          else if (dst_page < 0 || dst_page >= d.n_pool_pages) code = 401;
        }
        if (code != 0) {
          d.status[0] = kDevBounds;
          d.status[1] = code;
          continue;
        }
        v[u] = pool[((src_page * d.n_kv_heads + h) * kPage + t) * vec_per_row + c];
        to[u] = ((dst_page * d.n_kv_heads + h) * kPage + k % kPage) * vec_per_row + c;
      }
      __syncthreads();  // the round is in registers
#pragma unroll
      for (int u = 0; u < kRows; ++u)
        if (to[u] >= 0) pool[to[u]] = v[u];
    }
    __syncthreads();  // s_off is free again
  }
  if (blockIdx.x == 0 && tid == 0) {
    new_len[r] = carry;
    n_pages_kept[r] = (carry + kPage - 1) / kPage;
  }
}

}  // namespace

int launch_compact(lr_plan *p, const int32_t *keep_off, const int32_t *keep_pages, const int32_t *keep_valid, void *k_pool,
                   void *v_pool, int32_t *new_len, int32_t *n_pages_kept, cudaStream_t s) {
  const DevBatch &d = p->dev;
  if (d.n_req > kMaxReq) {
    set_error("lr_compact: more than %d requests in one pass", kMaxReq);
    return LR_EUNSUPPORTED;
  }
  // Rows are sliced while that gives idle SMs something to do: down to 64 bytes until there are two CTAs per SM (8 KV heads
  // of 128 channels, whole rows and sliced: one request with 360 displaced tokens 10.8 and 5.5 us, 16 with 160 each 7.6 and
  // 7.0, but sliced in four 8.8), down to one sector for half a CTA per SM (one request 5.5 and 4.5, with 4000 tokens 26 and
  // 17; four requests 4.2 and 5.1).
  int shift = d.head_dim == 128 ? 4 : 3;
  const int sides = k_pool == v_pool ? 1 : 2;
  const int64_t rows = (int64_t)d.n_req * d.n_kv_heads * sides;
  while (shift > 1 && rows * (d.head_dim / 8 >> shift) < (shift > 2 ? 2 * p->ctx->sm_count : p->ctx->sm_count / 2)) --shift;
  const dim3 grid((unsigned)(d.n_kv_heads * sides * (d.head_dim / 8 >> shift)), (unsigned)d.n_req);
  p->ctx->launches++;
  return cuda_fail(launch_dependent(compact_kernel, grid, dim3(kThreads), 0, s, d, keep_off, keep_pages, keep_valid, shift, sides,
                                    reinterpret_cast<uint4 *>(k_pool), reinterpret_cast<uint4 *>(v_pool), new_len, n_pages_kept),
                   "compact_kernel launch");
}

}  // namespace lr
