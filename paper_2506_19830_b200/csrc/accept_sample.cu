// Stochastic token-level acceptance (rejection sampling) for point-mass draft distributions.
//
// Two kernels.  accept_stats_kernel streams the bf16 logits once -- the HBM-bound part: a warp takes one chunk of a row
// at a time (2048 logits, or the next power-of-two multiple that leaves at most kMaxChunks chunks) and leaves the pair
// (raw maximum M_c, S_c = sum exp((x - M_c) / T)).  accept_sample_kernel, one CTA per branch, combines the pairs of a row
// into (m, Z), gets P_i(d_i) = exp((x_d - m) / T) / Z for the drafts, walks the acceptance chain u_i < P_i(d_i), and draws
// the final token by inverse CDF over the stop row with the rejected token removed: first over the chunk weights
// S_c exp((M_c - m) / T) (no second pass over the row), then inside the one chunk that holds the target, which is read
// again and prefix-summed.  Every reduction has a fixed order: same inputs, same output.  The second kernel is a chain of
// latencies (some 8 us behind the first); what does not depend on the statistics it reads while the first one drains, the
// statistics of a branch mostly come in one trip, one butterfly sums a row and one scan finds the chunk: 617 rows, both and the
// commit 51.7 -> 46.8 us.
#include <algorithm>

#include "lr_common.cuh"

namespace lr {

namespace {

constexpr int kThreads = 256;
constexpr int kVec = 8;                       // 16-byte vectors a lane loads at a time
constexpr int kStep = 32 * kVec * 8;          // logits a warp takes at a time
constexpr int kMaxChunks = 160;               // per row: the pairs of kRowBatch rows must fit into 40 KB
constexpr int kCtasPerSm = 4;
constexpr int kRowBatch = 32;                 // rows of a branch handled at a time in the chain
constexpr int kStats = 8;                     // chunk pairs a thread asks for at a time

__device__ __forceinline__ float bf_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf_hi(uint32_t u) { return __uint_as_float(u & 0xFFFF0000u); }
__device__ __forceinline__ float ex2_approx(float x) {  // one MUFU operation; -inf gives 0
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float denan(float x) { return fmaxf(x, -INFINITY); }  // NaN counts as -inf (max drops a NaN operand)

// the logits of vector vi of a row (-inf past its end)
__device__ __forceinline__ void unpack(const uint4 &v, float *x) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    x[2 * j] = denan(bf_lo(w[j]));
    x[2 * j + 1] = denan(bf_hi(w[j]));
  }
}
__device__ __forceinline__ void load_tail(const uint16_t *rp, int32_t vocab, int32_t vi, float *x) {
#pragma unroll
  for (int j = 0; j < 8; ++j) {  // ragged end of the row (vocab not a multiple of 8), or beyond it
    const int32_t e = vi * 8 + j;
    x[j] = e < vocab ? denan(bf_lo((uint32_t)rp[e])) : -INFINITY;
  }
}

__device__ __forceinline__ uint32_t max_bf2(uint32_t x, uint32_t y) {  // a NaN operand loses
  uint32_t r;
  asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(y));
  return r;
}
__device__ __forceinline__ uint4 ld_stream(const uint4 *p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

// One warp per chunk at a time, the grid's warps taking the chunks of all rows in turn: the 4 KB a warp has in flight come
// back while the 31 others of its SM compute, and no warp ever waits for another.  617 rows of 152064 logits: 35.4 us,
// 5.3 TB/s, bound by HBM and, close behind it, by the exponentials (21 us of the special-function units); one CTA per
// chunk of 8192 with its loads in registers and two block reductions behind them took 54.8 us.
__global__ void __launch_bounds__(kThreads, kCtasPerSm)
accept_stats_kernel(const uint16_t *__restrict__ logits, int64_t row_stride, int32_t vocab, float k_log2, uint32_t n_chunks, int steps,
                    uint32_t total, float2 *__restrict__ stats) {
  const int lane = threadIdx.x & 31;
  const int32_t n_vec = vocab >> 3, rem = vocab & 7;
  constexpr uint32_t kNegInf2 = 0xFF80FF80u;
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the logits may come from the kernel launched just before
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  for (uint32_t unit = blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5); unit < total; unit += gridDim.x * (kThreads / 32)) {
    const uint32_t row = unit / n_chunks;
    const uint16_t *rp = logits + (int64_t)row * row_stride;
    int32_t v0 = (int32_t)(unit - row * n_chunks) * steps * (kStep / 8) + lane;
    // Of this lane's share of the chunk: the maximum, an exponent near -m * k_log2 and the sum of 2^(x * k_log2 + off).  `off` is
    // rounded at its own magnitude, which for large logits or low temperatures is far above that of the differences:
    // whatever goes from one lane or step to another is scaled by what `off` really is, not by what it stands for.
    float m = -INFINITY, off = 0.f, sum = 0.f;
    for (int st = 0; st < steps; ++st, v0 += kStep / 8) {
      uint32_t x[kVec * 4];
#pragma unroll
      for (int k = 0; k < kVec; ++k) {
        const int32_t vi = v0 + k * 32;
        uint4 v = make_uint4(kNegInf2, kNegInf2, kNegInf2, kNegInf2);
        if (vi < n_vec) v = ld_stream(reinterpret_cast<const uint4 *>(rp) + vi);
        x[4 * k] = v.x;
        x[4 * k + 1] = v.y;
        x[4 * k + 2] = v.z;
        x[4 * k + 3] = v.w;
      }
      if (rem != 0 && v0 <= n_vec && v0 + kStep / 8 > n_vec && ((n_vec - v0) & 31) == 0) {  // this lane has the ragged end of the row
#pragma unroll
        for (int k = 0; k < kVec; ++k)
          if (v0 + k * 32 == n_vec)
#pragma unroll
            for (int j = 0; j < 7; ++j)
              if (j < rem) {
                const uint32_t h = rp[(int64_t)n_vec * 8 + j];
                x[4 * k + (j >> 1)] = (j & 1) ? ((x[4 * k + (j >> 1)] & 0xFFFFu) | (h << 16)) : ((x[4 * k + (j >> 1)] & 0xFFFF0000u) | h);
              }
      }
      uint32_t mx = kNegInf2;
#pragma unroll
      for (int i = 0; i < kVec * 4; ++i) {
        x[i] = max_bf2(x[i], kNegInf2);  // NaN counts as -inf
        mx = max_bf2(mx, x[i]);
      }
      const float mn = fmaxf(m, fmaxf(bf_lo(mx), bf_hi(mx)));
      const float off_before = off;
      off = mn > -INFINITY ? -mn * k_log2 : 0.f;
      float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
      for (int i = 0; i < kVec * 4; i += 2) {
        a0 += ex2_approx(fmaf(bf_lo(x[i]), k_log2, off));
        a1 += ex2_approx(fmaf(bf_hi(x[i]), k_log2, off));
        a2 += ex2_approx(fmaf(bf_lo(x[i + 1]), k_log2, off));
        a3 += ex2_approx(fmaf(bf_hi(x[i + 1]), k_log2, off));
      }
      sum = fmaf(sum, m > -INFINITY ? ex2_approx(off - off_before) : 0.f, (a0 + a1) + (a2 + a3));
      m = mn;
    }
    float M = m;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xFFFFFFFFu, M, o));
    float S = m > -INFINITY ? sum * ex2_approx(-fmaf(M, k_log2, off)) : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) S += __shfl_xor_sync(0xFFFFFFFFu, S, o);
    if (lane == 0) stats[unit] = make_float2(M, S);
  }
}

__global__ void __launch_bounds__(kThreads)
accept_sample_kernel(const uint16_t *__restrict__ logits, int64_t row_stride, int32_t vocab, float k_log2,
                     const float2 *stats, int n_chunks, int chunk, const int32_t *__restrict__ draft_ids,
                     const int32_t *__restrict__ cu_draft, const float *__restrict__ u_accept,
                     const float *__restrict__ u_final, int32_t *__restrict__ n_accept, int32_t *__restrict__ final_id,
                     float *__restrict__ p_draft) {
  extern __shared__ float2 s_st[];  // [kRowBatch][n_chunks]: the chunk pairs of a batch of rows
  __shared__ float s_red[kThreads / 32];
  __shared__ float s_m[kRowBatch], s_p[kRowBatch], s_u[kRowBatch], s_xd[kRowBatch];
  __shared__ int32_t s_tok[kRowBatch];
  __shared__ int s_n, s_stop;
  __shared__ int s_pick_chunk, s_pick_thread;
  __shared__ float s_pick_before;
  const int b = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // Only the statistics come from the kernel launched just before, and that kernel let this one start when everything older
  // had finished: all else is fetched while it drains.
  const int32_t d0 = cu_draft[b], L = cu_draft[b + 1] - d0, r0 = d0 + b;
  const float u_fin = u_final[b];
  static_assert(kRowBatch == 32, "the chain uses one lane per row of a batch");

  // ---- acceptance chain, kRowBatch rows at a time.  Everything a batch needs from global memory (the chunk
  //      pairs of its rows, the drafts, their logits, their uniforms) is fetched at once into shared memory.
  if (tid == 0) {
    s_n = L;
    s_stop = 0;
  }
  int i0 = 0;
  for (;; i0 += kRowBatch) {
    const int rows = min(kRowBatch, L + 1 - i0);
    __syncthreads();
    if (tid < rows) {
      const int i = i0 + tid;
      int32_t dtok = -1;
      float xd = -INFINITY, u = 2.f;  // row L has no draft: u = 2 never passes
      if (i < L) {
        dtok = draft_ids[d0 + i];
        u = u_accept[d0 + i];
        if (dtok >= 0 && dtok < vocab) xd = denan(bf_lo((uint32_t)logits[(int64_t)(r0 + i) * row_stride + dtok]));
        else dtok = -1;
      }
      s_tok[tid] = dtok;
      s_xd[tid] = xd;
      s_u[tid] = u;
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // lr_commit's grid may be set up meanwhile
    const float2 *src = stats + (int64_t)(r0 + i0) * n_chunks;  // consecutive rows are contiguous
    for (int at = tid; at < rows * n_chunks; at += kStats * kThreads) {
      // kStats loads in flight, which is one trip to L2 for 27 rows of 75 chunks; left to a loop of single loads, 617 rows took 49.4 us
      // with the commit, like this 46.7
      float2 v[kStats];
#pragma unroll
      for (int k = 0; k < kStats; ++k)
        if (at + k * kThreads < rows * n_chunks) v[k] = ld_behind_wait(src + at + k * kThreads);
#pragma unroll
      for (int k = 0; k < kStats; ++k)
        if (at + k * kThreads < rows * n_chunks) s_st[at + k * kThreads] = v[k];
    }
    __syncthreads();
    for (int k = warp; k < rows; k += kThreads / 32) {  // one warp per row combines the row's chunk pairs in order
      const float2 *st = s_st + k * n_chunks;
      float m = -INFINITY;
      for (int c = lane; c < n_chunks; c += 32) m = fmaxf(m, st[c].x);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
      float z = 0.f;
      for (int c = lane; c < n_chunks; c += 32) {
        const float2 v = st[c];
        if (v.y > 0.f) z += v.y * exp2f((v.x - m) * k_log2);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xFFFFFFFFu, z, o);
      if (lane == 0) {
        const float p = (s_tok[k] >= 0 && z > 0.f) ? exp2f((s_xd[k] - m) * k_log2) / z : 0.f;
        if (p_draft != nullptr && i0 + k < L) p_draft[d0 + i0 + k] = p;
        s_m[k] = m;
        s_p[k] = p;
      }
    }
    __syncthreads();
    if (warp == 0) {  // first rejected draft of the batch (kRowBatch == 32 rows = one per lane)
      const bool rej = lane < rows && !(s_u[lane] < s_p[lane]);  // row L has no draft: always "rejected"
      const unsigned mask = __ballot_sync(0xFFFFFFFFu, rej);
      if (lane == 0 && mask != 0u) {
        s_n = i0 + __ffs(mask) - 1;
        s_stop = 1;
      }
    }
    __syncthreads();
    if (s_stop) break;
  }
  const int n = s_n, kn = n - i0;  // the stop row is row kn of the batch in shared memory
  const float m = s_m[kn];
  const int64_t stop_row = r0 + n;
  const uint16_t *rp = logits + stop_row * row_stride;
  const int32_t dead = n < L ? s_tok[kn] : -1;  // the rejected token has weight 0 in the residual
  const float w_dead = dead >= 0 ? exp2f((s_xd[kn] - m) * k_log2) : 0.f;

  // ---- which chunk holds the target: warp 0 scans the chunk weights, 32 chunks at a time (inclusive prefix
  //      sums by shuffles, fixed order)
  if (warp == 0) {
    const float2 *st = s_st + kn * n_chunks;
    const int dead_chunk = dead >= 0 ? dead / chunk : -1;
    auto weight = [&](int c) -> float {
      if (c >= n_chunks) return 0.f;
      const float2 v = st[c];
      float w = v.y > 0.f ? v.y * exp2f((v.x - m) * k_log2) : 0.f;
      if (c == dead_chunk) w = fmaxf(w - w_dead, 0.f);
      return w;
    };
    constexpr int kSteps = kMaxChunks / 32;
    float w[kSteps], t[kSteps], total = 0.f;  // of the chunks c0 + lane: weight, inclusive sum over all chunks so far
#pragma unroll
    for (int k = 0; k < kSteps; ++k) t[k] = w[k] = weight(k * 32 + lane);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
      for (int k = 0; k < kSteps; ++k) {
        const float y = __shfl_up_sync(0xFFFFFFFFu, t[k], o);
        if (lane >= o) t[k] += y;
      }
    }
#pragma unroll
    for (int k = 0; k < kSteps; ++k) {
      const float base = total;
      total += __shfl_sync(0xFFFFFFFFu, t[k], 31);
      t[k] += base;
    }
    const float target = u_fin * total;
    int pick = -1, last_nonzero = 0;
    float before = 0.f;
#pragma unroll
    for (int k = 0; k < kSteps; ++k) {
      const unsigned nz = __ballot_sync(0xFFFFFFFFu, w[k] > 0.f), hit = __ballot_sync(0xFFFFFFFFu, w[k] > 0.f && t[k] > target);
      if (nz != 0u) last_nonzero = k * 32 + 31 - __clz(nz);
      const float less = t[k] - w[k];
      if (hit != 0u && pick < 0) {
        const int l = __ffs(hit) - 1;
        pick = k * 32 + l;
        before = __shfl_sync(0xFFFFFFFFu, less, l);
      }
    }
    if (pick < 0) {  // rounding pushed the target past the last chunk: take the last chunk with any weight
      pick = last_nonzero;
      before = target;
    }
    if (lane == 0) {
      s_pick_chunk = pick;
      s_pick_before = target - before;  // what is still to be covered inside the chunk
    }
  }
  __syncthreads();

  // ---- inside the chunk: thread t owns chunk / kThreads consecutive logits (a multiple of 8); exclusive scan of the
  //      thread sums, then a sequential walk in the one thread whose range holds the target
  const int pc = s_pick_chunk, own = chunk / kThreads;
  const float remain = s_pick_before;
  const int32_t n_vec = vocab >> 3, e0 = pc * chunk + tid * own;
  auto weights = [&](int i, float (&w)[8]) {  // of logits e0 + i .. e0 + i + 7
    const int32_t vi = (e0 + i) >> 3;
    float x[8];
    if (vi < n_vec) unpack(__ldg(reinterpret_cast<const uint4 *>(rp) + vi), x);
    else load_tail(rp, vocab, vi, x);
#pragma unroll
    for (int j = 0; j < 8; ++j) w[j] = (e0 + i + j == dead || x[j] == -INFINITY) ? 0.f : exp2f((x[j] - m) * k_log2);
  };
  float mine = 0.f;
  for (int i = 0; i < own; i += 8) {
    float w[8];
    weights(i, w);
#pragma unroll
    for (int j = 0; j < 8; ++j) mine += w[j];
  }
  float incl = mine;  // inclusive scan over the block, in thread order
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const float y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s_red[warp] = incl;
  if (tid == 0) s_pick_thread = -1;
  __syncthreads();
  float base = 0.f;
  for (int k = 0; k < warp; ++k) base += s_red[k];
  const float before = base + incl - mine;
  const bool holds = before <= remain && before + mine > remain && mine > 0.f;
  if (holds) atomicMax(&s_pick_thread, tid);  // rounding can make two neighbours claim it: the later one decides
  __syncthreads();
  int pt = s_pick_thread;
  if (pt < 0) {  // rounding pushed the target past the end of the chunk: the last thread with any weight
    if (mine > 0.f) atomicMax(&s_pick_thread, tid);
    __syncthreads();
    pt = s_pick_thread;
  }
  if (tid == max(pt, 0)) {
    float cum = before;
    int pick = -1, last = 0;
    for (int i = 0; i < own && pick < 0; i += 8) {
      float w[8];
      weights(i, w);
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (w[j] > 0.f) {
          last = i + j;
          if (pick < 0 && cum + w[j] > remain) pick = i + j;
          cum += w[j];
        }
    }
    if (pick < 0) pick = last;
    n_accept[b] = n;
    final_id[b] = e0 + pick;
  }
}

}  // namespace

// steps of kStep logits per chunk
static int chunk_steps(int32_t vocab) {
  int steps = 1;
  while ((vocab + (int64_t)steps * kStep - 1) / ((int64_t)steps * kStep) > kMaxChunks) steps *= 2;
  return steps;
}

size_t accept_sample_scratch_bytes(int32_t vocab, int32_t n_rows) {
  const size_t chunk = (size_t)chunk_steps(vocab) * kStep, n_chunks = ((size_t)vocab + chunk - 1) / chunk;
  return std::max<size_t>(8, (size_t)n_rows * n_chunks * sizeof(float2));
}

int launch_accept_sample(lr_ctx *ctx, const void *logits, int64_t stride, const int32_t *drafts, const int32_t *cu_draft,
                         int32_t n_branch, int32_t n_rows, float temperature, const float *u_accept, const float *u_final,
                         int32_t *n_accept, int32_t *final_id, float *p_draft, void *scratch, cudaStream_t s) {
  const int32_t vocab = ctx->model.vocab;
  const int steps = chunk_steps(vocab), chunk = steps * kStep, n_chunks = (int)(((int64_t)vocab + chunk - 1) / chunk);
  if (n_rows > 65535) {
    set_error("lr_accept_sample: more than 65535 logits rows in one call");
    return LR_EUNSUPPORTED;
  }
  const float k_log2 = 1.4426950408889634f / temperature;
  auto *lg = reinterpret_cast<const uint16_t *>(logits);
  auto *st = reinterpret_cast<float2 *>(scratch);
  const uint32_t total = (uint32_t)n_rows * n_chunks;  // at most 65535 * kMaxChunks
  const unsigned grid = std::min((total + kThreads / 32 - 1) / (kThreads / 32), (uint32_t)(ctx->sm_count * kCtasPerSm));
  // programmatic dependent launches: this grid is set up while whatever is before it drains (it waits at once: 617 rows with the
  // commit of the call before 47.0 -> 45.5 us), the per-branch grid while the streaming grid drains
  ctx->launches += 2;
  if (int rc = cuda_fail(launch_dependent(accept_stats_kernel, dim3(grid), dim3(kThreads), 0, s, lg, stride, vocab, k_log2, (uint32_t)n_chunks, steps, total, st),
                         "accept_stats_kernel launch"))
    return rc;
  return cuda_fail(launch_dependent(accept_sample_kernel, dim3((unsigned)n_branch), dim3(kThreads), (size_t)kRowBatch * n_chunks * sizeof(float2), s,
                                    lg, stride, vocab, k_log2, st, n_chunks, chunk, drafts, cu_draft, u_accept, u_final, n_accept, final_id,
                                    p_draft),
                   "accept_sample_kernel launch");
}

}  // namespace lr
