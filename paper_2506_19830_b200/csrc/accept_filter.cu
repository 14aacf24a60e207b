// Stochastic token-level acceptance with the sampling filters of Section 4 "Setup" (top-k, top-p) applied to
// the target distribution before the rejection-sampling rule of Background, "Speculative Decoding".
//
// The filters keep a leading part of the ranking of a row's tokens by probability (descending; equal
// probabilities in index order).  With bf16 logits the ranking is the ranking of a 16-bit ordered key (-0 and +0
// sharing one), so the kept set of a row is described by a cut: every token whose key is above cut_key, and of the
// tokens whose key equals cut_key those with an index up to cut_idx.  Masses are w = exp2((x - m) log2(e) / T) as
// integers in units of 2^-40 (m: the row maximum): integer sums do not depend on the order of the additions, so every
// route below gives the same cut and the same draw.
//
// The cut of a row is found by one of two routes.
//
// Candidates (filter_scan_kernel, filter_cut_kernel): the logits are read once for the largest key of every group of 64
// (or 8) tokens and, with top-k off, for the row's mass as an fp32 sum.  A CTA per row then finds the k_sel-th largest of the
// group maxima, reads the few groups that reach it once more and ranks their tokens.  With top-k on that is all there is
// to know.  With top-p alone the total mass is known to within kMassEps; the row is settled when both ends of that interval
// give the same cut.
//
// Windows (filter_window_kernel): a cluster of CTAs holds the row in shared memory, counts tokens per key, merges the
// counts through distributed shared memory and finds the cut in them, whatever the row looks like.  It takes the rows that
// the candidates leave open -- a kept set larger than the candidates, many equal logits, a cut within rounding of a
// step, no finite maximum -- and all rows of a call that cannot use the candidates or has few rows to settle by mass
// (launch_accept_filtered has the rule).
//
// accept_filtered_kernel (per branch) walks the acceptance chain with P'(d) = w_d / Z' for kept tokens and 0 for
// the others, and draws the final token by inverse CDF over the kept tokens of the stop row in index order: from the list of
// them when the candidates settled the row, else first over the kept mass of every slice of the row, then inside one slice.
#include <cooperative_groups.h>

#include <algorithm>

#include "lr_common.cuh"

namespace lr {

namespace {

constexpr int kT = 256;             // threads of every kernel but filter_window_kernel
constexpr int kWarps = kT / 32;
constexpr int kVec = 8;             // 16-byte vectors a lane of filter_scan_kernel takes at a time
constexpr int kChunk = 32 * kVec * 8;  // logits a warp takes at a time
constexpr int kScanCtasPerSm = 4;
constexpr int kGroupCap = 1344;     // groups filter_cut_kernel reads again (k_sel + k_sel / 4 + 4 at most, but for ties)
constexpr int kListCap = 1408;      // candidates of a row
constexpr int kSortCap = 2048;      // ... where many are looked for (a top-k of 1024 finds up to 1284 groups, and ties), to sort
constexpr int kListOut = 256;       // kept tokens that go out as a list
constexpr int kManyFrom = 128;      // top_k from which filter_cut_kernel reads many groups at a time and may sort
constexpr int64_t kManyBytes = 96 << 20;  // ... and the bytes of logits, with top-p alone
constexpr int kCountMax = 448;      // candidates ranked by counting; more may be sorted
constexpr int kSelMax = 1024;       // largest top_k the candidates serve
constexpr int kSelTopP = 128;       // leading tokens to look for when top-k is off
constexpr int kProbeRows = 16;      // rows the candidates are tried on first when top-k is off
constexpr int kWT = 512;            // threads of a CTA of filter_window_kernel
constexpr int kAT = 512;            // ... of accept_filtered_kernel
constexpr int kSlicesInFlight = 5;  // slices a warp of it works on at a time: one round for 163840 tokens and 8 CTAs
constexpr int kWin = 8192;          // keys per window
constexpr int kMaxSlices = 1024;    // slices a row is cut into for the draw
constexpr size_t kWindowSmemMax = 112 * 1024;  // two CTAs per SM
// Relative distance between the fp32 sum of a row's masses and their integer sum.  A token below the 2^-40th of the row's
// largest mass has none, so every argument that matters lies within 40 of 0, whatever the logits and the temperature: it is
// a difference scaled, rounded twice (2^-18.7 absolute, 1.7e-6 of the mass), on the way from the lane to its chunk and from
// there to the row twice more, and once in the integer masses (5.1e-6 together); ex2.approx is good to 2^-22 each time
// (1e-6), an fp32 sum of 64 terms and some 30 further additions to 5e-6, rounding masses to 2^-40 of the largest to 1e-7;
// rounded up.
constexpr double kMassEps = 2e-5;
typedef unsigned long long u64;
constexpr int32_t kNoKey = INT32_MIN;

struct RowCut {  // what the acceptance kernel needs to know about a row (32 bytes)
  float m;          // row maximum (finite: a row without a finite logit gets -3e38)
  int32_t cut_key;  // key32 of the last kept group of equal logits; kNoKey: everything is kept
  int32_t cut_idx;  // largest index kept inside that group
  int32_t n_kept;
  u64 z_fix;        // mass of the kept set
  int32_t listed;   // 1: the kept tokens were written as a list
  int32_t pad;
};

// Order-preserving key of a bf16 value given as fp32 bits (low 16 bits zero): sign-magnitude turned into two's
// complement, so that a larger value has a larger key and -0 and +0 share key 0.  A multiple of 65536; key32 >> 16
// ("key16") lies in [-32768, 32767].  A NaN lies beyond the infinities; its mass is 0 (below), so wherever it lands
// it changes no sum.
__device__ __forceinline__ int32_t key32(uint32_t f) {
  const uint32_t s = (uint32_t)((int32_t)f >> 31);
  return (int32_t)(((f & 0x7FFFFFFFu) ^ s) - s);
}
__device__ __forceinline__ uint32_t f_of_key16(int32_t key16) {
  return key16 >= 0 ? (uint32_t)key16 << 16 : (0x8000u | (uint32_t)(-key16)) << 16;
}
// mass of a token in units of 2^-40 relative to the row maximum (at most 2^40): a subtraction, a multiply-add, one
// exponential, one conversion.  The maximum turns NaN into 0 (the conversion alone would make it 2^63).
__device__ __forceinline__ u64 wfix_of(uint32_t f, float m, float k_log2) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(fmaf(__uint_as_float(f) - m, k_log2, 40.f)));
  u64 r;
  asm("cvt.rni.u64.f32 %0, %1;" : "=l"(r) : "f"(fmaxf(y, 0.f)));
  return r;
}

// a row's cut, behind the wait of a kernel that has loaded other things before (8-byte words: scratch is aligned to no more)
__device__ __forceinline__ RowCut cut_behind_wait(const RowCut *cut) {
  static_assert(sizeof(RowCut) == 32 && alignof(RowCut) == 8, "four words");
  u64 w[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) w[i] = ld_behind_wait(reinterpret_cast<const u64 *>(cut) + i);
  RowCut rc;
  memcpy(&rc, w, sizeof(rc));
  return rc;
}

__device__ __forceinline__ bool is_kept(int32_t key, int32_t e, const RowCut &rc) {
  return key > rc.cut_key || (key == rc.cut_key && e <= rc.cut_idx);
}

constexpr uint32_t kNegInf2 = 0xFF80FF80u;
__device__ __forceinline__ uint32_t max_bf2(uint32_t x, uint32_t y) {  // a NaN operand loses
  uint32_t r;
  asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(y));
  return r;
}
__device__ __forceinline__ float lo_f(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float hi_f(uint32_t u) { return __uint_as_float(u & 0xFFFF0000u); }
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// inclusive scan over the block in thread order; `total` receives the sum over the block
template <int kThreads, class T>
__device__ __forceinline__ T block_scan(T v, T *s_w, T &total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T y = __shfl_up_sync(0xFFFFFFFFu, v, o);
    if (lane >= o) v += y;
  }
  if (lane == 31) s_w[warp] = v;
  __syncthreads();
  T t = lane < kThreads / 32 ? s_w[lane] : 0;  // every warp scans the warps' sums
#pragma unroll
  for (int o = 1; o < kThreads / 32; o <<= 1) {
    const T y = __shfl_up_sync(0xFFFFFFFFu, t, o);
    if (lane >= o) t += y;
  }
  total = __shfl_sync(0xFFFFFFFFu, t, kThreads / 32 - 1);
  const T base = __shfl_sync(0xFFFFFFFFu, t, warp > 0 ? warp - 1 : 0);
  __syncthreads();
  return warp > 0 ? v + base : v;
}

// Candidates are ordered as 64-bit numbers: the key above, the complement of the index below, so that "larger" is
// "ranked before".
__device__ __forceinline__ u64 cand_of(uint32_t f, int32_t e) {
  return ((u64)(uint32_t)((key32(f) >> 16) + 32768) << 32) | (uint32_t)~(uint32_t)e;
}
__device__ __forceinline__ int32_t cand_key16(u64 c) { return (int32_t)(c >> 32) - 32768; }
__device__ __forceinline__ int32_t cand_idx(u64 c) { return (int32_t)~(uint32_t)c; }

// the last vector of a row whose length is not a multiple of 8, padded with -inf
__device__ __forceinline__ uint4 ragged_vec(const uint16_t *rp, int32_t n_vec, int32_t rem) {
  uint32_t w[4] = {kNegInf2, kNegInf2, kNegInf2, kNegInf2};
#pragma unroll
  for (int j = 0; j < 7; ++j)
    if (j < rem) {
      const uint32_t h = rp[(int64_t)n_vec * 8 + j];
      w[j >> 1] = (j & 1) ? ((w[j >> 1] & 0xFFFFu) | (h << 16)) : ((w[j >> 1] & 0xFFFF0000u) | h);
    }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// ---- one read of the logits -------------------------------------------------------------------------------
// A warp per chunk of 2048 logits at a time, no warp ever waiting for another.  A lane's kGV vectors of a chunk, 32 vectors
// apart, are a group: the group's largest logit goes out, and with kSum the chunk's pair (largest logit, sum of
// exp((x - largest) / T)).  Bound: HBM (kSum: and the special-function units close behind).
template <bool kSum, int kGV>
__global__ void __launch_bounds__(kT, kScanCtasPerSm)
filter_scan_kernel(const uint16_t *__restrict__ logits, int64_t row_stride, int32_t vocab, float k_log2, uint32_t n_chunks, uint32_t total,
                   uint16_t *__restrict__ group_max, float2 *__restrict__ stats, int32_t *n_open, int n_probe, int32_t *__restrict__ gave_up) {
  const int lane = threadIdx.x & 31;
  const int32_t n_vec = vocab >> 3, rem = vocab & 7;
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the logits may come from the kernel launched just before
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (gave_up == nullptr) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *n_open = 0;
  } else {  // the rows behind the probe: not worth reading when it left most of its rows open
    const bool skip = 2 * *n_open > n_probe;
    if (blockIdx.x == 0 && threadIdx.x == 0) *gave_up = skip;
    if (skip) return;
  }
  for (uint32_t unit = blockIdx.x * kWarps + (threadIdx.x >> 5); unit < total; unit += gridDim.x * kWarps) {
    const uint32_t row = unit / n_chunks;
    const uint16_t *rp = logits + (int64_t)row * row_stride;
    const int32_t v0 = (int32_t)(unit - row * n_chunks) * (kChunk / 8) + lane;
    uint32_t x[kVec * 4];
#pragma unroll
    for (int k = 0; k < kVec; ++k) {
      const int32_t vi = v0 + k * 32;
      uint4 v = make_uint4(kNegInf2, kNegInf2, kNegInf2, kNegInf2);
      if (vi < n_vec)
        asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                     : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(reinterpret_cast<const uint4 *>(rp) + vi));
      x[4 * k] = v.x;
      x[4 * k + 1] = v.y;
      x[4 * k + 2] = v.z;
      x[4 * k + 3] = v.w;
    }
    if (rem != 0 && v0 <= n_vec && v0 + kChunk / 8 > n_vec && ((n_vec - v0) & 31) == 0) {  // this lane has the ragged end of the row
#pragma unroll
      for (int k = 0; k < kVec; ++k)
        if (v0 + k * 32 == n_vec) {
          const uint4 v = ragged_vec(rp, n_vec, rem);
          x[4 * k] = v.x;
          x[4 * k + 1] = v.y;
          x[4 * k + 2] = v.z;
          x[4 * k + 3] = v.w;
        }
    }
    float top = -INFINITY;
#pragma unroll
    for (int k0 = 0; k0 < kVec; k0 += kGV) {
      uint32_t mx = kNegInf2;
#pragma unroll
      for (int i = 4 * k0; i < 4 * (k0 + kGV); ++i) {
        if (kSum) x[i] = max_bf2(x[i], kNegInf2);  // NaN counts as -inf
        mx = max_bf2(mx, x[i]);
      }
      const float g = fmaxf(lo_f(mx), hi_f(mx));
      top = fmaxf(top, g);
      group_max[(int64_t)unit * (32 * kVec / kGV) + (k0 / kGV) * 32 + lane] = (uint16_t)(__float_as_uint(g) >> 16);
    }
    if (kSum) {
      // subtracted before it is scaled: top * k_log2 would be rounded at its own magnitude, for all terms alike
      const float ref = top > -INFINITY ? top : 0.f;
      float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
      for (int i = 0; i < kVec * 4; i += 2) {
        a0 += ex2_approx((lo_f(x[i]) - ref) * k_log2);
        a1 += ex2_approx((hi_f(x[i]) - ref) * k_log2);
        a2 += ex2_approx((lo_f(x[i + 1]) - ref) * k_log2);
        a3 += ex2_approx((hi_f(x[i + 1]) - ref) * k_log2);
      }
      float M = top;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xFFFFFFFFu, M, o));
      float S = ((a0 + a1) + (a2 + a3)) * ex2_approx((top - (M > -INFINITY ? M : 0.f)) * k_log2);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) S += __shfl_xor_sync(0xFFFFFFFFu, S, o);
      if (lane == 0) stats[unit] = make_float2(M, S);
    }
  }
}

// tokens of a CTA's share of a row in a cluster of n (a multiple of 8)
__host__ __device__ __forceinline__ int32_t share_of(int32_t vocab, int n) { return ((vocab + 7) / 8 + n - 1) / n * 8; }
// tokens of a slice (a multiple of 256; at most kMaxSlices of them)
__host__ __device__ __forceinline__ int slice_len_of(int32_t vocab) { return 256 * ((vocab + 256 * kMaxSlices - 1) / (256 * kMaxSlices)); }

// ---- the cut of a row from its candidates -----------------------------------------------------------------
// A lower bound of the k_sel-th largest logit is any value that k_sel group maxima reach (they are logits of different
// tokens); it is raised by bisection on the key until little more than k_sel maxima reach it.  Only those groups hold tokens of at least that value: they are read again.  Bound: instructions, a few hundred per warp.
template <int kGV, bool kMany>
__global__ void __launch_bounds__(kT, kMany ? 4 : 0)
filter_cut_kernel(const uint16_t *__restrict__ logits, int64_t row_stride, int32_t vocab, float k_log2, int32_t top_k, float top_p, int k_sel,
                  int n_chunks, const uint16_t *__restrict__ group_max, const float2 *__restrict__ stats, RowCut *__restrict__ cuts,
                  u64 *__restrict__ lists, int32_t *__restrict__ n_kept_out, int32_t *__restrict__ n_open, int32_t *__restrict__ open_rows,
                  int row0, const int32_t *__restrict__ gave_up) {
  constexpr int kKeyWords = kGV == 4 || kGV == 2 ? 16 : 8;  // words of group maxima a thread keeps in registers
  constexpr int kCap = kMany ? kSortCap - 64 : kListCap;
  __shared__ u64 s_cand[kMany ? kSortCap : kListCap], s_ranked[kMany ? kCountMax : kListCap], s_cum[kCap];
  __shared__ int s_grp[kGroupCap];
  __shared__ int s_n, s_n_grp, s_cnt[2][kWarps], s_kept;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t row = row0 + (int)blockIdx.x;
  constexpr int kPerChunk = 32 * kVec / kGV;
  const int n_words = n_chunks * kPerChunk / 2;
  const bool by_k = top_k > 0 && top_k < vocab, by_p = top_p < 1.f;
  if (tid == 0) s_n = s_n_grp = 0;
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the maxima come from the kernel launched just before
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (gave_up != nullptr && *gave_up != 0) {  // every row is left to the windows, the tried ones in front of row0 too
    if (tid == 0) open_rows[row] = (int32_t)row;
    if (blockIdx.x == 0 && tid < row0) open_rows[tid] = tid;
    if (blockIdx.x == 0 && tid == 0) *n_open = row0 + (int)gridDim.x;
    return;
  }
  const uint32_t *src = reinterpret_cast<const uint32_t *>(group_max + row * n_chunks * kPerChunk);
  uint32_t g2[kKeyWords];  // word i of the thread is word i * kT + tid of the row
#pragma unroll
  for (int i = 0; i < kKeyWords; ++i) g2[i] = i * kT + tid < n_words ? __ldg(src + i * kT + tid) : kNegInf2;
  // mass of the whole row (top-p alone), to within kMassEps: warp 0, while the others wait for it to bisect
  float m_all = -INFINITY;
  double z_all = 0.0;
  if (!by_k && warp == 0) {
    for (int i = lane; i < n_chunks; i += 32) m_all = fmaxf(m_all, stats[row * n_chunks + i].x);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m_all = fmaxf(m_all, __shfl_xor_sync(0xFFFFFFFFu, m_all, o));
    for (int i = lane; i < n_chunks; i += 32) {
      const float2 h = stats[row * n_chunks + i];
      z_all += (double)(h.y * ex2_approx((h.x - m_all) * k_log2));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) z_all += __shfl_xor_sync(0xFFFFFFFFu, z_all, o);
  }
  // No token weighs more than 1 of z_all: a flat row keeps more than the list of candidates can hold.
  if (!by_k && __syncthreads_or((double)top_p * z_all > 1.01 * kCap)) {
    if (tid == 0) open_rows[atomicAdd(n_open, 1)] = (int32_t)row;
    return;
  }
  auto bf2_of = [](int32_t key16) -> __nv_bfloat162 {
    const uint32_t u = f_of_key16(key16) >> 16, uu = u | (u << 16);
    return *reinterpret_cast<const __nv_bfloat162 *>(&uu);
  };
  auto as_bf2 = [](const uint32_t &u) -> __nv_bfloat162 { return *reinterpret_cast<const __nv_bfloat162 *>(&u); };
  int32_t least = -32639;  // key16 of the smallest finite logit: all groups with one
  int reach = -1;          // groups that reach it
  int buf = 0;
  // keys from the largest finite one (32639) down to the smallest: 2^16 of them at most
#pragma unroll 1
  for (int step = 32768; step > 0; step >>= 1) {
    const int32_t u = least + step;
    if (u > 32640) continue;  // the key of +inf
    const __nv_bfloat162 t = bf2_of(u);
    __nv_bfloat162 c2 = __floats2bfloat162_rn(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < kKeyWords; ++i) c2 = __hadd2(c2, __hge2(as_bf2(g2[i]), t));
    int c = (int)(__low2float(c2) + __high2float(c2));
    for (int i = kKeyWords * kT + tid; i < n_words; i += kT) {
      const uint32_t w = __ldg(src + i);
      c += __popc(__hge2_mask(as_bf2(w), t)) >> 4;
    }
    c = __reduce_add_sync(0xFFFFFFFFu, c);
    if (lane == 0) s_cnt[buf][warp] = c;
    __syncthreads();
    c = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) c += s_cnt[buf][w];
    buf ^= 1;
    if (c >= k_sel) {
      least = u;
      reach = c;
      if (c <= k_sel + k_sel / 4 + 4) break;
    }
  }
  auto note = [&](uint32_t w, int word) {
    const uint32_t hit = __hge2_mask(as_bf2(w), bf2_of(least));
    if (hit != 0)
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (hit & (h ? 0x10000u : 1u)) {
          const int at = atomicAdd(&s_n_grp, 1);
          if (at < kGroupCap) s_grp[at] = 2 * word + h;
        }
  };
  if (reach <= kGroupCap) {
#pragma unroll
    for (int i = 0; i < kKeyWords; ++i) note(g2[i], i * kT + tid);
    for (int i = kKeyWords * kT + tid; i < n_words; i += kT) note(__ldg(src + i), i);
  }
  __syncthreads();
  const int n_grp = s_n_grp;
  const uint16_t *rp = logits + row * row_stride;
  if (n_grp <= kGroupCap) {
    const int32_t n_vec = vocab >> 3, rem = vocab & 7;
    const float least_x = __uint_as_float(f_of_key16(least));
    constexpr int kFly = kMany ? kGV : 1;  // vectors a thread asks for at a time
    for (int i0 = tid; i0 < n_grp * kGV; i0 += kFly * kT) {
      uint4 v[kFly];
      int32_t at_vec[kFly];
#pragma unroll
      for (int q = 0; q < kFly; ++q) {
        const int i = i0 + q * kT;
        v[q] = make_uint4(0x7FC07FC0u, 0x7FC07FC0u, 0x7FC07FC0u, 0x7FC07FC0u);  // NaN: never a candidate
        at_vec[q] = 0;
        if (i < n_grp * kGV) {
          const int g = s_grp[i / kGV];
          const int32_t vi = (g / kPerChunk) * (kChunk / 8) + (g % kPerChunk) / 32 * (32 * kGV) + g % 32 + (i % kGV) * 32;
          at_vec[q] = vi;
          if (vi < n_vec) v[q] = __ldg(reinterpret_cast<const uint4 *>(rp) + vi);
          else if (vi == n_vec && rem != 0) v[q] = ragged_vec(rp, n_vec, rem);
        }
      }
#pragma unroll
      for (int q = 0; q < kFly; ++q) {
        const uint32_t w[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const uint32_t f = (j & 1) ? (w[j >> 1] & 0xFFFF0000u) : (w[j >> 1] << 16);
          if (__uint_as_float(f) >= least_x) {  // (a NaN is not)
            const int at = atomicAdd(&s_n, 1);
            if (at < kCap) s_cand[at] = cand_of(f, at_vec[q] * 8 + j);
          }
        }
      }
    }
  }
  __syncthreads();
  const int n = s_n;
  const bool usable = n_grp <= kGroupCap && n >= 1 && n <= kCap && (!by_k || n >= top_k);
  const bool count = !kMany || n <= kCountMax;
  const u64 *s_sorted = count ? s_ranked : s_cand;
  if (usable && count) {
    for (int i = tid; i < n; i += kT) {  // rank by counting: the candidates are all different
      const u64 e = s_cand[i];
      int before = 0;
#pragma unroll 4
      for (int j = 0; j < n; ++j) before += s_cand[j] > e ? 1 : 0;
      s_ranked[before] = e;
    }
  } else if (kMany && usable) {  // bitonic, largest first
    int size = 512;
    while (size < n) size *= 2;
    for (int i = n + tid; i < size; i += kT) s_cand[i] = 0;  // behind every candidate
    for (int run = 2; run <= size; run *= 2)
      for (int step = run / 2; step > 0; step /= 2) {
        __syncthreads();
        for (int i = tid; i < size / 2; i += kT) {
          const int lo = 2 * i - (i & (step - 1)), hi = lo + step;
          const u64 x = s_cand[lo], y = s_cand[hi];
          if ((x < y) == ((lo & run) == 0)) {
            s_cand[lo] = y;
            s_cand[hi] = x;
          }
        }
      }
  }
  __syncthreads();
  // ---- warp 0: the last rank kept.  It is top_k - 1, or the first one at which the mass, itself included, reaches
  //      t = ceil(top_p W), where W is the mass of the leading top_k ranks, or -- to within kMassEps -- of the whole row.
  if (warp == 0) {
    bool ok = usable;
    const float m = ok ? __uint_as_float(f_of_key16(cand_key16(s_sorted[0]))) : 0.f;
    ok = ok && fabsf(m) < INFINITY;
    const int ranks = ok ? (by_k ? top_k : n) : 0;
    u64 sum = 0;
    for (int base = 0; base < ranks; base += 32) {
      const int i = base + lane;
      u64 c = i < ranks ? wfix_of(f_of_key16(cand_key16(s_sorted[i])), m, k_log2) : 0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const u64 y = __shfl_up_sync(0xFFFFFFFFu, c, o);
        if (lane >= o) c += y;
      }
      c += sum;
      if (i < ranks) s_cum[i] = c;
      sum = __shfl_sync(0xFFFFFFFFu, c, 31);
    }
    int r = ranks - 1;
    if (ok && by_p) {
      u64 t0, t1;
      if (by_k) {
        const double t_d = ceil((double)top_p * (double)sum);
        t0 = t_d < 1.0 ? 1ull : (u64)t_d;
        if (t0 > sum) t0 = sum;
        t1 = t0;
        ok = sum > 0;
      } else {
        const double z = z_all * 1099511627776.0;  // units of 2^-40
        t0 = (u64)((double)top_p * z * (1.0 - kMassEps));
        t1 = (u64)((double)top_p * z * (1.0 + kMassEps)) + 2;
        ok = t0 > 0 && t1 <= sum;  // else the cut may lie beyond the candidates
      }
      __syncwarp();
      int lo = 0, below = 0;  // ranks whose cumulative mass stays below t0, t1
      for (int i = lane; i < ranks; i += 32) {
        lo += s_cum[i] < t0 ? 1 : 0;
        below += s_cum[i] < t1 ? 1 : 0;
      }
      r = __reduce_add_sync(0xFFFFFFFFu, lo);
      ok = ok && r == __reduce_add_sync(0xFFFFFFFFu, below);
    }
    __syncwarp();
    if (lane == 0) {
      s_kept = ok ? r + 1 : 0;
      if (ok) {
        RowCut rc;
        rc.m = m;
        rc.cut_key = cand_key16(s_sorted[r]) * 65536;
        rc.cut_idx = cand_idx(s_sorted[r]);
        rc.n_kept = r + 1;
        rc.z_fix = s_cum[r];
        rc.listed = r < kListOut ? 1 : 0;
        rc.pad = 0;
        cuts[row] = rc;
        if (n_kept_out != nullptr) n_kept_out[row] = r + 1;
      } else {
        open_rows[atomicAdd(n_open, 1)] = (int32_t)row;
      }
    }
  }
  __syncthreads();
  if (tid < s_kept && s_kept <= kListOut) lists[row * kListOut + tid] = s_sorted[tid];
}

// ---- the cut of a row from counts per key: a cluster of kC CTAs per row --------------------------------------
struct KeyCut {  // the last token kept: a key, and how many of the tokens with that key
  int32_t key;         // key16
  uint32_t j;          // tokens of the key that are kept (0: not found here)
  uint32_t cnt_key;    // tokens of the key
  uint32_t cnt_above;  // tokens with a larger key
  u64 mass_above;      // their mass
  u64 w_key;           // mass of one token of the key
};

struct Xch {  // what a CTA tells the others in one exchange
  u64 mass;
  uint32_t cnt;
  int32_t key;
  KeyCut cut;
};

struct WindowShared {
  uint32_t cnt[kWin];  // counts of this CTA's tokens
  Xch xch[2];          // one for even, one for odd exchanges: a slot is written again only after every CTA has left the
                       // barrier of the exchange in between, hence has read it
  u64 w64[kWT / 32];
  uint32_t w32[kWT / 32];
  int32_t wi[kWT / 32];
};

// Counts cover kWin keys at a time.  The usual ones are fixed: position 0 is the largest key below 2^8, position 4095
// that of 2^-24, then -2^-24 down to above -2^8: one pass without branches, about nine instructions a token, and nothing
// to know in advance.  Tokens between -2^-24 and 2^-24 are counted as one group between positions 4095 and 4096: with a
// row maximum of at least 2 their masses are all that of 0 (x - m rounds to -m).  Where the cut falls into that group, the
// maximum is smaller, or a finite value lies beyond 2^8, the row is counted again over windows of kWin consecutive keys,
// hi down to hi - kWin + 1, from the row maximum down (a NaN is never counted).
constexpr uint32_t kMag0 = (127 - 24) << 7;  // bf16 bits of 2^-24
__device__ __forceinline__ int32_t fixed_key16(int pos) {
  return pos < 4096 ? (int32_t)kMag0 + 4095 - pos : -((int32_t)kMag0 + pos - 4096);
}
struct Window {
  int32_t hi;
  int32_t next_hi;     // the largest key below the window that occurs in the row; kNoKey if none
  uint32_t cnt_above;
  u64 mass_above;
  uint32_t cnt;        // tokens inside
  u64 mass;            // their mass
};

// The row is cut into kC contiguous shares, CTA rank order being index order; a share sits in shared memory when it fits
// (cached != 0), else every pass reads it from L2.  All exchanged values are the same in every CTA, so every CTA takes the
// same way through the cluster barriers.  Bound: the instructions of the count pass (about ten a token) and a chain of five
// cluster barriers.
template <int kC>
__global__ void __launch_bounds__(kWT, 2)
filter_window_kernel(const uint16_t *__restrict__ logits, int64_t row_stride, int32_t vocab, float k_log2, int32_t top_k, float top_p,
                     RowCut *__restrict__ cuts, int32_t *__restrict__ n_kept_out, const int32_t *__restrict__ n_open,
                     const int32_t *__restrict__ open_rows, int n_all, int cached, int n_min, int n_max) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  WindowShared &sh = *reinterpret_cast<WindowShared *>(smem_raw);
  uint16_t *s_row = reinterpret_cast<uint16_t *>(smem_raw + (sizeof(WindowShared) + 15) / 16 * 16);
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = kC == 1 ? 0 : (int)cluster.block_rank();
  auto sync_all = [&]() {
    if (kC == 1) __syncthreads();
    else cluster.sync();
  };
  constexpr int kPW = kWin / kC, kPer = kPW / kWT;  // positions of this CTA and of one thread
  const int32_t share = share_of(vocab, kC), e0 = min(vocab, rank * share), e1 = min(vocab, e0 + share);
  const int32_t n_vec = (e1 - e0) >> 3, rem = (e1 - e0) & 7;
  const bool by_k = top_k > 0 && top_k < vocab, by_p = top_p < 1.f;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int n_rows = n_all > 0 ? n_all : *n_open;
  if (n_rows < n_min || n_rows > n_max) return;  // another cluster size takes this many rows
  int ph = 0;

  auto peer = [&](int r) -> const Xch * { return kC == 1 ? &sh.xch[ph] : cluster.map_shared_rank(&sh.xch[ph], r); };
  auto block_max = [&](int32_t v) -> int32_t {
    v = __reduce_max_sync(0xFFFFFFFFu, v);
    if (lane == 0) sh.wi[warp] = v;
    __syncthreads();
    const int32_t r = __reduce_max_sync(0xFFFFFFFFu, lane < kWT / 32 ? sh.wi[lane] : INT32_MIN);
    __syncthreads();
    return r;
  };
  // key: maximum over the cluster; cnt, mass: sums over the cluster and over the CTAs of lower rank.  Lane q of every warp
  // reads what CTA q says.
  struct Sums { int32_t key; uint32_t cnt, cnt_before; u64 mass, mass_before; };
  auto exchange = [&](int32_t key, uint32_t cnt, u64 mass) -> Sums {
    if (tid == 0) {
      sh.xch[ph].key = key;
      sh.xch[ph].cnt = cnt;
      sh.xch[ph].mass = mass;
    }
    sync_all();
    Sums r = {INT32_MIN, 0, 0, 0, 0};
    if (lane < kC) {
      const Xch *x = peer(lane);
      r.key = x->key;
      r.cnt = x->cnt;
      r.mass = x->mass;
    }
    r.cnt_before = __reduce_add_sync(0xFFFFFFFFu, lane < rank ? r.cnt : 0u);
    r.cnt = __reduce_add_sync(0xFFFFFFFFu, r.cnt);
    r.key = __reduce_max_sync(0xFFFFFFFFu, r.key);
    u64 all = 0;
#pragma unroll
    for (int q = 0; q < kC; ++q) {
      if (q == rank) r.mass_before = all;
      all += __shfl_sync(0xFFFFFFFFu, r.mass, q);
    }
    r.mass = all;
    ph ^= 1;
    return r;
  };
  auto clear_counts = [&]() {
    for (int i = tid; i < kWin / 4; i += kWT) reinterpret_cast<uint4 *>(sh.cnt)[i] = make_uint4(0, 0, 0, 0);
  };

  for (int at = (int)blockIdx.x / kC; at < n_rows; at += (int)gridDim.x / kC) {
    const int64_t row = n_all > 0 ? at : open_rows[at];
    const uint16_t *gp = logits + row * row_stride + e0;
    const uint16_t *rp = cached ? s_row : gp;

    // ---- the share into shared memory; counts of the fixed keys; the row maximum
    if (cached) {
      const uint32_t dst = (uint32_t)__cvta_generic_to_shared(s_row);
      for (int32_t vi = tid; vi < n_vec; vi += kWT)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + vi * 16), "l"(gp + (int64_t)vi * 8) : "memory");
      if (tid < rem) s_row[n_vec * 8 + tid] = gp[n_vec * 8 + tid];
    }
    clear_counts();
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    uint32_t mx = kNegInf2;
    uint32_t far = 0;  // largest distance from the first fixed magnitude: from 4096 on not among them
    const uint32_t cnt_mid = (uint32_t)__cvta_generic_to_shared(sh.cnt) + 4096 * 4;
    auto count = [&](uint32_t mag4, int32_t sign) {  // 4 x the magnitude's bits; 0 or -1
      const uint32_t t4 = mag4 - 4 * kMag0;
      const uint32_t at = cnt_mid + ((t4 ^ ~(uint32_t)sign) & ~3u);  // 4096 + t, or 4095 - t when positive
      if (t4 < 4 * 4096u) asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(at) : "memory");
      far = max(far, t4);
    };
    constexpr int kFly = kC >= 4 ? 1 : 4;  // loads in flight: the share of a small cluster may come from HBM here
    for (int32_t v0 = tid; v0 < n_vec; v0 += kFly * kWT) {
      uint4 v[kFly];
#pragma unroll
      for (int k = 0; k < kFly; ++k)
        if (v0 + k * kWT < n_vec) v[k] = reinterpret_cast<const uint4 *>(rp)[v0 + k * kWT];
#pragma unroll
      for (int k = 0; k < kFly; ++k)
        if (v0 + k * kWT < n_vec) {
          mx = max_bf2(mx, max_bf2(max_bf2(v[k].x, v[k].y), max_bf2(v[k].z, v[k].w)));
          const uint32_t w[4] = {v[k].x, v[k].y, v[k].z, v[k].w};
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            count((w[j] << 2) & 0x1FFFCu, (int32_t)(w[j] << 16) >> 31);
            count((w[j] >> 14) & 0x1FFFCu, (int32_t)w[j] >> 31);
          }
        }
    }
    float top = fmaxf(lo_f(mx), hi_f(mx));
    if (tid < rem) {
      const uint32_t u = rp[n_vec * 8 + tid];
      count((u << 2) & 0x1FFFCu, (int32_t)(u << 16) >> 31);
      top = fmaxf(top, __uint_as_float(u << 16));
    }
    int odd = far >= 4 * 4096u ? 1 : 0;
    uint32_t n_zero = 0, zeros_here = 0;  // tokens of the middle group
    if (__syncthreads_or(odd)) {  // -inf and NaN do not matter (they have no mass), other values do
      odd = 0;
      auto look = [&](uint32_t u) {
        const uint32_t mag = u & 0x7FFFu;
        n_zero += mag < kMag0 ? 1u : 0u;
        if (mag >= kMag0 + 4096u && (mag < 0x7F80u || u == 0x7F80u)) odd = 1;
      };
#pragma unroll 1
      for (int32_t vi = tid; vi < n_vec; vi += kWT) {
        const uint4 v = reinterpret_cast<const uint4 *>(rp)[vi];
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          look(w[j] & 0xFFFFu);
          look(w[j] >> 16);
        }
      }
      if (tid < rem) look(rp[n_vec * 8 + tid]);
      odd = __syncthreads_or(odd);
      block_scan<kWT, uint32_t>(n_zero, sh.w32, zeros_here);
    }
    const Sums first = exchange(block_max(key32(__float_as_uint(top))), zeros_here, odd ? 1 : 0);
    const float m = fmaxf(__uint_as_float(f_of_key16(first.key >> 16)), -3.0e38f);  // finite: a row without a finite logit
    const int32_t key_top = key32(__float_as_uint(m)) >> 16;

    // ---- the cut
    KeyCut cut;
    cut.j = 0;
    bool have_cut = false;
    uint32_t n_kept_all = (uint32_t)vocab;
    u64 w_k = 0, t = 0;  // mass of what top-k keeps; the mass top-p's cut has to reach
    // rank r stays iff the mass ranked before it is below top_p W_k: the last one kept is the first rank at which the
    // mass, itself included, reaches t
    auto target_of = [&](u64 w) -> u64 {
      const double t_d = ceil((double)top_p * (double)w);
      return min(t_d < 1.0 ? 1ull : (u64)t_d, w);
    };
    const uint32_t zeros = first.cnt;
    bool fixed = first.mass == 0 && first.key > (-32640 * 65536) && (zeros == 0 || m >= 2.f);  // some finite logit, and all of them counted
    bool counting = by_k;   // looking for the k-th token; after it, or without it, for the mass t
    bool whole = !by_k;     // the first pass also gives the mass of the whole row
    Window win;
    win.hi = key_top;
    win.next_hi = kNoKey;
    win.cnt_above = 0;
    win.mass_above = 0;
    bool search = true;
#pragma unroll 1
    while (search) {
      u64 mass_below = 0;
      if (!fixed) {
        clear_counts();
        __syncthreads();
        int32_t nh = kNoKey;
        u64 rest = 0, rest_all = 0;
        const int32_t hi32 = win.hi * 65536;
        auto count_in = [&](uint32_t f) {
          const int32_t k32 = key32(f);
          const float x = __uint_as_float(f);
          if (k32 <= hi32 && x == x) {  // keys above the window were counted by an earlier pass
            const uint32_t d = ((uint32_t)hi32 - (uint32_t)k32) >> 16;
            if (d < (uint32_t)kWin) {
              atomicAdd(&sh.cnt[d], 1u);
            } else {
              nh = max(nh, k32);
              if (whole) rest += wfix_of(f, m, k_log2);
            }
          }
        };
#pragma unroll 1
        for (int32_t vi = tid; vi < n_vec; vi += kWT) {
          const uint4 v = reinterpret_cast<const uint4 *>(rp)[vi];
          const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll 1
          for (int j = 0; j < 4; ++j) {
            const uint32_t x = j == 0 ? w[0] : j == 1 ? w[1] : j == 2 ? w[2] : w[3];
            count_in(x << 16);
            count_in(x & 0xFFFF0000u);
          }
        }
        if (tid < rem) count_in((uint32_t)rp[n_vec * 8 + tid] << 16);
        if (whole) block_scan<kWT, u64>(rest, sh.w64, rest_all);
        const Sums below = exchange(block_max(nh), 0, rest_all);  // (its barrier also makes the counts visible to the cluster)
        win.next_hi = below.key == kNoKey ? kNoKey : below.key >> 16;
        mass_below = below.mass;
      }
      // every CTA sums the kPW positions it is given over the cluster; this thread has kPer of them, from pos0
      const int pos0 = rank * kPW + tid * kPer;
      auto key_of = [&](int i) -> int32_t { return fixed ? fixed_key16(pos0 + i) : win.hi - (pos0 + i); };
      auto w_of = [&](int i) -> u64 { return wfix_of(f_of_key16(key_of(i)), m, k_log2); };
      uint32_t c[kPer], c_sum = 0, c_all;
      u64 m_sum = 0, m_all;
#pragma unroll
      for (int i = 0; i < kPer; ++i) c[i] = 0;
#pragma unroll
      for (int q = 0; q < kC; ++q) {
        const uint32_t *rc = (kC == 1 ? sh.cnt : cluster.map_shared_rank(sh.cnt, q)) + pos0;
#pragma unroll
        for (int i = 0; i < kPer; ++i) c[i] += rc[i];
      }
#pragma unroll
      for (int i = 0; i < kPer; ++i)
        if (c[i] != 0) {
          c_sum += c[i];
          m_sum += (u64)c[i] * w_of(i);  // all tokens of a key weigh the same
        }
      uint32_t c_excl = block_scan<kWT, uint32_t>(c_sum, sh.w32, c_all) - c_sum;
      u64 m_excl = block_scan<kWT, u64>(m_sum, sh.w64, m_all) - m_sum;
      const Sums sums = exchange(0, c_all, m_all);  // (after it the counts may be cleared again)
      c_excl += sums.cnt_before;
      m_excl += sums.mass_before;
      win.cnt = sums.cnt;
      win.mass = sums.mass;
      if (fixed && zeros != 0) {
        const u64 z_mass = zeros * wfix_of(0, m, k_log2);
        if (pos0 >= 4096) {
          c_excl += zeros;
          m_excl += z_mass;
        }
        win.cnt += zeros;
        win.mass += z_mass;
      }
      if (whole) {
        whole = false;
        w_k = win.mass + mass_below;
        t = target_of(w_k);
        if (!by_p || w_k == 0) break;
      }
      if (fixed && counting && (uint32_t)top_k > win.cnt) {  // fewer finite logits than k
        fixed = false;
        continue;
      }
      // what lies here?  First the k-th token, then, perhaps in the same window, the mass t.
#pragma unroll 1
      for (;;) {
        const bool hit = counting ? (uint32_t)top_k <= win.cnt_above + win.cnt : t <= win.mass_above + win.mass;
        if (hit) {
          if (tid == 0) sh.xch[ph].cut.j = 0;
          __syncthreads();
          const uint32_t k_rel = (uint32_t)top_k - win.cnt_above;
          const u64 t_rel = t - win.mass_above;
          if (counting ? (c_excl < k_rel && k_rel <= c_excl + c_sum) : (m_sum > 0 && m_excl < t_rel && t_rel <= m_excl + m_sum)) {
            uint32_t cnt = c_excl;
            u64 mass = m_excl;
            bool done = false;
#pragma unroll
            for (int i = 0; i < kPer; ++i)
              if (c[i] != 0 && !done) {
                const u64 w = w_of(i);
                if (counting ? (cnt + c[i] >= k_rel) : (w > 0 && mass + (u64)c[i] * w >= t_rel)) {
                  KeyCut r;
                  r.key = key_of(i);
                  r.cnt_key = c[i];
                  r.cnt_above = win.cnt_above + cnt;
                  r.mass_above = win.mass_above + mass;
                  r.w_key = w;
                  r.j = counting ? (k_rel - cnt) : (uint32_t)((t_rel - mass + w - 1) / w);
                  sh.xch[ph].cut = r;
                  done = true;
                }
                cnt += c[i];
                mass += (u64)c[i] * w;
              }
          }
          sync_all();
          const unsigned has = __ballot_sync(0xFFFFFFFFu, lane < kC && peer(lane & (kC - 1))->cut.j != 0);
          if (has == 0) {  // it lies in the middle group: start over with windows
            ph ^= 1;
            fixed = have_cut = false;
            counting = by_k;
            whole = !by_k;
            break;
          }
          const KeyCut found = peer(__ffs(has) - 1)->cut;
          const uint32_t j_k = have_cut && found.key == cut.key ? cut.j : found.j;
          cut = found;
          cut.j = min(cut.j, j_k);  // top-p keeps no more of a key than top-k did (implied by t <= W_k)
          have_cut = true;
          ph ^= 1;
        }
        if (counting && (hit || win.next_hi == kNoKey)) {
          if (hit) {
            w_k = cut.mass_above + (u64)cut.j * cut.w_key;
          } else {  // fewer than k tokens that are numbers: every window was visited, nothing is cut
            w_k = win.mass_above + win.mass;
            n_kept_all = win.cnt_above + win.cnt;
          }
          counting = false;
          search = by_p && w_k > 0;
          t = target_of(w_k);
          if (search && t > win.mass_above) continue;  // look for it in this window first
          win.hi = key_top;  // the top-k search went past it: start again from the top
          win.cnt_above = 0;
          win.mass_above = 0;
          break;
        }
        if (hit || win.next_hi == kNoKey) {
          search = false;
          break;
        }
        win.cnt_above += win.cnt;
        win.mass_above += win.mass;
        win.hi = win.next_hi;
        break;
      }
    }
    const bool split = have_cut && cut.j < cut.cnt_key;
    if (rank == 0 && tid == 0) {
      RowCut *rc = cuts + row;
      rc->m = m;
      rc->cut_key = have_cut ? cut.key * 65536 : kNoKey;
      if (!split) rc->cut_idx = INT32_MAX;  // else whoever holds the last token kept of the group writes it
      rc->n_kept = have_cut ? (int32_t)(cut.cnt_above + cut.j) : (int32_t)n_kept_all;
      rc->z_fix = have_cut ? cut.mass_above + (u64)cut.j * cut.w_key : w_k;
      rc->listed = 0;
      if (n_kept_out != nullptr) n_kept_out[row] = have_cut ? (int32_t)(cut.cnt_above + cut.j) : (int32_t)n_kept_all;
    }
    // ---- only when the cut splits a group of equal keys (the usual thing with bf16): the index of the last one kept.
    //      Warps own contiguous runs of vectors (the last one the ragged end too); equality of the values is equality of
    //      the keys.
    if (split) {
      const uint32_t cb = f_of_key16(cut.key) >> 16, pat = cb | (cb << 16);
      const int32_t n_all_vec = n_vec + (rem ? 1 : 0), per = (n_all_vec + kWT / 32 - 1) / (kWT / 32);
      const int32_t v0 = min(n_all_vec, warp * per), v1 = min(n_all_vec, v0 + per);
      auto vec = [&](int32_t vi) -> uint4 {
        return vi < n_vec ? reinterpret_cast<const uint4 *>(rp)[vi] : vi < n_all_vec ? ragged_vec(rp, n_vec, rem) : make_uint4(kNegInf2, kNegInf2, kNegInf2, kNegInf2);
      };
      auto equal = [&](uint32_t x) -> uint32_t {  // 16 ones per value
        return __heq2_mask(*reinterpret_cast<const __nv_bfloat162 *>(&x), *reinterpret_cast<const __nv_bfloat162 *>(&pat));
      };
      auto equals = [&](const uint4 &v) -> uint32_t { return (__popc(equal(v.x)) + __popc(equal(v.y)) + __popc(equal(v.z)) + __popc(equal(v.w))) >> 4; };
      uint32_t mine = 0, all;
#pragma unroll 4
      for (int32_t vi = v0 + lane; vi < v1; vi += 32) mine += equals(vec(vi));
      mine = __reduce_add_sync(0xFFFFFFFFu, mine);
      uint32_t before = block_scan<kWT, uint32_t>(lane == 0 ? mine : 0, sh.w32, all);
      before = __shfl_sync(0xFFFFFFFFu, before, 0) - mine;  // in the warps in front of this one ...
      before += exchange(0, all, 0).cnt_before;             // ... and in the CTAs in front
      if (before < cut.j && cut.j <= before + mine) {
#pragma unroll 1
        for (int32_t vi = v0 + lane; __any_sync(0xFFFFFFFFu, vi < v1); vi += 32) {
          const uint4 v = vec(vi < v1 ? vi : n_all_vec);
          const uint32_t c = equals(v);
          uint32_t incl = c;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += y;
          }
          const uint32_t upto = before + incl;
          if (upto - c < cut.j && cut.j <= upto) {
            uint32_t seen = upto - c;
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int j = 0; j < 8; ++j)
              if ((equal(w[j >> 1]) & ((j & 1) ? 0x10000u : 1u)) && ++seen == cut.j) cuts[row].cut_idx = e0 + vi * 8 + j;
          }
          before = __shfl_sync(0xFFFFFFFFu, upto, 31);
          if (before >= cut.j) break;
        }
      }
    }
    sync_all();  // nobody leaves, or starts on the next row, while its shared memory is being read
  }
}

// ---- acceptance: a cluster of kC CTAs per branch ----------------------------------------------------------
// Every CTA walks the chain.  When the stop row's kept tokens are listed, the first CTA draws from the list; else the kept
// masses of the row's slices are summed first, each CTA taking a share of the row.
template <int kC>
__global__ void __launch_bounds__(kAT)
accept_filtered_kernel(const uint16_t *__restrict__ logits, int64_t row_stride, int32_t vocab, float k_log2,
                       const RowCut * cuts, const u64 * lists, int n_slices,
                       const int32_t *__restrict__ draft_ids, const int32_t *__restrict__ cu_draft,
                       const float *__restrict__ u_accept, const float *__restrict__ u_final, int32_t *__restrict__ n_accept,
                       int32_t *__restrict__ final_id, float *__restrict__ p_draft) {
  __shared__ u64 s_mass[kMaxSlices], s_w64[kAT / 32];
  __shared__ int32_t s_idx[kListOut];
  __shared__ u64 s_before, s_total;
  __shared__ int s_n, s_slice;
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  const int b = blockIdx.x / kC, rank = kC == 1 ? 0 : (int)cluster.block_rank(), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // Only the cuts come from the kernels launched just before, and the last of those let this one start when everything older
  // had finished: all else is fetched while it drains (with the commit behind it, 51 rows and top-p alone 35.4 -> 34.9 us).
  const int32_t d0 = cu_draft[b], L = cu_draft[b + 1] - d0, r0 = d0 + b;
  const double u_fin = (double)u_final[b];
  __shared__ int32_t s_draft[kAT];   // the first kAT drafts and their logits
  __shared__ uint32_t s_logit[kAT];
  __shared__ RowCut s_cut[kAT];      // and the cuts of the first kAT rows
  auto draft_of = [&](int i, int32_t &d, uint32_t &f) {
    d = draft_ids[d0 + i];
    f = d >= 0 && d < vocab ? (uint32_t)logits[(int64_t)(r0 + i) * row_stride + d] << 16 : 0u;
  };
  float u_first = 0.f;
  if (tid < L) {
    int32_t d;
    uint32_t f;
    draft_of(tid, d, f);
    s_draft[tid] = d;
    s_logit[tid] = f;
    u_first = u_accept[d0 + tid];
  }
  if (tid == 0) {
    s_n = L;
    s_slice = -1;
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  __syncthreads();

  // ---- acceptance chain: draft i passes iff u_i < P'_i(d_i); the first one that does not ends it
  for (int i = tid; i <= L; i += kAT) {
    const RowCut rc = cut_behind_wait(cuts + r0 + i);
    if (i < kAT) s_cut[i] = rc;
    if (i == L) break;  // no draft for the last row
    int32_t d;
    uint32_t f;
    if (i == tid) {
      d = s_draft[tid];
      f = s_logit[tid];
    } else {
      draft_of(i, d, f);
    }
    const float u = i == tid ? u_first : u_accept[d0 + i];
    float p = 0.f;
    if (d >= 0 && d < vocab && rc.z_fix > 0) {
      if (is_kept(key32(f), d, rc)) p = (float)wfix_of(f, rc.m, k_log2) / (float)rc.z_fix;
    }
    if (p_draft != nullptr && rank == 0) p_draft[d0 + i] = p;
    if (!(u < p)) atomicMin(&s_n, i);
  }
  __syncthreads();
  const int n = s_n;
  if (rank == 0 && tid == 0) n_accept[b] = n;

  // ---- the final token: inverse CDF over the kept tokens of the stop row, the rejected one removed
  const RowCut rc = n < kAT ? s_cut[n] : cut_behind_wait(cuts + r0 + n);
  const bool listed = rc.listed != 0;  // every CTA of the cluster sees the same
  if (listed && rank != 0) return;
  const uint16_t *rp = logits + (int64_t)(r0 + n) * row_stride;
  int32_t dead = -1;
  u64 w_dead = 0;
  if (n < L) {
    int32_t d;
    uint32_t f;
    if (n < kAT) {
      d = s_draft[n];
      f = s_logit[n];
    } else {
      draft_of(n, d, f);
    }
    if (d >= 0 && d < vocab) {
      if (is_kept(key32(f), d, rc)) {
        dead = d;
        w_dead = wfix_of(f, rc.m, k_log2);
      }
    }
  }
  const u64 total = rc.z_fix - w_dead;
  // smallest v whose cumulative mass exceeds u * total; the masses are integers, so "exceeds floor(u * total)"
  u64 target = (u64)(u_fin * (double)total);
  if (total > 0 && target >= total) target = total - 1;
  if (listed) {
    // the smallest index whose cumulative mass exceeds the target: every kept token sums those up to its own index
    const u64 *list = lists + (int64_t)(r0 + n) * kListOut;
    for (int i = tid; i < rc.n_kept; i += kAT) {
      const u64 e = ld_behind_wait(list + i);
      s_idx[i] = cand_idx(e);
      s_mass[i] = s_idx[i] == dead ? 0 : wfix_of(f_of_key16(cand_key16(e)), rc.m, k_log2);
    }
    __syncthreads();
    for (int i = tid; i < rc.n_kept; i += kAT) {
      u64 upto = 0;
#pragma unroll 4
      for (int j = 0; j < rc.n_kept; ++j) upto += s_idx[j] <= s_idx[i] ? s_mass[j] : 0;
      if (s_mass[i] > 0 && upto - s_mass[i] <= target && target < upto) final_id[b] = s_idx[i];
    }
    if (total == 0 && tid == 0) final_id[b] = 0;  // a row without mass
    return;
  }
  const int slice_len = slice_len_of(vocab);
  const int spc = (n_slices + kC - 1) / kC, sl0 = min(n_slices, rank * spc), n_here = min(spc, n_slices - sl0);
  const float cut_x = rc.cut_key == kNoKey ? -INFINITY : __uint_as_float(f_of_key16(rc.cut_key >> 16));
  for (int i0 = warp; i0 < n_here; i0 += kSlicesInFlight * (kAT / 32)) {  // a warp per slice, a lane per vector, several slices in flight
    u64 mass[kSlicesInFlight] = {};
    for (int32_t off = lane * 8; off < slice_len; off += 256) {
      uint4 v[kSlicesInFlight];
#pragma unroll
      for (int q = 0; q < kSlicesInFlight; ++q) {
        const int32_t e = (sl0 + i0 + q * (kAT / 32)) * slice_len + off;
        v[q] = make_uint4(kNegInf2, kNegInf2, kNegInf2, kNegInf2);
        if (i0 + q * (kAT / 32) < n_here && e < vocab)
          v[q] = e + 8 <= vocab ? __ldg(reinterpret_cast<const uint4 *>(rp + e)) : ragged_vec(rp, vocab >> 3, vocab & 7);
      }
#pragma unroll
      for (int q = 0; q < kSlicesInFlight; ++q) {
        const int32_t e = (sl0 + i0 + q * (kAT / 32)) * slice_len + off;
        const uint32_t w[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const uint32_t f = (j & 1) ? (w[j >> 1] & 0xFFFF0000u) : (w[j >> 1] << 16);
          const float x = __uint_as_float(f);
          if (x > cut_x || (x == cut_x && e + j <= rc.cut_idx)) mass[q] += wfix_of(f, rc.m, k_log2);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < kSlicesInFlight; ++q) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mass[q] += __shfl_xor_sync(0xFFFFFFFFu, mass[q], o);
      if (lane == 0 && i0 + q * (kAT / 32) < n_here) s_mass[i0 + q * (kAT / 32)] = mass[q];
    }
  }
  __syncthreads();
  const int spt = (n_here + kAT - 1) / kAT;  // slices per thread, consecutive
  u64 w[kMaxSlices / kAT], mine = 0, all, base = 0;
#pragma unroll
  for (int i = 0; i < kMaxSlices / kAT; ++i) {
    const int at = tid * spt + i;
    w[i] = 0;
    if (i < spt && at < n_here) {
      w[i] = s_mass[at];
      if (dead >= 0 && sl0 + at == dead / slice_len) w[i] -= w_dead;
    }
    mine += w[i];
  }
  u64 cum = block_scan<kAT, u64>(mine, s_w64, all) - mine;
  if (kC > 1) {
    if (tid == 0) s_total = all;
    cluster.sync();
    for (int q = 0; q < rank; ++q) base += *cluster.map_shared_rank(&s_total, q);
  }
  cum += base;
#pragma unroll
  for (int i = 0; i < kMaxSlices / kAT; ++i) {
    if (w[i] > 0 && cum <= target && target < cum + w[i]) {
      s_slice = sl0 + tid * spt + i;
      s_before = cum;
    }
    cum += w[i];
  }
  __syncthreads();
  const int sl = s_slice;
  if (sl >= 0) {  // inside the slice: one token per thread at a time
    u64 upto0 = s_before;
    for (int32_t x0 = sl * slice_len; x0 < min(vocab, (sl + 1) * slice_len); x0 += kAT) {
      const int32_t e = x0 + tid;
      u64 x = 0;
      if (e < vocab && e != dead) {
        const uint32_t f = (uint32_t)rp[e] << 16;
        if (is_kept(key32(f), e, rc)) x = wfix_of(f, rc.m, k_log2);
      }
      const u64 upto = upto0 + block_scan<kAT, u64>(x, s_w64, all);
      if (x > 0 && upto - x <= target && target < upto) final_id[b] = e;
      upto0 += all;
    }
  }
  if (total == 0 && rank == 0 && tid == 0) final_id[b] = 0;  // a row without mass
  if (kC > 1) cluster.sync();  // nobody leaves while its total is being read
}

// Vectors per group when k_sel leading tokens are looked for: the most, up to 8, that still make many more groups than that.
// Short rows have few groups anyway and go from 8 to 1.
int group_vecs(int32_t vocab, int k_sel) {
  for (const int v : {8, 4, 2})
    if (vocab / (8 * v) >= 4 * (int64_t)k_sel && (v == 8 || vocab > 65536)) return v;
  return 1;
}

struct ScratchLayout {
  size_t cuts, lists, maxima, stats, open, bytes;
  int n_chunks, n_slices;
};
ScratchLayout filter_layout(int32_t vocab, int32_t n_rows) {
  ScratchLayout s;
  s.n_chunks = (int)(((int64_t)vocab + kChunk - 1) / kChunk);
  s.n_slices = (int)(((int64_t)vocab + slice_len_of(vocab) - 1) / slice_len_of(vocab));
  size_t off = 0;
  auto take = [&](size_t n) {
    const size_t o = off;
    off += (n + 15) / 16 * 16;
    return o;
  };
  s.cuts = take((size_t)n_rows * sizeof(RowCut));
  s.lists = take((size_t)n_rows * kListOut * sizeof(u64));
  // in the smallest groups a top_k can ask for
  s.maxima = take((size_t)n_rows * s.n_chunks * (32 * kVec / group_vecs(vocab, std::min(vocab, kSelMax))) * sizeof(uint16_t));
  s.stats = take((size_t)n_rows * s.n_chunks * sizeof(float2));
  s.open = take(((size_t)n_rows + 2) * sizeof(int32_t));  // how many, which, and whether the probe gave up
  s.bytes = off;
  return s;
}

struct WindowShape {
  int cluster;
  size_t smem;
  bool cached;
  double us;  // estimated time
};
// Cluster size for n_rows rows through the windows: the one with the smallest estimate.  Two CTAs fit an SM.  A round of rows
// takes `two` with two CTAs on every SM and `one` with one, in us and us per 1000 tokens of a CTA's share, fitted to whole calls
// on flat rows less the 10 us of the draw (single CTAs, pairs, fours: 136 rows of 152064 tokens 63, 52 and 53 us, 340 of them
// 147, 142 and 158, 408 154, 143 and 198, 612 225, 232 and 316; 340 of 50000 57, 84 and 124; 68 of 20000 11, 21 and 18; eights:
// 17 of 152064 17 us, 272 223).  136 CTAs in pairs already share SMs, and so count as nearly all.  On other rows all are
// faster, single CTAs the most.
double window_us(const lr_ctx *ctx, int c, int64_t n_rows, bool flat) {
  const int64_t clusters = std::max(1, ctx->sm_count * 2 / c);
  const double k = share_of(ctx->model.vocab, c) * 1e-3;
  const double one = c == 1 ? 6 + 0.375 * k : c == 2 ? 10 + 0.34 * k : c == 4 ? 7.3 + 0.36 * k : 12 + 0.24 * k;
  const double two = c == 1 ? 11 + 0.467 * k : c == 2 ? 19.5 + 0.4 * k : c == 4 ? 26 + 0.23 * k : 22.8 + 0.41 * k;
  const int64_t rounds = n_rows / clusters, rest = n_rows % clusters;
  const double sms = ctx->sm_count, ctas = (double)(rest * c);
  const double full = c == 2 && rounds == 0 ? (ctas - 0.7 * sms) / (0.3 * sms) : (ctas - sms) / sms;
  const double all = (double)rounds * two + (rest ? one + std::min(1.0, std::max(0.0, full)) * (two - one) : 0.0);
  return c == 1 && !flat ? 0.92 * all : all;
}
WindowShape window_shape(const lr_ctx *ctx, int64_t n_rows, bool flat = false) {
  WindowShape best = {};
  for (const int c : {8, 4, 2, 1}) {
    const size_t fixed = (sizeof(WindowShared) + 15) / 16 * 16, share = (size_t)share_of(ctx->model.vocab, c) * 2;
    WindowShape w;
    w.cluster = c;
    w.cached = fixed + share <= kWindowSmemMax;
    w.smem = fixed + (w.cached ? share : 0);
    w.us = window_us(ctx, c, n_rows, flat);
    if (best.cluster == 0 || w.us < best.us) best = w;
  }
  return best;
}

template <class... KArgs, class... Args>
cudaError_t launch_clusters(void (*kernel)(KArgs...), int kc, int clusters, int threads, size_t smem, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(kc * clusters));
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)kc;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

}  // namespace

int init_accept_filter_kernels() {
  for (auto kernel : {filter_window_kernel<8>, filter_window_kernel<4>, filter_window_kernel<2>, filter_window_kernel<1>})
    if (int rc = cuda_fail(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWindowSmemMax),
                           "filter_window_kernel shared-memory attribute"))
      return rc;
  return LR_OK;
}

size_t accept_filtered_scratch_bytes(int32_t vocab, int32_t n_rows) { return filter_layout(vocab, n_rows).bytes; }

int launch_accept_filtered(lr_ctx *ctx, const void *logits, int64_t stride, const int32_t *drafts, const int32_t *cu_draft,
                           int32_t n_branch, int32_t n_rows, float temperature, int32_t top_k, float top_p,
                           const float *u_accept, const float *u_final, int32_t *n_accept, int32_t *final_id, float *p_draft,
                           int32_t *n_kept, void *scratch, cudaStream_t s) {
  const int32_t vocab = ctx->model.vocab;
  const float k_log2 = 1.4426950408889634f / temperature;
  const ScratchLayout L = filter_layout(vocab, n_rows);
  unsigned char *base = reinterpret_cast<unsigned char *>(scratch);
  auto *lg = reinterpret_cast<const uint16_t *>(logits);
  auto *cuts = reinterpret_cast<RowCut *>(base + L.cuts);
  auto *lists = reinterpret_cast<u64 *>(base + L.lists);
  auto *maxima = reinterpret_cast<uint16_t *>(base + L.maxima);
  auto *stats = reinterpret_cast<float2 *>(base + L.stats);
  auto *n_open = reinterpret_cast<int32_t *>(base + L.open);
  const bool by_k = top_k > 0 && top_k < vocab, by_p = top_p < 1.f;
  const int k_sel = by_k ? top_k : kSelTopP;
  const int gv = group_vecs(vocab, k_sel);
  // With too few groups of 8 tokens as well the bound is too low to be of use, unless the whole row fits the list of candidates.
  const bool enough = vocab / 8 >= 4 * (int64_t)k_sel || vocab <= kListCap;
  // Can a few leading tokens decide a row?  With a small top-k always: 16 us against 37 us through the windows for 51 rows
  // of 152064 tokens and top-k 20, 46 against 160 and more for 612.  Reading and ranking the groups of a larger one costs
  // about 10 us and 0.055 per k while every row has an SM, and more behind that (272 rows, top-k 200, 400 and 800: 49, 76 and
  // 96 us; 612 rows 84, 117 and 147; windows 93 and 184).  With top-p alone they mostly do, but the rows they leave open (taken
  // to be one in five) go through the windows all the same, and when a kept set is half the vocabulary that is every row.  So
  // they are tried on a few rows first and, if most of those stay open, on no more.  Rows of 152064 tokens, peaked, as a
  // language model's, flat: 408 of them 77, 134 and 183 us (windows alone 110, 138 and 153 to 165), 612 of them 106, 170 and
  // 262 (150, 177 and 236).
  WindowShape w = window_shape(ctx, n_rows);
  const WindowShape w_open = window_shape(ctx, (n_rows + 4) / 5, true);
  const double us_scan = (double)n_rows * vocab * 2 / 5.5e6;
  const int n_probe = !by_k && n_rows >= 4 * kProbeRows ? kProbeRows : 0;
  const double us_rank = gv == 1 ? (6.0 + 0.1 * top_k) * ((n_rows + 5 * ctx->sm_count - 1) / (5 * ctx->sm_count))
                                 : (10.0 + 0.055 * top_k) * (1.0 + 0.27 * std::max(0.0, (double)n_rows / ctx->sm_count - 1.0));
  const double us_candidates = by_k ? 12.0 + us_scan + us_rank
                                    : 24.0 + (n_probe ? 12.0 : 0.0) + us_scan + 0.02 * n_rows + w_open.us;
  const bool candidates = enough && (by_k ? top_k <= kSelMax : by_p) && ((by_k && top_k <= 128) || us_candidates < window_shape(ctx, n_rows, true).us);
  // The open rows are few or all of them; only the device knows.  Up to n_few rows take the shape for a few.
  WindowShape few = w;
  int n_few = n_rows;
  if (candidates) {
    auto scan = !by_k     ? (gv == 8 ? filter_scan_kernel<true, 8> : filter_scan_kernel<true, 1>)
                : gv == 8 ? filter_scan_kernel<false, 8>
                : gv == 4 ? filter_scan_kernel<false, 4>
                : gv == 2 ? filter_scan_kernel<false, 2>
                          : filter_scan_kernel<false, 1>;
    // Many vectors in flight pay where many groups are read (top-k 200, 272 rows of 152064 tokens: 61 and 49 us) or they come
    // from HBM (top-p, 408 peaked rows of 152064: 88 and 77 us, but 612 of 50000, which L2 holds, 63 and 66).
    const bool many = by_k ? top_k >= kManyFrom : (int64_t)n_rows * vocab * 2 > kManyBytes;
    auto cut = gv == 1            ? filter_cut_kernel<1, false>
               : gv == 8 && !many ? filter_cut_kernel<8, false>
               : gv == 8          ? filter_cut_kernel<8, true>
               : gv == 4          ? filter_cut_kernel<4, true>
                                  : filter_cut_kernel<2, true>;
    int32_t *gave_up = n_open + 1 + n_rows;
    const int64_t maxima_per_row = (int64_t)L.n_chunks * 32 * kVec / gv;
    auto settle = [&](int r0, int n, int32_t *verdict) -> int {
      const uint32_t total = (uint32_t)n * L.n_chunks;
      const unsigned grid = std::min((total + kWarps - 1) / kWarps, (uint32_t)(ctx->sm_count * kScanCtasPerSm));
      ctx->launches += 2;
      const uint16_t *from = lg + (int64_t)r0 * stride;
      uint16_t *to = maxima + r0 * maxima_per_row;
      float2 *to_stats = stats + (int64_t)r0 * L.n_chunks;
      // (also as the first kernel of a call it is set up while whatever is before it drains: 617 rows, top-k 20 and top-p 0.95, with
      // the commit of the call before 49.3 -> 47.9 us, 45 rows of 1081 tokens 18.6 -> 17.6)
      if (int rc = cuda_fail(launch_dependent(scan, dim3(grid), dim3(kT), 0, s, from, stride, vocab, k_log2, (uint32_t)L.n_chunks, total, to, to_stats,
                                              n_open, kProbeRows, verdict),
                             "filter_scan_kernel launch"))
        return rc;
      return cuda_fail(launch_dependent(cut, dim3((unsigned)n), dim3(kT), 0, s, lg, stride, vocab, k_log2, top_k, top_p, k_sel, L.n_chunks, maxima,
                                        stats, cuts, lists, n_kept, n_open, n_open + 1, r0, (const int32_t *)verdict),
                       "filter_cut_kernel launch");
    };
    if (n_probe)
      if (int rc = settle(0, n_probe, nullptr)) return rc;
    if (int rc = settle(n_probe, n_rows - n_probe, n_probe ? gave_up : nullptr)) return rc;
    few = by_k ? window_shape(ctx, 1) : w_open;  // after a top-k hardly ever a row is left
    if (n_probe) w = window_shape(ctx, n_rows, true);  // rows left open are mostly flat ones
    if (n_probe && few.cluster != w.cluster) {
      int lo = (n_rows + 4) / 5, hi = n_rows;  // `few` is the better one at lo, w at hi
      while (hi - lo > 1) {
        const int mid = lo + (hi - lo) / 2;
        if (window_us(ctx, few.cluster, mid, true) <= window_us(ctx, w.cluster, mid, true)) lo = mid;
        else hi = mid;
      }
      n_few = lo;
    }
  }
  auto windows = [&](const WindowShape &shape, int n_min, int n_max) -> int {
    auto kernel = shape.cluster == 8   ? filter_window_kernel<8>
                  : shape.cluster == 4 ? filter_window_kernel<4>
                  : shape.cluster == 2 ? filter_window_kernel<2>
                                       : filter_window_kernel<1>;
    const int clusters = std::max(1, ctx->sm_count * 2 / shape.cluster);
    ctx->launches++;
    return cuda_fail(launch_clusters(kernel, shape.cluster, candidates ? clusters : std::min(n_rows, clusters), kWT, shape.smem, s, lg, stride, vocab,
                                     k_log2, top_k, top_p, cuts, n_kept, n_open, n_open + 1, candidates ? 0 : n_rows, shape.cached ? 1 : 0, n_min, n_max),
                     "filter_window_kernel launch");
  };
  if (int rc = windows(few, 0, n_few)) return rc;
  if (n_few < n_rows)
    if (int rc = windows(w, n_few + 1, n_rows)) return rc;
  ctx->launches++;
  // one CTA per branch when there is no stop row to walk (hardly ever after the candidates of a small top-k) or it is short
  if ((candidates && by_k && top_k <= kListOut) || vocab <= 16384)
    return cuda_fail(launch_dependent(accept_filtered_kernel<1>, dim3((unsigned)n_branch), dim3(kAT), 0, s, lg, stride, vocab, k_log2, cuts, lists,
                                      L.n_slices, drafts, cu_draft, u_accept, u_final, n_accept, final_id, p_draft),
                     "accept_filtered_kernel launch");
  return cuda_fail(launch_clusters(accept_filtered_kernel<8>, 8, n_branch, kAT, 0, s, lg, stride, vocab, k_log2, cuts, lists, L.n_slices, drafts,
                                   cu_draft, u_accept, u_final, n_accept, final_id, p_draft),
                   "accept_filtered_kernel launch");
}

}  // namespace lr
