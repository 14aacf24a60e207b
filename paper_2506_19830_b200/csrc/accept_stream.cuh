// The streaming part of greedy acceptance, for the kernels that take part in it: a warp reduces a stretch of a logits row to
// (maximum, lowest index) and publishes it with one 64-bit atomicMax on the row's key; and what the keys say of a branch.
#pragma once

#include "lr_common.cuh"

namespace lr {

// Monotone map of a float (already NaN-free, -0 folded to +0) to an unsigned key.
__device__ __forceinline__ uint32_t order_key(float x) {
  uint32_t u = __float_as_uint(x == 0.0f ? 0.0f : x);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ uint4 ld_stream(const uint4 *p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

__device__ __forceinline__ __nv_bfloat162 as_bf2(uint32_t u) {
  __nv_bfloat162 r;
  *reinterpret_cast<uint32_t *>(&r) = u;
  return r;
}

__device__ __forceinline__ float bf_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf_hi(uint32_t u) { return __uint_as_float(u & 0xFFFF0000u); }

// NaN counts as -inf.
__device__ __forceinline__ float denan(float x) { return (x != x) ? -INFINITY : x; }

// max over the 8 bf16 of a vector; NaNs are ignored by the packed max (an all-NaN
// vector gives NaN, which then fails every "greater than" test).
__device__ __forceinline__ float vec_max(const uint4 &v) {
  __nv_bfloat162 a = __hmax2(as_bf2(v.x), as_bf2(v.y));
  __nv_bfloat162 b = __hmax2(as_bf2(v.z), as_bf2(v.w));
  a = __hmax2(a, b);
  uint32_t u = *reinterpret_cast<uint32_t *>(&a);
  return fmaxf(bf_lo(u), bf_hi(u));
}

// index (0..7) of the first element of v equal to x (x is the vector's max, not NaN)
__device__ __forceinline__ int first_equal(const uint4 &v, float x) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
  int idx = 7;
#pragma unroll
  for (int i = 3; i >= 0; --i) {
    if (bf_hi(w[i]) == x) idx = 2 * i + 1;
    if (bf_lo(w[i]) == x) idx = 2 * i;
  }
  return idx;
}

struct Best {
  float v;
  int32_t i;
};

__device__ __forceinline__ Best better(Best a, Best b) {
  // higher value wins; equal values: lower index wins
  if (b.v > a.v || (b.v == a.v && b.i < a.i)) return b;
  return a;
}

// What a launch streams: `total` units, n_chunks of them a row, one after another.
struct AcceptWork {
  const uint16_t *logits;
  int64_t row_stride;
  unsigned long long *scratch;  // [0] counters, [1..] row keys; zeros between calls
  int32_t vocab;
  uint32_t n_chunks, total;
};

// A unit: a stretch of kVec x 32 vectors of a row, one load instruction a lane and vector, all in flight together.
template <int kVec>
__device__ __forceinline__ void accept_load(const AcceptWork &w, uint32_t unit, int lane, uint4 (&v)[kVec]) {
  const uint32_t row = unit / w.n_chunks, c = unit - row * w.n_chunks;
  const int32_t n_vec = w.vocab >> 3, v0 = (int32_t)c * (32 * kVec) + lane;
  const uint4 *vp = reinterpret_cast<const uint4 *>(w.logits + (int64_t)row * w.row_stride);
#pragma unroll
  for (int k = 0; k < kVec; ++k)
    if (v0 + k * 32 < n_vec) v[k] = ld_stream(vp + v0 + k * 32);
}

// What a lane has of a unit: its largest logit and where that is first.
template <int kVec>
__device__ __forceinline__ Best accept_best(const AcceptWork &w, uint32_t unit, int lane, const uint4 (&v)[kVec]) {
  const uint32_t row = unit / w.n_chunks, c = unit - row * w.n_chunks;
  const int32_t n_vec = w.vocab >> 3, rem = w.vocab & 7, v0 = (int32_t)c * (32 * kVec) + lane;
  // Vectors are visited in increasing index order and only a strictly
  // greater maximum replaces the current one, so the earliest maximum is kept.
  Best best;
  best.v = -INFINITY;
  best.i = 0x7FFFFFFF;  // "owns no element": loses every tie
  uint4 bv = make_uint4(0, 0, 0, 0);
  int32_t bvi = -1;
#pragma unroll
  for (int k = 0; k < kVec; ++k) {
    const int32_t vi = v0 + k * 32;
    if (vi < n_vec) {
      const float m = denan(vec_max(v[k]));
      if (m > best.v || bvi < 0) {
        best.v = m;
        bv = v[k];
        bvi = vi;
      }
    }
  }
  // a maximum of -inf means every element is -inf or NaN: the first one wins
  if (bvi >= 0) best.i = bvi * 8 + (best.v == -INFINITY ? 0 : first_equal(bv, best.v));
  if (c == w.n_chunks - 1 && lane < rem) {  // ragged end of the row: up to 7 single elements
    const uint16_t *rp = w.logits + (int64_t)row * w.row_stride;
    Best t;
    t.v = denan(bf_lo((uint32_t)rp[n_vec * 8 + lane]));
    t.i = n_vec * 8 + lane;
    best = better(best, t);
  }
  return best;
}

// The best of a warp's lanes, to the row's key.
__device__ __forceinline__ void accept_publish(const AcceptWork &w, uint32_t row, int lane, Best best) {
  const uint32_t key = order_key(best.v), top = __reduce_max_sync(0xFFFFFFFFu, key);
  const uint32_t first = __reduce_min_sync(0xFFFFFFFFu, key == top ? (uint32_t)best.i : 0x7FFFFFFFu);
  if (lane == 0 && first != 0x7FFFFFFFu) atomicMax(w.scratch + 1 + row, ((unsigned long long)top << 32) | (unsigned long long)(0xFFFFFFFFu - first));
}

// Consecutive units: one atomic a row, not one a unit.
template <int kVec>
__device__ __forceinline__ void accept_run(const AcceptWork &w, uint32_t unit, uint32_t end, int lane) {
  while (unit < end) {
    const uint32_t row = unit / w.n_chunks, stop = min(end, (row + 1u) * w.n_chunks);
    Best best;
    best.v = -INFINITY;
    best.i = 0x7FFFFFFF;
    for (; unit < stop; ++unit) {
      uint4 v[kVec];
      accept_load(w, unit, lane, v);
      best = better(best, accept_best(w, unit, lane, v));
    }
    accept_publish(w, row, lane, best);
  }
}

// Longest matching prefix of a branch whose drafts are draft_ids[d0 .. d0 + L) and whose row keys start at `keys`, and its
// bonus token.  The rows are read eight at a time -- keys and drafts of a chunk are loaded together, so a chunk costs one round
// trip to L2 -- and the scan stops at the first mismatch.
__device__ __forceinline__ int accept_branch(const unsigned long long *keys, const int32_t *draft_ids, int32_t d0, int32_t L, int32_t &bonus) {
  int32_t n = L;
  bool found = false;
  bonus = 0;
  for (int32_t i0 = 0; i0 <= L && !found; i0 += 8) {
    int32_t t[8], dr[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int32_t i = i0 + k;
      t[k] = 0;
      dr[k] = -1;
      if (i <= L) t[k] = (int32_t)(0xFFFFFFFFu - (uint32_t)ld_behind_wait(keys + i));
      if (i < L) dr[k] = ld_behind_wait(draft_ids + d0 + i);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int32_t i = i0 + k;
      // row L has no draft: the scan always stops there
      if (!found && i <= L && (i == L || dr[k] != t[k])) {
        found = true;
        n = i;
        bonus = t[k];
      }
    }
  }
  return n;
}

inline AcceptWork accept_work(const lr_ctx *ctx, const void *logits, int64_t row_stride, int32_t n_rows, void *scratch, int vecs) {
  AcceptWork w = {reinterpret_cast<const uint16_t *>(logits), row_stride, reinterpret_cast<unsigned long long *>(scratch), ctx->model.vocab};
  w.n_chunks = ((w.vocab >> 3) + 32 * vecs - 1) / (32 * vecs);
  if (w.n_chunks == 0) w.n_chunks = 1;
  w.total = w.n_chunks * (uint32_t)n_rows;
  return w;
}

}  // namespace lr
