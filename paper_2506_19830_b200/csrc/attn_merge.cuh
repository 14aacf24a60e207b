// The merge of the partial results of an M-tile, as a part of the kernels that do it (attn_tc.cu, pass_tail.cu).
#pragma once

#include "lr_common.cuh"

namespace lr {

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t *>(&t);
}

// Merge of the partials of one M-tile: O = sum_j 2^(m_j - M) O_j / sum_j 2^(m_j - M) l_j.
// One thread per (query row, 16-byte chunk of channels); a warp holds 32 consecutive rows of one chunk, which
// is how the partials are laid out ([slot][chunk][row]).  Grid: targets x (head size / 8) CTAs of 256 threads.  The
// slots are combined in a fixed order.
// What bounds it is the latency of a thread's two trips to memory times the waves of CTAs, not the bytes, which L2 holds.  Where no
// M-tile has more than four slots, which is what a large batch gives (it has hundreds of M-tiles), a thread therefore has four in
// flight, in 43 registers: five CTAs on an SM.  Eight take 70 registers, three CTAs.  With eight for every plan and as it is, in
// turn: 16 ragged requests 171.8 -> 169.6 us a pass (two runs of one side differ by 0.3 %), a cycle of 8 ragged requests over four
// layers 483 -> 475 (1 %), 8 trees 588 both; same results.  The rule looks at the target with most slots, so one long
// request among many short ones takes all of them through the wider form.  Where a target has more slots, as few long requests
// give, eight at a time make one trip of two.
template <int kBatch>
constexpr int kMergeCtas = kBatch == 4 ? 5 : 3;
template <int kD, int kBatch>
__device__ __forceinline__ void merge_cta(const DevBatch &d, const DevTcPlan &tc, int target, int part, uint16_t *__restrict__ out, float *__restrict__ lse) {
  const TcTarget g = tc.targets[target];
  const int T = tc.tokens_per_mtile, G = d.group;
  const int item = part * 256 + threadIdx.x;  // 0 .. kD / 4 * 128 - 1
  const int k = item >> 7, r = item & 127;           // chunk of 4 channels, row
  const int tok = g.mtile * T + r / G;
  const bool live = r < T * G && tok < g.n_q;
  // the partials come from the kernel launched just before this one
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (!live) return;
  const int64_t qi = (int64_t)(g.q_row0 + tok) * d.n_q_heads + g.kv_head * G + r % G;
  const float2 *ml = reinterpret_cast<const float2 *>(tc.partial_ml) + (int64_t)g.slot_begin * 128 + r;
  const float4 *po = reinterpret_cast<const float4 *>(tc.partial_o) + ((int64_t)g.slot_begin * (kD / 4) + k) * 128 + r;
  // kBatch slots at a time, the (exponent, sum) pairs and the partial outputs of a batch requested together: one
  // round trip to memory per batch.  The running maximum moves between batches (never within one), in slot order,
  // so the result depends on nothing but the partials.
  float M = -INFINITY, L = 0.f;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int j0 = 0; j0 < g.n_slots; j0 += kBatch) {
    float4 o[kBatch];
    float2 v[kBatch];
#pragma unroll
    for (int jj = 0; jj < kBatch; ++jj)
      if (j0 + jj < g.n_slots) {
        v[jj] = ml[(int64_t)(j0 + jj) * 128];
        o[jj] = po[(int64_t)(j0 + jj) * (kD / 4) * 128];
      }
    float mb = M;
#pragma unroll
    for (int jj = 0; jj < kBatch; ++jj)
      if (j0 + jj < g.n_slots && v[jj].y > 0.f) mb = fmaxf(mb, v[jj].x);  // a stream that saw no key of the row contributes nothing
    if (mb > M) {
      const float a = exp2f(M - mb);  // 0 while nothing has been accumulated (M = -inf)
      L *= a;
      acc.x *= a;
      acc.y *= a;
      acc.z *= a;
      acc.w *= a;
      M = mb;
    }
#pragma unroll
    for (int jj = 0; jj < kBatch; ++jj)
      if (j0 + jj < g.n_slots && v[jj].y > 0.f) {
        const float w = exp2f(v[jj].x - M);
        L = fmaf(w, v[jj].y, L);
        acc.x = fmaf(w, o[jj].x, acc.x);
        acc.y = fmaf(w, o[jj].y, acc.y);
        acc.z = fmaf(w, o[jj].z, acc.z);
        acc.w = fmaf(w, o[jj].w, acc.w);
      }
  }
  const float inv = 1.0f / L;
  uint2 pk = make_uint2(pack_bf16(acc.x * inv, acc.y * inv), pack_bf16(acc.z * inv, acc.w * inv));
  *reinterpret_cast<uint2 *>(out + qi * kD + k * 4) = pk;
  if (lse != nullptr && k == 0) lse[qi] = (M + log2f(L)) * 0.6931471805599453f;
}

}  // namespace lr
