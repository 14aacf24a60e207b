// Host side of the C ABI: contexts, batch validation, plan images, launch
// wrappers and the host-buffer pass.  No device memory is allocated here; every
// device byte the library touches lies in caller-provided buffers.
#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <new>

#include "lr_common.cuh"

namespace lr {

static thread_local char g_err[512] = "";

void set_error(const char *fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof(g_err), fmt, ap);
  va_end(ap);
}

int cuda_fail(cudaError_t e, const char *what) {
  if (e == cudaSuccess) return LR_OK;
  set_error("%s: %s", what, cudaGetErrorString(e));
  return LR_ECUDA;
}

static inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }
static inline int pages_of(int64_t n) { return (int)((n + kPage - 1) / kPage); }

// ---- batch validation --------------------------------------------------------
#define LR_REQUIRE(cond, ...)          \
  do {                                 \
    if (!(cond)) {                     \
      set_error(__VA_ARGS__);          \
      return LR_EINVAL;                \
    }                                  \
  } while (0)

static int validate_batch(const lr_batch *b) {
  LR_REQUIRE(b != nullptr, "null batch");
  LR_REQUIRE(b->n_req >= 1 && b->n_branch >= 1 && b->n_span >= b->n_req && b->n_page_slots >= 1,
             "batch needs at least one request, one branch and one page slot");
  LR_REQUIRE(b->req_span_off && b->span_len && b->span_slot && b->br_req && b->br_depth && b->br_own_len &&
                 b->br_own_slot && b->br_n_draft && b->cu_q && b->page_ids,
             "null table pointer in batch");
  LR_REQUIRE(b->n_pool_pages >= 1 && b->n_pool_pages <= (int64_t)1 << 31, "n_pool_pages out of range");
  LR_REQUIRE(b->req_span_off[0] == 0 && b->req_span_off[b->n_req] == b->n_span, "req_span_off must run from 0 to n_span");
  std::vector<unsigned char> slot_used((size_t)b->n_page_slots, 0);
  auto claim = [&](int64_t first, int64_t len, const char *what, int idx) -> int {
    int n = pages_of(len);
    LR_REQUIRE(first >= 0 && first + n <= b->n_page_slots, "%s %d: page slots [%lld, %lld) outside [0, %d)", what, idx,
               (long long)first, (long long)(first + n), b->n_page_slots);
    for (int i = 0; i < n; ++i) {
      LR_REQUIRE(!slot_used[first + i], "%s %d: page slot %lld is claimed twice", what, idx, (long long)(first + i));
      slot_used[first + i] = 1;
    }
    return LR_OK;
  };
  for (int r = 0; r < b->n_req; ++r) {
    int s0 = b->req_span_off[r], s1 = b->req_span_off[r + 1];
    LR_REQUIRE(s1 > s0, "request %d has no prefix span", r);
    LR_REQUIRE(s1 - s0 - 1 <= 255, "request %d: more than 255 draft step segments", r);
    for (int s = s0; s < s1; ++s) {
      LR_REQUIRE(b->span_len[s] >= (s == s0 ? 0 : 1), "span %d of request %d has length %d", s - s0, r, b->span_len[s]);
      if (int rc = claim(b->span_slot[s], b->span_len[s], "span", s)) return rc;
    }
    if (b->seg_parent) {
      std::vector<int> level((size_t)(s1 - s0), 0);
      for (int c = 1; c < s1 - s0; ++c) {
        const int par = b->seg_parent[s0 + c];
        LR_REQUIRE(par >= 0 && par < c, "request %d: segment %d continues %d, which is not the prefix or an earlier segment", r, c, par);
        level[c] = level[par] + 1;
        LR_REQUIRE(level[c] <= kMaxTreeDepth, "request %d: segment %d lies %d steps below the prefix (tree mode allows %d)", r,
                   c, level[c], kMaxTreeDepth);
      }
    }
  }
  LR_REQUIRE(b->cu_q[0] == 0, "cu_q[0] must be 0");
  for (int i = 0; i < b->n_branch; ++i) {
    int r = b->br_req[i];
    LR_REQUIRE(r >= 0 && r < b->n_req, "branch %d: request %d out of range", i, r);
    LR_REQUIRE(i == 0 || b->br_req[i - 1] <= r, "branches must be grouped by request (br_req non-decreasing)");
    int gamma = b->req_span_off[r + 1] - b->req_span_off[r] - 1;
    LR_REQUIRE(b->br_depth[i] >= 0 && b->br_depth[i] <= gamma, "branch %d: depth %d outside [0, %d]", i, b->br_depth[i], gamma);
    int q_len = b->cu_q[i + 1] - b->cu_q[i];
    LR_REQUIRE(q_len >= 1, "branch %d: q_len %d < 1", i, q_len);
    LR_REQUIRE(b->br_own_len[i] >= q_len, "branch %d: own_len %d < q_len %d", i, b->br_own_len[i], q_len);
    LR_REQUIRE(b->br_n_draft[i] >= 0 && b->br_n_draft[i] <= b->br_own_len[i], "branch %d: n_draft %d outside [0, own_len]", i,
               b->br_n_draft[i]);
    if (int rc = claim(b->br_own_slot[i], b->br_own_len[i], "branch tail", i)) return rc;
  }
  std::vector<unsigned char> page_used((size_t)((b->n_pool_pages + 7) / 8), 0);
  for (int i = 0; i < b->n_page_slots; ++i) {
    if (!slot_used[i]) continue;  // slots no span refers to are ignored
    int64_t p = b->page_ids[i];
    LR_REQUIRE(p >= 0 && p < b->n_pool_pages, "page_ids[%d] = %lld outside the pool of %lld pages", i, (long long)p,
               (long long)b->n_pool_pages);
    LR_REQUIRE(!(page_used[p >> 3] & (1u << (p & 7))), "physical page %lld is referenced by two page slots", (long long)p);
    page_used[p >> 3] |= (unsigned char)(1u << (p & 7));
  }
  return LR_OK;
}

// ---- plan image --------------------------------------------------------------
// lr_plan_bytes needs the sizes only, lr_plan_create the sizes first (for the buffer) and then the tables: layout() works
// out the structure of the plan once, sections() lays the image out and, given a buffer, fills it in place.
struct Layout {
  size_t o_req_span_off, o_span_len, o_span_slot, o_br_req, o_br_depth, o_br_own_len, o_br_own_slot, o_br_n_draft, o_cu_q,
      o_cu_draft, o_page_ids, o_req_br_off, o_span_req, o_status, o_slot_item, o_chain_pg, o_chain_tok, o_tail_pg,
      o_span_tin, o_span_last, o_child_off, o_child_list;
  std::vector<int32_t> cu_draft, req_br_off, span_tin, span_last, child_off, child_list;
  TcHostPlan tc;
  size_t image_bytes, pair_cap, scratch_cap, total_bytes;
};

static void sections(const lr_batch *b, Layout &L, Image &g) {
  L.o_req_span_off = g.copy(b->req_span_off, b->n_req + 1);
  L.o_span_len = g.copy(b->span_len, b->n_span);
  L.o_span_slot = g.copy(b->span_slot, b->n_span);
  L.o_br_req = g.copy(b->br_req, b->n_branch);
  L.o_br_depth = g.copy(b->br_depth, b->n_branch);
  L.o_br_own_len = g.copy(b->br_own_len, b->n_branch);
  L.o_br_own_slot = g.copy(b->br_own_slot, b->n_branch);
  L.o_br_n_draft = g.copy(b->br_n_draft, b->n_branch);
  L.o_cu_q = g.copy(b->cu_q, b->n_branch + 1);
  L.o_cu_draft = g.copy(L.cu_draft.data(), L.cu_draft.size());
  L.o_page_ids = g.copy(b->page_ids, b->n_page_slots);
  L.o_req_br_off = g.copy(L.req_br_off.data(), L.req_br_off.size());
  L.o_span_tin = g.copy(L.span_tin.data(), L.span_tin.size());
  L.o_span_last = g.copy(L.span_last.data(), L.span_last.size());
  L.o_child_off = g.copy(L.child_off.data(), L.child_off.size());
  L.o_child_list = g.copy(L.child_list.data(), L.child_list.size());
  int32_t *span_req = g.add<int32_t>(b->n_span, L.o_span_req);
  int32_t *slot_item = g.add<int32_t>(b->n_page_slots, L.o_slot_item);
  int32_t *chain_pg = g.add<int32_t>((size_t)b->n_span + b->n_req, L.o_chain_pg);
  int32_t *chain_tok = g.add<int32_t>((size_t)b->n_span + b->n_req, L.o_chain_tok);
  int32_t *tail_pg = g.add<int32_t>((size_t)b->n_branch + b->n_req, L.o_tail_pg);
  int32_t *status = g.add<int32_t>(2, L.o_status);
  if (g.base) {
    status[0] = status[1] = 0;
    std::fill(slot_item, slot_item + b->n_page_slots, -1);
    for (int r = 0; r < b->n_req; ++r) {
      const int s0 = b->req_span_off[r], s1 = b->req_span_off[r + 1], base = s0 + r;
      const int b0 = L.req_br_off[r], b1 = L.req_br_off[r + 1], tb = b0 + r;
      chain_pg[base] = chain_tok[base] = tail_pg[tb] = 0;
      for (int s = s0; s < s1; ++s) {
        const int npg = pages_of(b->span_len[s]);
        span_req[s] = r;
        chain_pg[base + (s - s0) + 1] = chain_pg[base + (s - s0)] + npg;
        chain_tok[base + (s - s0) + 1] = chain_tok[base + (s - s0)] + b->span_len[s];
        std::fill(slot_item + b->span_slot[s], slot_item + b->span_slot[s] + npg, s);
      }
      for (int i = b0; i < b1; ++i) {
        const int npg = pages_of(b->br_own_len[i]);
        tail_pg[tb + (i - b0) + 1] = tail_pg[tb + (i - b0)] + npg;
        std::fill(slot_item + b->br_own_slot[i], slot_item + b->br_own_slot[i] + npg, b->n_span + i);
      }
    }
  }
  tc_plan_tables(b, L.req_br_off.data(), L.span_tin.data(), L.tc, g);
}

static int layout(const lr_ctx *ctx, const lr_batch *b, Layout &L) {
  if (!ctx) {
    set_error("null context");
    return LR_EINVAL;
  }
  if (int rc = validate_batch(b)) return rc;
  L.cu_draft.assign(b->n_branch + 1, 0);
  L.req_br_off.assign(b->n_req + 1, 0);
  for (int i = 0; i < b->n_branch; ++i) {
    L.cu_draft[i + 1] = L.cu_draft[i] + b->br_n_draft[i];
    L.req_br_off[b->br_req[i] + 1]++;
  }
  for (int r = 0; r < b->n_req; ++r) L.req_br_off[r + 1] += L.req_br_off[r];
  // depth-first interval labels and child lists of the draft-step trees (a chain when seg_parent is absent)
  L.span_tin.assign((size_t)b->n_span, 0);
  L.span_last.assign((size_t)b->n_span, 0);
  L.child_off.assign((size_t)b->n_span + 1, 0);
  L.child_list.assign((size_t)b->n_span, 0);
  std::vector<int> n_child, fill, size;
  for (int r = 0; r < b->n_req; ++r) {
    const int s0 = b->req_span_off[r], n = b->req_span_off[r + 1] - s0;
    auto parent_of = [&](int c) { return b->seg_parent ? b->seg_parent[s0 + c] : c - 1; };
    n_child.assign((size_t)n, 0);
    for (int c = 1; c < n; ++c) n_child[parent_of(c)]++;
    for (int c = 0; c < n; ++c) L.child_off[s0 + c + 1] = L.child_off[s0 + c] + n_child[c];
    fill.assign((size_t)n, 0);
    for (int c = 1; c < n; ++c) {  // increasing c: every list comes out sorted
      const int par = parent_of(c);
      L.child_list[L.child_off[s0 + par] + fill[par]++] = c;
    }
    size.assign((size_t)n, 1);  // subtree sizes: children have larger indices than parents
    for (int c = n - 1; c >= 1; --c) size[parent_of(c)] += size[c];
    // pre-order numbers: a node's number is its parent's + 1 + the subtree sizes of its earlier siblings
    for (int c = 0; c < n; ++c) {
      int next = L.span_tin[s0 + c] + 1;
      for (int k = L.child_off[s0 + c]; k < L.child_off[s0 + c + 1]; ++k) {
        L.span_tin[s0 + L.child_list[k]] = next;
        next += size[L.child_list[k]];
      }
      L.span_last[s0 + c] = L.span_tin[s0 + c] + size[c] - 1;
    }
  }
  tc_plan_structure(ctx, b, L.req_br_off.data(), L.span_tin.data(), L.span_last.data(), L.tc);
  Image sizes;
  sections(b, L, sizes);
  L.image_bytes = align_up(sizes.bytes, 256);
  const PairBytes pair = pair_bytes_bound(ctx, b, L.req_br_off.data());
  L.pair_cap = align_up(pair.image, 256);
  L.scratch_cap = align_up(std::max(L.tc.scratch_bytes, pair.scratch), 256);
  L.total_bytes = L.image_bytes + L.pair_cap + L.scratch_cap;
  return LR_OK;
}

}  // namespace lr

using namespace lr;

static int check_model(const lr_model *m, const char *who) {
  if (m->n_q_heads < 1 || m->n_kv_heads < 1 || m->vocab < 1) {
    set_error("%s: non-positive model dimension", who);
    return LR_EINVAL;
  }
  if ((m->head_dim != 64 && m->head_dim != 128) || m->page_size != kPage || m->n_q_heads % m->n_kv_heads != 0 ||
      m->n_q_heads / m->n_kv_heads > 16) {
    set_error("%s: unsupported geometry (head_dim %d, page_size %d, heads %d/%d)", who, m->head_dim, m->page_size,
              m->n_q_heads, m->n_kv_heads);
    return LR_EUNSUPPORTED;
  }
  return LR_OK;
}

extern "C" int lr_validate_batch(const lr_model *m, const lr_batch *b) {
  if (!m) {
    set_error("lr_validate_batch: null model");
    return LR_EINVAL;
  }
  if (int rc = check_model(m, "lr_validate_batch")) return rc;
  return validate_batch(b);
}

static void destroy_side(const SideStream &side) {
  for (cudaEvent_t ev : {side.fork, side.part, side.join})
    if (ev) cudaEventDestroy(ev);
  if (side.s) cudaStreamDestroy(side.s);
}

static int make_side(SideStream &side) {
  side = SideStream{};
  cudaError_t e = cudaStreamCreateWithFlags(&side.s, cudaStreamNonBlocking);
  for (cudaEvent_t *ev : {&side.fork, &side.part, &side.join})
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(ev, cudaEventDisableTiming);
  if (e == cudaSuccess) return LR_OK;
  destroy_side(side);
  side = SideStream{};
  return cuda_fail(e, "side stream");
}

// The plan's side stream: the one the context was made with, that of an earlier plan, or a new one (about 90 us).  Also while
// the caller's stream is being captured, which making a stream is no part of.
static int take_side(lr_plan *p) {
  if (p->side.s) return LR_OK;
  std::vector<SideStream> &idle = p->ctx->side_free;
  if (idle.empty()) {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    if (int rc = cuda_fail(cudaThreadExchangeStreamCaptureMode(&mode), "cudaThreadExchangeStreamCaptureMode")) return rc;
    const int rc = make_side(p->side);
    const cudaError_t e = cudaThreadExchangeStreamCaptureMode(&mode);
    return rc != LR_OK ? rc : cuda_fail(e, "cudaThreadExchangeStreamCaptureMode");
  }
  p->side = idle.back();
  idle.pop_back();
  return LR_OK;
}

// ---- context -------------------------------------------------------------------
extern "C" int lr_create(lr_ctx **out, const lr_model *m, int device) {
  if (!out || !m) {
    set_error("lr_create: null argument");
    return LR_EINVAL;
  }
  *out = nullptr;
  if (int rc = check_model(m, "lr_create")) return rc;
  int n_dev = 0;
  if (int rc = cuda_fail(cudaGetDeviceCount(&n_dev), "cudaGetDeviceCount")) return rc;
  if (device < 0 || device >= n_dev) {
    set_error("lr_create: device %d not present (%d devices)", device, n_dev);
    return LR_EINVAL;
  }
  int major = 0, minor = 0, sms = 0;  // (cudaGetDeviceProperties takes milliseconds)
  cudaError_t e = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  if (int rc = cuda_fail(e, "cudaDeviceGetAttribute")) return rc;
  if (major != 10) {
    set_error("lr_create: device %d is sm_%d%d; this library is built for sm_100a only", device, major, minor);
    return LR_EUNSUPPORTED;
  }
  if (int rc = cuda_fail(cudaSetDevice(device), "cudaSetDevice")) return rc;
  lr_ctx *c = new (std::nothrow) lr_ctx();
  if (!c) return LR_ENOMEM;
  c->model = *m;
  c->device = device;
  c->sm_count = sms;
  c->launches = 0;
  c->tmap_encode = nullptr;
  if (int rc = init_commit_kernel()) { delete c; return rc; }
  if (int rc = init_attn_tc_kernel()) { delete c; return rc; }
  if (int rc = init_attn_pair_kernel()) { delete c; return rc; }
  if (int rc = init_accept_filter_kernels()) { delete c; return rc; }
  SideStream side;
  if (int rc = make_side(side)) { delete c; return rc; }
  c->side_free.push_back(side);
  *out = c;
  return LR_OK;
}

static void give_back_side(lr_plan *p) {
  if (!p->side.s) return;
  if (p->ctx->side_free.size() < 8) p->ctx->side_free.push_back(p->side);
  else destroy_side(p->side);  // work still queued on it is finished all the same
}

extern "C" int lr_destroy(lr_ctx *ctx) {
  if (ctx) {
    for (auto &pb : ctx->pinned_free) {
      cudaEventSynchronize(pb.uploaded);
      cudaEventDestroy(pb.uploaded);
      cudaFreeHost(pb.ptr);
    }
    for (auto &side : ctx->side_free) destroy_side(side);
  }
  delete ctx;
  return LR_OK;
}

// A pinned buffer of at least `bytes`: the smallest cached one that fits, else a new one (capacity rounded up to a
// power of two, at least 64 KB, so that the next plan of a similar batch fits too).
static int take_pinned(lr_ctx *ctx, size_t bytes, void **ptr, size_t *cap, cudaEvent_t *ev) {
  int best = -1;
  for (int i = 0; i < (int)ctx->pinned_free.size(); ++i)
    if (ctx->pinned_free[i].cap >= bytes && (best < 0 || ctx->pinned_free[i].cap < ctx->pinned_free[best].cap)) best = i;
  if (best >= 0) {
    lr_ctx::PinnedBuf pb = ctx->pinned_free[best];
    ctx->pinned_free.erase(ctx->pinned_free.begin() + best);
    if (int rc = cuda_fail(cudaEventSynchronize(pb.uploaded), "cudaEventSynchronize(pinned buffer)")) return rc;
    *ptr = pb.ptr; *cap = pb.cap; *ev = pb.uploaded;
    return LR_OK;
  }
  size_t c = 64 << 10;
  while (c < bytes) c <<= 1;
  if (int rc = cuda_fail(cudaMallocHost(ptr, c), "cudaMallocHost(plan image)")) return rc;
  if (int rc = cuda_fail(cudaEventCreateWithFlags(ev, cudaEventDisableTiming), "cudaEventCreate")) {
    cudaFreeHost(*ptr);
    return rc;
  }
  *cap = c;
  return LR_OK;
}

static void give_back_pinned(lr_ctx *ctx, void *ptr, size_t cap, cudaEvent_t ev) {
  if (ctx->pinned_free.size() < 8) {
    ctx->pinned_free.push_back({ptr, cap, ev});
    return;
  }
  cudaEventSynchronize(ev);
  cudaEventDestroy(ev);
  cudaFreeHost(ptr);
}

extern "C" int64_t lr_launch_count(const lr_ctx *ctx) { return ctx ? ctx->launches : 0; }

// ---- plan ----------------------------------------------------------------------
extern "C" int lr_plan_bytes(const lr_ctx *ctx, const lr_batch *b, size_t *bytes_out) {
  if (!bytes_out) {
    set_error("lr_plan_bytes: null bytes_out");
    return LR_EINVAL;
  }
  Layout L;
  if (int rc = layout(ctx, b, L)) return rc;
  *bytes_out = L.total_bytes;
  return LR_OK;
}

struct lr_plan_draft {
  lr_ctx *ctx;
  lr_batch batch;
  Layout layout;
};

extern "C" int lr_plan_begin(lr_ctx *ctx, const lr_batch *b, size_t *bytes_out, lr_plan_draft **out) {
  if (!bytes_out || !out) {
    set_error("lr_plan_begin: null argument");
    return LR_EINVAL;
  }
  *out = nullptr;
  lr_plan_draft *draft = new (std::nothrow) lr_plan_draft();
  if (!draft) return LR_ENOMEM;
  if (int rc = layout(ctx, b, draft->layout)) {
    delete draft;
    return rc;
  }
  draft->ctx = ctx;
  draft->batch = *b;
  *bytes_out = draft->layout.total_bytes;
  *out = draft;
  return LR_OK;
}

extern "C" int lr_plan_drop(lr_plan_draft *draft) {
  delete draft;
  return LR_OK;
}

static int plan_build(lr_ctx *ctx, const lr_batch *b, Layout &L, void *ws, size_t ws_bytes, void *stream, lr_plan **out);
static int build_pair(lr_plan *p);
static cudaError_t queue_pair_upload(lr_plan *p, cudaStream_t s);

static int check_workspace(const void *ws, lr_plan **out) {
  if (!out || !ws) {
    set_error("lr_plan_create: null argument");
    return LR_EINVAL;
  }
  *out = nullptr;
  if (((uintptr_t)ws & 255) != 0) {
    set_error("lr_plan_create: workspace must be 256-byte aligned");
    return LR_EINVAL;
  }
  return LR_OK;
}

extern "C" int lr_plan_finish(lr_plan_draft *draft, void *ws, size_t ws_bytes, void *stream, lr_plan **out) {
  if (!draft) {
    set_error("lr_plan_finish: null draft");
    return LR_EINVAL;
  }
  int rc = check_workspace(ws, out);
  if (rc == LR_OK) rc = plan_build(draft->ctx, &draft->batch, draft->layout, ws, ws_bytes, stream, out);
  delete draft;
  return rc;
}

extern "C" int lr_plan_create(lr_ctx *ctx, const lr_batch *b, void *ws, size_t ws_bytes, void *stream, lr_plan **out) {
  if (int rc = check_workspace(ws, out)) return rc;
  Layout L;
  if (int rc = layout(ctx, b, L)) return rc;
  return plan_build(ctx, b, L, ws, ws_bytes, stream, out);
}

static int plan_build(lr_ctx *ctx, const lr_batch *b, Layout &L, void *ws, size_t ws_bytes, void *stream, lr_plan **out) {
  if (ws_bytes < L.total_bytes) {
    set_error("lr_plan_create: workspace of %zu bytes, %zu needed", ws_bytes, L.total_bytes);
    return LR_ENOMEM;
  }
  if (int rc = cuda_fail(cudaSetDevice(ctx->device), "cudaSetDevice")) return rc;
  lr_plan *p = new (std::nothrow) lr_plan();
  if (!p) return LR_ENOMEM;
  p->ctx = ctx;
  p->pinned = nullptr;
  p->results_pinned = nullptr;
  p->results_pinned_cap = 0;
  p->side = SideStream{};
  p->image_bytes = L.image_bytes;
  p->workspace_d = ws;
  p->workspace_bytes = ws_bytes;
  p->attention_path = 0;
  p->o_page_ids = L.o_page_ids;
  if (int rc = take_pinned(ctx, L.image_bytes + 64, &p->pinned, &p->pinned_cap, &p->uploaded)) {
    delete p;
    return rc;
  }
  Image img;
  img.base = reinterpret_cast<unsigned char *>(p->pinned);
  sections(b, L, img);
  unsigned char *base = reinterpret_cast<unsigned char *>(ws);
  auto at = [&](size_t off) { return reinterpret_cast<const int32_t *>(base + off); };
  DevBatch &d = p->dev;
  d.req_span_off = at(L.o_req_span_off);
  d.span_len = at(L.o_span_len);
  d.span_slot = at(L.o_span_slot);
  d.br_req = at(L.o_br_req);
  d.br_depth = at(L.o_br_depth);
  d.br_own_len = at(L.o_br_own_len);
  d.br_own_slot = at(L.o_br_own_slot);
  d.br_n_draft = at(L.o_br_n_draft);
  d.cu_q = at(L.o_cu_q);
  d.cu_draft = at(L.o_cu_draft);
  d.page_ids = at(L.o_page_ids);
  d.req_br_off = at(L.o_req_br_off);
  d.span_req = at(L.o_span_req);
  d.slot_item = at(L.o_slot_item);
  d.chain_pg = at(L.o_chain_pg);
  d.chain_tok = at(L.o_chain_tok);
  d.tail_pg = at(L.o_tail_pg);
  d.span_tin = at(L.o_span_tin);
  d.span_last = at(L.o_span_last);
  d.child_off = at(L.o_child_off);
  d.child_list = at(L.o_child_list);
  d.tree = b->seg_parent ? 1 : 0;
  d.status = reinterpret_cast<int32_t *>(base + L.o_status);
  d.n_req = b->n_req;
  d.n_branch = b->n_branch;
  d.n_span = b->n_span;
  d.n_page_slots = b->n_page_slots;
  d.n_q_rows = b->cu_q[b->n_branch];
  d.n_q_heads = ctx->model.n_q_heads;
  d.n_kv_heads = ctx->model.n_kv_heads;
  d.head_dim = ctx->model.head_dim;
  d.group = ctx->model.n_q_heads / ctx->model.n_kv_heads;
  d.n_pool_pages = b->n_pool_pages;
  p->cu_draft_h = L.cu_draft;
  p->n_drafts = L.cu_draft[b->n_branch];
  p->n_rows_logits = p->n_drafts + b->n_branch;
  p->n_verdicts = b->n_span - b->n_req;
  p->pair_off = L.image_bytes;
  p->pair_cap = L.pair_cap;
  p->scratch_off = L.image_bytes + L.pair_cap;
  p->scratch_cap = L.scratch_cap;
  tc_bind_device_plan(L.tc, base, base + p->scratch_off, p);
  p->pair_ok = p->pair_built = false;
  memset(&p->pr, 0, sizeof(p->pr));
  p->pr.wait_limit_us = p->tc.wait_limit_us = p->tc_pass.wait_limit_us = 1000000u;  // one second per wait
  p->o_req_span_off = L.o_req_span_off;
  p->o_span_len = L.o_span_len;
  p->o_span_slot = L.o_span_slot;
  p->o_br_req = L.o_br_req;
  p->o_br_depth = L.o_br_depth;
  p->o_br_own_len = L.o_br_own_len;
  p->o_br_own_slot = L.o_br_own_slot;
  p->o_br_n_draft = L.o_br_n_draft;
  p->o_cu_q = L.o_cu_q;
  p->o_req_br_off = L.o_req_br_off;
  p->o_span_tin = L.o_span_tin;
  p->o_span_last = L.o_span_last;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  cudaError_t e = cudaMemcpyAsync(ws, p->pinned, L.image_bytes, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaEventRecord(p->uploaded, s);
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  if (e == cudaSuccess) e = cudaStreamIsCapturing(s, &capture);
  // a captured upload has to bring the CTA-pair tables along: nothing tells when it will have run
  if (e == cudaSuccess && capture != cudaStreamCaptureStatusNone && build_pair(p) == LR_OK) {
    if (p->pair_ok) e = queue_pair_upload(p, s);
    p->pair_built = true;
  }
  if (e != cudaSuccess) {
    give_back_pinned(ctx, p->pinned, p->pinned_cap, p->uploaded);
    delete p;
    return cuda_fail(e, "plan upload");
  }
  *out = p;
  return LR_OK;
}

extern "C" int lr_plan_destroy(lr_plan *p) {
  if (!p) return LR_OK;
  if (p->pinned) give_back_pinned(p->ctx, p->pinned, p->pinned_cap, p->uploaded);
  give_back_side(p);
  if (p->results_pinned) give_back_pinned(p->ctx, p->results_pinned, p->results_pinned_cap, p->results_copied);
  delete p;
  return LR_OK;
}

// Plans the CTA-pair path from the batch tables of the plan's host image.
static int build_pair(lr_plan *p) {
  const unsigned char *img = reinterpret_cast<const unsigned char *>(p->pinned);
  auto at = [&](size_t off) { return reinterpret_cast<const int32_t *>(img + off); };
  lr_batch b = {};
  b.n_req = p->dev.n_req;
  b.n_branch = p->dev.n_branch;
  b.n_span = p->dev.n_span;
  b.n_page_slots = p->dev.n_page_slots;
  b.req_span_off = at(p->o_req_span_off);
  b.span_len = at(p->o_span_len);
  b.span_slot = at(p->o_span_slot);
  b.br_req = at(p->o_br_req);
  b.br_depth = at(p->o_br_depth);
  b.br_own_len = at(p->o_br_own_len);
  b.br_own_slot = at(p->o_br_own_slot);
  b.br_n_draft = at(p->o_br_n_draft);
  b.cu_q = at(p->o_cu_q);
  b.page_ids = at(p->o_page_ids);
  b.n_pool_pages = p->dev.n_pool_pages;
  PairHostPlan h;
  p->pr_image.clear();
  if (int rc = pair_build_host_plan(p->ctx, &b, at(p->o_req_br_off), at(p->o_span_tin), at(p->o_span_last), h, p->pr_image)) return rc;
  if (h.ok && (p->pr_image.size() > p->pair_cap || h.scratch_bytes > p->scratch_cap)) {
    set_error("lr_plan_set_attention_path: the CTA-pair plan needs %zu and %zu bytes of workspace, %zu and %zu are set aside", p->pr_image.size(),
              h.scratch_bytes, p->pair_cap, p->scratch_cap);
    return LR_ENOMEM;
  }
  unsigned char *ws = reinterpret_cast<unsigned char *>(p->workspace_d);
  const uint32_t wait_limit_us = p->pr.wait_limit_us, phantom = p->pr.phantom_tx_bytes;
  pair_bind_device_plan(h, ws + p->pair_off, ws + p->scratch_off, p);
  p->pr.wait_limit_us = wait_limit_us;
  p->pr.phantom_tx_bytes = phantom;
  return LR_OK;
}

static cudaError_t queue_pair_upload(lr_plan *p, cudaStream_t s) {
  return cudaMemcpyAsync(reinterpret_cast<unsigned char *>(p->workspace_d) + p->pair_off, p->pr_image.data(), p->pr_image.size(), cudaMemcpyHostToDevice, s);
}

// Uploads the tables on a stream of their own, behind the plan's image (before which the workspace may still be another's), and
// waits: whatever launches the path later, on whichever stream and captured or not, finds them.
static int upload_pair(lr_plan *p) {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;  // the caller may be capturing: none of this is part of it
  if (int rc = cuda_fail(cudaThreadExchangeStreamCaptureMode(&mode), "cudaThreadExchangeStreamCaptureMode")) return rc;
  int rc = cuda_fail(cudaEventSynchronize(p->uploaded), "cudaEventSynchronize(plan image)");
  cudaStream_t own = nullptr;
  if (rc == LR_OK) rc = cuda_fail(cudaStreamCreateWithFlags(&own, cudaStreamNonBlocking), "cudaStreamCreate");
  if (rc == LR_OK) rc = cuda_fail(queue_pair_upload(p, own), "CTA-pair plan upload");
  if (rc == LR_OK) rc = cuda_fail(cudaStreamSynchronize(own), "CTA-pair plan upload");
  if (own) cudaStreamDestroy(own);
  const cudaError_t e = cudaThreadExchangeStreamCaptureMode(&mode);
  return rc != LR_OK ? rc : cuda_fail(e, "cudaThreadExchangeStreamCaptureMode");
}

extern "C" int lr_plan_set_attention_path(lr_plan *p, int path) {
  if (!p || path < 0 || path > 3) {
    set_error("lr_plan_set_attention_path: bad argument");
    return LR_EINVAL;
  }
  if (path == 3 && !p->pair_built) {
    if (int rc = build_pair(p)) return rc;
    if (p->pair_ok)
      if (int rc = upload_pair(p)) return rc;
    p->pair_built = true;
  }
  p->attention_path = path;
  return LR_OK;
}

extern "C" int lr_plan_describe(const lr_plan *p, lr_plan_info *info) {
  if (!p || !info) {
    set_error("lr_plan_describe: null argument");
    return LR_EINVAL;
  }
  memset(info, 0, sizeof(*info));
  info->tensor_core_ok = p->tc_ok ? 1 : 0;
  info->path = p->attention_path;
  if (p->attention_path == 3) {
    info->uses_tensor_core = p->pair_ok ? 1 : 0;
    if (p->pair_ok) {
      info->n_cta = 2 * p->pr.n_pairs;
      info->n_pieces = p->pr_pieces;
      info->n_merge_targets = p->pr.n_targets;
      info->n_partial_slots = p->pr_partial_slots;
    }
    return LR_OK;
  }
  info->uses_tensor_core = (p->tc_ok && p->attention_path != 1) ? 1 : 0;
  if (info->uses_tensor_core) {
    info->n_cta = p->tc.n_cta;
    info->n_pieces = p->tc_pieces;
    info->n_merge_targets = p->tc.n_targets;
    info->n_partial_slots = p->tc_partial_slots;
  }
  return LR_OK;
}

extern "C" int lr_debug_partitions(const lr_model *m, const lr_batch *b, int32_t n_sm, lr_partition_info *attention, lr_partition_info *pass,
                                   int32_t *small_pass) {
  if (!m || !attention || !pass || !small_pass || n_sm < 1) {
    set_error("lr_debug_partitions: bad argument");
    return LR_EINVAL;
  }
  if (int rc = check_model(m, "lr_debug_partitions")) return rc;
  lr_ctx ctx = {};
  ctx.model = *m;
  ctx.sm_count = n_sm;
  Layout L;
  if (int rc = layout(&ctx, b, L)) return rc;
  auto info = [](const TcPartition &p) { return lr_partition_info{p.n_cta, (int32_t)p.targets.size(), p.n_partial_slots, p.longest}; };
  *attention = info(L.tc.all);
  *pass = info(L.tc.beside.n_cta > 0 ? L.tc.beside : L.tc.all);
  *small_pass = (int32_t)L.tc.small;
  return LR_OK;
}

extern "C" int lr_plan_debug_set_wait_limit(lr_plan *p, uint32_t microseconds) {
  if (!p || microseconds == 0) {
    set_error("lr_plan_debug_set_wait_limit: bad argument");
    return LR_EINVAL;
  }
  p->tc.wait_limit_us = p->tc_pass.wait_limit_us = microseconds;
  p->pr.wait_limit_us = microseconds;
  return LR_OK;
}

extern "C" int lr_plan_debug_set_phantom_bytes(lr_plan *p, uint32_t bytes) {
  if (!p) {
    set_error("lr_plan_debug_set_phantom_bytes: null plan");
    return LR_EINVAL;
  }
  p->tc.phantom_tx_bytes = p->tc_pass.phantom_tx_bytes = bytes;
  p->pr.phantom_tx_bytes = bytes;
  return LR_OK;
}

extern "C" int lr_plan_debug_set_page(lr_plan *p, int32_t page_slot, int32_t new_id, void *stream) {
  if (!p || page_slot < 0 || page_slot >= p->dev.n_page_slots) {
    set_error("lr_plan_debug_set_page: bad argument");
    return LR_EINVAL;
  }
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  // the pinned image is the source of the last upload: wait until that copy has read it
  if (int rc = cuda_fail(cudaEventSynchronize(p->uploaded), "cudaEventSynchronize(plan image)")) return rc;
  unsigned char *img = reinterpret_cast<unsigned char *>(p->pinned);
  int32_t *ids = reinterpret_cast<int32_t *>(img + p->o_page_ids);
  const int32_t old_id = ids[page_slot];
  ids[page_slot] = new_id;
  // physical page ids are distinct within a batch, so the old id names this slot in the attention tables too
  TcPage *pages = reinterpret_cast<TcPage *>(img + p->o_tc_pages);
  for (int i = 0; i < p->n_tc_pages; ++i)
    if (pages[i].page == old_id && (pages[i].meta & 31u) != 0u) pages[i].page = new_id;
  for (int part = 0; part < 2; ++part) {
    TcCtaHead *heads = reinterpret_cast<TcCtaHead *>(img + p->o_tc_heads[part]);
    for (int c = 0; c < p->n_tc_heads[part]; ++c)
      for (int k = 0; k < 32; ++k)
        if (heads[c].first_pages[k] == old_id && heads[c].piece1 > heads[c].piece0) heads[c].first_pages[k] = new_id;
  }
  cudaError_t e = cudaMemcpyAsync(p->workspace_d, p->pinned, p->image_bytes, cudaMemcpyHostToDevice, s);
  if (p->pair_built) {
    if (int rc = build_pair(p)) return rc;
    if (e == cudaSuccess && p->pair_ok) e = queue_pair_upload(p, s);
  }
  if (e == cudaSuccess) e = cudaEventRecord(p->uploaded, s);
  return cuda_fail(e, "lr_plan_debug_set_page upload");
}

// ---- steps ---------------------------------------------------------------------
static int check_attention(const lr_plan *p, const void *q, const void *k, const void *v, const void *out, const float *lse) {
  if (!p || !q || !k || !v || !out) {
    set_error("lr_verify_attention: null argument");
    return LR_EINVAL;
  }
  if ((((uintptr_t)q | (uintptr_t)k | (uintptr_t)v | (uintptr_t)out) & 15) != 0 || ((uintptr_t)lse & 3) != 0) {
    set_error("lr_verify_attention: q, pools and out must be 16-byte aligned");
    return LR_EINVAL;
  }
  return LR_OK;
}

extern "C" int lr_verify_attention(lr_plan *p, const void *q, const void *k, const void *v, void *out, float *lse,
                                   float scale, void *stream) {
  if (int rc = check_attention(p, q, k, v, out, lse)) return rc;
  if (!(scale > 0.f)) scale = 1.0f / sqrtf((float)p->dev.head_dim);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (p->attention_path == 3) {
    if (!p->pair_ok) {
      set_error("lr_verify_attention: the CTA-pair tensor-core path does not support this shape");
      return LR_EUNSUPPORTED;
    }
    return launch_attn_pair(p, q, k, v, out, lse, scale, s);
  }
  bool use_tc = p->attention_path == 2 || (p->attention_path == 0 && p->tc_ok);
  if (use_tc) {
    if (!p->tc_ok) {
      set_error("lr_verify_attention: the tensor-core path does not support this shape");
      return LR_EUNSUPPORTED;
    }
    return launch_attn_tc(p, p->tc, q, k, v, out, lse, scale, true, s);
  }
  return launch_attn_generic(p, q, k, v, out, lse, scale, s);
}

extern "C" int lr_accept_scratch_bytes(int32_t n_rows, size_t *bytes_out) {
  if (!bytes_out || n_rows < 0) {
    set_error("lr_accept_scratch_bytes: bad argument");
    return LR_EINVAL;
  }
  *bytes_out = 8 * ((size_t)n_rows + 1);
  return LR_OK;
}

static int check_accept(const lr_ctx *ctx, const void *logits, int64_t stride, const int32_t *drafts, const int32_t *cu_draft, int32_t n_branch,
                        int32_t n_rows, const int32_t *n_accept, const int32_t *bonus, const void *scratch) {
  if (!ctx || !logits || !cu_draft || !n_accept || !bonus || !scratch || (!drafts && n_rows > n_branch)) {
    set_error("lr_accept_greedy: null argument");
    return LR_EINVAL;
  }
  if (n_branch < 0 || n_rows < n_branch) {
    set_error("lr_accept_greedy: n_rows %d < n_branch %d", n_rows, n_branch);
    return LR_EINVAL;
  }
  if (((uintptr_t)logits & 15) != 0 || (stride & 7) != 0 || stride < ctx->model.vocab || ((uintptr_t)scratch & 7) != 0) {
    set_error("lr_accept_greedy: logits must be 16-byte aligned with a row stride that is a multiple of 8 and >= vocab");
    return LR_EINVAL;
  }
  return LR_OK;
}

extern "C" int lr_accept_greedy(lr_ctx *ctx, const void *logits, int64_t stride, const int32_t *drafts,
                                const int32_t *cu_draft, int32_t n_branch, int32_t n_rows, int32_t *n_accept,
                                int32_t *bonus, int32_t *row_argmax, void *scratch, void *stream) {
  if (int rc = check_accept(ctx, logits, stride, drafts, cu_draft, n_branch, n_rows, n_accept, bonus, scratch)) return rc;
  if (n_branch == 0) return LR_OK;
  return launch_accept(ctx, logits, stride, drafts, cu_draft, n_branch, n_rows, 0, n_accept, bonus, row_argmax, scratch,
                       reinterpret_cast<cudaStream_t>(stream));
}

extern "C" int lr_accept_greedy_static(lr_ctx *ctx, const void *logits, int64_t stride, const int32_t *drafts,
                                       const int32_t *cu_draft, int32_t n_branch, int32_t n_rows, int32_t *n_accept,
                                       int32_t *bonus, int32_t *row_argmax, void *stream) {
  if (!ctx || !logits || !cu_draft || !n_accept || !bonus || (!drafts && n_rows > n_branch)) {
    set_error("lr_accept_greedy_static: null argument");
    return LR_EINVAL;
  }
  if (n_branch < 0 || n_rows < n_branch) {
    set_error("lr_accept_greedy_static: n_rows %d < n_branch %d", n_rows, n_branch);
    return LR_EINVAL;
  }
  if (((uintptr_t)logits & 15) != 0 || (stride & 7) != 0 || stride < ctx->model.vocab) {
    set_error("lr_accept_greedy_static: logits must be 16-byte aligned with a row stride that is a multiple of 8 and >= vocab");
    return LR_EINVAL;
  }
  if (n_branch == 0) return LR_OK;
  return launch_accept_static(ctx, logits, stride, drafts, cu_draft, n_branch, n_rows, n_accept, bonus, row_argmax,
                              reinterpret_cast<cudaStream_t>(stream));
}

extern "C" int lr_accept_sample_scratch_bytes(const lr_ctx *ctx, int32_t n_rows, size_t *bytes_out) {
  if (!ctx || !bytes_out || n_rows < 0) {
    set_error("lr_accept_sample_scratch_bytes: bad argument");
    return LR_EINVAL;
  }
  *bytes_out = accept_sample_scratch_bytes(ctx->model.vocab, n_rows);
  return LR_OK;
}

extern "C" int lr_accept_sample(lr_ctx *ctx, const void *logits, int64_t stride, const int32_t *drafts, const int32_t *cu_draft,
                                int32_t n_branch, int32_t n_rows, float temperature, const float *u_accept,
                                const float *u_final, int32_t *n_accept, int32_t *final_id, float *p_draft, void *scratch,
                                void *stream) {
  if (!ctx || !logits || !cu_draft || !u_final || !n_accept || !final_id || !scratch ||
      ((!drafts || !u_accept) && n_rows > n_branch)) {
    set_error("lr_accept_sample: null argument");
    return LR_EINVAL;
  }
  if (n_branch < 0 || n_rows < n_branch) {
    set_error("lr_accept_sample: n_rows %d < n_branch %d", n_rows, n_branch);
    return LR_EINVAL;
  }
  if (!(temperature > 0.f)) {
    set_error("lr_accept_sample: temperature must be positive (use lr_accept_greedy for the greedy rule)");
    return LR_EINVAL;
  }
  if (((uintptr_t)logits & 15) != 0 || (stride & 7) != 0 || stride < ctx->model.vocab || ((uintptr_t)scratch & 7) != 0) {
    set_error("lr_accept_sample: logits must be 16-byte aligned with a row stride that is a multiple of 8 and >= vocab");
    return LR_EINVAL;
  }
  if (n_branch == 0) return LR_OK;
  return launch_accept_sample(ctx, logits, stride, drafts, cu_draft, n_branch, n_rows, temperature, u_accept, u_final, n_accept,
                              final_id, p_draft, scratch, reinterpret_cast<cudaStream_t>(stream));
}

extern "C" int lr_accept_sample_filtered_scratch_bytes(const lr_ctx *ctx, int32_t n_rows, size_t *bytes_out) {
  if (!ctx || !bytes_out || n_rows < 0) {
    set_error("lr_accept_sample_filtered_scratch_bytes: bad argument");
    return LR_EINVAL;
  }
  *bytes_out = accept_filtered_scratch_bytes(ctx->model.vocab, n_rows);
  return LR_OK;
}

extern "C" int lr_accept_sample_filtered(lr_ctx *ctx, const void *logits, int64_t stride, const int32_t *drafts,
                                         const int32_t *cu_draft, int32_t n_branch, int32_t n_rows, float temperature,
                                         int32_t top_k, float top_p, const float *u_accept, const float *u_final,
                                         int32_t *n_accept, int32_t *final_id, float *p_draft, int32_t *n_kept, void *scratch,
                                         void *stream) {
  if (!ctx || !logits || !cu_draft || !u_final || !n_accept || !final_id || !scratch ||
      ((!drafts || !u_accept) && n_rows > n_branch)) {
    set_error("lr_accept_sample_filtered: null argument");
    return LR_EINVAL;
  }
  if (n_branch < 0 || n_rows < n_branch) {
    set_error("lr_accept_sample_filtered: n_rows %d < n_branch %d", n_rows, n_branch);
    return LR_EINVAL;
  }
  if (!(temperature > 0.f) || top_k < 0 || !(top_p > 0.f) || top_p > 1.f) {
    set_error("lr_accept_sample_filtered: temperature must be positive, top_k >= 0 (0 = off), top_p in (0, 1] (1 = off)");
    return LR_EINVAL;
  }
  if (((uintptr_t)logits & 15) != 0 || (stride & 7) != 0 || stride < ctx->model.vocab || ((uintptr_t)scratch & 7) != 0) {
    set_error("lr_accept_sample_filtered: logits must be 16-byte aligned with a row stride that is a multiple of 8 and >= vocab");
    return LR_EINVAL;
  }
  if (n_branch == 0) return LR_OK;
  return launch_accept_filtered(ctx, logits, stride, drafts, cu_draft, n_branch, n_rows, temperature, top_k, top_p, u_accept,
                                u_final, n_accept, final_id, p_draft, n_kept, scratch, reinterpret_cast<cudaStream_t>(stream));
}

static int check_commit(const lr_plan *p, const uint8_t *verdict, const int32_t *n_accept, const CommitOut &o) {
  if (!p || !n_accept || !o.n_steps || !o.survivor || !o.committed || !o.keep_off || !o.keep_pages || !o.keep_valid || !o.free_off ||
      !o.free_pages || (!verdict && p->n_verdicts > 0)) {
    set_error("lr_commit: null argument");
    return LR_EINVAL;
  }
  return LR_OK;
}

static int commit(lr_plan *p, const uint8_t *verdict, const int32_t *n_accept, const CommitOut &o, bool after_accept, void *stream) {
  if (int rc = check_commit(p, verdict, n_accept, o)) return rc;
  return launch_commit(p, verdict, n_accept, o, after_accept, reinterpret_cast<cudaStream_t>(stream));
}

extern "C" int lr_commit(lr_plan *p, const uint8_t *verdict, const int32_t *n_accept, int32_t *n_steps, int32_t *survivor,
                         int32_t *committed, int32_t *keep_off, int32_t *keep_pages, int32_t *keep_valid,
                         int32_t *free_off, int32_t *free_pages, void *stream) {
  return commit(p, verdict, n_accept, CommitOut{n_steps, survivor, committed, keep_off, keep_pages, keep_valid, free_off, free_pages}, false, stream);
}

extern "C" int lr_compact_scratch_bytes(const lr_plan *p, size_t *bytes_out) {
  if (!p || !bytes_out) {
    set_error("lr_compact_scratch_bytes: null argument");
    return LR_EINVAL;
  }
  *bytes_out = 256;  // the tokens move in place; the argument stays in the interface
  return LR_OK;
}

extern "C" int lr_compact(lr_plan *p, const int32_t *keep_off, const int32_t *keep_pages, const int32_t *keep_valid, void *k_pool,
                          void *v_pool, int32_t *new_len, int32_t *n_pages_kept, void *scratch, void *stream) {
  if (!p || !keep_off || !keep_pages || !keep_valid || !k_pool || !v_pool || !new_len || !n_pages_kept || !scratch) {
    set_error("lr_compact: null argument");
    return LR_EINVAL;
  }
  if ((((uintptr_t)k_pool | (uintptr_t)v_pool) & 15) != 0 || ((uintptr_t)scratch & 255) != 0) {
    set_error("lr_compact: pools must be 16-byte aligned and the scratch 256-byte aligned");
    return LR_EINVAL;
  }
  return launch_compact(p, keep_off, keep_pages, keep_valid, k_pool, v_pool, new_len, n_pages_kept,
                        reinterpret_cast<cudaStream_t>(stream));
}

// ---- status --------------------------------------------------------------------
extern "C" int lr_poll_status(lr_plan *p, void *stream, int32_t *detail) {
  if (!p) {
    set_error("lr_poll_status: null plan");
    return LR_EINVAL;
  }
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  // the last 64 bytes of the pinned buffer are for this (pageable memory would be staged by the driver)
  volatile int32_t *st = reinterpret_cast<int32_t *>(reinterpret_cast<unsigned char *>(p->pinned) + p->pinned_cap - 64);
  cudaError_t e = cudaMemcpyAsync(const_cast<int32_t *>(st), p->dev.status, 8, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_fail(e, "lr_poll_status");
  if (detail) *detail = st[1];
  if (st[0] == kDevOk) return LR_OK;
  e = cudaMemsetAsync(p->dev.status, 0, 8, s);
  if (e != cudaSuccess) return cuda_fail(e, "lr_poll_status clear");
  if (st[0] == kDevTimeout) {
    set_error("device wait expired (detail %d)", st[1]);
    return LR_ETIMEOUT;
  }
  set_error("device bounds check failed (detail %d)", st[1]);
  return LR_EBOUNDS;
}

// ---- whole pass on device buffers ----------------------------------------------------
static CommitOut commit_out(const lr_pass_io *io) {
  return {io->n_steps_accepted_d, io->survivor_d, io->committed_len_d, io->keep_off_d, io->keep_pages_d, io->keep_valid_d, io->free_off_d, io->free_pages_d};
}

// Acceptance and commit on a second stream beside attention: they fill the SMs that it leaves idle.  (Which of the two comes first
// makes no difference.)  As one kernel they run on the few SMs that a small pass leaves them, so they have to start with attention.
static int pass_side_by_side(lr_ctx *ctx, lr_plan *p, const lr_pass_io *io, float scale, bool one_kernel, cudaStream_t side, cudaStream_t s) {
  if (int rc = take_side(p)) return rc;
  cudaError_t e = cudaEventRecord(p->side.fork, s);
  if (e != cudaSuccess) return cuda_fail(e, "lr_verify_pass: fork");
  if (one_kernel) {  // (its arguments have been checked)
    if (int rc = launch_attn_tc(p, p->tc_pass, io->q_d, io->k_pool_d, io->v_pool_d, io->out_d, io->lse_d, scale, /*merge=*/true, s)) return rc;
  } else if (int rc = lr_verify_attention(p, io->q_d, io->k_pool_d, io->v_pool_d, io->out_d, io->lse_d, scale, s)) {
    return rc;
  }
  if (!side) side = p->side.s;
  e = cudaStreamWaitEvent(side, p->side.fork, 0);
  if (e != cudaSuccess) return cuda_fail(e, "lr_verify_pass: fork");
  int rc;
  if (one_kernel) {
    rc = launch_pass_tail(ctx, p, io, /*behind_attention=*/false, side);
  } else {
    rc = lr_accept_greedy(ctx, io->logits_d, io->logits_stride, io->draft_ids_d, io->cu_draft_d, p->dev.n_branch, (int32_t)io->n_rows, io->n_accept_d,
                          io->bonus_id_d, io->row_argmax_d, io->accept_scratch_d, side);
    if (rc == LR_OK) rc = commit(p, io->verdict_d, io->n_accept_d, commit_out(io), /*after_accept=*/p->dev.n_branch > 0, side);
  }
  e = cudaEventRecord(p->side.join, side);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(s, p->side.join, 0);
  return rc != LR_OK ? rc : cuda_fail(e, "lr_verify_pass: join");
}

extern "C" int lr_verify_pass(lr_ctx *ctx, lr_plan *p, const lr_pass_io *io, float scale, void *side_stream, void *stream) {
  if (!ctx || !p || !io) {
    set_error("lr_verify_pass: null argument");
    return LR_EINVAL;
  }
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream), side = reinterpret_cast<cudaStream_t>(side_stream);
  const bool tc = p->tc_ok && (p->attention_path == 0 || p->attention_path == 2);
  if (!tc || !pass_tail_fits(ctx, p, io->n_rows)) return pass_side_by_side(ctx, p, io, scale, false, side, s);
  if (int rc = check_attention(p, io->q_d, io->k_pool_d, io->v_pool_d, io->out_d, io->lse_d)) return rc;
  if (int rc = check_accept(ctx, io->logits_d, io->logits_stride, io->draft_ids_d, io->cu_draft_d, p->dev.n_branch, (int32_t)io->n_rows, io->n_accept_d,
                            io->bonus_id_d, io->accept_scratch_d))
    return rc;
  if (int rc = check_commit(p, io->verdict_d, io->n_accept_d, commit_out(io))) return rc;
  if (!(scale > 0.f)) scale = 1.0f / sqrtf((float)p->dev.head_dim);
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  if (int rc = cuda_fail(cudaStreamIsCapturing(s, &capture), "cudaStreamIsCapturing")) return rc;
  // On one stream, two kernels in a row of which the second is set up, and mostly done, while the first runs (pass_tail.cu), there
  // are no events between two passes, and the next attention is set up early too.  A caller who gives a second stream has a reason
  // to order work with it.  In a graph events cost nothing and both streams' kernels start together: where the acceptance has SMs
  // of its own it is one kernel with the commit there (one request of 4 K tokens, head size 64, 18.9 -> 16.6 us), and beside an
  // attention of few CTAs a root of its own; where it has not, two kernels on a second stream are as good (4 K tokens, head size 128,
  // 19.2 us and 19.6).
  // Launched one by one, the second stream's kernel often comes when CTAs of the merge, which wait for attention, already sit on
  // the SMs left free, and then runs behind all of it on a few SMs: a pass by itself, head size 64, 32.2 us with acceptance and commit
  // as two kernels and 35.2 with one.  So they are two there, unless there is no merge and few logits.
  const bool captured = capture != cudaStreamCaptureStatusNone, beside = p->small == kBesideAttention;
  if (side || (captured && (!beside || 2 * p->tc_pass.n_cta <= p->ctx->sm_count)))
    return pass_side_by_side(ctx, p, io, scale, /*one_kernel=*/captured ? beside : pass_tail_apart(ctx, p, (int32_t)io->n_rows), side, s);
  if (int rc = launch_attn_tc(p, p->tc_pass, io->q_d, io->k_pool_d, io->v_pool_d, io->out_d, io->lse_d, scale, /*merge=*/false, s)) return rc;
  return launch_pass_tail(ctx, p, io, /*behind_attention=*/true, s);
}

// ---- whole pass from host buffers --------------------------------------------------
namespace {
struct Staging {
  size_t q, logits, drafts, verdict, out, n_accept, bonus, n_steps, survivor, committed, keep_off, free_off, keep_pages,
      keep_valid, free_pages, scratch, total;
};
Staging staging_layout(const lr_plan *p) {
  Staging s;
  size_t off = 0;
  auto take = [&](size_t n) {
    size_t o = off;
    off = align_up(off + n, 256);
    return o;
  };
  const DevBatch &d = p->dev;
  const size_t qo = (size_t)d.n_q_rows * d.n_q_heads * d.head_dim * 2;
  s.q = take(qo);
  s.logits = take((size_t)p->n_rows_logits * p->ctx->model.vocab * 2 + 16);
  s.drafts = take((size_t)p->n_drafts * 4 + 4);
  s.verdict = take((size_t)p->n_verdicts + 4);
  s.out = take(qo);
  s.n_accept = take((size_t)d.n_branch * 4);
  s.bonus = take((size_t)d.n_branch * 4);
  s.n_steps = take((size_t)d.n_req * 4);
  s.survivor = take((size_t)d.n_req * 4);
  s.committed = take((size_t)d.n_req * 4);
  s.keep_off = take((size_t)(d.n_req + 1) * 4);
  s.free_off = take((size_t)(d.n_req + 1) * 4);
  s.keep_pages = take((size_t)d.n_page_slots * 4);
  s.keep_valid = take((size_t)d.n_page_slots * 4);
  s.free_pages = take((size_t)d.n_page_slots * 4);
  s.scratch = take(8 * ((size_t)p->n_rows_logits + 1));
  s.total = off;
  return s;
}
}  // namespace

extern "C" int lr_pass_staging_bytes(const lr_plan *p, size_t *bytes_out) {
  if (!p || !bytes_out) {
    set_error("lr_pass_staging_bytes: null argument");
    return LR_EINVAL;
  }
  *bytes_out = staging_layout(p).total;
  return LR_OK;
}

// From this many bytes of logits on the acceptance runs in two parts, so that only the last sixteenth of the rows is still
// to be read when the upload ends.  Whole pass on a B200, one part and two: 62 MB 1225 and 1228 us, 124 MB 2398 and 2379,
// 248 MB 4725 and 4685; 3 MB 126 and 131.
constexpr size_t kAcceptInPartsBytes = 64 << 20;

// Queues the whole pass.  The logits are nearly all of what crosses the host link (188 MB against 5 MB of queries for 16
// ragged requests), so they are uploaded on the plan's side stream while attention runs and its output goes back on the
// caller's.  All on one stream and so: that batch 3815 and 3570 us (the upload alone 3.5 ms), one 4 K-token request with
// 16 MB of logits 375 and 346, with 0.2 MB 94 and 90, the smallest request 62 to 70 and 62.
static int issue_pass_host(lr_plan *p, const lr_pass_host_io *io, const void *k_pool, const void *v_pool, unsigned char *b, const Staging &L,
                           float scale, void *stream) {
  lr_ctx *ctx = p->ctx;
  const DevBatch &d = p->dev;
  const int vocab = ctx->model.vocab;
  const size_t qo = (size_t)d.n_q_rows * d.n_q_heads * d.head_dim * 2, row_bytes = (size_t)vocab * 2, logit_bytes = p->n_rows_logits * row_bytes;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream), c = p->side.s;
  auto I = [&](size_t off) { return reinterpret_cast<int32_t *>(b + off); };
  // branches of the first part of the acceptance
  int b_part = 0;
  if (logit_bytes >= kAcceptInPartsBytes)
    while (b_part + 1 < d.n_branch && 16ll * (p->cu_draft_h[b_part + 1] + b_part + 1) <= 15ll * p->n_rows_logits) ++b_part;
  const size_t part_rows = b_part ? (size_t)(p->cu_draft_h[b_part] + b_part) : 0, part_bytes = part_rows * row_bytes;

  cudaError_t e = cudaMemcpyAsync(b + L.q, io->q_h, qo, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess && p->n_drafts) e = cudaMemcpyAsync(b + L.drafts, io->draft_ids_h, (size_t)p->n_drafts * 4, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess && p->n_verdicts) e = cudaMemcpyAsync(b + L.verdict, io->verdict_h, (size_t)p->n_verdicts, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaEventRecord(p->side.fork, s);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(c, p->side.fork, 0);
  const unsigned char *logits_h = reinterpret_cast<const unsigned char *>(io->logits_h);
  if (e == cudaSuccess && part_bytes) e = cudaMemcpyAsync(b + L.logits, logits_h, part_bytes, cudaMemcpyHostToDevice, c);
  if (e == cudaSuccess && part_bytes) e = cudaEventRecord(p->side.part, c);
  if (e == cudaSuccess) e = cudaMemcpyAsync(b + L.logits + part_bytes, logits_h + part_bytes, logit_bytes - part_bytes, cudaMemcpyHostToDevice, c);
  if (e == cudaSuccess) e = cudaEventRecord(p->side.join, c);
  if (e != cudaSuccess) return cuda_fail(e, "lr_verify_pass_host: host-to-device copies");

  if (int rc = lr_verify_attention(p, b + L.q, k_pool, v_pool, b + L.out, nullptr, scale, stream)) return rc;
  e = cudaMemcpyAsync(io->out_h, b + L.out, qo, cudaMemcpyDeviceToHost, s);
  if (e != cudaSuccess) return cuda_fail(e, "lr_verify_pass_host: device-to-host copy of the output");
  // rows and branches of a part are counted from its first branch, drafts from the batch's first one
  auto accept = [&](int b0, int b1, size_t row0, size_t n_rows) {
    return launch_accept(ctx, b + L.logits + row0 * row_bytes, vocab, I(L.drafts), d.cu_draft + b0, b1 - b0, (int32_t)n_rows,
                         p->cu_draft_h[b0], I(L.n_accept) + b0, I(L.bonus) + b0, nullptr, b + L.scratch, s);
  };
  if (part_bytes) {
    if (int rc = cuda_fail(cudaStreamWaitEvent(s, p->side.part, 0), "cudaStreamWaitEvent")) return rc;
    if (int rc = accept(0, b_part, 0, part_rows)) return rc;
  }
  if (int rc = cuda_fail(cudaStreamWaitEvent(s, p->side.join, 0), "cudaStreamWaitEvent")) return rc;
  if (int rc = accept(b_part, d.n_branch, part_rows, p->n_rows_logits - part_rows)) return rc;
  const CommitOut lists = {I(L.n_steps), I(L.survivor), I(L.committed), I(L.keep_off), I(L.keep_pages), I(L.keep_valid), I(L.free_off), I(L.free_pages)};
  if (int rc = commit(p, b + L.verdict, I(L.n_accept), lists, /*after_accept=*/true, stream)) return rc;
  // The ten integer arrays lie next to one another in the staging buffer and leave in one copy, through a pinned buffer the
  // plan keeps, then to the caller's arrays.
  e = cudaMemcpyAsync(p->results_pinned, b + L.n_accept, L.scratch - L.n_accept, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaEventRecord(p->results_copied, s);
  return cuda_fail(e, "lr_verify_pass_host: device-to-host copy of the integer results");
}

extern "C" int lr_verify_pass_host(lr_plan *p, const lr_pass_host_io *io, const void *k_pool, const void *v_pool,
                                   void *staging, size_t staging_bytes, float scale, void *stream) {
  if (!p || !io || !k_pool || !v_pool || !staging) {
    set_error("lr_verify_pass_host: null argument");
    return LR_EINVAL;
  }
  if (!io->q_h || !io->logits_h || !io->out_h || !io->n_accept_h || !io->bonus_id_h || !io->n_steps_accepted_h ||
      !io->survivor_h || !io->committed_len_h || !io->keep_off_h || !io->free_off_h || !io->keep_pages_h ||
      !io->keep_valid_h || !io->free_pages_h || (!io->draft_ids_h && p->n_drafts) || (!io->verdict_h && p->n_verdicts)) {
    set_error("lr_verify_pass_host: null host buffer");
    return LR_EINVAL;
  }
  const Staging L = staging_layout(p);
  if (staging_bytes < L.total || ((uintptr_t)staging & 255) != 0) {
    set_error("lr_verify_pass_host: staging of %zu bytes (256-byte aligned) needed", L.total);
    return LR_ENOMEM;
  }
  if (p->ctx->model.vocab % 8 != 0) {
    set_error("lr_verify_pass_host: dense logits rows need vocab to be a multiple of 8");
    return LR_EUNSUPPORTED;
  }
  unsigned char *b = reinterpret_cast<unsigned char *>(staging);
  const DevBatch &d = p->dev;
  const size_t small_bytes = L.scratch - L.n_accept;
  if (p->results_pinned_cap < small_bytes)
    if (int rc = take_pinned(p->ctx, small_bytes, &p->results_pinned, &p->results_pinned_cap, &p->results_copied)) return rc;
  if (int rc = take_side(p)) return rc;
  if (int issued = issue_pass_host(p, io, k_pool, v_pool, b, L, scale, stream)) {
    // whatever was queued beside the caller's stream still comes before what the caller does next
    cudaEventRecord(p->side.join, p->side.s);
    cudaStreamWaitEvent(reinterpret_cast<cudaStream_t>(stream), p->side.join, 0);
    return issued;
  }
  const int rc = lr_poll_status(p, stream, nullptr);  // waits for the stream
  if (rc != LR_OK && rc != LR_ETIMEOUT && rc != LR_EBOUNDS) return rc;
  struct Back { void *dst; size_t off, n; } back[] = {
      {io->n_accept_h, L.n_accept, (size_t)d.n_branch * 4},
      {io->bonus_id_h, L.bonus, (size_t)d.n_branch * 4},
      {io->n_steps_accepted_h, L.n_steps, (size_t)d.n_req * 4},
      {io->survivor_h, L.survivor, (size_t)d.n_req * 4},
      {io->committed_len_h, L.committed, (size_t)d.n_req * 4},
      {io->keep_off_h, L.keep_off, (size_t)(d.n_req + 1) * 4},
      {io->free_off_h, L.free_off, (size_t)(d.n_req + 1) * 4},
      {io->keep_pages_h, L.keep_pages, (size_t)d.n_page_slots * 4},
      {io->keep_valid_h, L.keep_valid, (size_t)d.n_page_slots * 4},
      {io->free_pages_h, L.free_pages, (size_t)d.n_page_slots * 4},
  };
  for (const Back &k : back) memcpy(k.dst, reinterpret_cast<unsigned char *>(p->results_pinned) + (k.off - L.n_accept), k.n);
  return rc;
}

extern "C" const char *lr_strerror(int st) {
  switch (st) {
    case LR_OK: return "ok";
    case LR_EINVAL: return "invalid argument";
    case LR_EUNSUPPORTED: return "unsupported shape or device";
    case LR_ECUDA: return "CUDA error";
    case LR_ETIMEOUT: return "device-side wait expired";
    case LR_EBOUNDS: return "device-side bounds check failed";
    case LR_ENOMEM: return "buffer too small or out of host memory";
    default: return "unknown status";
  }
}

extern "C" const char *lr_last_error(void) { return lr::g_err; }
