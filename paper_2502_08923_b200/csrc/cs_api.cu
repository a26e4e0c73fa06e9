// C ABI of the copy-and-verify library: argument checks, workspace layout, the chain of
// kernels of one verification step and the device-resident generation loop.
#include <math.h>
#include <stdlib.h>

#include <mutex>
#include <new>

#include <string.h>

#include "cs_common.cuh"
#include "cs_loop_host.h"

namespace {

struct WsLayout {
  size_t x, xn, attn_out, act, qbuf, partial, attn_o, attn_ml, ssq, rope_cs, inv_freq, tile_max, tile_idx,
      row_tok, row_pos, row_lim, row_write, seq_ok, iota, pair_part, pair_flag, chain_part, chain_epoch, chain_ctl, status, loop_last, loop_draft, loop_dlen, loop_mpos,
      loop_emitted, loop_done, loop_accept, loop_out, loop_argmax, loop_stats, total;
  size_t qkv_elems;
  int attn_splits;
};

bool config_ok(const cs_model_config* c) {
  if (c == nullptr) return false;
  if (c->n_layers < 1 || c->d_model < 8 || c->n_heads < 1 || c->n_kv_heads < 1 || c->d_ffn < 8 ||
      c->vocab < 1 || c->max_seq < 1 || c->max_batch < 1 || c->k_max < 0)
    return false;
  if (c->head_dim != 32 && c->head_dim != 64 && c->head_dim != 128) return false;
  if (c->n_heads % c->n_kv_heads) return false;
  if ((long)c->max_batch * (c->k_max + 1) > CS_MAX_ROWS) return false;
  if (c->d_model % 8 || c->d_ffn % 8 || (c->n_heads * c->head_dim) % 8) return false;
  return true;
}

size_t take(size_t* off, size_t bytes) {
  const size_t at = *off;
  *off = (at + bytes + 1023) & ~(size_t)1023;
  return at;
}

// CS_CHAIN: chained projections 0 = by the shape of the layer, -1 = never, 1 = always
int chain_switch() {
  const char* v = getenv("CS_CHAIN");
  return v == nullptr ? 0 : (v[0] == '0' ? -1 : (v[0] == '1' ? 1 : 0));
}

WsLayout ws_layout(const cs_model_config* c) {
  WsLayout L;
  const size_t rows = CS_MAX_ROWS;
  const size_t d = c->d_model, qd = (size_t)c->n_heads * c->head_dim, F = c->d_ffn;
  const size_t qkv = qd + 2 * (size_t)c->n_kv_heads * c->head_dim;
  L.qkv_elems = rows * (qkv > 4096 ? qkv : 4096);
  int as = cs_ceil_div(c->max_seq, c->head_dim == 128 ? 128 : 64);   // key tiles of the attention kernels
  L.attn_splits = as < 1 ? 1 : (as > 64 ? 64 : as);
  const size_t lm_tiles = cs_ceil_div(c->vocab, CS_GEMM_BM);
  size_t off = 0;
  L.x = take(&off, rows * d * 4);
  // operands carried as two bf16 terms: hi rows then lo rows
  L.xn = take(&off, 2 * rows * d * 2);
  L.attn_out = take(&off, 2 * rows * qd * 2);
  L.act = take(&off, 2 * rows * F * 2);
  L.qbuf = take(&off, 2 * rows * qd * 2);
  L.partial = take(&off, L.qkv_elems * 4);
  L.attn_o = take(&off, (size_t)L.attn_splits * rows * qd * 4);
  L.attn_ml = take(&off, (size_t)L.attn_splits * rows * c->n_heads * 2 * 4);
  L.ssq = take(&off, rows * (size_t)cs_ceil_div(c->d_model, CS_GEMM_BM) * CS_MAX_SPLITS * 4);
  L.rope_cs = take(&off, rows * c->head_dim * 4);
  L.inv_freq = take(&off, (size_t)c->head_dim / 2 * 8);
  L.tile_max = take(&off, lm_tiles * rows * 4);
  L.tile_idx = take(&off, lm_tiles * rows * 4);
  L.row_tok = take(&off, rows * 4);
  L.row_pos = take(&off, rows * 4);
  L.row_lim = take(&off, rows * 4);
  L.row_write = take(&off, rows * 4);
  L.seq_ok = take(&off, rows * 4);
  L.iota = take(&off, rows * 4);
  L.pair_part = take(&off, (size_t)CS_MAX_PAIRS * 2 * CS_MAX_ROWS * CS_GEMM_BM * 4);
  L.pair_flag = take(&off, CS_MAX_PAIRS * 2 * 4);
  const size_t chained = cs_chain_max_rows(*c, chain_switch()) > 0 ? 1 : 0;   // (21 MB that other models need not hold)
  L.chain_part = take(&off, chained * 4 * CS_CHAIN_MAX_RUNS * CS_CHAIN_MAX_ROWS / 2 * CS_GEMM_BM * sizeof(uint4));
  L.chain_epoch = take(&off, chained * 256);
  L.chain_ctl = take(&off, chained * c->n_layers * cs_chain_words(c) * 4);
  L.status = take(&off, 256);
  L.loop_last = take(&off, rows * 4);
  L.loop_draft = take(&off, rows * 4);
  L.loop_dlen = take(&off, rows * 4);
  L.loop_mpos = take(&off, rows * 4);
  L.loop_emitted = take(&off, rows * 4);
  L.loop_done = take(&off, (rows + 2) * 4);
  L.loop_accept = take(&off, rows * 4);
  L.loop_out = take(&off, rows * 4);
  L.loop_argmax = take(&off, rows * 4);
  L.loop_stats = take(&off, sizeof(cs_stats));
  L.total = off;
  return L;
}

// Pinned host memory of the contexts, in slots of one block per device: cs_create takes a slot and cs_destroy gives it
// back; a context that finds none left pins its own.  A block stays (0.3 MB, one per device) because pinning is slow:
// with memory of its own for every context, creating one takes 2.8 ms instead of 0.25 and destroying it 0.5 instead
// of 0.06, each up to 0.9 s now and then.  A block belongs to the CUDA context it was pinned in and goes with it when
// the process resets the device, so a block is known by that context's id.
constexpr size_t kStepInAt = 2048, kStepOutAt = kStepInAt + CS_STEP_IN_MAX * sizeof(int);
constexpr size_t kSlotBytes = kStepOutAt + 2 * CS_MAX_ROWS * sizeof(int) + 1024;
constexpr int kSlots = 32, kBlocks = 64;
static_assert(sizeof(cs_stats) + 8 <= 2 * CS_MAX_ROWS * sizeof(int), "report of a whole loop");
static_assert(64 + (CS_MAX_ROWS + 1) * sizeof(int) <= kStepInAt && kSlotBytes % 1024 == 0, "progress word and host scratch");
struct PinnedBlock {
  char* at;
  unsigned taken;
  unsigned long long owner;
};
std::mutex g_pinned_lock;
PinnedBlock g_pinned[kBlocks] = {};

// id of the current CUDA context, never given twice in a process; 0 = the driver does not say
unsigned long long cuda_context_id() {
  void* p = nullptr;
  cudaDriverEntryPointQueryResult q;
  unsigned long long id = 0;
  if (cudaGetDriverEntryPoint("cuCtxGetId", &p, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  return reinterpret_cast<CUresult (*)(CUcontext, unsigned long long*)>(p)(nullptr, &id) == CUDA_SUCCESS ? id : 0;
}

cudaError_t take_pinned(PinnedSlot* out, int dev) {
  const unsigned flags = cudaHostAllocMapped | cudaHostAllocPortable;
  const unsigned long long id = dev < kBlocks ? cuda_context_id() : 0;
  std::lock_guard<std::mutex> hold(g_pinned_lock);
  if (id != 0) {
    PinnedBlock& k = g_pinned[dev];
    if (k.owner != id) k = PinnedBlock{};              // (there is none yet, or it went with the context before this one)
    if (k.at == nullptr) {
      const cudaError_t e = cudaHostAlloc(reinterpret_cast<void**>(&k.at), kSlotBytes * kSlots, flags);
      if (e != cudaSuccess) { k = PinnedBlock{}; return e; }
      k.owner = id;
    }
    for (int i = 0; i < kSlots; ++i)
      if (!(k.taken >> i & 1u)) {
        k.taken |= 1u << i;
        *out = PinnedSlot{k.at + i * kSlotBytes, id, dev, i};
        return cudaSuccess;
      }
  }
  void* own = nullptr;
  const cudaError_t e = cudaHostAlloc(&own, kSlotBytes, flags);
  if (e == cudaSuccess) *out = PinnedSlot{static_cast<char*>(own), 0, dev, -1};
  return e;
}

void give_pinned(const PinnedSlot& s) {
  if (s.at == nullptr) return;
  if (s.index < 0) { cudaFreeHost(s.at); return; }
  std::lock_guard<std::mutex> hold(g_pinned_lock);
  PinnedBlock& k = g_pinned[s.block];
  if (k.owner == s.owner) k.taken &= ~(1u << s.index);   // (or else the block is gone already)
}

// cs_create has no context to leave an error text in: the last failure of this thread is kept here
thread_local char g_create_err[256] = "";

cs_status fail(cs_ctx* ctx, cs_status s, const char* msg) {
  if (ctx) snprintf(ctx->err, sizeof(ctx->err), "%s", msg);
  return s;
}

bool aligned(const void* p, unsigned bytes) { return (reinterpret_cast<uintptr_t>(p) & (bytes - 1)) == 0; }

cs_status ensure_act_maps(cs_ctx* ctx, int rows) {
  const int box = cs_gemm_act_box(CS_EPI_RESIDUAL, rows, true);
  if (ctx->act_box == box) return CS_OK;
  const cs_model_config& c = ctx->cfg;
  cs_status s;
  if ((s = cs_make_act_map(ctx, &ctx->tmXn, ctx->xn, 2 * CS_MAX_ROWS, c.d_model, box)) != CS_OK) return s;
  if ((s = cs_make_act_map(ctx, &ctx->tmAttn, ctx->attn_out, 2 * CS_MAX_ROWS, c.n_heads * c.head_dim, box)) != CS_OK)
    return s;
  if ((s = cs_make_act_map(ctx, &ctx->tmAct, ctx->act, 2 * CS_MAX_ROWS, c.d_ffn, box)) != CS_OK) return s;
  ctx->act_box = box;
  return CS_OK;
}

// The forward of Sec. 3.2 over the rows prepared by a *_setup kernel: B sequences of R
// rows each.  With `with_lm` the LM head leaves per-tile (max, id) pairs for k_accept.
cs_status enqueue_forward(cs_ctx* ctx, int B, int R, void* kv_cache, bool with_lm, float* logits,
                          cudaStream_t st) {
  const cs_model_config& c = ctx->cfg;
  const int rows = B * R;
  const int lo_row = CS_MAX_ROWS;      // second bf16 term of every activation operand: row offset in the operand maps
  cs_status s = ensure_act_maps(ctx, rows);
  if (s != CS_OK) return s;
  // Only the first RMSNorm runs as a kernel.  Every later one is folded into the GEMMs around
  // it: the residual GEMM before it writes gain * x (two bf16 terms) and sums of squares, the
  // GEMM after it scales its accumulators by 1/rms.
  NormFuse take_norm = {};           // how the next norm-consuming GEMM finds its 1/rms
  auto qkv_epi = [&](int l) {
    return QkvEpi{ctx->rope_cs, ctx->row_pos, ctx->row_write, ctx->qbuf, static_cast<__nv_bfloat16*>(kv_cache),
                  R, l, c.n_heads, c.n_kv_heads, c.head_dim, c.max_batch, c.max_seq};
  };
  const bool chained = cs_chain_takes(ctx, rows);
  if (chained) {
    // short blocks: two launches per layer, the attention and everything up to the next one
    cs_launch_embed_rmsnorm(ctx, ctx->layers[0].attn_norm, rows, st);
    const QkvEpi q0 = qkv_epi(0);
    s = cs_launch_gemm(ctx, &ctx->layers[0].qkv, &ctx->tmXn, lo_row, rows, CS_EPI_QKV, nullptr, nullptr, nullptr, 0, &q0, &take_norm, st);
    for (int l = 0; l < c.n_layers && s == CS_OK; ++l) {
      const int nsplit = cs_launch_attention(ctx, kv_cache, l, B, R, false, st);
      const bool last = l + 1 == c.n_layers;
      const QkvEpi qn = qkv_epi(l + 1);
      s = cs_launch_chain(ctx, l, nsplit, rows, last ? nullptr : &qn,
                          !last ? ctx->layers[l + 1].attn_norm : (with_lm ? ctx->final_norm : nullptr), st);
    }
    if (s != CS_OK) return s;
    take_norm.ssq_in = ctx->ssq;
    take_norm.slots_in = cs_ceil_div(c.d_model, CS_GEMM_BM);
    take_norm.slot_stride = ctx->ssq_stride;
    take_norm.inv_d = 1.f / (float)c.d_model;
    take_norm.eps = c.rms_eps;
  }
  for (int l = 0; l < c.n_layers && !chained; ++l) {
    const LayerPlan& L = ctx->layers[l];
    if (l == 0) {
      cs_launch_embed_rmsnorm(ctx, L.attn_norm, rows, st);
    }
    const QkvEpi qe = qkv_epi(l);
    s = cs_launch_gemm(ctx, &L.qkv, &ctx->tmXn, lo_row, rows, CS_EPI_QKV, nullptr, nullptr, nullptr, 0, &qe,
                       &take_norm, st);
    if (s != CS_OK) return s;
    cs_launch_attention(ctx, kv_cache, l, B, R, true, st);
    NormFuse give = {};
    give.gain_out = L.ffn_norm;
    give.xn_out = ctx->xn;
    give.ssq_out = ctx->ssq;
    give.slot_stride = ctx->ssq_stride;
    s = cs_launch_gemm(ctx, &L.o, &ctx->tmAttn, lo_row, rows, CS_EPI_RESIDUAL, ctx->x, nullptr, nullptr, 0, nullptr,
                       &give, st);
    if (s != CS_OK) return s;
    take_norm = NormFuse{};
    take_norm.ssq_in = ctx->ssq;
    take_norm.slots_in = cs_norm_slots(&L.o, rows);
    take_norm.slot_stride = ctx->ssq_stride;
    take_norm.inv_d = 1.f / (float)c.d_model;
    take_norm.eps = c.rms_eps;
    s = cs_launch_gemm(ctx, &L.gate_up, &ctx->tmXn, lo_row, rows, CS_EPI_SWIGLU, nullptr, ctx->act,
                       ctx->act + (size_t)CS_MAX_ROWS * c.d_ffn, c.d_ffn, nullptr, &take_norm, st);
    if (s != CS_OK) return s;
    // the norm after this layer: the next layer's, or the final one before the LM head
    const __nv_bfloat16* next_gain = (l + 1 < c.n_layers) ? ctx->layers[l + 1].attn_norm : (with_lm ? ctx->final_norm : nullptr);
    give.gain_out = next_gain;
    s = cs_launch_gemm(ctx, &L.down, &ctx->tmAct, lo_row, rows, CS_EPI_RESIDUAL, ctx->x, nullptr, nullptr, 0, nullptr,
                       &give, st);
    if (s != CS_OK) return s;
    take_norm.slots_in = cs_norm_slots(&L.down, rows);
  }
  if (with_lm) {
    s = cs_launch_gemm(ctx, &ctx->lm, &ctx->tmXn, lo_row, rows, CS_EPI_ARGMAX, logits, nullptr, nullptr, 0, nullptr,
                       &take_norm, st);
    if (s != CS_OK) return s;
  }
  CS_CUDA_OK(ctx, cudaGetLastError());
  return CS_OK;
}

// One iteration of the generation loop (App. B.3 steps 1, 2, 4) on device-resident state.
// `report`: the commit also reports the loop's progress to the host.
cs_status enqueue_loop_step(cs_ctx* ctx, cudaStream_t st, bool report = false) {
  const LoopState& L = ctx->loop;
  ctx->stamp_n = 0;
  // App. B.3 step 1: the scan, or the lookup in the gamma-gram index (Sec. 3.1) - same outputs
  cs_status r = L.use_index
                    ? cs_launch_gram_lookup(ctx->match_index, L.B, ctx->match_index_cap, L.hist, L.hist_len, L.stride, L.gamma,
                                            L.k, L.policy, ctx->loop_mpos, ctx->loop_draft, ctx->loop_dlen, ctx->loop_last,
                                            ctx->loop_done, st)
                    : cs_launch_find_match(L.hist, L.hist_len, L.B, L.stride, L.gamma, L.k, L.policy, ctx->loop_mpos,
                                           ctx->loop_draft, ctx->loop_dlen, ctx->loop_last, ctx->loop_done, st,
                                           cs_next_stamp(ctx, CS_FAM_OTHER));
  if (r != CS_OK) return fail(ctx, r, "match kernel launch failed");
  cs_launch_block_setup(ctx, ctx->loop_last, ctx->loop_draft, ctx->loop_dlen, L.kv_len, ctx->loop_done, L.B, L.k, false, st);
  // k_block_setup lets nothing pass that was enqueued before the step, and nothing before k_loop_commit changes kv_len
  ctx->kv_len_early = L.kv_len;
  r = enqueue_forward(ctx, L.B, L.k + 1, L.kv_cache, true, nullptr, st);
  ctx->kv_len_early = nullptr;
  if (r != CS_OK) return r;
  cs_launch_accept(ctx, L.B, L.k, ctx->loop_draft, ctx->loop_dlen, L.script, L.max_new, ctx->loop_emitted, L.max_new,
                   ctx->loop_accept, ctx->loop_out, ctx->loop_argmax, L.kv_len, 0, st);
  cs_launch_loop_commit(ctx, L.hist, L.hist_len, L.B, L.stride, L.kv_len, L.k, L.max_new, L.eos_id,
                        L.script != nullptr, report ? ctx->progress_dev : nullptr, st);
  if (L.use_index) {
    // App. B.3 step 2(d): the grams that the appended tokens made admissible enter the index
    r = cs_launch_gram_update(ctx->match_index, L.B, ctx->match_index_cap, L.hist, L.hist_len, L.stride, L.gamma, 1,
                              ctx->d_status, st);
    if (r != CS_OK) return fail(ctx, r, "index update launch failed");
  }
  CS_CUDA_OK(ctx, cudaGetLastError());
  return CS_OK;
}

cs_status status_from_bits(cs_ctx* ctx, int bits) {
  if (bits & CS_DEV_TIMEOUT) return fail(ctx, CS_ERR_TIMEOUT, "a bounded device-side wait ran out");
  if (bits & CS_DEV_CAPACITY) return fail(ctx, CS_ERR_CAPACITY, "KV cache or history row too small for a sequence");
  if (bits & CS_DEV_SMEM) return fail(ctx, CS_ERR_UNSUPPORTED, "attention kernel could not place its barriers in shared memory");
  if (bits & CS_DEV_BADARG) return fail(ctx, CS_ERR_ARG, "device-side argument check failed (lengths inconsistent)");
  return CS_OK;
}

// Reads and clears the status word; synchronises.
cs_status take_status(cs_ctx* ctx, int* bits, cudaStream_t st) {
  CS_CUDA_OK(ctx, cudaMemcpyAsync(bits, ctx->d_status, sizeof(int), cudaMemcpyDeviceToHost, st));
  CS_CUDA_OK(ctx, cudaMemsetAsync(ctx->d_status, 0, sizeof(int), st));
  CS_CUDA_OK(ctx, cudaStreamSynchronize(st));
  // a wait that ran out may have left a hand-over flag of the two-SM GEMM raised
  if (*bits & CS_DEV_TIMEOUT) CS_CUDA_OK(ctx, cudaMemsetAsync(ctx->pair_flag, 0, CS_MAX_PAIRS * 2 * sizeof(int), st));
  return CS_OK;
}

// One reporting step of the loop as a graph (captured on the context's own stream: the legacy default stream
// cannot).  Without it the loop goes on enqueueing, so a failure here is not one of the call.
void capture_step(cs_ctx* ctx) {
  LoopState& L = ctx->loop;
  if (cudaStreamBeginCapture(ctx->cap_stream, cudaStreamCaptureModeRelaxed) != cudaSuccess) { (void)cudaGetLastError(); return; }
  const cs_status s = enqueue_loop_step(ctx, ctx->cap_stream, true);
  const cudaError_t e = cudaStreamEndCapture(ctx->cap_stream, &L.graph);
  if (s != CS_OK || e != cudaSuccess || cudaGraphInstantiate(&L.exec, L.graph, 0) != cudaSuccess) L.exec = nullptr;
  if (L.graph) cudaGraphDestroy(L.graph);    // (while the first steps run; what replays is a copy)
  L.graph = nullptr;
  (void)cudaGetLastError();
}

// Waits until the progress word tells of more steps than *at, and takes it over.  Ends with an error when the
// stream failed, or ran dry without a report.
cs_status wait_progress(cs_ctx* ctx, LoopProgress* at, cudaStream_t st) {
  cudaError_t state = cudaErrorNotReady;
  for (unsigned spin = 0;; ++spin) {
    if (newer_report([ctx] { return __atomic_load_n(ctx->progress, __ATOMIC_ACQUIRE); }, at)) return CS_OK;
    if (state != cudaErrorNotReady) break;      // (looked once more after the stream had ended)
    if ((spin & 1023u) == 1023u) state = cudaStreamQuery(st);
#if defined(__x86_64__)
    else __builtin_ia32_pause();
#endif
  }
  CS_CUDA_OK(ctx, state);
  return fail(ctx, CS_ERR_CUDA, "a step of the loop ended without reporting its progress");
}

}  // namespace

extern "C" {

size_t cs_workspace_bytes(const cs_model_config* cfg) {
  if (!config_ok(cfg)) return 0;
  return ws_layout(cfg).total;
}

const char* cs_last_error(const cs_ctx* ctx) { return ctx ? ctx->err : g_create_err; }

cs_status cs_create(cs_ctx** out, const cs_model_config* cfg, const cs_weights* w, void* workspace,
                    size_t workspace_bytes) {
  auto create_fail = [](cs_status st, const char* msg) {
    snprintf(g_create_err, sizeof(g_create_err), "cs_create: %s", msg);
    return st;
  };
  if (out == nullptr) return create_fail(CS_ERR_ARG, "NULL output pointer");
  *out = nullptr;
  if (cfg == nullptr || w == nullptr || workspace == nullptr) return create_fail(CS_ERR_ARG, "NULL argument");
  if (!config_ok(cfg)) return create_fail(CS_ERR_SHAPE, "model configuration outside what the kernels support");
  if (w->embed == nullptr || w->lm_head == nullptr || w->final_norm == nullptr || w->attn_norm == nullptr ||
      w->wqkv == nullptr || w->wo == nullptr || w->ffn_norm == nullptr || w->w_gate_up == nullptr ||
      w->w_down == nullptr)
    return create_fail(CS_ERR_ARG, "NULL weight pointer");
  // what the kernels' loads of these need (the matrices' 16 bytes are checked where their operand maps are made)
  bool rows_ok = aligned(w->embed, 8) && aligned(w->final_norm, 8);
  for (int l = 0; l < cfg->n_layers; ++l) rows_ok = rows_ok && aligned(w->attn_norm[l], l == 0 ? 4 : 8) && aligned(w->ffn_norm[l], 8);
  if (!rows_ok) return create_fail(CS_ERR_ARG, "embedding or norm gain not aligned (16 bytes)");
  const WsLayout L = ws_layout(cfg);
  if (workspace_bytes < L.total) return create_fail(CS_ERR_CAPACITY, "workspace smaller than cs_workspace_bytes");
  if (reinterpret_cast<uintptr_t>(workspace) & 1023) return create_fail(CS_ERR_ARG, "workspace not 1024-byte aligned");

  cs_ctx* ctx = new (std::nothrow) cs_ctx();
  if (ctx == nullptr) return create_fail(CS_ERR_ARG, "out of host memory");
  memset(static_cast<void*>(ctx), 0, sizeof(*ctx));
  ctx->cfg = *cfg;
  ctx->max_rows = cfg->max_batch * (cfg->k_max + 1);
  ctx->rows_pad = CS_MAX_ROWS;
  ctx->attn_splits = L.attn_splits;
  {
    // the environment switches of the library, all read here (CS_CHAIN for the size of the workspace too) and nowhere else
    const char* k = getenv("CS_ATTN_KERNEL");
    ctx->attn_force = (k == nullptr) ? 0 : (strcmp(k, "mma") == 0 ? 1 : (strcmp(k, "tc") == 0 ? 2 : (strcmp(k, "tcw") == 0 ? 3 : 0)));
    const char* ng = getenv("CS_NO_GRAPH");
    ctx->no_graph = ng != nullptr && ng[0] == '1';
    ctx->chain_force = chain_switch();
    const char* sm = getenv("CS_SMALL");
    ctx->small_force = sm == nullptr ? 0 : (sm[0] == '0' ? -1 : (sm[0] == '1' ? 1 : 0));
    const char* wl = getenv("CS_WAIT_LIMIT_US");
    const long long us = (wl != nullptr) ? atoll(wl) : 0;
    ctx->wait_limit_ns = (us > 0) ? (unsigned long long)us * 1000ull : 2000000000ull;
    ctx->debug_drop_kb = -1;
    ctx->debug_drop_chain = -1;
  }
  ctx->qkv_elems = L.qkv_elems;
  ctx->layers = new (std::nothrow) LayerPlan[cfg->n_layers];
  cs_status s = CS_OK;
  int dev = 0, major = 0, minor = 0;
#define CREATE_OK(call)                                                                        \
  do {                                                                                         \
    cudaError_t e__ = (call);                                                                  \
    if (e__ != cudaSuccess) {                                                                  \
      snprintf(g_create_err, sizeof(g_create_err), "cs_create: %s: %s", #call, cudaGetErrorString(e__)); \
      cs_destroy(ctx);                                                                         \
      return CS_ERR_CUDA;                                                                      \
    }                                                                                          \
  } while (0)
  if (ctx->layers == nullptr) { cs_destroy(ctx); return create_fail(CS_ERR_ARG, "out of host memory"); }
  CREATE_OK(cudaGetDevice(&dev));
  // (single attributes: reading the whole property table takes milliseconds)
  CREATE_OK(cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev));
  CREATE_OK(cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev));
  CREATE_OK(cudaDeviceGetAttribute(&ctx->num_sms, cudaDevAttrMultiProcessorCount, dev));
  if (major != 10) {
    snprintf(g_create_err, sizeof(g_create_err), "cs_create: this library is built for sm_100a only (device is sm_%d%d)",
             major, minor);
    cs_destroy(ctx);
    return CS_ERR_UNSUPPORTED;
  }
  CREATE_OK(cudaStreamCreateWithFlags(&ctx->cap_stream, cudaStreamNonBlocking));
  CREATE_OK(take_pinned(&ctx->pinned, dev));
  ctx->progress = reinterpret_cast<unsigned long long*>(ctx->pinned.at);
  CREATE_OK(cudaHostGetDevicePointer(reinterpret_cast<void**>(&ctx->progress_dev), ctx->progress, 0));
  ctx->host_ints = reinterpret_cast<int*>(reinterpret_cast<char*>(ctx->progress) + 64);
  ctx->step_in = reinterpret_cast<int*>(reinterpret_cast<char*>(ctx->progress) + kStepInAt);
  ctx->step_in_dev = reinterpret_cast<int*>(reinterpret_cast<char*>(ctx->progress_dev) + kStepInAt);
  ctx->step_out = reinterpret_cast<int*>(reinterpret_cast<char*>(ctx->progress) + kStepOutAt);
  ctx->step_out_dev = reinterpret_cast<int*>(reinterpret_cast<char*>(ctx->progress_dev) + kStepOutAt);
  char* base = static_cast<char*>(workspace);
  ctx->ws = base;
  ctx->ws_bytes = L.total;
  CREATE_OK(cudaMemset(base, 0, L.total));
  ctx->x = reinterpret_cast<float*>(base + L.x);
  ctx->xn = reinterpret_cast<__nv_bfloat16*>(base + L.xn);
  ctx->attn_out = reinterpret_cast<__nv_bfloat16*>(base + L.attn_out);
  ctx->act = reinterpret_cast<__nv_bfloat16*>(base + L.act);
  ctx->qbuf = reinterpret_cast<__nv_bfloat16*>(base + L.qbuf);
  ctx->qkv = reinterpret_cast<float*>(base + L.partial);
  ctx->attn_o = reinterpret_cast<float*>(base + L.attn_o);
  ctx->attn_ml = reinterpret_cast<float*>(base + L.attn_ml);
  ctx->ssq = reinterpret_cast<float*>(base + L.ssq);
  ctx->ssq_stride = cs_ceil_div(ctx->cfg.d_model, CS_GEMM_BM) * CS_MAX_SPLITS;
  ctx->rope_cs = reinterpret_cast<float*>(base + L.rope_cs);
  ctx->inv_freq = reinterpret_cast<double*>(base + L.inv_freq);
  ctx->tile_max = reinterpret_cast<float*>(base + L.tile_max);
  ctx->tile_idx = reinterpret_cast<int*>(base + L.tile_idx);
  ctx->row_tok = reinterpret_cast<int*>(base + L.row_tok);
  ctx->row_pos = reinterpret_cast<int*>(base + L.row_pos);
  ctx->row_lim = reinterpret_cast<int*>(base + L.row_lim);
  ctx->row_write = reinterpret_cast<int*>(base + L.row_write);
  ctx->seq_ok = reinterpret_cast<int*>(base + L.seq_ok);
  ctx->iota = reinterpret_cast<int*>(base + L.iota);
  ctx->pair_part = reinterpret_cast<float*>(base + L.pair_part);
  ctx->pair_flag = reinterpret_cast<int*>(base + L.pair_flag);
  ctx->chain_part = reinterpret_cast<uint4*>(base + L.chain_part);
  ctx->chain_epoch = reinterpret_cast<int*>(base + L.chain_epoch);
  ctx->chain_ctl = reinterpret_cast<int*>(base + L.chain_ctl);
  ctx->d_status = reinterpret_cast<int*>(base + L.status);
  ctx->loop_last = reinterpret_cast<int*>(base + L.loop_last);
  ctx->loop_draft = reinterpret_cast<int*>(base + L.loop_draft);
  ctx->loop_dlen = reinterpret_cast<int*>(base + L.loop_dlen);
  ctx->loop_mpos = reinterpret_cast<int*>(base + L.loop_mpos);
  ctx->loop_emitted = reinterpret_cast<int*>(base + L.loop_emitted);
  ctx->loop_done = reinterpret_cast<int*>(base + L.loop_done);
  ctx->loop_accept = reinterpret_cast<int*>(base + L.loop_accept);
  ctx->loop_out = reinterpret_cast<int*>(base + L.loop_out);
  ctx->loop_argmax = reinterpret_cast<int*>(base + L.loop_argmax);
  ctx->loop_stats = reinterpret_cast<unsigned long long*>(base + L.loop_stats);

  // rotary frequencies theta^(-2i/Dh), in double
  {
    const int half = cfg->head_dim / 2;
    double f[64];
    for (int i = 0; i < half; ++i) f[i] = pow((double)cfg->rope_theta, -2.0 * i / cfg->head_dim);
    CREATE_OK(cudaMemcpy(ctx->inv_freq, f, sizeof(double) * half, cudaMemcpyHostToDevice));
  }
  {
    int ramp[CS_MAX_ROWS];
    for (int i = 0; i < CS_MAX_ROWS; ++i) ramp[i] = i;
    CREATE_OK(cudaMemcpy(ctx->iota, ramp, sizeof(ramp), cudaMemcpyHostToDevice));
  }
  ctx->embed = static_cast<const __nv_bfloat16*>(w->embed);
  ctx->final_norm = static_cast<const __nv_bfloat16*>(w->final_norm);
  const int d = cfg->d_model, qd = cfg->n_heads * cfg->head_dim, F = cfg->d_ffn;
  const int qkv = qd + 2 * cfg->n_kv_heads * cfg->head_dim;
  for (int l = 0; l < cfg->n_layers && s == CS_OK; ++l) {
    LayerPlan& P = ctx->layers[l];
    if (!w->attn_norm[l] || !w->wqkv[l] || !w->wo[l] || !w->ffn_norm[l] || !w->w_gate_up[l] || !w->w_down[l]) {
      s = CS_ERR_ARG;
      break;
    }
    P.attn_norm = static_cast<const __nv_bfloat16*>(w->attn_norm[l]);
    P.ffn_norm = static_cast<const __nv_bfloat16*>(w->ffn_norm[l]);
    if ((s = cs_gemm_plan(ctx, &P.qkv, w->wqkv[l], qkv, d, true)) != CS_OK) break;
    if ((s = cs_gemm_plan(ctx, &P.o, w->wo[l], d, qd, true)) != CS_OK) break;
    if ((s = cs_gemm_plan(ctx, &P.gate_up, w->w_gate_up[l], cs_ceil_div(F, 64) * 128, d, true)) != CS_OK) break;
    if ((s = cs_gemm_plan(ctx, &P.down, w->w_down[l], d, F, true)) != CS_OK) break;
  }
  if (s == CS_OK) s = cs_gemm_plan(ctx, &ctx->lm, w->lm_head, cfg->vocab, d, false);
  if (s != CS_OK) {
    snprintf(g_create_err, sizeof(g_create_err), "cs_create: %.200s", ctx->err[0] ? ctx->err : "NULL layer weight pointer");
    cs_destroy(ctx);
    return s;
  }
#undef CREATE_OK
  *out = ctx;
  return CS_OK;
}

void cs_destroy(cs_ctx* ctx) {
  if (ctx == nullptr) return;
  cs_loop_end(ctx);
  if (ctx->cap_stream) cudaStreamDestroy(ctx->cap_stream);
  give_pinned(ctx->pinned);
  cs_small_free(ctx);
  delete[] ctx->layers;
  delete ctx;
}

cs_status cs_sync_status(cs_ctx* ctx, void* stream) {
  if (ctx == nullptr) return CS_ERR_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int bits = 0;
  const cs_status s = take_status(ctx, &bits, st);
  if (s != CS_OK) return s;
  return status_from_bits(ctx, bits);
}

cs_status cs_find_match(const int32_t* hist, const int32_t* hist_len, int B, int stride, int gamma, int k,
                        cs_match_policy policy, int32_t* match_pos, int32_t* draft, int32_t* draft_len,
                        void* stream) {
  if (B < 0 || k < 0 || stride < 0) return CS_ERR_ARG;
  if (gamma < 1 || gamma > CS_MAX_GAMMA) return CS_ERR_ARG;
  if (policy != CS_MATCH_LATEST && policy != CS_MATCH_FIRST) return CS_ERR_ARG;
  if (B == 0) return CS_OK;
  if (B > 65535) return CS_ERR_ARG;
  if (hist == nullptr || hist_len == nullptr || match_pos == nullptr || draft_len == nullptr ||
      (draft == nullptr && k > 0))
    return CS_ERR_ARG;
  return cs_launch_find_match(hist, hist_len, B, stride, gamma, k, (int)policy, match_pos, draft, draft_len,
                              nullptr, nullptr, static_cast<cudaStream_t>(stream));
}

cs_status cs_verify_step(cs_ctx* ctx, const int32_t* last_tok, const int32_t* draft, const int32_t* draft_len,
                         int B, int k, void* kv_cache, int32_t* kv_len, const int32_t* target_script,
                         int32_t* accept_len, int32_t* out_tokens, int32_t* argmax_ids, float* logits_dbg,
                         void* stream) {
  if (ctx == nullptr) return CS_ERR_ARG;
  if (B < 1 || B > ctx->cfg.max_batch || k < 0 || k > ctx->cfg.k_max) return fail(ctx, CS_ERR_ARG, "B or k out of range");
  if (last_tok == nullptr || draft_len == nullptr || (draft == nullptr && k > 0) || kv_cache == nullptr ||
      kv_len == nullptr || accept_len == nullptr || out_tokens == nullptr || argmax_ids == nullptr)
    return fail(ctx, CS_ERR_ARG, "NULL argument");
  if (!aligned(kv_cache, 16)) return fail(ctx, CS_ERR_ARG, "KV cache not 16-byte aligned");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  ctx->stamp_n = 0;
  cs_launch_block_setup(ctx, last_tok, draft, draft_len, kv_len, nullptr, B, k, true, st);
  ctx->kv_len_early = kv_len;      // the step opened stream-ordered and nothing before the acceptance changes it
  cs_status s = enqueue_forward(ctx, B, k + 1, kv_cache, true, logits_dbg, st);
  ctx->kv_len_early = nullptr;
  if (s != CS_OK) return s;
  cs_launch_accept(ctx, B, k, draft, draft_len, target_script, k + 1, nullptr, k + 1, accept_len, out_tokens,
                   argmax_ids, kv_len, 1, st);
  CS_CUDA_OK(ctx, cudaGetLastError());
  return CS_OK;
}

cs_status cs_step_host(cs_ctx* ctx, int32_t* hist_host, int32_t* hist_len_host, int B, int stride,
                       int32_t* hist_dev, int32_t* hist_len_dev, void* kv_cache, int32_t* kv_len, int gamma, int k,
                       cs_match_policy policy, const int32_t* script_host, int32_t* accept_len_host,
                       int32_t* out_tokens_host, void* stream) {
  if (ctx == nullptr) return CS_ERR_ARG;
  if (B < 1 || B > ctx->cfg.max_batch || k < 0 || k > ctx->cfg.k_max || gamma < 1 || gamma > CS_MAX_GAMMA || stride < 1)
    return fail(ctx, CS_ERR_ARG, "B, k, gamma or stride out of range");
  if (policy != CS_MATCH_LATEST && policy != CS_MATCH_FIRST) return fail(ctx, CS_ERR_ARG, "bad policy");
  if (hist_host == nullptr || hist_len_host == nullptr || hist_dev == nullptr || hist_len_dev == nullptr ||
      kv_cache == nullptr || kv_len == nullptr || accept_len_host == nullptr || out_tokens_host == nullptr)
    return fail(ctx, CS_ERR_ARG, "NULL argument");
  if (!aligned(kv_cache, 16)) return fail(ctx, CS_ERR_ARG, "KV cache not 16-byte aligned");
  for (int b = 0; b < B; ++b)
    if (hist_len_host[b] < 1 || hist_len_host[b] + k + 1 > stride)
      return fail(ctx, CS_ERR_CAPACITY, "history row too short for one more block");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // ---- host -> device: the tokens the device copy of each history lacks (everything on the first
  // call with these buffers, afterwards what the previous call appended), the lengths, this step's
  // script rows
  HostStep& G = ctx->host_step;
  const bool known = G.host == hist_host && G.dev == hist_dev && G.B == B && G.stride == stride;
  G.host = nullptr;                                    // (a call that fails on its way leaves nothing to rely on)
  // ends the call with an error; the input kernel may still be reading the pinned words
  auto give_up = [&](cs_status e) { (void)cudaStreamSynchronize(st); (void)cudaGetLastError(); return e; };
  int* in = ctx->step_in;                              // (every earlier step of this context has been waited for)
  int tokens = 0;
  for (int b = 0; b < B; ++b) {
    const int n = hist_len_host[b];
    int have = (known && G.host_len[b] == n && G.uploaded[b] <= n) ? G.uploaded[b] : 0;
    if (n - have > k + 1) {
      const cudaError_t e = cudaMemcpyAsync(hist_dev + (size_t)b * stride + have, hist_host + (size_t)b * stride + have,
                                            (size_t)(n - have) * 4, cudaMemcpyHostToDevice, st);
      if (e != cudaSuccess) return give_up(fail(ctx, CS_ERR_CUDA, cudaGetErrorString(e)));
      have = n;
    }
    in[b] = n;
    in[B + b] = have;
    in[2 * B + b] = tokens;
    if (n > have) memcpy(in + 3 * B + tokens, hist_host + (size_t)b * stride + have, (size_t)(n - have) * 4);
    tokens += n - have;
    G.uploaded[b] = n;
  }
  const int script_ints = script_host != nullptr ? B * (k + 1) : 0;
  const int32_t* script_dev = script_host != nullptr ? ctx->loop_emitted : nullptr;
  if (script_host != nullptr) memcpy(in + 3 * B + tokens, script_host, (size_t)script_ints * 4);
  *ctx->progress = 0ull;
  cs_launch_host_in(ctx->step_in_dev, B, tokens, script_ints, stride, hist_dev, hist_len_dev, ctx->loop_emitted, st);
  // ---- App. B.3 step 1 (search, gather), step 2 (verify, accept, truncate).  Enqueued launch by launch:
  // the device starts on the first kernel while the rest is enqueued (0.16 ms of host time beside 3.0 ms
  // on the device at the 8B shape, 0.45 beside 3.4 with a launch per projection; a graph replay took 0.16 ms before the first kernel began).
  ctx->stamp_n = 0;
  cs_status s = cs_launch_find_match(hist_dev, hist_len_dev, B, stride, gamma, k, (int)policy, ctx->loop_mpos,
                                     ctx->loop_draft, ctx->loop_dlen, ctx->loop_last, nullptr, st);
  if (s != CS_OK) return give_up(fail(ctx, s, "match kernel launch failed"));
  cs_launch_block_setup(ctx, ctx->loop_last, ctx->loop_draft, ctx->loop_dlen, kv_len, nullptr, B, k, false, st);
  // every call ends when its last kernel has reported, and k_block_setup lets nothing pass that was enqueued
  // earlier, so the cached rows and kv_len are settled while the forward runs
  ctx->kv_len_early = kv_len;
  s = enqueue_forward(ctx, B, k + 1, kv_cache, true, nullptr, st);
  ctx->kv_len_early = nullptr;
  if (s != CS_OK) return give_up(s);
  cs_launch_accept(ctx, B, k, ctx->loop_draft, ctx->loop_dlen, script_dev, k + 1, nullptr, k + 1, ctx->loop_accept,
                   ctx->loop_out, ctx->loop_argmax, kv_len, 1, st);
  // ---- device -> host, then step 4 on the host: append what was emitted
  cs_launch_host_out(ctx->loop_accept, ctx->loop_out, B, k, ctx->step_out_dev, ctx->progress_dev, st);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return give_up(fail(ctx, CS_ERR_CUDA, cudaGetErrorString(e)));
  LoopProgress done = {0, 0};
  s = wait_progress(ctx, &done, st);
  if (s != CS_OK) return give_up(s);
  memcpy(accept_len_host, ctx->step_out, (size_t)B * 4);
  memcpy(out_tokens_host, ctx->step_out + CS_MAX_ROWS, (size_t)B * (k + 1) * 4);
  for (int b = 0; b < B; ++b) {
    const int tau = accept_len_host[b];
    if (tau < 0 || tau > k) continue;                  // the device skipped this sequence (status word)
    const int n = hist_len_host[b];
    for (int i = 0; i <= tau; ++i) hist_host[(size_t)b * stride + n + i] = out_tokens_host[(size_t)b * (k + 1) + i];
    hist_len_host[b] = n + tau + 1;
  }
  for (int b = 0; b < B; ++b) G.host_len[b] = hist_len_host[b];
  G.host = hist_host; G.dev = hist_dev; G.B = B; G.stride = stride;
  return CS_OK;
}

void cs_step_host_reset(cs_ctx* ctx) {
  if (ctx != nullptr) ctx->host_step.host = nullptr;
}

cs_status cs_debug_drop_tile(cs_ctx* ctx, int k_block) {
  if (ctx == nullptr) return CS_ERR_ARG;
  ctx->debug_drop_kb = k_block < 0 ? -1 : k_block;
  return CS_OK;
}

cs_status cs_debug_drop_chain_tile(cs_ctx* ctx, int unit) {
  if (ctx == nullptr) return CS_ERR_ARG;
  ctx->debug_drop_chain = unit < 0 ? -1 : unit;
  return CS_OK;
}

cs_status cs_debug_leave_shares(cs_ctx* ctx, int mask) {
  if (ctx == nullptr || mask < 0 || mask >= 1 << CS_PAIR_MAX_SPLITS) return CS_ERR_ARG;
  ctx->debug_leave = mask;
  return CS_OK;
}

cs_status cs_kv_truncate(cs_ctx* ctx, int32_t* kv_len, const int32_t* new_len, int B, void* stream) {
  if (ctx == nullptr) return CS_ERR_ARG;
  if (B < 0 || kv_len == nullptr || new_len == nullptr) return fail(ctx, CS_ERR_ARG, "bad argument");
  if (B == 0) return CS_OK;
  cs_launch_truncate(ctx, kv_len, new_len, B, static_cast<cudaStream_t>(stream));
  CS_CUDA_OK(ctx, cudaGetLastError());
  return CS_OK;
}

cs_status cs_prefill(cs_ctx* ctx, const int32_t* hist, const int32_t* hist_len, int B, int stride, int max_len,
                     void* kv_cache, int32_t* kv_len, void* stream) {
  if (ctx == nullptr) return CS_ERR_ARG;
  if (B < 1 || B > ctx->cfg.max_batch || hist == nullptr || hist_len == nullptr || kv_cache == nullptr ||
      kv_len == nullptr || max_len < 0 || stride < max_len)
    return fail(ctx, CS_ERR_ARG, "bad argument");
  if (!aligned(kv_cache, 16)) return fail(ctx, CS_ERR_ARG, "KV cache not 16-byte aligned");
  if (max_len - 1 > ctx->cfg.max_seq) return fail(ctx, CS_ERR_CAPACITY, "history longer than the KV cache");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int R = CS_MAX_ROWS / B;
  const int total = max_len - 1;   // positions whose K/V are cached
  for (int start = 0; start < total; start += R) {
    const int r = (total - start < R) ? total - start : R;
    ctx->stamp_n = 0;
    cs_launch_prefill_setup(ctx, hist, hist_len, B, stride, start, r, st);
    cs_status s = enqueue_forward(ctx, B, r, kv_cache, false, nullptr, st);
    if (s != CS_OK) return s;
  }
  if (total <= 0) cs_launch_prefill_setup(ctx, hist, hist_len, B, stride, 0, 1, st);   // sets seq_ok
  cs_launch_prefill_finish(ctx, hist_len, kv_len, B, st);
  CS_CUDA_OK(ctx, cudaGetLastError());
  return CS_OK;
}

// Checks a loop's arguments, sets its state up and enqueues the initialisation.
static cs_status loop_prepare(cs_ctx* ctx, int32_t* hist, int32_t* hist_len, int B, int stride, void* kv_cache,
                              int32_t* kv_len, int gamma, int k, cs_match_policy policy, int max_new, int eos_id,
                              const int32_t* script, void* stream) {
  if (ctx == nullptr) return CS_ERR_ARG;
  if (B < 1 || B > ctx->cfg.max_batch || k < 0 || k > ctx->cfg.k_max || gamma < 1 || gamma > CS_MAX_GAMMA ||
      max_new < 0 || stride < 1)
    return fail(ctx, CS_ERR_ARG, "B, k, gamma, max_new or stride out of range");
  if (policy != CS_MATCH_LATEST && policy != CS_MATCH_FIRST) return fail(ctx, CS_ERR_ARG, "bad policy");
  if (hist == nullptr || hist_len == nullptr || kv_cache == nullptr || kv_len == nullptr)
    return fail(ctx, CS_ERR_ARG, "NULL argument");
  if (!aligned(kv_cache, 16)) return fail(ctx, CS_ERR_ARG, "KV cache not 16-byte aligned");
  cs_loop_end(ctx);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  LoopState& L = ctx->loop;
  L.hist = hist; L.hist_len = hist_len; L.B = B; L.stride = stride; L.kv_cache = kv_cache; L.kv_len = kv_len;
  L.gamma = gamma; L.k = k; L.policy = (int)policy; L.max_new = max_new; L.eos_id = eos_id; L.script = script;
  L.use_graph = false;
  L.use_index = ctx->match_index != nullptr;
  if (L.use_index) {
    if (ctx->match_index_cap < stride) return fail(ctx, CS_ERR_CAPACITY, "the gamma-gram index is sized for fewer tokens than a history row holds");
    // built afresh from the histories as they stand
    cs_status r = cs_gram_index_reset(ctx->match_index, B, ctx->match_index_cap, st);
    if (r == CS_OK) r = cs_launch_gram_update(ctx->match_index, B, ctx->match_index_cap, hist, hist_len, stride, gamma, 64, ctx->d_status, st);
    if (r != CS_OK) return fail(ctx, r, "index build failed");
  }

  cs_launch_loop_init(ctx, hist_len, kv_len, B, stride, max_new, k, st);
  CS_CUDA_OK(ctx, cudaGetLastError());
  // the activation maps must exist before a capture (encoding them is host work)
  return ensure_act_maps(ctx, B * (k + 1));
}

cs_status cs_loop_begin(cs_ctx* ctx, int32_t* hist, int32_t* hist_len, int B, int stride, void* kv_cache,
                        int32_t* kv_len, int gamma, int k, cs_match_policy policy, int max_new, int eos_id,
                        const int32_t* script, void* stream) {
  cs_status s = loop_prepare(ctx, hist, hist_len, B, stride, kv_cache, kv_len, gamma, k, policy, max_new, eos_id, script, stream);
  if (s != CS_OK) return s;
  LoopState& L = ctx->loop;
  L.use_graph = !ctx->no_graph;
  if (L.use_graph) {
    // captured on the context's own stream (the legacy default stream cannot capture),
    // replayed on the caller's
    CS_CUDA_OK(ctx, cudaStreamBeginCapture(ctx->cap_stream, cudaStreamCaptureModeRelaxed));
    s = enqueue_loop_step(ctx, ctx->cap_stream);
    cudaError_t e = cudaStreamEndCapture(ctx->cap_stream, &L.graph);
    if (s != CS_OK) { cs_loop_end(ctx); return s; }
    if (e != cudaSuccess) { cs_loop_end(ctx); CS_CUDA_OK(ctx, e); }
    e = cudaGraphInstantiate(&L.exec, L.graph, 0);
    if (e != cudaSuccess) { cs_loop_end(ctx); CS_CUDA_OK(ctx, e); }
    size_t nodes = 0;
    if (cudaGraphGetNodes(L.graph, nullptr, &nodes) == cudaSuccess) L.graph_nodes = (int)nodes;
    // the same step CS_LOOP_UNROLL times over in one graph, for runs of several steps
    CS_CUDA_OK(ctx, cudaStreamBeginCapture(ctx->cap_stream, cudaStreamCaptureModeRelaxed));
    for (int i = 0; i < CS_LOOP_UNROLL && s == CS_OK; ++i) s = enqueue_loop_step(ctx, ctx->cap_stream);
    e = cudaStreamEndCapture(ctx->cap_stream, &L.graph_n);
    if (s != CS_OK) { cs_loop_end(ctx); return s; }
    if (e != cudaSuccess) { cs_loop_end(ctx); CS_CUDA_OK(ctx, e); }
    e = cudaGraphInstantiate(&L.exec_n, L.graph_n, 0);
    if (e != cudaSuccess) { cs_loop_end(ctx); CS_CUDA_OK(ctx, e); }
  }
  L.active = true;
  return CS_OK;
}

cs_status cs_loop_steps(cs_ctx* ctx, int n_steps, void* stream) {
  if (ctx == nullptr) return CS_ERR_ARG;
  if (!ctx->loop.active || n_steps < 0) return fail(ctx, CS_ERR_ARG, "no loop in progress");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  for (int i = 0; i < n_steps; ++i) {
    if (ctx->loop.use_graph) {
      if (n_steps - i >= CS_LOOP_UNROLL && ctx->loop.exec_n != nullptr) {
        CS_CUDA_OK(ctx, cudaGraphLaunch(ctx->loop.exec_n, st));
        i += CS_LOOP_UNROLL - 1;
        continue;
      }
      CS_CUDA_OK(ctx, cudaGraphLaunch(ctx->loop.exec, st));
    } else {
      cs_status s = enqueue_loop_step(ctx, st);
      if (s != CS_OK) return s;
    }
  }
  return CS_OK;
}

cs_status cs_loop_poll(cs_ctx* ctx, cs_stats* stats_out, int* n_done_out, void* stream) {
  if (ctx == nullptr) return CS_ERR_ARG;
  if (!ctx->loop.active) return fail(ctx, CS_ERR_ARG, "no loop in progress");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int done = 0, bits = 0;
  CS_CUDA_OK(ctx, cudaMemcpyAsync(&done, ctx->loop_done + ctx->cfg.max_batch, sizeof(int), cudaMemcpyDeviceToHost, st));
  if (stats_out != nullptr)
    CS_CUDA_OK(ctx, cudaMemcpyAsync(stats_out, ctx->loop_stats, sizeof(cs_stats), cudaMemcpyDeviceToHost, st));
  const cs_status s = take_status(ctx, &bits, st);   // (one synchronisation for all three)
  if (s != CS_OK) return s;
  if (n_done_out != nullptr) *n_done_out = done;
  return status_from_bits(ctx, bits);
}

cs_status cs_loop_last_step(cs_ctx* ctx, int32_t* match_pos_host, int32_t* draft_len_host, int32_t* accept_len_host,
                            int32_t* out_tokens_host, int32_t* argmax_ids_host, void* stream) {
  if (ctx == nullptr) return CS_ERR_ARG;
  if (!ctx->loop.active) return fail(ctx, CS_ERR_ARG, "no loop in progress");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const size_t B = (size_t)ctx->loop.B, R = (size_t)ctx->loop.k + 1;
  const struct { int32_t* dst; const int* src; size_t n; } copies[5] = {
      {match_pos_host, ctx->loop_mpos, B},        {draft_len_host, ctx->loop_dlen, B},
      {accept_len_host, ctx->loop_accept, B},     {out_tokens_host, ctx->loop_out, B * R},
      {argmax_ids_host, ctx->loop_argmax, B * R}};
  for (const auto& c : copies)
    if (c.dst != nullptr) CS_CUDA_OK(ctx, cudaMemcpyAsync(c.dst, c.src, c.n * 4, cudaMemcpyDeviceToHost, st));
  CS_CUDA_OK(ctx, cudaStreamSynchronize(st));
  return CS_OK;
}

int cs_loop_launches_per_step(const cs_ctx* ctx) {
  return (ctx != nullptr && ctx->loop.active) ? ctx->loop.graph_nodes : 0;
}

void cs_loop_end(cs_ctx* ctx) {
  if (ctx == nullptr) return;
  if (ctx->loop.exec) cudaGraphExecDestroy(ctx->loop.exec);
  if (ctx->loop.graph) cudaGraphDestroy(ctx->loop.graph);
  if (ctx->loop.exec_n) cudaGraphExecDestroy(ctx->loop.exec_n);
  if (ctx->loop.graph_n) cudaGraphDestroy(ctx->loop.graph_n);
  ctx->loop.exec = nullptr;
  ctx->loop.graph = nullptr;
  ctx->loop.exec_n = nullptr;
  ctx->loop.graph_n = nullptr;
  ctx->loop.active = false;
}

cs_status cs_decode_loop(cs_ctx* ctx, int32_t* hist, int32_t* hist_len, int B, int stride, void* kv_cache,
                         int32_t* kv_len, int gamma, int k, cs_match_policy policy, int max_new, int eos_id,
                         const int32_t* script, cs_stats* stats_out, void* stream) {
  cs_status s = loop_prepare(ctx, hist, hist_len, B, stride, kv_cache, kv_len, gamma, k, policy, max_new, eos_id,
                             script, stream);
  if (s != CS_OK) return s;
  // The first two steps are enqueued launch by launch (0.16 ms of host time each against 3.0 ms on the device at
  // the 8B shape, 0.45 against 3.4 with a launch per projection, 42 against 72 us for two small layers), at most two ahead of the device.  The device
  // reports after every step how many tokens are still wanted, and a step is enqueued ahead of that report
  // only where it is needed whatever the steps in flight accept: the loop used to look every four
  // steps and ran up to three whole forwards for nothing.
  // While those two run the host captures the step and replays it from then on: with a launch per projection a step
  // enqueued directly takes 3.44 instead of 3.35 ms.  (Chained layers do not need it: calls of 4, 8, 11 and 24 steps at the 8B shape
  // take 2.97, 2.97, 2.95 and 2.96 ms a step with a graph, 2.97, 2.96, 2.96 and 2.96 without.)  Building the graph takes 1 - 2 ms, so it is only done where
  // two steps last longer (32 MB of weights a layer; at 2 MB they last 0.15 ms) and at least three more are certain.
  // Calls of 8 steps with a graph and without, us a step: 24 layers of 34 MB 957 / 1,006, 28 of 93 MB 1,393 / 1,442, 16 of
  // 122 MB 935 / 965.  Destroying the graph takes 0.1 - 0.6 ms, so that is done while what will likely be the last steps
  // run (it may be in flight then: the driver frees it when they are done); steps still needed after that are enqueued.
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  ctx->loop.active = true;
  *ctx->progress = 0ull;               // (every earlier loop of this context has been waited for)
  bool whole = false;
  s = cs_launch_small_loop(ctx, &whole, st);
  if (whole) {
    // a small model: all steps are in one launch, which reports once
    LoopProgress at = {0, max_new};
    s = wait_progress(ctx, &at, st);
    if (s == CS_OK) {
      const unsigned long long* report = reinterpret_cast<const unsigned long long*>(ctx->step_out);
      if (stats_out != nullptr) memcpy(stats_out, report + 1, sizeof(cs_stats));
      const int bits = (int)report[0];
      // (as in take_status: the bit may be an earlier forward's)
      if ((bits & CS_DEV_TIMEOUT) && (cudaMemsetAsync(ctx->pair_flag, 0, CS_MAX_PAIRS * 2 * sizeof(int), st) != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess))
        (void)cudaGetLastError();
      s = status_from_bits(ctx, bits);
    } else {
      (void)cudaStreamSynchronize(st);
    }
    cs_loop_end(ctx);
    return s;
  }
  if (s != CS_OK) { cs_loop_end(ctx); return s; }
  auto send = [&](int sent, int wanted) {
    cs_status r;
    if (ctx->loop.exec != nullptr) {
      const cudaError_t e = cudaGraphLaunch(ctx->loop.exec, st);
      r = e == cudaSuccess ? CS_OK : fail(ctx, CS_ERR_CUDA, cudaGetErrorString(e));
    } else {
      r = enqueue_loop_step(ctx, st, true);
    }
    if (sent == 2 && r == CS_OK && wanted > (long)4 * (k + 1) && !ctx->no_graph && cs_layer_bytes(ctx->cfg) >= (32ll << 20))
      capture_step(ctx);
    return r;
  };
  auto wait = [&](LoopProgress* at, int sent) {
    if (ctx->loop.exec != nullptr && likely_last(*at, sent, max_new)) {
      cudaGraphExecDestroy(ctx->loop.exec);
      ctx->loop.exec = nullptr;
    }
    return wait_progress(ctx, at, st);
  };
  s = (cs_status)drive_loop(max_new, k, send, wait);
  // A status that concerns single sequences (no room, inconsistent lengths: those were marked
  // finished and left alone while the others ran to their end) is returned here as well.
  if (s == CS_OK) s = cs_loop_poll(ctx, stats_out, nullptr, stream);
  else (void)cudaStreamSynchronize(st);
  cs_loop_end(ctx);
  return s;
}

cs_status cs_set_match_index(cs_ctx* ctx, void* index, int capacity_tokens) {
  if (ctx == nullptr || (index != nullptr && capacity_tokens < 1)) return CS_ERR_ARG;
  if (ctx->loop.active) return fail(ctx, CS_ERR_ARG, "the search method cannot change while a loop is in progress");
  ctx->match_index = index;
  ctx->match_index_cap = index != nullptr ? capacity_tokens : 0;
  return CS_OK;
}

cs_status cs_set_stamps(cs_ctx* ctx, unsigned long long* stamps, int capacity) {
  if (ctx == nullptr || capacity < 0) return CS_ERR_ARG;
  if (ctx->loop.active) return fail(ctx, CS_ERR_ARG, "stamps cannot change while a loop is in progress (its graph holds the slots)");
  ctx->stamp_buf = (capacity > 0) ? stamps : nullptr;
  ctx->stamp_cap = (stamps != nullptr) ? capacity : 0;
  ctx->stamp_n = 0;
  return CS_OK;
}

int cs_stamp_layout(const cs_ctx* ctx, int* family, int capacity) {
  if (ctx == nullptr) return 0;
  for (int i = 0; i < ctx->stamp_n && i < capacity && family != nullptr; ++i) family[i] = ctx->stamp_fam[i];
  return ctx->stamp_n;
}

cs_status cs_linear(cs_ctx* ctx, const void* X, const void* W, int rows, int N, int K, float* Y, void* stream) {
  if (ctx == nullptr) return CS_ERR_ARG;
  if (X == nullptr || W == nullptr || Y == nullptr || rows < 1 || rows > CS_MAX_ROWS || N < 1 || K < 8 || (K % 8))
    return fail(ctx, CS_ERR_ARG, "bad argument");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  GemmPlan g;
  cs_status s = cs_gemm_plan(ctx, &g, W, N, K, true);
  if (s != CS_OK) return s;
  const int n_tok = cs_ceil_div(rows, 16) * 16;
  CUtensorMap tmX;
  if ((s = cs_make_act_map(ctx, &tmX, X, n_tok, K, cs_gemm_act_box(CS_EPI_STORE, rows, false))) != CS_OK) return s;
  return cs_launch_gemm(ctx, &g, &tmX, -1, rows, CS_EPI_STORE, Y, nullptr, nullptr, 0, nullptr, nullptr, st);
}

cs_status cs_lm_head(cs_ctx* ctx, const void* X, int rows, int32_t* ids, float* logits_dbg, void* stream) {
  if (ctx == nullptr) return CS_ERR_ARG;
  if (X == nullptr || ids == nullptr || rows < 1 || rows > CS_MAX_ROWS) return fail(ctx, CS_ERR_ARG, "bad argument");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int n_tok = cs_ceil_div(rows, 16) * 16;
  CUtensorMap tmX;
  cs_status s = cs_make_act_map(ctx, &tmX, X, n_tok, ctx->cfg.d_model, cs_gemm_act_box(CS_EPI_ARGMAX, rows, false));
  if (s != CS_OK) return s;
  if ((s = cs_launch_gemm(ctx, &ctx->lm, &tmX, -1, rows, CS_EPI_ARGMAX, logits_dbg, nullptr, nullptr, 0, nullptr, nullptr, st)) != CS_OK) return s;
  cs_launch_tile_reduce(ctx, rows, ids, st);
  CS_CUDA_OK(ctx, cudaGetLastError());
  return CS_OK;
}

}  // extern "C"
