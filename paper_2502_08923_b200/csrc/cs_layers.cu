// The small kernels around the GEMMs and the attention of the verification forward
// (Sec. 3.2; App. B.2): block assembly (rows, positions, rotary table), embedding lookup with
// the first RMSNorm, the merge of the attention's key slices, the reduction of the LM-head
// tile maxima with prefix acceptance, KV truncation, and the loop's init and commit steps.
// RoPE, the K/V append, SwiGLU, the residual adds and every later RMSNorm live in the GEMM
// epilogues (cs_gemm.cu, cs_gemm_pair.cu); attention is in cs_attn_tc.cu, cs_attn_tcw.cu and cs_attn.cu.
#include <math.h>

#include <algorithm>

#include "cs_common.cuh"

namespace {

// A wait that ran out may have left words raised by which the two-SM GEMM's pairs hand sums over, and the
// next forward would take sums of the one before.  Everything enqueued earlier is complete where this is called.
__device__ __forceinline__ void lower_pair_flags(const int* status, int* pair_flag) {
  if (blockIdx.x == 0 && (__ldcg(status) & CS_DEV_TIMEOUT) != 0)
    for (int i = threadIdx.x; i < 2 * CS_MAX_PAIRS; i += blockDim.x) pair_flag[i] = 0;
}

// Counters and "done" words of the forward's chained projections (cs_chain.cu) start at zero.  Their kernels may take runs
// ahead of their own wait, so a set-up kernel clears the words before it lets its dependents go.
__device__ __forceinline__ void clear_chain_words(int4* words, int quads, int* epoch) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *epoch = __ldcg(epoch) + 1;   // (marks the sums of this forward)
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < quads; i += gridDim.x * blockDim.x) words[i] = make_int4(0, 0, 0, 0);
  __threadfence();
  __syncthreads();
}

// ----------------------------------------------------------------- block assembly
// Rows of sequence b: r = 0 is the last accepted token, r = 1..draft_len[b] the draft
// (Sec. 3.2: the speculative tokens are appended to the context).  Rows past the draft
// are dead: they are computed but attend to nothing and write nothing.  The first CTA fills in the
// rows, all share the rotary table, whose fp64 sincos bound the kernel (one CTA for everything before:
// 17.8 -> 3.4 us at 168 rows, 22.0 -> 2.6 at 256).  Dependents are let go behind the wait and not ahead of it: the search in front of this
// kernel is launched early itself, and kernels further down the chain read cached rows and lengths
// ahead of their own waits, relying on the step before being complete.
// Words that other kernels of the chain write (the search's results, lengths, rows, tile maxima) are read through L2, here
// and in every kernel of the library that starts early: it may be resident while they still change, and the read-only
// path, which a const __restrict__ pointer allows the compiler, is not coherent across that.
constexpr int kSetupThreads = 256;
__global__ void __launch_bounds__(kSetupThreads)
k_block_setup(const int* last_tok, const int* draft, const int* draft_len, const int* kv_len,
                              const int* skip, int B, int k, int max_seq, int vocab,
                              int half, const double* __restrict__ inv_freq, int* row_tok, int* row_pos,
                              int* row_lim, int* row_write, int* seq_ok, float* rope_cs, int* status,
                              int* pair_flag, int4* chain_words, int chain_quads, int* chain_epoch, unsigned long long* stamp) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (chain_quads > 0) clear_chain_words(chain_words, chain_quads, chain_epoch);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  lower_pair_flags(status, pair_flag);
  const int R = k + 1, rows = B * R;
  for (int row = threadIdx.x; row < rows && blockIdx.x == 0; row += kSetupThreads) {
    const int b = row / R, r = row % R;
    int dl = __ldcg(draft_len + b);
    dl = dl < 0 ? 0 : (dl > k ? k : dl);
    const int kv = __ldcg(kv_len + b);
    const bool skipped = (skip != nullptr && __ldcg(skip + b) != 0);
    const bool fits = (kv >= 0 && kv + dl + 1 <= max_seq);
    const bool ok = fits && !skipped;
    if (r == 0) {
      seq_ok[b] = ok ? 1 : 0;
      if (!fits && !skipped) atomicOr(status, CS_DEV_CAPACITY);
    }
    const bool valid = ok && r <= dl;
    int tok = __ldcg((r == 0 || !valid) ? last_tok + b : draft + (size_t)b * k + r - 1);
    tok = tok < 0 ? 0 : (tok >= vocab ? vocab - 1 : tok);
    row_tok[row] = tok;
    row_pos[row] = (kv < 0 ? 0 : kv) + r;
    row_lim[row] = valid ? kv + r + 1 : 0;
    row_write[row] = valid ? 1 : 0;
  }
  for (int i = blockIdx.x * kSetupThreads + threadIdx.x; i < rows * half; i += gridDim.x * kSetupThreads) {
    const int row = i / half, j = i % half;
    const int b = row / R, r = row % R;
    const int kv = __ldcg(kv_len + b);
    const double ang = (double)((kv < 0 ? 0 : kv) + r) * inv_freq[j];
    double s, c;
    sincos(ang, &s, &c);
    rope_cs[2 * i] = (float)c;
    rope_cs[2 * i + 1] = (float)s;
  }
  if (stamp != nullptr) {
    __syncthreads();
    if (threadIdx.x == 0) cs_stamp_end(stamp);
  }
}

// Forced rows for filling the cache from a history: row r of sequence b is token
// hist[b][start + r]; only positions below hist_len[b] - 1 are computed.
__global__ void __launch_bounds__(kSetupThreads)
k_prefill_setup(const int* hist, const int* hist_len, int B,
                                int stride, int start, int R, int max_seq, int vocab, int half,
                                const double* __restrict__ inv_freq, int* row_tok, int* row_pos,
                                int* row_lim, int* row_write, int* seq_ok, float* rope_cs, int* status, int* pair_flag,
                                int4* chain_words, int chain_quads, int* chain_epoch) {
  if (chain_quads == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (chain_quads > 0) {
    clear_chain_words(chain_words, chain_quads, chain_epoch);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  }
  lower_pair_flags(status, pair_flag);
  const int rows = B * R;
  for (int row = threadIdx.x; row < rows && blockIdx.x == 0; row += kSetupThreads) {
    const int b = row / R, r = row % R;
    const int p = start + r;
    const int n = __ldcg(hist_len + b);
    const bool fits = (n - 1 <= max_seq && n <= stride);
    if (r == 0) {
      seq_ok[b] = fits ? 1 : 0;
      if (!fits) atomicOr(status, CS_DEV_CAPACITY);
    }
    const bool valid = fits && p < n - 1;
    int tok = valid ? __ldcg(hist + (size_t)b * stride + p) : 0;
    tok = tok < 0 ? 0 : (tok >= vocab ? vocab - 1 : tok);
    row_tok[row] = tok;
    row_pos[row] = p;
    row_lim[row] = valid ? p + 1 : 0;
    row_write[row] = valid ? 1 : 0;
  }
  for (int i = blockIdx.x * kSetupThreads + threadIdx.x; i < rows * half; i += gridDim.x * kSetupThreads) {
    const int row = i / half, j = i % half;
    const double ang = (double)(start + row % R) * inv_freq[j];
    double s, c;
    sincos(ang, &s, &c);
    rope_cs[2 * i] = (float)c;
    rope_cs[2 * i + 1] = (float)s;
  }
}

// Embedding lookup and the first RMSNorm in one pass: x = E[token] (fp32 residual stream) and
// xn = x * rsqrt(mean(x^2) + eps) * g as two bf16 terms (hi, lo).  One CTA per row; the row is
// read once and kept in registers (up to 4 float4 per thread).  Every later norm is folded
// into the GEMMs around it.
constexpr int kNormThreads = 1024;
__global__ void __launch_bounds__(kNormThreads)
k_embed_rmsnorm(const __nv_bfloat16* __restrict__ E, const int* row_tok, float* __restrict__ x, int d,
                const __nv_bfloat16* __restrict__ gain, float eps, __nv_bfloat16* __restrict__ xn,
                __nv_bfloat16* __restrict__ xn_lo, unsigned long long* stamp) {
  CS_PDL_PROLOGUE();
  const int row = blockIdx.x;
  const __nv_bfloat16* er = E + (size_t)__ldcg(row_tok + row) * d;
  float* xr = x + (size_t)row * d;
  auto fetch = [&](int i) {
    const uint2 w = *reinterpret_cast<const uint2*>(er + i);          // four bf16
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w.y));
    const float4 v = make_float4(a.x, a.y, b.x, b.y);
    *reinterpret_cast<float4*>(xr + i) = v;
    return v;
  };
  float4 v[4];
  float ss = 0.f;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = (q * kNormThreads + threadIdx.x) * 4;
    v[q] = (i < d) ? fetch(i) : make_float4(0.f, 0.f, 0.f, 0.f);
    ss += v[q].x * v[q].x + v[q].y * v[q].y + v[q].z * v[q].z + v[q].w * v[q].w;
  }
  for (int i = 4 * kNormThreads * 4 + threadIdx.x * 4; i < d; i += kNormThreads * 4) {   // d > 16384
    const float4 w = fetch(i);
    ss += w.x * w.x + w.y * w.y + w.z * w.z + w.w * w.w;
  }
  __shared__ float red[32];
  __shared__ float s_scale;
  for (int off = 16; off > 0; off >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  if (threadIdx.x < 32) {
    float t = red[threadIdx.x];
    for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
    if (threadIdx.x == 0) s_scale = rsqrtf(t / (float)d + eps);
  }
  __syncthreads();
  const float sc = s_scale;
  auto emit = [&](int i, const float4& w) {
    const float2 g0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(gain + i));
    const float2 g1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(gain + i + 2));
    const float y0 = w.x * sc * g0.x, y1 = w.y * sc * g0.y, y2 = w.z * sc * g1.x, y3 = w.w * sc * g1.y;
    const __nv_bfloat162 o0 = __floats2bfloat162_rn(y0, y1), o1 = __floats2bfloat162_rn(y2, y3);
    *reinterpret_cast<__nv_bfloat162*>(xn + (size_t)row * d + i) = o0;
    *reinterpret_cast<__nv_bfloat162*>(xn + (size_t)row * d + i + 2) = o1;
    // second term: what the first rounding lost
    const float2 h0 = __bfloat1622float2(o0), h1 = __bfloat1622float2(o1);
    *reinterpret_cast<__nv_bfloat162*>(xn_lo + (size_t)row * d + i) = __floats2bfloat162_rn(y0 - h0.x, y1 - h0.y);
    *reinterpret_cast<__nv_bfloat162*>(xn_lo + (size_t)row * d + i + 2) = __floats2bfloat162_rn(y2 - h1.x, y3 - h1.y);
  };
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = (q * kNormThreads + threadIdx.x) * 4;
    if (i < d) emit(i, v[q]);
  }
  for (int i = 4 * kNormThreads * 4 + threadIdx.x * 4; i < d; i += kNormThreads * 4)
    emit(i, *reinterpret_cast<const float4*>(xr + i));
  if (stamp != nullptr) {
    __syncthreads();
    if (threadIdx.x == 0) cs_stamp_end(stamp);
  }
}

// Combine the key slices: o = sum_s o_s e^(m_s - M) / sum_s l_s e^(m_s - M).  W warps per (row, head), each
// taking every W-th slice, at most NS of them; a lane holds four dims.  All of a thread's partial outputs
// are requested at once, so their latencies overlap each other and the weight computation.  Bound by
// that latency.  Measured (one thread per dim and all slices before): at 11 rows x 32 heads x 33 slices 5.8 -> 5.5 us (4.6
// with the 18 slices that the tcgen05 kernels leave of one sequence now); at 176 rows and one slice 5.6 -> 3.1, at 256 rows and
// four slices 8.5 -> 3.6 (and the next kernel starts 2 us earlier: a quarter of the CTAs hold thread slots).
constexpr int kMergeThreads = 128;
template <int W, int NS>
__global__ void __launch_bounds__(kMergeThreads)
k_attn_merge(const float* __restrict__ in_o, const float* __restrict__ in_ml, int nsplit, int rows, int H, int Dh,
             __nv_bfloat16* __restrict__ attn_out, unsigned long long* stamp) {
  CS_PDL_PROLOGUE();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, part = warp % W;
  const long long rh = (long long)blockIdx.x * (kMergeThreads / 32 / W) + warp / W, total = (long long)rows * H;   // (row, head)
  const bool live = rh < total, has = live && 4 * lane < Dh;
  float4 v[NS];
#pragma unroll
  for (int i = 0; i < NS; ++i) {
    const int s = part + i * W;
    v[i] = has && s < nsplit ? __ldcg(reinterpret_cast<const float4*>(in_o + ((size_t)s * total + rh) * Dh + 4 * lane))
                             : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  // every warp works out the slice weights e^(m_s - M) / L itself: lane s owns slices s, s + 32
  float2 a = make_float2(-INFINITY, 0.f), b = a;
  if (live && lane < nsplit) a = __ldcg(reinterpret_cast<const float2*>(in_ml) + (size_t)lane * total + rh);
  if (W * NS > 32 && live && lane + 32 < nsplit) b = __ldcg(reinterpret_cast<const float2*>(in_ml) + (size_t)(lane + 32) * total + rh);
  float M = fmaxf(a.x, b.x);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, off));
  float w0 = (a.x == -INFINITY) ? 0.f : expf(a.x - M), w1 = (b.x == -INFINITY) ? 0.f : expf(b.x - M);
  float L = a.y * w0 + b.y * w1;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) L += __shfl_xor_sync(0xffffffffu, L, off);
  const float inv = L > 0.f ? 1.f / L : 0.f;
  w0 *= inv; w1 *= inv;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int i = 0; i < NS; ++i) {
    const int s = part + i * W;
    const float w = __shfl_sync(0xffffffffu, s < 32 ? w0 : w1, s & 31);
    acc.x = fmaf(v[i].x, w, acc.x); acc.y = fmaf(v[i].y, w, acc.y);
    acc.z = fmaf(v[i].z, w, acc.z); acc.w = fmaf(v[i].w, w, acc.w);
  }
  if (W > 1) {
    __shared__ float4 sums[kMergeThreads];
    sums[threadIdx.x] = acc;
    __syncthreads();
    if (part == 0) {
#pragma unroll
      for (int q = 1; q < W; ++q) {
        const float4 o = sums[threadIdx.x + 32 * q];
        acc.x += o.x; acc.y += o.y; acc.z += o.z; acc.w += o.w;
      }
    }
  }
  if (part == 0 && has) {
    const __nv_bfloat162 h0 = __floats2bfloat162_rn(acc.x, acc.y), h1 = __floats2bfloat162_rn(acc.z, acc.w);
    const float2 f0 = __bfloat1622float2(h0), f1 = __bfloat1622float2(h1);
    const __nv_bfloat162 l0 = __floats2bfloat162_rn(acc.x - f0.x, acc.y - f0.y), l1 = __floats2bfloat162_rn(acc.z - f1.x, acc.w - f1.y);
    __nv_bfloat16* dst = attn_out + rh * Dh + 4 * lane;
    *reinterpret_cast<uint2*>(dst) = make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1));
    *reinterpret_cast<uint2*>(dst + (size_t)CS_MAX_ROWS * H * Dh) = make_uint2(*reinterpret_cast<const uint32_t*>(&l0), *reinterpret_cast<const uint32_t*>(&l1));
  }
  if (stamp != nullptr) {
    __syncthreads();
    if (threadIdx.x == 0) cs_stamp_end(stamp);
  }
}

// ------------------------------------------------------------------ acceptance
// Reduce the LM-head tile maxima to the greedy token of each row (lowest id on ties),
// then accept the longest prefix of the draft that agrees with the target tokens and
// emit it plus one extra token (Sec. 3.2; App. B.2).  One CTA per sequence.
// Bound by the latency of its loads: as many warps per row as fit, eight tiles of a lane at a time, and
// the comparison with the draft one thread per row (one warp per row and a serial comparison before, us at a
// vocabulary of 128,256: 11 rows 12.4 -> 6.9, 16 x 11 rows 17.4 -> 8.4, 8 x 21 rows 36 -> 11.5).
constexpr int kAcceptThreads = 1024;
__global__ void __launch_bounds__(kAcceptThreads)
k_accept(const float* tile_max, const int* tile_idx, int tiles, int tile_stride,
         int k, const int* draft, const int* draft_len, const int* seq_ok, const int* script, int script_stride,
         const int* script_off, int script_limit, int* __restrict__ accept_len,
         int* __restrict__ out_tokens, int* __restrict__ argmax_ids, int* __restrict__ kv_len,
         int update_kv, unsigned long long* stamp) {
  CS_PDL_PROLOGUE();
  const int b = blockIdx.x, R = k + 1, tid = threadIdx.x;
  constexpr int kWarps = kAcceptThreads / 32;
  const int warp = tid >> 5, lane = tid & 31;
  __shared__ unsigned long long s_key[CS_MAX_ROWS];   // (largest logit, lowest id) as one ordered number; 0 = none
  __shared__ int s_tau;
  int dl = __ldcg(draft_len + b);
  dl = dl < 0 ? 0 : (dl > k ? k : dl);
  const bool ok = __ldcg(seq_ok + b) != 0;
  if (tid < R) s_key[tid] = 0ull;
  if (tid == 0) s_tau = dl;
  __syncthreads();
  const int live = ok ? dl + 1 : 0;
  int per = 1;                                        // warps per row
  while (2 * per * live <= kWarps && per < kWarps) per *= 2;
  constexpr int kAtOnce = 8;
  for (int r = warp / per; r < live; r += kWarps / per) {
    const float* mx = tile_max + (size_t)(b * R + r) * tile_stride;
    const int* ids = tile_idx + (size_t)(b * R + r) * tile_stride;
    float val = -INFINITY;
    int idx = INT32_MAX;
    for (int t0 = (warp % per) * 32 + lane; t0 < tiles; t0 += 32 * per * kAtOnce) {
      float v[kAtOnce];
      int id[kAtOnce];
#pragma unroll
      for (int q = 0; q < kAtOnce; ++q) {
        const int t = t0 + 32 * per * q;
        v[q] = t < tiles ? __ldcg(mx + t) : -INFINITY;
        id[q] = t < tiles ? __ldcg(ids + t) : INT32_MAX;
      }
#pragma unroll
      for (int q = 0; q < kAtOnce; ++q)
        if (v[q] > val || (v[q] == val && id[q] < idx)) { val = v[q]; idx = id[q]; }
    }
    for (int off = 16; off > 0; off >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, val, off);
      const int oi = __shfl_xor_sync(0xffffffffu, idx, off);
      if (ov > val || (ov == val && oi < idx)) { val = ov; idx = oi; }
    }
    if (lane == 0 && idx != INT32_MAX) {
      const uint32_t u = __float_as_uint(val == 0.f ? 0.f : val);   // (-0 and 0 tie)
      const uint32_t order = u & 0x80000000u ? ~u : u | 0x80000000u;
      atomicMax(&s_key[r], (unsigned long long)order << 32 | (uint32_t)~idx);
    }
  }
  __syncthreads();
  // thread r: the greedy token of row r and whether the draft's next token agrees with it; the first row that
  // does not is the number of accepted tokens
  int tgt = -1;
  if (tid < R) {
    const int arg = s_key[tid] != 0ull ? (int)~(uint32_t)s_key[tid] : -1;
    argmax_ids[(size_t)b * R + tid] = arg;
    if (tid < live) {
      tgt = arg;
      if (script != nullptr) {
        const int at = (script_off != nullptr ? __ldcg(script_off + b) : 0) + tid;
        tgt = at < script_limit ? __ldcg(script + (size_t)b * script_stride + at) : -1;
      }
      if (tid < dl && __ldcg(draft + (size_t)b * k + tid) != tgt) atomicMin(&s_tau, tid);
    }
  }
  __syncthreads();
  const int tau = s_tau;
  if (tid < R) out_tokens[(size_t)b * R + tid] = tid <= tau ? tgt : -1;
  if (tid == 0) {
    accept_len[b] = ok ? tau : -1;
    if (ok && update_kv) kv_len[b] += tau + 1;
  }
  if (stamp != nullptr) {
    __syncthreads();
    if (tid == 0) cs_stamp_end(stamp);
  }
}

// Greedy token of each row from the LM head's per-tile (max, id) pairs (lowest id on ties).
__global__ void __launch_bounds__(128)
k_tile_reduce(const float* tile_max, const int* tile_idx, int tiles, int tile_stride,
              int* __restrict__ ids) {
  CS_PDL_PROLOGUE();
  const int row = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float val = -INFINITY;
  int idx = INT32_MAX;
  for (int t = threadIdx.x; t < tiles; t += 128) {
    const float v = __ldcg(tile_max + (size_t)row * tile_stride + t);
    const int id = __ldcg(tile_idx + (size_t)row * tile_stride + t);
    if (v > val || (v == val && id < idx)) { val = v; idx = id; }
  }
  __shared__ float sv[4];
  __shared__ int si[4];
  for (int off = 16; off > 0; off >>= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, val, off);
    const int oi = __shfl_xor_sync(0xffffffffu, idx, off);
    if (ov > val || (ov == val && oi < idx)) { val = ov; idx = oi; }
  }
  if (lane == 0) { sv[warp] = val; si[warp] = idx; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 4; ++w)
      if (sv[w] > val || (sv[w] == val && si[w] < idx)) { val = sv[w]; idx = si[w]; }
    ids[row] = (idx == INT32_MAX) ? -1 : idx;
  }
}

__global__ void k_truncate(int* kv_len, const int* new_len, int B, int* status) {
  CS_PDL_PROLOGUE();
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  const int nl = new_len[b];
  if (nl < 0 || nl > kv_len[b]) atomicOr(status, CS_DEV_BADARG);
  else kv_len[b] = nl;
}

// Host-ordered loop, end of a step: the emitted tokens go to the history, the lengths of history and
// cache follow, and so does a second model's cache length when it has one to cut.
__global__ void k_append(int* hist, int* hist_len, int n, const int* tokens, int count, int* kv_len, int* kv_len_2, int new_len_2) {
  CS_PDL_PROLOGUE();
  const int i = threadIdx.x;
  if (i < count) hist[n + i] = tokens[i];
  if (i == 0) {
    *hist_len = n + count;
    *kv_len = n + count - 1;
    if (kv_len_2 != nullptr) *kv_len_2 = new_len_2;
  }
}

__global__ void k_prefill_finish(const int* hist_len, const int* seq_ok, int* kv_len, int B) {
  CS_PDL_PROLOGUE();
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < B && seq_ok[b]) kv_len[b] = max(0, hist_len[b] - 1);
}

// ------------------------------------------------------------------ loop bookkeeping
__global__ void k_loop_init(const int* hist_len, const int* kv_len, int B, int stride, int max_new, int k,
                            int max_seq, int max_batch, int* emitted, int* done,
                            unsigned long long* stats, int* status) {
  CS_PDL_PROLOGUE();
  const int t = threadIdx.x;
  for (int i = t; i < (int)(sizeof(cs_stats) / 8); i += blockDim.x) stats[i] = 0ull;
  __shared__ int s_done;
  if (t == 0) s_done = 0;
  __syncthreads();
  for (int b = t; b < B; b += blockDim.x) {
    const int n = hist_len[b];
    const bool fits = n >= 1 && (long long)n + max_new <= stride && (long long)n + max_new + k <= max_seq;
    const bool consistent = kv_len[b] == n - 1;
    emitted[b] = 0;
    int d = 0;
    if (!fits) { atomicOr(status, CS_DEV_CAPACITY); d = 1; }
    else if (!consistent) { atomicOr(status, CS_DEV_BADARG); d = 1; }
    else if (max_new <= 0) d = 1;
    done[b] = d;
    if (d) atomicAdd(&s_done, 1);
  }
  __syncthreads();
  if (t == 0) { done[max_batch] = s_done; done[max_batch + 1] = 0; }
}

// Append the step's tokens to the history (App. B.3 step 4), clip at max_new, stop at
// EOS in real mode, advance the lengths (the KV truncation of App. B.2) and count.
// One CTA (a batch has at most CS_MAX_ROWS sequences).  With `progress`, a word in pinned host memory, the
// step also reports how many tokens the sequence furthest from its end still wants, so that the
// host knows without a synchronisation whether another step is needed.
__global__ void __launch_bounds__(CS_MAX_ROWS)
k_loop_commit(int* hist, int* hist_len, int B, int stride, int* kv_len, int k, int max_new,
              int eos_id, int scripted, const int* accept, const int* out, const int* mpos,
              int* emitted, int* done, int max_batch, unsigned long long* stats,
              const int* status, unsigned long long* progress, unsigned long long* stamp) {
  CS_PDL_PROLOGUE();
  const int b = threadIdx.x;
  if (b == 0) cs_stamp_end(stamp);   // (the kernel is a few dozen instructions: its start stands for its end)
  int wanted = 0;
  if (b < B && !done[b]) {
    cs_stats* st = reinterpret_cast<cs_stats*>(stats);
    const int tau = accept[b];
    bool fin = tau < 0;     // the step skipped this sequence (capacity): it stops here
    if (!fin) {
      const int R = k + 1;
      const int n = hist_len[b], e = emitted[b];
      int c = min(tau + 1, max_new - e);
      if (!scripted && eos_id >= 0) {
        for (int i = 0; i < c; ++i)
          if (out[(size_t)b * R + i] == eos_id) { c = i + 1; fin = true; break; }
      }
      for (int i = 0; i < c; ++i) hist[(size_t)b * stride + n + i] = out[(size_t)b * R + i];
      hist_len[b] = n + c;
      kv_len[b] = n + c - 1;
      emitted[b] = e + c;
      if (e + c >= max_new) fin = true;
      atomicAdd((unsigned long long*)&st->steps, 1ull);
      atomicAdd((unsigned long long*)&st->emitted, (unsigned long long)c);
      if (mpos[b] >= 0) {
        atomicAdd((unsigned long long*)&st->attempts, 1ull);
        atomicAdd((unsigned long long*)&st->accepted, (unsigned long long)(c - 1));
        atomicAdd((unsigned long long*)&st->tau_hist[min(c - 1, CS_TAU_HIST - 1)], 1ull);
      } else {
        atomicAdd((unsigned long long*)&st->no_match, 1ull);
      }
      if (!fin) wanted = max_new - e - c;
    }
    if (fin) {
      done[b] = 1;
      atomicAdd(&done[max_batch], 1);
    }
  }
  if (progress != nullptr) {
    __shared__ int s_wanted;
    if (b == 0) s_wanted = 0;
    __syncthreads();
    if (wanted > 0) atomicMax(&s_wanted, wanted);
    __syncthreads();
    if (b == 0) {
      const int step = ++done[max_batch + 1];            // steps of this loop
      const unsigned rest = (*status & CS_DEV_TIMEOUT) ? 0u : (unsigned)s_wanted;   // (a wait that ran out ends the loop)
      *reinterpret_cast<volatile unsigned long long*>(progress) = ((unsigned long long)(unsigned)step << 32) | rest;
    }
  }
}

// The two ends of a step that a client drives from host memory.  Its few words travel in one kernel each way
// instead of three copies in and two out, and the host waits for a word that the last kernel writes instead of
// for the stream: every copy hands the stream from the SMs to a copy engine and back.  (Four steps of the 8B shape at 3,001 tokens:
// 13.78 -> 13.72 ms, with two runs of one build 0.01 apart.)
__global__ void __launch_bounds__(CS_MAX_ROWS)
k_host_in(const int* in, int B, int tokens, int script_ints, int stride, int* hist, int* hist_len, int* script) {
  __shared__ int s_in[CS_STEP_IN_MAX];
  const int n = 3 * B + tokens + script_ints, tid = threadIdx.x;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  int v[CS_STEP_IN_MAX / CS_MAX_ROWS];                 // (one trip over the bus, and ahead of the wait)
#pragma unroll
  for (int q = 0; q < CS_STEP_IN_MAX / CS_MAX_ROWS; ++q)
    v[q] = q * CS_MAX_ROWS + tid < n ? *reinterpret_cast<const volatile int*>(in + q * CS_MAX_ROWS + tid) : 0;
#pragma unroll
  for (int q = 0; q < CS_STEP_IN_MAX / CS_MAX_ROWS; ++q) s_in[q * CS_MAX_ROWS + tid] = v[q];
  __syncthreads();
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (tid < B) {
    const int len = s_in[tid], from = s_in[B + tid], at = 3 * B + s_in[2 * B + tid];
    for (int i = from; i < len; ++i) hist[(size_t)tid * stride + i] = s_in[at + i - from];
    hist_len[tid] = len;
  }
  if (tid < script_ints) script[tid] = s_in[3 * B + tokens + tid];
}

__global__ void __launch_bounds__(CS_MAX_ROWS)
k_host_out(const int* accept_len, const int* out_tokens, int B, int n_out, int* out, unsigned long long* progress) {
  CS_PDL_PROLOGUE();
  const int tid = threadIdx.x;
  if (tid < B) out[tid] = __ldcg(accept_len + tid);
  if (tid < n_out) out[CS_MAX_ROWS + tid] = __ldcg(out_tokens + tid);
  __threadfence_system();
  __syncthreads();
  if (tid == 0) *reinterpret_cast<volatile unsigned long long*>(progress) = 1ull << 32;
}

}  // namespace

// one angle, or four words to clear, per thread up to a quarter of the chip
static dim3 setup_grid(int rows, int half, int quads) { return dim3(std::min(cs_ceil_div(std::max(rows * half, quads), kSetupThreads), 37)); }
// chained projections' words that a forward over so many rows needs cleared, in fours
static int chain_quads(const cs_ctx* ctx, int rows) {
  return cs_chain_takes(ctx, rows) ? (int)(ctx->cfg.n_layers * cs_chain_words(&ctx->cfg) / 4) : 0;
}

void cs_launch_block_setup(cs_ctx* ctx, const int32_t* last_tok, const int32_t* draft,
                           const int32_t* draft_len, const int32_t* kv_len, const int32_t* skip, int B,
                           int k, bool opens_step, cudaStream_t st) {
  const cs_model_config& c = ctx->cfg;
  const int quads = chain_quads(ctx, B * (k + 1));
  // A step that opens here (no search in front of it) opens with an ordinary stream-ordered launch, so
  // that kernels further down the chain may rely on everything enqueued earlier being complete.
  cs_launch_chained(k_block_setup, setup_grid(B * (k + 1), c.head_dim / 2, quads), dim3(kSetupThreads), 0, st, !opens_step, last_tok, draft, draft_len, kv_len, skip, B, k, c.max_seq,
                c.vocab, c.head_dim / 2, ctx->inv_freq, ctx->row_tok, ctx->row_pos, ctx->row_lim, ctx->row_write,
                ctx->seq_ok, ctx->rope_cs, ctx->d_status, ctx->pair_flag, reinterpret_cast<int4*>(ctx->chain_ctl), quads, ctx->chain_epoch,
                cs_next_stamp(ctx, CS_FAM_OTHER));
}

void cs_launch_prefill_setup(cs_ctx* ctx, const int32_t* hist, const int32_t* hist_len, int B, int stride,
                             int start, int R, cudaStream_t st) {
  const cs_model_config& c = ctx->cfg;
  const int quads = chain_quads(ctx, B * R);
  cs_launch_pdl(k_prefill_setup, setup_grid(B * R, c.head_dim / 2, quads), dim3(kSetupThreads), 0, st, hist, hist_len, B, stride, start, R, c.max_seq, c.vocab,
                c.head_dim / 2, ctx->inv_freq, ctx->row_tok, ctx->row_pos, ctx->row_lim, ctx->row_write, ctx->seq_ok,
                ctx->rope_cs, ctx->d_status, ctx->pair_flag, reinterpret_cast<int4*>(ctx->chain_ctl), quads, ctx->chain_epoch);
}

void cs_launch_embed_rmsnorm(cs_ctx* ctx, const __nv_bfloat16* gain, int rows, cudaStream_t st) {
  cs_launch_pdl(k_embed_rmsnorm, dim3(rows), dim3(kNormThreads), 0, st, ctx->embed, ctx->row_tok, ctx->x, ctx->cfg.d_model, gain,
                ctx->cfg.rms_eps, ctx->xn, ctx->xn + (size_t)CS_MAX_ROWS * ctx->cfg.d_model,
                cs_next_stamp(ctx, CS_FAM_OTHER));
}

void cs_launch_attn_merge(cs_ctx* ctx, int nsplit, int rows, cudaStream_t st) {
  const cs_model_config& c = ctx->cfg;
  // a handful of slices: one warp per (row, head); more: four warps share them
  auto kernel = nsplit <= 1 ? k_attn_merge<1, 1> : nsplit <= 2 ? k_attn_merge<1, 2> : nsplit <= 4 ? k_attn_merge<1, 4>
              : nsplit <= 16 ? k_attn_merge<4, 4> : nsplit <= 36 ? k_attn_merge<4, 9> : k_attn_merge<4, 16>;
  const int per_cta = nsplit <= 4 ? kMergeThreads / 32 : 1;
  cs_launch_pdl(kernel, dim3(cs_ceil_div(rows * c.n_heads, per_cta)), dim3(kMergeThreads), 0, st, ctx->attn_o, ctx->attn_ml, nsplit, rows,
                c.n_heads, c.head_dim, ctx->attn_out, cs_next_stamp(ctx, CS_FAM_MERGE));
}

void cs_launch_accept(cs_ctx* ctx, int B, int k, const int32_t* draft, const int32_t* draft_len,
                      const int32_t* script, int script_stride, const int32_t* script_off, int script_limit,
                      int32_t* accept_len, int32_t* out_tokens, int32_t* argmax_ids, int32_t* kv_len,
                      int update_kv, cudaStream_t st) {
  cs_launch_pdl(k_accept, dim3(B), dim3(kAcceptThreads), 0, st, ctx->tile_max, ctx->tile_idx,
                cs_ceil_div(ctx->cfg.vocab, CS_GEMM_BM), cs_ceil_div(ctx->cfg.vocab, CS_GEMM_BM), k, draft, draft_len, ctx->seq_ok, script,
                script_stride, script_off, script_limit, accept_len, out_tokens, argmax_ids, kv_len, update_kv,
                cs_next_stamp(ctx, CS_FAM_OTHER));
}

void cs_launch_tile_reduce(cs_ctx* ctx, int rows, int32_t* ids, cudaStream_t st) {
  cs_launch_pdl(k_tile_reduce, dim3(rows), dim3(128), 0, st, ctx->tile_max, ctx->tile_idx,
                cs_ceil_div(ctx->cfg.vocab, CS_GEMM_BM), cs_ceil_div(ctx->cfg.vocab, CS_GEMM_BM), ids);
}

void cs_launch_truncate(cs_ctx* ctx, int32_t* kv_len, const int32_t* new_len, int B, cudaStream_t st) {
  cs_launch_pdl(k_truncate, dim3(cs_ceil_div(B, 128)), dim3(128), 0, st, kv_len, new_len, B, ctx->d_status);
}

void cs_launch_append(int32_t* hist, int32_t* hist_len, int n, const int32_t* tokens, int count, int32_t* kv_len,
                      int32_t* kv_len_2, int new_len_2, cudaStream_t st) {
  cs_launch_pdl(k_append, dim3(1), dim3(CS_MAX_ROWS), 0, st, hist, hist_len, n, tokens, count, kv_len, kv_len_2, new_len_2);
}

void cs_launch_host_in(const int* in, int B, int tokens, int script_ints, int stride, int32_t* hist, int32_t* hist_len,
                       int32_t* script, cudaStream_t st) {
  cs_launch_pdl(k_host_in, dim3(1), dim3(CS_MAX_ROWS), 0, st, in, B, tokens, script_ints, stride, hist, hist_len, script);
}

void cs_launch_host_out(const int32_t* accept_len, const int32_t* out_tokens, int B, int k, int* out,
                        unsigned long long* progress, cudaStream_t st) {
  cs_launch_pdl(k_host_out, dim3(1), dim3(CS_MAX_ROWS), 0, st, accept_len, out_tokens, B, B * (k + 1), out, progress);
}

void cs_launch_prefill_finish(cs_ctx* ctx, const int32_t* hist_len, int32_t* kv_len, int B, cudaStream_t st) {
  cs_launch_pdl(k_prefill_finish, dim3(cs_ceil_div(B, 128)), dim3(128), 0, st, hist_len, ctx->seq_ok, kv_len, B);
}

void cs_launch_loop_init(cs_ctx* ctx, const int32_t* hist_len, const int32_t* kv_len, int B, int stride,
                         int max_new, int k, cudaStream_t st) {
  cs_launch_pdl(k_loop_init, dim3(1), dim3(256), 0, st, hist_len, kv_len, B, stride, max_new, k, ctx->cfg.max_seq,
                ctx->cfg.max_batch, ctx->loop_emitted, ctx->loop_done, ctx->loop_stats, ctx->d_status);
}

void cs_launch_loop_commit(cs_ctx* ctx, int32_t* hist, int32_t* hist_len, int B, int stride, int32_t* kv_len,
                           int k, int max_new, int eos_id, int scripted, unsigned long long* progress,
                           cudaStream_t st) {
  cs_launch_pdl(k_loop_commit, dim3(1), dim3(cs_ceil_div(B, 32) * 32), 0, st, hist, hist_len, B, stride, kv_len, k,
                max_new, eos_id, scripted, ctx->loop_accept, ctx->loop_out, ctx->loop_mpos, ctx->loop_emitted,
                ctx->loop_done, ctx->cfg.max_batch, ctx->loop_stats, ctx->d_status, progress,
                cs_next_stamp(ctx, CS_FAM_OTHER));
}
