// Everything between two attentions of a short block (at most 32 token rows) in one launch: the merge of the
// attention's key slices, the attention-output, gate/up and down projections of a layer and the QKV
// projection of the next one (Sec. 3.2).
//
// What bounds it: the weights, 436 MB a layer at the 8B shape, read from HBM once.  As one launch per
// projection every boundary left HBM idle for 4 - 5 us (last epilogue, release, first activations, restart),
// 29 of 98 us a layer.  Here the weight stream does not stop: a producer warp per SM walks the weight
// tiles of all four projections in order, held back by nothing but its ring (192 KB of 16 KB tiles on
// each of 148 SMs: 4 us of HBM), and only the activations wait for what they depend on.
// Measured, us a layer with its attention, launch per projection -> this kernel (4,096 keys): 1 row 93.6 -> 82.9, 8 rows
// 95.7 -> 85.0, 11 rows 97.9 -> 87.4, 16 rows 99.2 -> 88.6, 32 rows 108.0 -> 100.3.  What made it pay, in the order found
// (11 rows): runs taken one at a time behind the wait and not ahead of it (150 -> 109), sums handed over without fences and
// what finishing needs asked for early (98), two K blocks per ring slot and activations without padding rows (93.5), weights
// that leave L2 first (89.2), sums asked for again only where they were missing (88.1).
//
// Work: each projection's (128-feature tile, 64-wide K block) units are dealt out in equal contiguous runs, one
// per SM, so a tile is shared by the runs that cover it.  The run that holds the tile's head collects the others' sums
// through the workspace (they stay in L2), adds them up in the order of K (deterministic) and finishes the tile.  What a projection
// needs of the one before is tracked by 128-feature tile (gate/up to down: 64 features), not by a barrier over the grid: the
// activation producer polls the word of the tile that its next K block comes from.  The RMSNorm between
// projections is folded into them as in cs_gemm.cu, so a projection's MMAs can start before the
// norm's sums are complete.
//
// Nothing relies on all CTAs running at once.  Runs are taken from a counter in the order of the chain, a projection's last
// K range first, and a run depends only on runs that were taken before it, by CTAs that run; shares of the merge are
// taken from a counter of their own until none is left, before anything waits for them.
//
// Warps: eight read-out (TMEM lane quarter x half of the tokens), weight producer (which also takes the runs),
// activation producer, MMA issuer, and one that tells the other SMs of finished tiles.  The two bf16 terms of a token's
// activations are neighbouring rows of one operand.
//
// Counters and "done" words live in the workspace, a set per layer; the set-up kernel of a forward clears them.
// Every wait is bounded as in cs_gemm.cu; polls have the same limit.
#include <algorithm>

#include "cs_common.cuh"
#include "cs_tcgen.cuh"

using std::max;
using std::min;

namespace {

constexpr int kEpiWarps = 8, kWWarp = 8, kXWarp = 9, kMmaWarp = 10, kDoneWarp = 11, kThreads = 384;
constexpr int kWBytes = CS_GEMM_BM * CS_GEMM_BK * 2;   // 16 KB: one weight tile
constexpr int kQueue = 4;                              // runs taken ahead of their use
constexpr int kStep = 2;                               // K blocks of a ring slot
constexpr int kMaxW = 6, kMaxX = 8;
// Slots of weights asked for and not landed, at most.  Three (96 KB per SM) keep HBM busy; more only lengthen the queue in
// which everything else waits, 11 rows: layer 94.1 / 93.1 / 93.8 us with 2 / 3 / 4.  During the first run, while the
// attention's slices are merged, two: 89.5 / 89.2 / 89.6 us with 1 / 2 / 3.
constexpr int kFlight = 3, kFlightFirst = 2;
constexpr int kCtlBytes = 512;
constexpr int kMinRun = 4;                             // K blocks of a run, at least
constexpr int kSlices = 18;                            // merge: slices a warp has in flight
constexpr int kMergeBytes = kEpiWarps * 32 * 24;       // and what its warps hand to one another
constexpr int kTicket = 0, kMergeTicket = 32, kWords = 64;   // control words of a layer: the counters, then the rest

struct ChainPhase {
  int mode, num_kb, units, items, first;               // first = number of this projection's first run
  int dep, dep_shift, dep_target, dep_n;               // words of the input's groups: K block kb needs word[dep + (kb >> dep_shift)] >= dep_target
  int done;                                            // words per tile: finished (-1 = nobody asks)
  int norm_tiles;                                      // > 0: scaled by 1/rms over so many tiles of the input
  unsigned long long* stamp;
};
struct ChainArgs {
  ChainPhase ph[4];
  int phases, runs, rows, w_stages, x_stages, x_block, smem_bytes;
  int merge_word, merge_per, merge_shares, merge_groups, warps_per_item, nsplit, H, Dh, qd;
  const float *attn_o, *attn_ml;
  __nv_bfloat16* attn_out;
  float* x;
  __nv_bfloat16 *xn, *act;
  int d, F;
  float* ssq;
  int ssq_stride;
  const __nv_bfloat16* gain[2];                        // norm behind the attention output, norm behind down (NULL = none)
  float inv_d, eps;
  QkvEpi q;
  uint4* part;                                         // sums handed over, [projection][run][16 pairs of tokens][128 features]
  int* ctl;
  const int* epoch;                                    // counts forwards
  int layer, n_layers;
  int drop;                                            // test hook: unit of every run whose weights are left out (-1 = none)
  int* status;
  unsigned long long wait_ns;
  unsigned long long* merge_stamp;
};
struct ChainMaps {
  CUtensorMap w[4], x[4];
};

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// Results written by ordinary stores are fetched by TMA on other SMs: both sides put this fence between their
// accesses and the word that hands over.
__device__ __forceinline__ void fence_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }
__device__ __forceinline__ void red_release(int* p, int v) {
  asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void epi_sync() {
  __syncwarp();
  asm volatile("bar.sync 1, 256;" ::: "memory");
}
__device__ __forceinline__ bool epi_all(bool p) {
  uint32_t r;
  __syncwarp();
  asm volatile("{\n.reg .pred p, q;\nsetp.ne.b32 p, %1, 0;\nbar.red.and.pred q, 1, 256, p;\nselp.u32 %0, 1, 0, q;\n}"
               : "=r"(r) : "r"((uint32_t)p) : "memory");
  return r != 0;
}
// the words [base, base + n) of a warp's 32 that have reached `target`; `want` are the bits waited for.  0 = gave up.
__device__ __noinline__ uint32_t poll_words(const int* base, int n, int target, uint32_t want, volatile int* abort_flag, unsigned long long limit_ns) {
  const int lane = threadIdx.x & 31;
  unsigned long long t0 = 0;
  for (uint32_t it = 0;; ++it) {
    const int v = lane < n ? ld_acquire(base + lane) : target - 1;
    const uint32_t got = __ballot_sync(0xffffffffu, v >= target);
    if ((got & want) == want) {
      __syncwarp();                                    // what one lane has acquired, all of them may read now (a vote orders no memory)
      return got;
    }
    if ((it & 63u) == 63u) {
      bool stop = *abort_flag != 0;
      const unsigned long long now = globaltimer_ns();
      if (t0 == 0) t0 = now;
      else stop = stop || now - t0 > limit_ns;
      if (__any_sync(0xffffffffu, stop)) return 0;
    }
  }
}
// NT tokens of this thread's feature: two columns each, one per term of the activations; added up
template <int NT>
__device__ __forceinline__ void read_acc(uint32_t taddr, float (&v)[NT]) {
  float w[2 * NT];
#pragma unroll
  for (int c = 0; c < 2 * NT; c += 8)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(w[c]), "=f"(w[c + 1]), "=f"(w[c + 2]), "=f"(w[c + 3]), "=f"(w[c + 4]), "=f"(w[c + 5]), "=f"(w[c + 6]), "=f"(w[c + 7])
                 : "r"(taddr + (uint32_t)c));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
  // (the registers are valid only behind the wait)
#pragma unroll
  for (int c = 0; c < 2 * NT; ++c) asm volatile("" : "+f"(w[c]) :: "memory");
#pragma unroll
  for (int c = 0; c < NT; ++c) v[c] = w[2 * c] + w[2 * c + 1];
}
// four values as leading bf16 pairs and the pairs of what that rounding lost
__device__ __forceinline__ void split4(const float (&v)[4], uint2& hi, uint2& lo) {
  const __nv_bfloat162 h0 = __floats2bfloat162_rn(v[0], v[1]), h1 = __floats2bfloat162_rn(v[2], v[3]);
  const float2 f0 = __bfloat1622float2(h0), f1 = __bfloat1622float2(h1);
  const __nv_bfloat162 l0 = __floats2bfloat162_rn(v[0] - f0.x, v[1] - f0.y), l1 = __floats2bfloat162_rn(v[2] - f1.x, v[3] - f1.y);
  hi = make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1));
  lo = make_uint2(*reinterpret_cast<const uint32_t*>(&l0), *reinterpret_cast<const uint32_t*>(&l1));
}
// Sums that one run hands to another: every value travels with a word that is different in every launch, so that the
// reader polls the values themselves and neither side needs a fence.  A value and its word are one 64-bit element of the
// access: the elements of a vector access are accesses of their own, in no stated order, but each is written and read whole.
__device__ __forceinline__ void put_pair(uint4* p, float v0, float v1, uint32_t mark) {
  asm volatile("{\n.reg .b64 a, b;\nmov.b64 a, {%1, %2};\nmov.b64 b, {%3, %4};\nst.volatile.global.v2.b64 [%0], {a, b};\n}"
               ::"l"(p), "r"(__float_as_uint(v0)), "r"(mark), "r"(__float_as_uint(v1)), "r"(mark) : "memory");
}
__device__ __forceinline__ uint4 peek_pair(const uint4* p) {
  uint4 v;
  asm volatile("{\n.reg .b64 a, b;\nld.volatile.global.v2.b64 {a, b}, [%4];\nmov.b64 {%0, %1}, a;\nmov.b64 {%2, %3}, b;\n}"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}
// Adds the sums of the runs behind this one that cover the tile, in the order of K: `n` of them, `step` apart, NT tokens of
// this thread's feature from `from` on (only `pairs` pairs of tokens are real).  false = gave up.
template <int NT>
__device__ __forceinline__ bool take_sums(const uint4* from, size_t step, int n, int pairs, uint32_t mark, float (&v)[NT],
                                          volatile int* abort_flag, unsigned long long limit_ns) {
  constexpr int kB = NT == 4 ? 6 : NT == 8 ? 5 : 2, kP = NT / 2;   // runs whose sums are in flight together
  unsigned long long t0 = 0;
#pragma unroll 1
  for (int c0 = 0; c0 < n; c0 += kB) {
    uint4 w[kB][kP];
#pragma unroll
    for (int c = 0; c < kB; ++c)
#pragma unroll
      for (int q = 0; q < kP; ++q) w[c][q] = make_uint4(0u, mark, 0u, c0 + c < n && q < pairs ? ~mark : mark);
    for (uint32_t it = 0;; ++it) {
      // (asks again only for what was not there: the others' sums come at different times)
#pragma unroll
      for (int c = 0; c < kB; ++c)
#pragma unroll
        for (int q = 0; q < kP; ++q)
          if (w[c][q].w != mark || w[c][q].y != mark) w[c][q] = peek_pair(from + (size_t)(c0 + c) * step + q * CS_GEMM_BM);
      bool there = true;
#pragma unroll
      for (int c = 0; c < kB; ++c)
#pragma unroll
        for (int q = 0; q < kP; ++q) there = there && w[c][q].y == mark && w[c][q].w == mark;
      if (there) break;
      if ((it & 63u) == 63u) {
        if (*abort_flag) return false;
        const unsigned long long now = globaltimer_ns();
        if (t0 == 0) t0 = now;
        else if (now - t0 > limit_ns) return false;
      }
    }
#pragma unroll
    for (int c = 0; c < kB; ++c)
#pragma unroll
      for (int q = 0; q < kP; ++q) { v[2 * q] += __uint_as_float(w[c][q].x); v[2 * q + 1] += __uint_as_float(w[c][q].z); }
  }
  return true;
}

// a run: its projection and its units, from K block kb0 of tile t0 on.  (Behind a division the compiler no longer
// knows that a value is uniform, and instructions that want it in a uniform register loop over the lanes.)
__device__ __forceinline__ int uni(int v) { return (int)uniform((uint32_t)v); }
struct Run {
  int p, i, u0, u1, num_kb, t0, kb0;
};
__device__ __forceinline__ Run decode(const ChainArgs& a, int run) {
  int p = 0;
  for (int q = 1; q < 4; ++q)
    if (q < a.phases && run >= a.ph[q].first) p = q;
  Run r;
  r.p = uni(p);
  const ChainPhase& P = a.ph[r.p];
  r.i = uni(P.items - 1 - (run - P.first));            // (from the end: a run waits for sums of those behind it in K)
  r.u0 = uni((int)((long long)r.i * P.units / P.items));
  r.u1 = uni((int)((long long)(r.i + 1) * P.units / P.items));
  r.num_kb = uni(P.num_kb);
  r.t0 = uni(r.u0 / r.num_kb);
  r.kb0 = r.u0 - r.t0 * r.num_kb;
  return r;
}

// The merge of one share of (row, 128 features) items: o = sum_s o_s e^(m_s - M) / sum_s l_s e^(m_s - M).  Several warps per
// item where a share leaves warps over, each with its share of the slices; a lane holds four features.
__device__ __forceinline__ void merge_share(const ChainArgs& a, int share, bool first, uint8_t* scratch, int warp, int lane) {
  const int W = a.warps_per_item, part = warp % W, total = a.rows * a.merge_groups;
  float4* s_acc = reinterpret_cast<float4*>(scratch);
  float2* s_ml = reinterpret_cast<float2*>(scratch + kEpiWarps * 32 * 16);
  const int hi = min(total, (share + 1) * a.merge_per);
  for (int base = share * a.merge_per; base < hi; base += kEpiWarps / W) {
    const int item = base + warp / W;
    const int row = item / a.merge_groups, g = item - row * a.merge_groups, f = 128 * g + 4 * lane;
    const bool live = item < hi, has = live && f < a.qd;
    const int head = has ? f / a.Dh : 0;
    const float* from_o = a.attn_o + (size_t)row * a.qd + f;
    const float2* from_ml = reinterpret_cast<const float2*>(a.attn_ml) + (size_t)row * a.H + head;
    if (first) asm volatile("griddepcontrol.wait;" ::: "memory");
    float M = -INFINITY, L = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s0 = part; s0 < a.nsplit; s0 += W * kSlices) {
      float4 v[kSlices];
      float2 ml[kSlices];
#pragma unroll
      for (int q = 0; q < kSlices; ++q) {
        const int s = s0 + q * W;
        const bool in = has && s < a.nsplit;
        const size_t at = (size_t)s * a.rows;
        v[q] = in ? __ldcg(reinterpret_cast<const float4*>(from_o + at * a.qd)) : make_float4(0.f, 0.f, 0.f, 0.f);
        ml[q] = in ? __ldcg(from_ml + at * a.H) : make_float2(-INFINITY, 0.f);
      }
      float m = M;
#pragma unroll
      for (int q = 0; q < kSlices; ++q) m = fmaxf(m, ml[q].x);
      const float c = M == -INFINITY ? 0.f : expf(M - m);
      L *= c;
      acc.x *= c; acc.y *= c; acc.z *= c; acc.w *= c;
#pragma unroll
      for (int q = 0; q < kSlices; ++q) {
        const float w = ml[q].x == -INFINITY ? 0.f : expf(ml[q].x - m);
        L = fmaf(ml[q].y, w, L);
        acc.x = fmaf(v[q].x, w, acc.x); acc.y = fmaf(v[q].y, w, acc.y);
        acc.z = fmaf(v[q].z, w, acc.z); acc.w = fmaf(v[q].w, w, acc.w);
      }
      M = m;
    }
    if (W > 1) {
      s_acc[warp * 32 + lane] = acc;
      s_ml[warp * 32 + lane] = make_float2(M, L);
      epi_sync();
      if (part == 0) {
        float m = M;
        for (int q = 1; q < W; ++q) m = fmaxf(m, s_ml[(warp + q) * 32 + lane].x);
        const float c = M == -INFINITY ? 0.f : expf(M - m);
        L *= c;
        acc.x *= c; acc.y *= c; acc.z *= c; acc.w *= c;
        for (int q = 1; q < W; ++q) {
          const float2 o = s_ml[(warp + q) * 32 + lane];
          const float4 v = s_acc[(warp + q) * 32 + lane];
          const float w = o.x == -INFINITY ? 0.f : expf(o.x - m);
          L = fmaf(o.y, w, L);
          acc.x = fmaf(v.x, w, acc.x); acc.y = fmaf(v.y, w, acc.y);
          acc.z = fmaf(v.z, w, acc.z); acc.w = fmaf(v.w, w, acc.w);
        }
      }
    }
    if (part == 0 && has) {
      const float inv = L > 0.f ? 1.f / L : 0.f;
      const float o4[4] = {acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv};
      uint2 h, l;
      split4(o4, h, l);
      __nv_bfloat16* dst = a.attn_out + (size_t)row * a.qd + f;
      *reinterpret_cast<uint2*>(dst) = h;
      *reinterpret_cast<uint2*>(dst + (size_t)CS_MAX_ROWS * a.qd) = l;
      fence_async_global();
    }
    __syncwarp();
    if (part == 0 && live && lane == 0) {
      cs_stamp_end(a.merge_stamp);
      red_release(a.ctl + a.merge_word + g, 1);
    }
    if (W > 1) epi_sync();                             // (the scratch is written again)
  }
}

// Residual update of a parked tile: a warp per token, four features per lane; leaves the next norm's operand and the
// row's sum of squares over the tile.  The residual rows and the norm's gain were asked for long before.
template <int Q, int P>
__device__ __forceinline__ void finish_residual(const ChainArgs& a, bool feeds, int tile, const float* park, const float4 (&x)[P], uint2 g, int warp, int lane) {
  const int n0 = tile * CS_GEMM_BM, f = 4 * lane;
  const bool in = n0 + f < a.d;                        // (d is a multiple of 8)
  const float2 g01 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&g.x));
  const float2 g23 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&g.y));
#pragma unroll
  for (int u = 0; u < Q; ++u) {
    const int tok = warp + u * kEpiWarps;              // (the same for the whole warp)
    if (tok >= a.rows) break;
    const float4 y = *reinterpret_cast<const float4*>(park + tok * CS_GEMM_BM + f);
    const float o[4] = {y.x + x[u].x, y.y + x[u].y, y.z + x[u].z, y.w + x[u].w};
    if (in) *reinterpret_cast<float4*>(a.x + (size_t)tok * a.d + n0 + f) = make_float4(o[0], o[1], o[2], o[3]);
    if (!feeds) continue;
    float ss = 0.f;
    if (in) {
      const float w[4] = {o[0] * g01.x, o[1] * g01.y, o[2] * g23.x, o[3] * g23.y};
      uint2 h, l;
      split4(w, h, l);
      __nv_bfloat16* xo = a.xn + (size_t)tok * a.d + n0 + f;
      *reinterpret_cast<uint2*>(xo) = h;
      *reinterpret_cast<uint2*>(xo + (size_t)CS_MAX_ROWS * a.d) = l;
      ss = (o[0] * o[0] + o[1] * o[1]) + (o[2] * o[2] + o[3] * o[3]);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
    if (lane == 0) a.ssq[(size_t)tok * a.ssq_stride + tile] = ss;
  }
}

// SwiGLU of a tile of 64 gate features and the 64 matching up features: two tokens per warp, four feature pairs per lane
__device__ __forceinline__ void finish_swiglu(const ChainArgs& a, int tile, const float* park, const float* rstd, int warp, int lane) {
  const int j = 4 * (lane & 15), col = tile * 64 + j;
  for (int tok = 2 * warp + (lane >> 4); tok < a.rows; tok += 2 * kEpiWarps) {
    const float4 y[2] = {*reinterpret_cast<const float4*>(park + tok * CS_GEMM_BM + j),
                         *reinterpret_cast<const float4*>(park + tok * CS_GEMM_BM + 64 + j)};
    const float r = rstd[tok];
    const float gv[4] = {y[0].x * r, y[0].y * r, y[0].z * r, y[0].w * r}, uv[4] = {y[1].x * r, y[1].y * r, y[1].z * r, y[1].w * r};
    float v4[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) v4[e] = __fdividef(gv[e], 1.f + __expf(-gv[e])) * uv[e];
    if (col < a.F) {                                   // (F is a multiple of 8)
      uint2 h, l;
      split4(v4, h, l);
      __nv_bfloat16* dst = a.act + (size_t)tok * a.F + col;
      *reinterpret_cast<uint2*>(dst) = h;
      *reinterpret_cast<uint2*>(dst + (size_t)CS_MAX_ROWS * a.F) = l;
    }
  }
}

// Rotation, query split and K/V append of a tile: RoPE pairs feature i of a head with i + Dh/2, both in this tile.  Two
// tokens per warp; their rotation factors and places in the cache were asked for ahead of the sums.
template <int T>
__device__ __forceinline__ void ask_qkv(const ChainArgs& a, int warp, int lane, float4 (&cs)[2 * T], int2 (&place)[T]) {
  const int half = a.q.Dh >> 1, i = (4 * (lane & 15)) % half;
#pragma unroll
  for (int q = 0; q < T; ++q) {
    const int tok = min(2 * warp + (lane >> 4) + 2 * kEpiWarps * q, a.rows - 1);
    const float4* csp = reinterpret_cast<const float4*>(a.q.rope_cs + 2 * ((size_t)tok * half + i));
    cs[2 * q] = __ldcg(csp);                           // (cos, sin) of dims i .. i + 3
    cs[2 * q + 1] = __ldcg(csp + 1);
    place[q] = make_int2(__ldcg(a.q.row_write + tok), __ldcg(a.q.row_pos + tok));
  }
}
template <int T>
__device__ __forceinline__ void finish_qkv(const ChainArgs& a, int tile, const float* park, const float* rstd, const float4 (&cs)[2 * T],
                                           const int2 (&place)[T], int warp, int lane) {
  const QkvEpi& Q = a.q;
  const int n0 = tile * CS_GEMM_BM, j = 4 * (lane & 15), half = Q.Dh >> 1, i = j % half, f1 = (j / half) * Q.Dh + i, f2 = f1 + half;
  const int head = (n0 + f1) / Q.Dh;
  const bool is_v = head >= Q.H + Q.Hkv;
  if (head >= Q.H + 2 * Q.Hkv) return;
#pragma unroll
  for (int q = 0; q < T; ++q) {
    const int tok = 2 * warp + (lane >> 4) + 2 * kEpiWarps * q;
    if (tok >= a.rows) break;
    const float4 cs01 = cs[2 * q], cs23 = cs[2 * q + 1];
    const int row_w = place[q].x, row_p = place[q].y;
    const float4 y[2] = {*reinterpret_cast<const float4*>(park + tok * CS_GEMM_BM + f1),
                         *reinterpret_cast<const float4*>(park + tok * CS_GEMM_BM + f2)};
    const float r = rstd[tok];
    const float a4[4] = {y[0].x * r, y[0].y * r, y[0].z * r, y[0].w * r}, b4[4] = {y[1].x * r, y[1].y * r, y[1].z * r, y[1].w * r};
    const float cc[4] = {cs01.x, cs01.z, cs23.x, cs23.z}, sn[4] = {cs01.y, cs01.w, cs23.y, cs23.w};
    float r0[4], r1[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      r0[e] = is_v ? a4[e] : a4[e] * cc[e] - b4[e] * sn[e];
      r1[e] = is_v ? b4[e] : b4[e] * cc[e] + a4[e] * sn[e];
    }
    uint2 h0, l0, h1, l1;
    split4(r0, h0, l0);
    split4(r1, h1, l1);
    if (head < Q.H) {                                  // rotated query as two bf16 terms
      __nv_bfloat16* qd = Q.qbuf + ((size_t)tok * Q.H + head) * Q.Dh + i;
      __nv_bfloat16* ql = qd + (size_t)CS_MAX_ROWS * Q.H * Q.Dh;
      *reinterpret_cast<uint2*>(qd) = h0;
      *reinterpret_cast<uint2*>(qd + half) = h1;
      *reinterpret_cast<uint2*>(ql) = l0;
      *reinterpret_cast<uint2*>(ql + half) = l1;
    } else if (row_w) {                                // new K (rotated) / V row of the cache, stored in bf16
      const int kvh = is_v ? head - Q.H - Q.Hkv : head - Q.H;
      __nv_bfloat16* dst = Q.kv + ((((size_t)Q.layer * 2 + (is_v ? 1 : 0)) * Q.max_batch + tok / Q.R) * Q.Hkv + kvh) *
                                      (size_t)Q.max_seq * Q.Dh + (size_t)row_p * Q.Dh + i;
      *reinterpret_cast<uint2*>(dst) = h0;
      *reinterpret_cast<uint2*>(dst + half) = h1;
    }
  }
}

template <int NT>                                      // token columns per read-out group: half of the padded rows
__global__ void __launch_bounds__(kThreads, 1)
k_chain(const __grid_constant__ ChainMaps maps, const __grid_constant__ ChainArgs a) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  constexpr int n_tok = 2 * NT, kAccCols = 2 * n_tok, kParkBytes = n_tok * CS_GEMM_BM * 4 > kMergeBytes ? n_tok * CS_GEMM_BM * 4 : kMergeBytes;
  constexpr uint32_t kTmemCols = 2 * kAccCols;
  constexpr int kPre = n_tok > 16 ? 4 : 2;             // 16-byte operands of the epilogue asked for ahead of time
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  uint8_t* smem = smem_raw + (((raw + 1023u) & ~1023u) - raw);   // operand tiles need 1024-byte alignment
  const int WS = a.w_stages, XS = a.x_stages, xblock = a.x_block;   // (bytes from one K block of the activations to the next)
  uint8_t* xring = smem + (size_t)WS * (kStep * kWBytes);
  uint8_t* parkb = xring + (size_t)XS * (kStep * xblock);
  float* park = reinterpret_cast<float*>(parkb);       // a whole tile, [n_tok][128]; scratch of the merge
  uint8_t* ctlb = parkb + kParkBytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(ctlb);
  int* s_run = reinterpret_cast<int*>(bars + 2 * kMaxW + 2 * kMaxX + 8 + 2 * kQueue);   // [kQueue]
  volatile int* s_done = reinterpret_cast<volatile int*>(s_run + kQueue);               // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(s_run + kQueue + 2);
  volatile int* s_abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* s_never = reinterpret_cast<volatile int*>(tmem_slot + 2);   // stays 0: drains wait on time only
  volatile int* s_word = reinterpret_cast<volatile int*>(tmem_slot + 3);
  float* rstd = reinterpret_cast<float*>(ctlb + kCtlBytes);    // [n_tok]
  if ((size_t)(reinterpret_cast<uint8_t*>(rstd + n_tok) - smem_raw) > (size_t)a.smem_bytes) {
    if (threadIdx.x == 0) atomicOr(a.status, CS_DEV_SMEM);     // the launcher sizes the window for exactly this layout
    return;
  }
  const uint32_t b_wf = smem_u32(bars), b_we = b_wf + 8 * kMaxW, b_xf = b_we + 8 * kMaxW, b_xe = b_xf + 8 * kMaxX,
                 b_af = b_xe + 8 * kMaxX, b_ae = b_af + 16, b_df = b_ae + 16, b_de = b_df + 16, b_qf = b_de + 16, b_qe = b_qf + 8 * kQueue;
  const int tid = threadIdx.x, warp = (int)uniform(tid >> 5), lane = tid & 31;

  if (tid == kWWarp * 32) {
    for (int s = 0; s < WS; ++s) { mbar_init(b_wf + 8 * s, 1); mbar_init(b_we + 8 * s, 1); }
    for (int s = 0; s < XS; ++s) { mbar_init(b_xf + 8 * s, 1); mbar_init(b_xe + 8 * s, 1); }
    for (int s = 0; s < 2; ++s) { mbar_init(b_af + 8 * s, 1); mbar_init(b_ae + 8 * s, kEpiWarps); }
    for (int s = 0; s < 2; ++s) { mbar_init(b_df + 8 * s, kEpiWarps); mbar_init(b_de + 8 * s, 1); }
    for (int s = 0; s < kQueue; ++s) { mbar_init(b_qf + 8 * s, 1); mbar_init(b_qe + 8 * s, kEpiWarps + 2); }
    *s_abort = 0;
    *s_never = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_base = uniform(*tmem_slot);

  // the next run as the weight producer announced it; -1 = none is left, -2 = gave up
  int qn = 0;
  uint32_t qph = 0;
  auto next_run = [&]() -> int {
    if (!mbar_wait_warp(b_qf + 8 * qn, qph, s_abort, a.wait_ns)) return -2;
    const int r = (int)uniform((uint32_t)*reinterpret_cast<volatile int*>(s_run + qn));
    __syncwarp();
    if (lane == 0) mbar_arrive(b_qe + 8 * qn);
    if (++qn == kQueue) { qn = 0; qph ^= 1u; }
    return r;
  };
  auto give_up = [&]() {                               // (one lane)
    *s_abort = 1;
    atomicOr(a.status, CS_DEV_TIMEOUT);
  };

  if (warp == kWWarp) {
    // ------------------------------------------------------------- weights: take runs, stream their tiles
    // Weights are read once per forward: they leave L2 first, so that what the layers pass to one another (and the norms' gains
    // and rotation factors) is still there when it is wanted, instead of waiting in the queue that the weights keep full.
    const uint64_t policy = l2_evict_first();
    auto take = [&]() -> int { return lane == 0 ? atomicAdd(a.ctl + kTicket, 1) : 0; };
    int s = 0, issued = 0, landed = 0, sl = 0;         // slots filled, slots known to have landed, the next one to
    uint32_t ph = 1, eph = 1, lph = 0;                 // (the rings start empty)
    bool ok = true;
    while (ok) {
      // (CTAs start as SMs fall free: the first ones must not take the runs of those that follow)
      if (issued > 0) asm volatile("griddepcontrol.wait;" ::: "memory");
      const int run = uni(take());
      ok = mbar_wait_warp(b_qe + 8 * qn, eph, s_abort, a.wait_ns);
      if (!ok) break;
      if (lane == 0) {
        *reinterpret_cast<volatile int*>(s_run + qn) = run < a.runs ? run : -1;
        mbar_arrive(b_qf + 8 * qn);
      }
      if (++qn == kQueue) { qn = 0; eph ^= 1u; }
      if (run >= a.runs) break;
      const Run r = decode(a, run);
      const CUtensorMap* tm = &maps.w[r.p];
      int t = r.t0, kb = r.kb0, nk;
      for (int u = r.u0; u < r.u1; u += nk) {
        nk = min(kStep, min(r.u1 - u, r.num_kb - kb));
        ok = mbar_wait_warp(b_we + 8 * s, ph, s_abort, a.wait_ns);
        for (const int most = r.p == 0 ? kFlightFirst : kFlight; ok && issued - landed >= most; ++landed) {
          ok = mbar_wait_warp(b_wf + 8 * sl, lph, s_abort, a.wait_ns);
          if (++sl == WS) { sl = 0; lph ^= 1u; }
        }
        if (!ok) break;
        if ((a.drop < u - r.u0 || a.drop >= u - r.u0 + nk) && elect_one()) {
          const uint32_t dst = smem_u32(smem) + (uint32_t)(s * kStep * kWBytes);
          mbar_expect_tx(b_wf + 8 * s, (uint32_t)(nk * kWBytes));
          tma_load_2d_hint(dst, tm, b_wf + 8 * s, kb * CS_GEMM_BK, t * CS_GEMM_BM, policy);
          if (nk > 1) tma_load_2d_hint(dst + kWBytes, tm, b_wf + 8 * s, (kb + 1) * CS_GEMM_BK, t * CS_GEMM_BM, policy);
        }
        ++issued;
        kb += nk;
        if (kb == r.num_kb) { kb = 0; ++t; }
        if (++s == WS) { s = 0; ph ^= 1u; }
      }
    }
    if (!ok && lane == 0) give_up();
    __syncwarp();
    // copies in flight land before the shared memory goes away (a tile that the test hook left out never does)
    if (*s_abort && lane == 0)
      for (int i = max(0, issued - WS); i < issued; ++i)
        mbar_wait(b_wf + 8 * (i % WS), (uint32_t)(i / WS) & 1u, s_never, a.drop >= 0 ? 1000000ull : a.wait_ns);
  } else if (warp == kXWarp) {
    // ------------------------------------------------------------- activations: each K block once its tile is finished
    asm volatile("griddepcontrol.wait;" ::: "memory");
    int s = 0, issued = 0;
    uint32_t ph = 1;
    bool ok = true;
    while (ok) {
      const int run = next_run();
      if (run < 0) { ok = run == -1; break; }
      const Run r = decode(a, run);
      const ChainPhase& P = a.ph[r.p];
      const CUtensorMap* tm = &maps.x[r.p];
      const int dep_n = P.dep_n, dep_shift = uni(P.dep_shift), dep_target = P.dep_target;
      const int* dep = a.ctl + P.dep;
      int kb = r.kb0, window = -1, nk;
      uint32_t ready = 0;                              // finished groups of the window
      for (int u = r.u0; u < r.u1; u += nk) {
        nk = min(kStep, min(r.u1 - u, r.num_kb - kb));
        for (int g = kb >> dep_shift; g <= (kb + nk - 1) >> dep_shift && ok; ++g)
          if (g >> 5 != window || !(ready >> (g & 31) & 1u)) {
            window = g >> 5;
            ready = poll_words(dep + 32 * window, dep_n - 32 * window, dep_target, 1u << (g & 31), s_abort, a.wait_ns);
            ok = ready != 0;
            fence_async_global();
          }
        ok = ok && mbar_wait_warp(b_xe + 8 * s, ph, s_abort, a.wait_ns);
        if (!ok) break;
        if (elect_one()) {
          const uint32_t dst = smem_u32(xring) + (uint32_t)(s * kStep * xblock);
          mbar_expect_tx(b_xf + 8 * s, (uint32_t)(nk * a.rows * 256));
          tma_load_3d(dst, tm, b_xf + 8 * s, kb * CS_GEMM_BK, 0, 0);
          if (nk > 1) tma_load_3d(dst + (uint32_t)xblock, tm, b_xf + 8 * s, (kb + 1) * CS_GEMM_BK, 0, 0);
        }
        ++issued;
        kb += nk;
        if (kb == r.num_kb) kb = 0;
        if (++s == XS) { s = 0; ph ^= 1u; }
      }
    }
    if (!ok && lane == 0) give_up();
    __syncwarp();
    if (*s_abort && lane == 0)
      for (int i = max(0, issued - XS); i < issued; ++i) mbar_wait(b_xf + 8 * (i % XS), (uint32_t)(i / XS) & 1u, s_never, a.wait_ns);
  } else if (warp == kMmaWarp) {
    // ------------------------------------------------------------- MMA issuer: bf16 x bf16 -> fp32, both K-major, M = 128 features
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)((2 * a.rows + 15) >> 4) << 18) | ((uint32_t)(CS_GEMM_BM >> 4) << 24);
    const uint64_t dw0 = desc_kmajor(smem_u32(smem)), dx0 = desc_kmajor(smem_u32(xring));
    int sw = 0, sx = 0, j = 0;
    uint32_t phw = 0, phx = 0;
    bool ok = true;
    while (ok) {
      const int run = next_run();
      if (run < 0) { ok = run == -1; break; }
      const Run r = decode(a, run);
      int todo = r.u1 - r.u0, here = min(todo, r.num_kb - r.kb0);   // K blocks of the run, of its next tile
      for (; todo > 0 && ok; ++j) {
        const int buf = j & 1;
        const uint32_t acc = tmem_base + (uint32_t)(buf * kAccCols);
        if (j >= 2) ok = mbar_wait_warp(b_ae + 8 * buf, (uint32_t)((j >> 1) - 1) & 1u, s_abort, a.wait_ns);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        uint32_t acc_on = 0;
        for (int n = here; n > 0 && ok; n -= kStep) {
          ok = mbar_wait_warp(b_wf + 8 * sw, phw, s_abort, a.wait_ns) && mbar_wait_warp(b_xf + 8 * sx, phx, s_abort, a.wait_ns);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          if (elect_one()) {
            const uint64_t dw = dw0 + (uint64_t)(uint32_t)(sw * (kStep * kWBytes >> 4)), dx = dx0 + (uint64_t)(uint32_t)(sx * (kStep * xblock >> 4));
#pragma unroll
            for (int kk = 0; kk < CS_GEMM_BK / 16; ++kk)           // 16 K-elements = 32 bytes per instruction
              umma_bf16(acc, dw + 2 * kk, dx + 2 * kk, idesc, kk == 0 ? acc_on : 1u);
            if (n > 1) {
              const uint64_t ew = dw + (kWBytes >> 4), ex = dx + (uint64_t)(uint32_t)(xblock >> 4);
#pragma unroll
              for (int kk = 0; kk < CS_GEMM_BK / 16; ++kk) umma_bf16(acc, ew + 2 * kk, ex + 2 * kk, idesc, 1u);
            }
            umma_commit(b_we + 8 * sw);
            umma_commit(b_xe + 8 * sx);
          }
          acc_on = 1u;
          if (++sw == WS) { sw = 0; phw ^= 1u; }
          if (++sx == XS) { sx = 0; phx ^= 1u; }
        }
        todo -= here;
        here = min(todo, r.num_kb);
        if (!ok && lane == 0) give_up();               // (known before the accumulator looks finished)
        __syncwarp();
        if (elect_one()) umma_commit(b_af + 8 * buf);
        if (!ok) mbar_wait(b_af + 8 * buf, (uint32_t)(j >> 1) & 1u, s_never, a.wait_ns);   // what was issued has retired
      }
    }
    if (!ok && lane == 0) give_up();
  } else if (warp == kDoneWarp) {
    // ------------------------------------------------------------- tells the other SMs of finished tiles: what makes their results visible
    // takes 1 - 2 us while weights stream, and the read-out warps have the next tile to see to
    bool ok = true;
    for (int i = 0;; ++i) {
      ok = mbar_wait_warp(b_df + 8 * (i & 1), (uint32_t)(i >> 1) & 1u, s_abort, a.wait_ns);
      if (!ok) break;
      const int word = s_done[i & 1];
      __syncwarp();
      if (word < 0) break;
      if (lane == 0) {
        red_release(a.ctl + word, 1);
        mbar_arrive(b_de + 8 * (i & 1));
      }
    }
    if (!ok && lane == 0) give_up();
  } else {
    // ------------------------------------------------------------- read-out warps
    int share = tid == 0 ? atomicAdd(a.ctl + kMergeTicket, 1) : 0;
    // Ahead of the wait: the residual rows and the norm's gain come back to L2 (a layer's weights have passed through it since
    // they were written), and the arguments into the constant cache
    {
      const int lines = (a.rows * a.d * 4 + 127) >> 7, gl = (a.d * 2 + 127) >> 7;
      for (int i = (int)blockIdx.x * (kEpiWarps * 32) + tid; i < lines + gl; i += (int)gridDim.x * kEpiWarps * 32)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(i < lines ? reinterpret_cast<const char*>(a.x) + (size_t)i * 128
                                                                   : reinterpret_cast<const char*>(a.gain[0]) + (size_t)(i - lines) * 128));
#pragma unroll
      for (int p = 0; p < 4; ++p) asm volatile("" ::"r"(a.ph[p].first), "r"(a.ph[p].units), "r"(a.ph[p].done), "r"(a.ph[p].mode));
      asm volatile("" ::"r"(a.nsplit), "l"(a.attn_o), "l"(a.attn_ml), "l"(a.attn_out), "r"(a.merge_word), "l"(a.part), "l"(a.epoch), "l"(a.merge_stamp));
    }
    for (bool first = true;; first = false) {          // the merge, until nobody has a share left to take
      if (tid == 0) *s_word = share;
      epi_sync();
      const int m = *s_word;
      if (m >= a.merge_shares) break;
      merge_share(a, m, first, parkb, warp, lane);
      if (tid == 0) share = atomicAdd(a.ctl + kMergeTicket, 1);
      epi_sync();
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int wq = warp & 3, cg = warp >> 2, feat = wq * 32 + lane;
    const uint32_t lane_base = tmem_base + ((uint32_t)(wq * 32) << 16) + (uint32_t)(cg * 2 * NT);
    const uint32_t mark = (uint32_t)__ldcg(a.epoch) * (uint32_t)a.n_layers + (uint32_t)a.layer + 1u;
    int finished = 0;                                  // tiles handed to the warp that tells of them
    auto tell = [&](int word) {
      __syncwarp();
      if (lane == 0) {
        const int b = finished & 1;
        if (finished >= 2 && !mbar_wait(b_de + 8 * b, (uint32_t)((finished >> 1) - 1) & 1u, s_abort, a.wait_ns)) *s_abort = 1;
        if (warp == 0) s_done[b] = word;
        mbar_arrive(b_df + 8 * b);
      }
      __syncwarp();
      ++finished;
    };
    int j = 0, normed = -1;                            // accumulators read; projection whose 1/rms is in shared memory
    bool ok = true;
    while (ok) {
      const int run = next_run();
      ok = epi_all(run != -2);                         // (one decision for all: they meet at barriers below)
      if (!ok || run < 0) break;
      const Run r = decode(a, run);
      const ChainPhase& P = a.ph[r.p];
      if (P.norm_tiles > 0 && normed != r.p) {
        // 1/rms of every token row, while the MMAs run: one sum of squares per tile of the input, in a fixed order
        for (int w0 = 0; w0 < P.norm_tiles && ok && warp == 0; w0 += 32) {
          const int n = min(32, P.norm_tiles - w0);
          ok = poll_words(a.ctl + P.dep + w0, n, P.dep_target, n == 32 ? 0xffffffffu : (1u << n) - 1u, s_abort, a.wait_ns) != 0;
        }
        epi_sync();                                    // (the projection before has been finished with the old values)
        float ss[n_tok / kEpiWarps];
#pragma unroll
        for (int q = 0; q < n_tok / kEpiWarps; ++q) {
          ss[q] = 0.f;
          const int tok = warp + q * kEpiWarps;
          for (int sl = lane; sl < P.norm_tiles && tok < a.rows; sl += 32) ss[q] += __ldcg(a.ssq + (size_t)tok * a.ssq_stride + sl);
        }
#pragma unroll
        for (int q = 0; q < n_tok / kEpiWarps; ++q) {
#pragma unroll
          for (int off = 16; off > 0; off >>= 1) ss[q] += __shfl_xor_sync(0xffffffffu, ss[q], off);
          if (lane == 0) rstd[warp + q * kEpiWarps] = rsqrtf(ss[q] * a.inv_d + a.eps);
        }
        normed = r.p;
      }
      for (int u = r.u0; u < r.u1; ++j) {
        const int tile = u / P.num_kb, lo = tile * P.num_kb, hi = lo + P.num_kb, buf = j & 1;
        const bool head = r.u0 <= lo;                  // the run that holds a tile's head finishes it, at the run's end
        u = min(r.u1, hi);
        const bool resid = P.mode == CS_EPI_RESIDUAL, feeds = a.gain[r.p == 0 ? 0 : 1] != nullptr;
        const int xf = tile * CS_GEMM_BM + 4 * lane;
        if (resid && head) {
          // (the rows behind down are those that the attention output left, and L2 may have lost them to the weights)
          if (r.p != 0) ok = ok && poll_words(a.ctl + a.ph[0].done + tile, 1, 1, 1u, s_abort, a.wait_ns) != 0;
          for (int tok = warp; tok < a.rows && (lane & 7) == 0 && xf < a.d; tok += kEpiWarps)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(a.x + (size_t)tok * a.d + xf));
        }
        ok = ok && mbar_wait(b_af + 8 * buf, (uint32_t)(j >> 1) & 1u, s_abort, a.wait_ns) && *s_abort == 0;
        ok = epi_all(ok);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        float v[NT];
        read_acc<NT>(lane_base + (uint32_t)(buf * kAccCols), v);
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(b_ae + 8 * buf);
        constexpr size_t kSlot = CS_CHAIN_MAX_ROWS / 2 * CS_GEMM_BM;
        uint4* mine = a.part + ((size_t)r.p * CS_CHAIN_MAX_RUNS + r.i) * kSlot + (size_t)(cg * NT / 2) * CS_GEMM_BM + feat;
        const int pairs = (max(0, min(NT, a.rows - cg * NT)) + 1) >> 1;
        if (!head) {
#pragma unroll
          for (int q = 0; q < NT / 2; ++q)
            if (q < pairs) put_pair(mine + q * CS_GEMM_BM, v[2 * q], v[2 * q + 1], mark);
          continue;
        }
        // what finishing needs besides the sums, asked for ahead of them
        float4 pre[kPre];
        uint2 gain = make_uint2(0u, 0u);
        int2 place[kPre / 2];
        if (resid) {
#pragma unroll
          for (int q = 0; q < n_tok / kEpiWarps; ++q) {
            const int tok = warp + q * kEpiWarps;
            pre[q] = xf < a.d && tok < a.rows ? __ldcg(reinterpret_cast<const float4*>(a.x + (size_t)tok * a.d + xf)) : make_float4(0.f, 0.f, 0.f, 0.f);
          }
          if (feeds && xf < a.d) gain = *reinterpret_cast<const uint2*>(a.gain[r.p == 0 ? 0 : 1] + xf);
        } else if (P.mode == CS_EPI_QKV) {
          ask_qkv<kPre / 2>(a, warp, lane, pre, place);
        }
        if (r.u1 < hi)                                 // the runs behind this one, up to the one that holds the tile's last K block
          ok = take_sums<NT>(mine + kSlot, kSlot, (int)(((long long)hi * P.items - 1) / P.units) - r.i, pairs, mark, v, s_abort, a.wait_ns);
#pragma unroll
        for (int q = 0; q < NT; ++q) park[(cg * NT + q) * CS_GEMM_BM + feat] = v[q];
        ok = epi_all(ok);
        if (!ok) break;
        if (resid) finish_residual<n_tok / kEpiWarps, kPre>(a, feeds, tile, park, pre, gain, warp, lane);
        else if (P.mode == CS_EPI_SWIGLU) finish_swiglu(a, tile, park, rstd, warp, lane);
        else finish_qkv<kPre / 2>(a, tile, park, rstd, pre, place, warp, lane);
        fence_async_global();
        if (tid == 0) cs_stamp_end(P.stamp);
        if (P.done >= 0) tell(P.done + tile);
      }
    }
    if (!ok && lane == 0) give_up();
    if (ok) tell(-1);
  }
  // ---------------------------------------------------------------- teardown
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
  }
}

typedef void (*ChainKernel)(const ChainMaps, const ChainArgs);
ChainKernel chain_kernel(int nt) { return nt == 4 ? k_chain<4> : nt == 8 ? k_chain<8> : k_chain<16>; }

// control words of a layer, in the order of the phases
struct ChainWords {
  int merge, o_done, gu_done, down_done, total;
};
ChainWords chain_words(int d, int qd, int F) {
  auto pad = [](int n) { return (n + 31) & ~31; };
  const int dt = cs_ceil_div(d, CS_GEMM_BM), ft = cs_ceil_div(F, 64);
  ChainWords w;
  int at = kWords;
  w.merge = at; at += pad(cs_ceil_div(qd, 128));
  w.o_done = at; at += pad(dt);
  w.gu_done = at; at += pad(ft);
  w.down_done = at; at += pad(dt);
  w.total = at;
  return w;
}

}  // namespace

size_t cs_chain_words(const cs_model_config* c) {
  return (size_t)chain_words(c->d_model, c->n_heads * c->head_dim, c->d_ffn).total;
}

// Highest block that is chained.  A hand-over between two projections takes 5 - 6 us whatever they hold, a launch boundary
// 4 - 5, and only the weights streamed meanwhile make up for it; the taller the block, the more sums it has to hand over,
// and heads of 64 come in more key slices, whose merge is part of the launch.  Verify steps of 8 layers over 500 to 30,000 keys,
// 1 to 32 sequences, launch per projection / chained, us at 2,000 keys (rows of one sequence; S = one row each of so many):
//   MiB a layer              1        8       11      12 S     16       24       32       32 S
//   416                   779/685  807/703  817/721  963/885  827/731  868/780  897/809  1293/1230
//   288, heads of 64      602/530  660/571  681/604  710/651  696/626  754/696  794/736   908/886
//   245, narrow (d 2,048) 597/528  624/548  633/584  690/655  642/593  664/652  678/680   834/876
//   245, heads of 64      559/507  613/545  643/602  669/644  650/615  706/689  718/719   848/881
//   192                   502/441  532/461  540/490  683/657  549/500  573/534  592/560   940/940
//   195, heads of 64      487/442  537/483  561/539  586/582  568/554  625/630  636/654   770/822
//   154                   449/418  478/442  482/468  545/540  494/479  520/535  536/549   682/743
//   135                   429/398  454/420  458/446  524/514  472/458  496/514  514/528   662/722
//   122                   416/370  438/387  436/415  505/498  443/428  471/474  486/506   639/726
//   116, heads of 64      395/365  426/400  436/442  494/479  451/461  491/494  504/539   672/727
//   112, QKV of 3 d       409/394  434/418  440/447  594/624  447/463  482/518  493/558   843/939
//   108, heads of 64      386/389  416/430  424/480  483/492  434/505  482/489  495/546   662/727
//    98                   390/346  404/366  411/393  474/483  420/406  443/458  462/483   617/689
//    92, heads of 64      367/363  400/399  404/455  466/461  417/476  462/489  477/593   645/728
// The lines lie where the worst of the lengths and batches of 42 shapes is no loss (at most 1 %: 154 MiB, heads of 64, 12
// sequences; 192 MiB, 8 x 4 rows; 222 MiB with a QKV of 2 d, 4 x 6 rows).  A narrow model's tiles of O and down are few, so more runs share each
// (232 MiB, d 2,560, 4 x 6 rows 0.98x, 16 rows 1.02x); a QKV of 2 d and more has more slices to merge (198 MiB, 3 d, 4 x 8
// rows 0.97x).  Below the lines some layers gain (92 MiB with heads of 128 at 1 row 381/334, 98 MiB at 11 rows 411/393) and others lose
// up to a quarter (103 MiB, d 2,304, 10 sequences 0.91x; 32 MiB at 22 rows 360/485).
int cs_chain_max_rows(const cs_model_config& c, int force) {
  if (force != 0) return force > 0 ? CS_CHAIN_MAX_ROWS : 0;
  const long long mib = cs_layer_bytes(c) >> 20;
  const bool wide = c.head_dim == 128, lean = (c.n_heads + 2 * c.n_kv_heads) * c.head_dim < 2 * c.d_model;
  if (mib >= 280 && c.d_model >= 3072) return CS_CHAIN_MAX_ROWS;
  if (mib >= 192 && wide) return c.d_model < 3072 ? 16 : lean ? CS_CHAIN_MAX_ROWS : 24;
  if (mib >= 128) return 12;
  return lean && mib >= (wide ? 96 : 112) ? 8 : 0;
}
bool cs_chain_takes(const cs_ctx* ctx, int rows) { return rows <= cs_chain_max_rows(ctx->cfg, ctx->chain_force); }

cs_status cs_launch_chain(cs_ctx* ctx, int layer, int nsplit, int rows, const QkvEpi* next_q, const __nv_bfloat16* next_gain, cudaStream_t st) {
  const cs_model_config& c = ctx->cfg;
  const LayerPlan& L = ctx->layers[layer];
  const int d = c.d_model, qd = c.n_heads * c.head_dim, F = c.d_ffn;
  const ChainWords w = chain_words(d, qd, F);
  const int nt = rows <= 8 ? 4 : rows <= 16 ? 8 : 16, n_tok = 2 * nt;
  if (ctx->chain_box != rows) {
    const struct { CUtensorMap* tm; const __nv_bfloat16* base; int K; } ops[3] = {
        {&ctx->tmChainAttn, ctx->attn_out, qd}, {&ctx->tmChainXn, ctx->xn, d}, {&ctx->tmChainAct, ctx->act, F}};
    for (const auto& o : ops) {
      // a row's two terms lie next to one another in the copy
      const unsigned long long dims[3] = {(unsigned long long)o.K, 2ull, (unsigned long long)CS_MAX_ROWS};
      const unsigned long long strides[2] = {(unsigned long long)o.K * 2 * CS_MAX_ROWS, (unsigned long long)o.K * 2};
      const unsigned box[3] = {(unsigned)CS_GEMM_BK, 2u, (unsigned)rows};
      const cs_status s = cs_encode_tiled(ctx, o.tm, o.base, 3, dims, strides, box);
      if (s != CS_OK) return s;
    }
    ctx->chain_box = rows;
  }
  ChainMaps m;
  ChainArgs a = {};
  a.phases = next_q != nullptr ? 4 : 3;
  const GemmPlan* plans[4] = {&L.o, &L.gate_up, &L.down, next_q != nullptr ? &ctx->layers[layer + 1].qkv : nullptr};
  const CUtensorMap* xs[4] = {&ctx->tmChainAttn, &ctx->tmChainXn, &ctx->tmChainAct, &ctx->tmChainXn};
  const int fit = min(ctx->num_sms, CS_CHAIN_MAX_RUNS);
  a.merge_stamp = cs_next_stamp(ctx, CS_FAM_MERGE);
  for (int p = 0; p < a.phases; ++p) {
    ChainPhase& P = a.ph[p];
    m.w[p] = plans[p]->tmW;
    m.x[p] = *xs[p];
    P.num_kb = cs_ceil_div(plans[p]->K, CS_GEMM_BK);
    P.units = cs_ceil_div(plans[p]->N, CS_GEMM_BM) * P.num_kb;
    P.items = max(1, min(fit, P.units / kMinRun));
    P.first = a.runs;
    a.runs += P.items;
    P.stamp = cs_next_stamp(ctx, CS_FAM_GEMM);
  }
  for (int p = a.phases; p < 4; ++p) { m.w[p] = m.w[0]; m.x[p] = m.x[0]; }
  const int dt = cs_ceil_div(d, CS_GEMM_BM);
  a.ph[0].mode = CS_EPI_RESIDUAL; a.ph[0].dep = w.merge; a.ph[0].dep_shift = 1; a.ph[0].dep_target = rows; a.ph[0].dep_n = cs_ceil_div(qd, 128);
  a.ph[0].done = w.o_done;
  a.ph[1].mode = CS_EPI_SWIGLU; a.ph[1].dep = w.o_done; a.ph[1].dep_shift = 1; a.ph[1].dep_target = 1; a.ph[1].dep_n = dt;
  a.ph[1].done = w.gu_done; a.ph[1].norm_tiles = dt;
  a.ph[2].mode = CS_EPI_RESIDUAL; a.ph[2].dep = w.gu_done; a.ph[2].dep_shift = 0; a.ph[2].dep_target = 1; a.ph[2].dep_n = cs_ceil_div(F, 64);
  a.ph[2].done = w.down_done;
  a.ph[3].mode = CS_EPI_QKV; a.ph[3].dep = w.down_done; a.ph[3].dep_shift = 1; a.ph[3].dep_target = 1; a.ph[3].dep_n = dt;
  a.ph[3].done = -1; a.ph[3].norm_tiles = dt;
  const int grid = min(fit, a.runs);
  a.rows = rows;
  a.merge_word = w.merge;
  a.merge_groups = cs_ceil_div(qd, 128);
  a.merge_per = cs_ceil_div(rows * a.merge_groups, grid);
  a.merge_shares = cs_ceil_div(rows * a.merge_groups, a.merge_per);
  a.warps_per_item = 1;
  while (2 * a.warps_per_item * min(a.merge_per, kEpiWarps) <= kEpiWarps && a.warps_per_item < nsplit) a.warps_per_item *= 2;
  a.nsplit = nsplit; a.H = c.n_heads; a.Dh = c.head_dim; a.qd = qd;
  a.attn_o = ctx->attn_o; a.attn_ml = ctx->attn_ml; a.attn_out = ctx->attn_out;
  a.x = ctx->x; a.xn = ctx->xn; a.act = ctx->act; a.d = d; a.F = F;
  a.ssq = ctx->ssq; a.ssq_stride = ctx->ssq_stride;
  a.gain[0] = L.ffn_norm; a.gain[1] = next_gain;
  a.inv_d = 1.f / (float)d; a.eps = c.rms_eps;
  if (next_q != nullptr) a.q = *next_q;
  a.part = ctx->chain_part;
  a.epoch = ctx->chain_epoch; a.layer = layer; a.n_layers = c.n_layers;
  a.ctl = ctx->chain_ctl + (size_t)layer * w.total;
  a.drop = ctx->debug_drop_chain;
  ctx->debug_drop_chain = -1;         // the hook covers one launch
  a.status = ctx->d_status;
  a.wait_ns = ctx->wait_limit_ns;
  // weights: six slots of 32 KB where they fit; activations get the rest
  const int park = max(n_tok * CS_GEMM_BM * 4, kMergeBytes), fixed = 1024 + kCtlBytes + n_tok * 4 + park, room = 227 * 1024 - fixed;
  a.x_block = (rows * 256 + 1023) & ~1023;
  a.w_stages = min(kMaxW, (room - 3 * kStep * a.x_block) / (kStep * kWBytes));
  a.x_stages = min(kMaxX, (room - a.w_stages * kStep * kWBytes) / (kStep * a.x_block));
  a.smem_bytes = fixed + a.x_stages * kStep * a.x_block + a.w_stages * kStep * kWBytes;
  if (!ctx->chain_attr_set) {
    for (int q : {4, 8, 16}) CS_CUDA_OK(ctx, cudaFuncSetAttribute(chain_kernel(q), cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
    ctx->chain_attr_set = true;
  }
  CS_CUDA_OK(ctx, cs_launch_pdl(chain_kernel(nt), dim3(grid), dim3(kThreads), (size_t)a.smem_bytes, st, m, a));
  return CS_OK;
}
