// Projections of tall blocks (Sec. 3.2: batches of verification blocks, wide copy windows, prefill
// chunks) on pairs of SMs: Y = X W^T with up to 256 token rows, tcgen05.mma with cta_group::2.
//
// What bounds them.  At 16 rows a projection waits for its weights (HBM).  From a few dozen rows on
// the activations, two bf16 terms of every row, outgrow the 16 KB weight tile they are multiplied
// with: one SM needed a 61 KB stage per 64-wide K block at 176 rows, had room for three of them and
// drew 87 bytes per clock from L2.  Here two CTAs of a cluster form one tensor-core unit of 256
// features (128 each): each loads half of the token rows and the hardware multiplies both halves
// on both SMs, so a stage is 16 KB of weights + 64 bytes x rows x terms, five stages fit at 176 rows.
// Up to 128 rows the two terms of the activations are one operand of twice the rows (CTA 0 loads
// the leading terms, CTA 1 the second ones): one instruction does the work of two and the halves
// of the accumulator are added at read-out.
//
// Two launch forms share the pipeline (TMA producer warp, MMA warp on the even CTA, sixteen read-out
// warps), one pair of CTAs per two SMs:
//   split form (STORE, RESIDUAL, QKV: few feature tiles, long K): S pairs share a 256-feature tile, each
//     takes a K range, leaves its sums in the workspace (they stay in L2) and finishes a share of the
//     tokens from everybody's.  A pair waits for the others of its tile only once all of them have
//     started; otherwise it leaves its share to whoever comes last, so nobody ever holds an SM for a
//     CTA that has none.  (Clusters of 2 x S CTAs that add up over distributed shared memory were
//     slower: a cluster lies in one GPC, so only 96 of 148 SMs took part at S = 3.)
//   stream form (SWIGLU, ARGMAX: many feature tiles): the (tile, K block) units of the whole matrix are
//     dealt out in equal contiguous runs, so 112 tiles on 74 pairs take 1.51 turns instead of two.  The
//     tail of a tile cut by a run's start comes first in its run and its sums go to the workspace;
//     the tile is finished by the pair that holds its head, at the end of its run, long after.  Runs are
//     numbered against the block index, so that a pair only ever waits for one that was dispatched
//     earlier.  Two accumulators in TMEM: a tile is read out while the next one is multiplied.
//
// Measured on the 8B shape (us per launch: QKV / attention output / gate/up / down / LM head), one-SM
// tiles with launch shapes by a cost model -> this kernel:
//    88 rows  23.5 19.9 54.9 36.5 272 -> 17.4 16.5 49.3 28.2 184
//   176 rows  31.8 26.7 90.7 49.1 509 -> 24.2 20.6 66.6 38.5 257   (two-term tensor floor 10.6 7.1 49 25 222)
//   256 rows  42.2 36.4 114 70.7 791  -> 25.7 23.7 75.0 45.4 287 with 2,048 keys cached
// (the power cap's share differs from GPU to GPU: 21.7 18.9 61.0 36.1 250 at 176 rows on another one)
// and the stream form at 11 rows: gate/up 42.2 -> 41.1, LM head 168 -> 157 us (6.7 TB/s).  Clusters that
// add up over distributed shared memory instead of the split form's exchange: 24.2, 25.6, 45.5 us at
// 176 rows, 29.5, 32.7, 60.4 at 256 (QKV, output, down).
//
// Weights leave L2 first, so that activations and sums stay, and so do K and V in the attention between (us a layer, both at
// normal priority / both first): 44 rows over 4 x 4,096 keys 121.7 / 116.2, over 4 x 16,384 152.6 / 144.0, 176 rows over
// 16 x 8,192 241.5 / 235.6, 256 rows behind 2,048 202.7 / 200.5, 168 rows over 8 x 16,384 no difference (267.5 / 268.7, +-3).
//
// Every wait is bounded as in cs_gemm.cu; waits for other pairs' sums are polls with the same limit.
#include <algorithm>

#include "cs_common.cuh"
#include "cs_tcgen.cuh"

using std::max;
using std::min;

namespace {

constexpr int kABytes = CS_GEMM_BM * CS_GEMM_BK * 2;         // 16 KB: this CTA's weight tile of one K block
constexpr int kMaxStages = 10;
constexpr int kBatch = 3;                                    // tokens a warp of the split form's epilogue has in flight
constexpr int kCtlBytes = (2 * kMaxStages + 4) * 8 + 32;

struct PairArgs {
  int rows, n_tok, N, num_kb;
  int splits, kb_per_split;   // split form
  int units;                  // stream form: pair tiles x K blocks
  int stages, terms, stacked, mode;
  int lo_row;                 // row coordinate of the activations' second term
  float* out;
  bool vec_out;               // four values of a row of `out` lie on a 16-byte boundary (a caller's buffer may start anywhere)
  __nv_bfloat16 *act, *act_lo;
  int F;
  QkvEpi q;
  NormFuse nf;
  float* tile_max;
  int* tile_idx;
  int tile_stride;
  float* part;                // sums handed to other pairs, [pair][half][256 tokens][128 features]
  int* part_flag;             // stream form: "written", [pair][half]; split form: who is where, [tile][half]; 0 between launches
  int drop_kb;                // test hook: K block of a run whose loads are left out, by every pair (split form) or every second one (stream form); -1 = none
  int leave;                  // test hook, split form: K ranges whose pairs leave their shares to others (bit mask; 0 = as they come)
  int* status;
  unsigned long long wait_ns;
  unsigned long long* stamp;
};

__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {   // barrier of any CTA of the cluster
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Hand-over words in global memory: low byte = arrivals, next = shares left to others, top = pairs started.
// count_wait polls until `count` have arrived and returns the second byte, -1 when it gave up (bounded like mbar_wait).
__device__ __noinline__ int count_wait(const int* word, int count, volatile int* abort_flag, unsigned long long limit_ns) {
  const unsigned long long t0 = globaltimer_ns();
  for (;;) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(word) : "memory");
    if ((v & 0xff) >= count) return v >> 8 & 0xff;
    if (*abort_flag || globaltimer_ns() - t0 > limit_ns) return -1;
  }
}
__device__ __forceinline__ int started(const int* word) {
  return (int)((unsigned)*reinterpret_cast<const volatile int*>(word) >> 24);
}
// a copy of the pair: it lands in this CTA's shared memory and counts on the even CTA's barrier
__device__ __forceinline__ void tma_load_pair(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(tm), "r"(bar), "r"(c0), "r"(c1) : "memory");
}
__device__ __forceinline__ void tma_load_pair_hint(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int c0, int c1, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4}], [%2], %5;"
      ::"r"(dst), "l"(tm), "r"(bar), "r"(c0), "r"(c1), "l"(policy) : "memory");
}
__device__ __forceinline__ void umma_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// arrives on the barrier at this offset in both CTAs of the pair once the MMAs issued so far have retired
__device__ __forceinline__ void umma_commit_pair(uint32_t bar, uint16_t mask) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar), "h"(mask)
      : "memory");
}
__device__ __forceinline__ void tmem_ld8_nowait(uint32_t taddr, float* v) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]) : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_landed(float* v) {   // the registers are valid only behind the wait
  asm volatile("" : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]) :: "memory");
}
// like every barrier the cluster barrier counts warps: each executes both halves once, converged
__device__ __forceinline__ void cluster_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the peer's abort flag; seen by whoever sees an arrival that follows
__device__ __forceinline__ void abort_peer(uint32_t flag) {
  asm volatile("st.shared::cluster.u32 [%0], 1;" ::"r"(flag) : "memory");
  asm volatile("fence.acq_rel.cluster;" ::: "memory");
}
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
template <int THREADS>
__device__ __forceinline__ void epi_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory"); }   // all read-out warps
__device__ __forceinline__ void group_barrier(int g) { asm volatile("bar.sync %0, 128;" ::"r"(2 + g) : "memory"); }   // one group of four warps

// four values as two leading bf16 pairs and the pairs of what that rounding lost
__device__ __forceinline__ void split4(const float (&v)[4], uint2& hi, uint2& lo) {
  const __nv_bfloat162 h0 = __floats2bfloat162_rn(v[0], v[1]), h1 = __floats2bfloat162_rn(v[2], v[3]);
  const float2 f0 = __bfloat1622float2(h0), f1 = __bfloat1622float2(h1);
  const __nv_bfloat162 l0 = __floats2bfloat162_rn(v[0] - f0.x, v[1] - f0.y), l1 = __floats2bfloat162_rn(v[2] - f1.x, v[3] - f1.y);
  hi = make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1));
  lo = make_uint2(*reinterpret_cast<const uint32_t*>(&l0), *reinterpret_cast<const uint32_t*>(&l1));
}

// C token columns of this thread's feature: the accumulator and, `lo` columns further, its second term's half
// (stacked terms; -1 = none), added up.  Each branch waits for its own loads: a register loaded in one
// branch and waited for behind it could be copied before it has landed.
template <int C>
__device__ __forceinline__ void read_chunk(uint32_t taddr, int lo, float (&v)[C]) {
  if (lo >= 0) {
    float w[C];
#pragma unroll
    for (int c = 0; c < C; c += 8) {
      tmem_ld8_nowait(taddr + (uint32_t)c, v + c);
      tmem_ld8_nowait(taddr + (uint32_t)(lo + c), w + c);
    }
    tmem_ld_wait();
#pragma unroll
    for (int c = 0; c < C; c += 8) { tmem_landed(v + c); tmem_landed(w + c); }
#pragma unroll
    for (int j = 0; j < C; ++j) v[j] += w[j];
  } else {
#pragma unroll
    for (int c = 0; c < C; c += 8) tmem_ld8_nowait(taddr + (uint32_t)c, v + c);
    tmem_ld_wait();
#pragma unroll
    for (int c = 0; c < C; c += 8) tmem_landed(v + c);
  }
}

// SwiGLU of eight parked tokens ([8][64 gate, 64 up features]): thread = four features of a token
__device__ __forceinline__ void finish_swiglu(const PairArgs& a, const float* park, int tile, int c0, int t) {
  const int j = 4 * (t & 15), jj0 = tile * 64 + j, lt = t >> 4, tok = c0 + lt;
  if (tok >= a.rows || jj0 >= a.F) return;
  const float4 g = *reinterpret_cast<const float4*>(park + lt * CS_GEMM_BM + j);
  const float4 up = *reinterpret_cast<const float4*>(park + lt * CS_GEMM_BM + 64 + j);
  const float gv[4] = {g.x, g.y, g.z, g.w}, uv[4] = {up.x, up.y, up.z, up.w};
  float v4[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) v4[i] = __fdividef(gv[i], 1.f + __expf(-gv[i])) * uv[i];
  uint2 hi, lo;
  split4(v4, hi, lo);
  // (F is a multiple of 8, so four features are written together or not at all)
  *reinterpret_cast<uint2*>(a.act + (size_t)tok * a.F + jj0) = hi;
  *reinterpret_cast<uint2*>(a.act_lo + (size_t)tok * a.F + jj0) = lo;
}

// largest logit (lowest id on ties) of eight parked tokens: 16 threads per token, eight features each
__device__ __forceinline__ void finish_argmax(const PairArgs& a, const float* park, int tile, int c0, int t) {
  const int lt = t >> 4, i = t & 15, tok = c0 + lt, n0 = tile * CS_GEMM_BM;
  float best = -INFINITY;
  int idx = INT32_MAX;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int f = 4 * i + 64 * q;
    const float4 y = *reinterpret_cast<const float4*>(park + lt * CS_GEMM_BM + f);
    const float v[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (n0 + f + e < a.N && v[e] > best) { best = v[e]; idx = n0 + f + e; }
    if (a.out != nullptr && tok < a.rows) {
      float* dst = a.out + (size_t)tok * a.N + n0 + f;
      if (a.vec_out && n0 + f < a.N) {
        *reinterpret_cast<float4*>(dst) = y;
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (n0 + f + e < a.N) dst[e] = v[e];
      }
    }
  }
#pragma unroll
  for (int off = 8; off > 0; off >>= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, best, off);
    const int oi = __shfl_xor_sync(0xffffffffu, idx, off);
    if (ov > best || (ov == best && oi < idx)) { best = ov; idx = oi; }
  }
  if (i == 0 && tok < a.rows && n0 < a.N) {
    a.tile_max[(size_t)tok * a.tile_stride + tile] = best;
    a.tile_idx[(size_t)tok * a.tile_stride + tile] = idx;
  }
}

// threads of a launch with G read-out groups of four warps (one warp per TMEM lane quarter), producer, MMA issuer
constexpr int pair_threads(int G) { return 128 * G + 64; }

// C = token columns per read-out step of a group
template <bool STREAM, int G, int C>
__global__ void __launch_bounds__(pair_threads(G), 1)
k_gemm_pair(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX, PairArgs a) {
  constexpr int kEpiWarps = 4 * G, kEpiThreads = 128 * G, kProdWarp = kEpiWarps, kMmaWarp = kEpiWarps + 1;
  constexpr int kChunk = C, kChunkBytes = C * CS_GEMM_BM * 4;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  uint8_t* smem = smem_raw + (((raw + 1023u) & ~1023u) - raw);   // operand tiles need 1024-byte alignment
  const int n_tok = a.n_tok, stages = a.stages;
  const int xbytes = a.terms * n_tok * 64;                       // this CTA's share of the activations of one K block
  const int stage_bytes = kABytes + xbytes;
  float* park = reinterpret_cast<float*>(smem + (size_t)stages * stage_bytes);   // stream form: two chunk buffers per group
  uint8_t* ctl = smem + (size_t)stages * stage_bytes + (STREAM ? 2 * G * kChunkBytes : 0);
  uint64_t* bars = reinterpret_cast<uint64_t*>(ctl);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kMaxStages + 4);
  volatile int* s_abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* s_never = reinterpret_cast<volatile int*>(tmem_slot + 2);   // stays 0: drains wait on time only
  volatile int* s_shares = reinterpret_cast<volatile int*>(tmem_slot + 3);
  float* rstd_s = reinterpret_cast<float*>(ctl + kCtlBytes);     // [n_tok]
  const uint32_t b_full = smem_u32(bars), b_empty = smem_u32(bars + kMaxStages), b_accf = smem_u32(bars + 2 * kMaxStages),
                 b_acce = b_accf + 16;

  const int tid = threadIdx.x, warp = (int)uniform(tid >> 5), lane = tid & 31;
  const int half = (int)(blockIdx.x & 1u);                       // which 128 features of the pair's 256, which half of the tokens
  const int pair = STREAM ? (int)((gridDim.x - 1 - blockIdx.x) >> 1) : (int)(blockIdx.x >> 1);
  // this pair's run of (tile, K block) units
  int u0, u1;
  if (STREAM) {
    const long long pairs = gridDim.x >> 1;
    u0 = (int)(pair * (long long)a.units / pairs);
    u1 = (int)((pair + 1) * (long long)a.units / pairs);
  } else {
    const int t = pair / a.splits, kb0 = (pair - t * a.splits) * a.kb_per_split;
    u0 = t * a.num_kb + kb0;
    u1 = t * a.num_kb + min(a.num_kb, kb0 + a.kb_per_split);
  }
  const int t_lo = u0 / a.num_kb, t_hi = (u1 - 1) / a.num_kb;
  const int accw = a.stacked ? 2 * n_tok : n_tok;
  uint32_t tmem_cols = 32;
  while ((int)tmem_cols < (STREAM ? 2 : 1) * accw) tmem_cols <<= 1;

  if (tid == kProdWarp * 32) {
    for (int s = 0; s < stages; ++s) { mbar_init(b_full + 8 * s, 1); mbar_init(b_empty + 8 * s, 1); }
    for (int s = 0; s < 2; ++s) { mbar_init(b_accf + 8 * s, 1); mbar_init(b_acce + 8 * s, 2 * kEpiWarps); }
    *s_abort = 0;
    *s_never = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmW) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmX) : "memory");
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  cluster_sync();                                                // the peer's barriers exist before anything arrives on them
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  // (after the allocation: the successor's CTAs must not take tensor memory ahead of this kernel's)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const uint32_t tmem_base = uniform(*tmem_slot);

  if (warp == kProdWarp) {
    // ------------------------------------------------------------- TMA producer (both CTAs)
    const uint32_t full_even = uniform(map_rank(b_full, 0)), ring = smem_u32(smem);
    const uint64_t policy = l2_evict_first();                    // (of the weights: each byte is read once)
    const int xrow = a.stacked ? half * a.lo_row : half * (n_tok >> 1);
    const bool second = a.terms == 2 && !a.stacked;
    int tw = t_lo, kw = u0 - tw * a.num_kb, kx = kw;             // next weight tile and its K block; next K block of the activations
    const int drop = STREAM && !(pair & 1) ? -1 : a.drop_kb;
    auto load_w = [&](int i, int s) {
      if (i != drop && elect_one()) {
        if (half == 0) mbar_expect_tx(b_full + 8 * s, 2u * (uint32_t)stage_bytes);   // both CTAs' copies of the stage
        tma_load_pair_hint(ring + (uint32_t)(s * stage_bytes), &tmW, full_even + 8 * s, kw * CS_GEMM_BK, (2 * tw + half) * CS_GEMM_BM, policy);
      }
      if (++kw == a.num_kb) { kw = 0; ++tw; }
    };
    auto load_x = [&](int i, int s) {
      if (i != drop && elect_one()) {
        const uint32_t sx = ring + (uint32_t)(s * stage_bytes) + kABytes;
        tma_load_pair(sx, &tmX, full_even + 8 * s, kx * CS_GEMM_BK, xrow);
        if (second) tma_load_pair(sx + (uint32_t)n_tok * 64u, &tmX, full_even + 8 * s, kx * CS_GEMM_BK, a.lo_row + xrow);
      }
      if (++kx == a.num_kb) kx = 0;
    };
    const int n = u1 - u0, npre = min(n, stages);
    bool ok = true;
    int i = 0, s = 0;
    uint32_t ph = 0;
    for (; i < npre; ++i) load_w(i, i);                             // weights depend on nothing
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (i = 0; i < npre; ++i) load_x(i, i);
    for (; i < n; ++i) {
      ok = mbar_wait_warp(b_empty + 8 * s, ph, s_abort, a.wait_ns);
      if (!ok) break;
      load_w(i, s);
      load_x(i, s);
      if (++s == stages) { s = 0; ph ^= 1u; }
    }
    if (!ok && lane == 0) { *s_abort = 1; atomicOr(a.status, CS_DEV_TIMEOUT); }
    __syncwarp();
    if (*s_abort && lane == 0) {
      // copies in flight land before this CTA's shared memory goes away: the even CTA sees them on its
      // barriers, the odd one gives them a thousand times their latency
      if (half == 0) {
        for (int j = max(0, i - stages); j < i; ++j)
          if (j != drop) mbar_wait(b_full + 8 * (j % stages), (uint32_t)(j / stages) & 1u, s_never, 1000000ull);
      } else {
        const unsigned long long t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 1000000ull) {}
      }
    }
  } else if (warp == kMmaWarp) {
    // ------------------------------------------------------------- MMA issuer (even CTA only)
    if (half == 0) {
      const uint16_t mask = 3;                                   // (both CTAs of the cluster)
      // bf16 x bf16 -> fp32, both operands K-major, M = 256 over the pair
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(accw >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
      const bool second = a.terms == 2 && !a.stacked;
      const uint64_t desc0 = desc_kmajor(smem_u32(smem));
      const uint64_t x_off = kABytes >> 4, lo_off = (uint64_t)(uint32_t)((kABytes + n_tok * 64) >> 4);
      bool ok = true;
      int j = 0, s = 0;
      uint32_t ph = 0;
      for (int t = t_lo; t <= t_hi && ok; ++t, ++j) {
        int todo = min(u1 - t * a.num_kb, a.num_kb) - max(u0 - t * a.num_kb, 0);
        const int buf = STREAM ? (j & 1) : 0;
        const uint32_t acc = tmem_base + (uint32_t)(buf * accw);
        if (j >= 2) ok = mbar_wait_warp(b_acce + 8 * buf, (uint32_t)((j >> 1) - 1) & 1u, s_abort, a.wait_ns);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        uint32_t acc_on = 0;
        for (; todo > 0; --todo) {
          ok = mbar_wait_warp(b_full + 8 * s, ph, s_abort, a.wait_ns);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          if (elect_one()) {
            const uint64_t da = desc0 + (uint64_t)(uint32_t)(s * (stage_bytes >> 4));
#pragma unroll
            for (int kk = 0; kk < CS_GEMM_BK / 16; ++kk) {       // 16 K-elements = 32 bytes per instruction
              umma_pair(acc, da + 2 * kk, da + x_off + 2 * kk, idesc, kk == 0 ? acc_on : 1u);
              if (second) umma_pair(acc, da + 2 * kk, da + lo_off + 2 * kk, idesc, 1u);   // x = hi + lo
            }
            umma_commit_pair(b_empty + 8 * s, mask);
          }
          acc_on = 1u;
          if (++s == stages) { s = 0; ph ^= 1u; }
        }
        if (!ok && lane == 0) {                                  // (both CTAs know before the accumulator looks finished)
          *s_abort = 1;
          abort_peer(map_rank(smem_u32(const_cast<int*>(s_abort)), 1));
          atomicOr(a.status, CS_DEV_TIMEOUT);
        }
        __syncwarp();
        if (elect_one()) umma_commit_pair(b_accf + 8 * buf, mask);
        if (!ok) {
          mbar_wait(b_accf + 8 * buf, (uint32_t)(j >> 1) & 1u, s_never, a.wait_ns);   // what was issued has retired
        }
      }
    }
  } else {
    // ------------------------------------------------------------- read-out warps (both CTAs)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int wq = warp & 3, g = warp >> 2, t = tid & 127;
    const bool scaled = a.nf.ssq_in != nullptr;
    if (scaled) {
      // 1/rms of every token row while the main loop runs: slots summed in a fixed order, eight rows at a time
      for (int tok0 = warp * 8; tok0 < a.rows; tok0 += 8 * kEpiWarps) {
        float ss[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) ss[r] = 0.f;
        for (int sl = lane; sl < a.nf.slots_in; sl += 32) {
#pragma unroll
          for (int r = 0; r < 8; ++r)
            if (tok0 + r < a.rows) ss[r] += a.nf.ssq_in[(size_t)(tok0 + r) * a.nf.slot_stride + sl];
        }
#pragma unroll
        for (int r = 0; r < 8; ++r) {
#pragma unroll
          for (int off = 16; off > 0; off >>= 1) ss[r] += __shfl_xor_sync(0xffffffffu, ss[r], off);
          if (lane == 0 && tok0 + r < a.rows) rstd_s[tok0 + r] = rsqrtf(ss[r] * a.nf.inv_d + a.nf.eps);
        }
      }
      epi_barrier<kEpiThreads>();
    }
    const uint32_t lane_base = tmem_base + ((uint32_t)(wq * 32) << 16);
    const int feat = wq * 32 + lane;                             // this thread's feature within the CTA's tile
    const int nchunk = (min(n_tok, a.rows) + kChunk - 1) / kChunk;
    bool ok = true;
    if constexpr (STREAM) {
      const uint32_t acce_even = map_rank(b_acce, 0);
      const bool ends_in_head = u1 < (t_hi + 1) * a.num_kb;      // the last tile's tail is with the next pair
      const int own = 2 * pair + half, next = own + 2;
      const float* theirs = a.part + (size_t)next * CS_GEMM_BM * CS_MAX_ROWS;
      int j = 0, turn = 0;
      for (int tp = t_lo; tp <= t_hi; ++tp, ++j) {
        const int tile = 2 * tp + half, buf = j & 1;
        const bool give = u0 > tp * a.num_kb;                    // the tail of a tile that the pair before finishes
        const bool take = ends_in_head && tp == t_hi;            // (a run is at least a tile long: never walked first)
        const uint32_t acc = lane_base + (uint32_t)(buf * accw);
        ok = mbar_wait(b_accf + 8 * buf, (uint32_t)(j >> 1) & 1u, s_abort, a.wait_ns);
        // (the other pair's sums are asked for now and not ahead of time: polling for them while the MMAs run
        //  costs 2 us at 11 rows)
        if (ok && take && lane == 0) ok = count_wait(a.part_flag + next, 1, s_abort, a.wait_ns) >= 0;
        ok = __all_sync(0xffffffffu, ok) && *s_abort == 0;
        if (!ok) {
          *s_abort = 1;
          if (lane == 0) atomicOr(a.status, CS_DEV_TIMEOUT);
        }
        // the decision to go on is one for all read-out warps: they meet at barriers below
        uint32_t go;
        asm volatile("{\n.reg .pred p, q;\nsetp.ne.b32 p, %1, 0;\nbar.red.and.pred q, 1, %2, p;\nselp.u32 %0, 1, 0, q;\n}"
                     : "=r"(go) : "r"((uint32_t)ok), "n"(kEpiThreads) : "memory");
        if (!go) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        float w[C];
        auto fetch = [&](int c) {                                // the other pair's sums of chunk c
#pragma unroll
          for (int q = 0; q < C; ++q) w[q] = __ldcg(theirs + (size_t)(c * C + q) * CS_GEMM_BM + feat);
        };
        if (take && g < nchunk) fetch(g);
        for (int c = g; c < nchunk; c += G, ++turn) {
          const int c0 = c * C;
          float v[C];
          read_chunk<C>(acc + (uint32_t)c0, a.stacked ? n_tok : -1, v);
          if (take) {
#pragma unroll
            for (int q = 0; q < C; ++q) v[q] += w[q];
            if (c + G < nchunk) fetch(c + G);                    // (on its way while this chunk is finished)
          }
          if (give) {
            float* mine = a.part + (size_t)own * CS_GEMM_BM * CS_MAX_ROWS;
#pragma unroll
            for (int q = 0; q < C; ++q) mine[(size_t)(c0 + q) * CS_GEMM_BM + feat] = v[q];
            continue;
          }
          float* pk = park + (size_t)(2 * g + (turn & 1)) * (C * CS_GEMM_BM);
#pragma unroll
          for (int q = 0; q < C; ++q) {
            const float r = (scaled && c0 + q < a.rows) ? rstd_s[c0 + q] : 1.f;
            pk[q * CS_GEMM_BM + feat] = v[q] * r;
          }
          group_barrier(g);                                      // (two buffers: a thread that runs ahead fills the other one)
#pragma unroll
          for (int q = 0; q < C; q += 8) {
            if (a.mode == CS_EPI_SWIGLU) finish_swiglu(a, pk + q * CS_GEMM_BM, tile, c0 + q, t);
            else finish_argmax(a, pk + q * CS_GEMM_BM, tile, c0 + q, t);
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(acce_even + 8 * buf);
        if (give || take) {
          epi_barrier<kEpiThreads>();                            // all of this CTA's sums are written, or read
          if (tid == 0) {
            __threadfence();
            asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(a.part_flag + (give ? own : next)), "r"(give ? 1 : 0) : "memory");
          }
        }
      }
    } else {
      const int S = a.splits, tile = 2 * t_lo + half, n0 = tile * CS_GEMM_BM, split = pair - t_lo * S;
      int* word = a.part_flag + tile;                            // (S > 1: arrivals | shares left to others << 8 | leavers << 16 | started << 24)
      if (S > 1 && tid == 0) atomicAdd(word, 1 << 24);
      const int share = (a.rows + S - 1) / S;                    // tokens a pair finishes
      const int f = 4 * lane;                                    // STORE, RESIDUAL: a warp per token, four features per lane
      const bool resid = a.mode == CS_EPI_RESIDUAL, feeds = a.nf.gain_out != nullptr;
      const bool vec = a.vec_out && n0 + f + 3 < a.N;
      // the residual rows and the next norm's gain are asked for while the MMAs still run
      float4 x_pre[kBatch];
      uint2 gain = make_uint2(0u, 0u);
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const int tok = min(split * share + warp + u * kEpiWarps, a.rows - 1);
        x_pre[u] = resid && vec ? *reinterpret_cast<const float4*>(a.out + (size_t)tok * a.N + n0 + f) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
      if (feeds && vec) gain = *reinterpret_cast<const uint2*>(a.nf.gain_out + n0 + f);
      bool all_started = S > 1 && tid == 0 && started(word) == S;
      ok = mbar_wait(b_accf, 0, s_abort, a.wait_ns);
      ok = __all_sync(0xffffffffu, ok) && *s_abort == 0;
      if (!ok && lane == 0) atomicOr(a.status, CS_DEV_TIMEOUT);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      // Every pair's sums as [token][128 features]: in the workspace, or with S = 1 in the ring (the MMAs have
      // retired, it is free)
      float* dump = S > 1 ? a.part + (size_t)blockIdx.x * CS_GEMM_BM * CS_MAX_ROWS : reinterpret_cast<float*>(smem);
      for (int c = g; c < nchunk; c += G) {
        const int c0 = c * kChunk;
        float v[kChunk];
        if (ok) {
          read_chunk<C>(lane_base + (uint32_t)c0, a.stacked ? n_tok : -1, v);
        } else {
#pragma unroll
          for (int q = 0; q < kChunk; ++q) v[q] = 0.f;
        }
#pragma unroll
        for (int q = 0; q < kChunk; ++q) {
          const float r = (scaled && c0 + q < a.rows) ? rstd_s[c0 + q] : 1.f;
          dump[(size_t)(c0 + q) * CS_GEMM_BM + feat] = v[q] * r;
        }
      }
      epi_barrier<kEpiThreads>();
      if (tid == 0) {
        int mine = 1;                                            // bit r: this CTA finishes share r
        if (S > 1) {
          __threadfence();
          all_started = all_started || started(word) == S;
          if (a.leave != 0) all_started = !(a.leave >> split & 1);
          atomicAdd(word, all_started ? 1 : 1 + (1 << (8 + split)));
          mine = 0;
          if (all_started) {
            // (shares left behind go to the first pair that waits; the last one to come always does)
            const int left = count_wait(word, S, s_abort, a.wait_ns);
            if (left >= 0) mine = 1 << split | (__ffs(~left) - 1 == split ? left : 0);
            else { *s_abort = 1; atomicOr(a.status, CS_DEV_TIMEOUT); }
          }
        }
        *s_shares = mine;
      }
      epi_barrier<kEpiThreads>();
      const float* sums = a.part + (size_t)(2 * t_lo * S + half) * CS_GEMM_BM * CS_MAX_ROWS;
      // four features of one token from four pairs (requests only; S is rarely above 4), and their sum in
      // the order of the K ranges
      auto ask = [&](int q0, int tok, int feat0, float4 (&v)[4]) {
        const size_t at = (size_t)tok * CS_GEMM_BM + feat0;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          v[e] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (S == 1 && e == 0) v[e] = *reinterpret_cast<const float4*>(dump + at);
          else if (q0 + e < S) v[e] = __ldcg(reinterpret_cast<const float4*>(sums + (size_t)(q0 + e) * 2 * CS_GEMM_BM * CS_MAX_ROWS + at));
        }
      };
      auto add = [](float4 y, const float4 (&v)[4]) {
#pragma unroll
        for (int e = 0; e < 4; ++e) { y.x += v[e].x; y.y += v[e].y; y.z += v[e].z; y.w += v[e].w; }
        return y;
      };
      const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
      // The own share first: x_pre holds its residual rows, and other shares load theirs over them
      for (int todo = *s_shares, r = split; todo != 0; todo &= ~(1 << r), r = __ffs(todo) - 1) {
        const int lo = r * share, hi = min(a.rows, lo + share);
        if (a.mode == CS_EPI_QKV) {
          // RoPE pairs feature i of a head with i + Dh/2: both lie in this tile; j in [0, 64) walks the first
          // halves, two tokens per warp
          const QkvEpi& Q = a.q;
          const int j = 4 * (lane & 15), hd = Q.Dh >> 1, i = j % hd, f1 = (j / hd) * Q.Dh + i, f2 = f1 + hd;
          const int head = (n0 + f1) / Q.Dh;
          const bool is_v = head >= Q.H + Q.Hkv;
          if (head >= Q.H + 2 * Q.Hkv) continue;
          for (int tok = lo + 2 * warp + (lane >> 4); tok < hi; tok += 2 * kEpiWarps) {
            const float4* csp = reinterpret_cast<const float4*>(Q.rope_cs + 2 * ((size_t)tok * hd + i));
            const float4 cs01 = csp[0], cs23 = csp[1];           // (cos, sin) of dims i .. i + 3
            const int row_w = Q.row_write[tok], row_p = Q.row_pos[tok];
            float4 va[4], vb[4];
            ask(0, tok, f1, va);
            ask(0, tok, f2, vb);
            float4 av = add(zero, va), bv = add(zero, vb);
            if (S > 4) {
              ask(4, tok, f1, va);
              ask(4, tok, f2, vb);
              av = add(av, va); bv = add(bv, vb);
            }
            const float a4[4] = {av.x, av.y, av.z, av.w}, b4[4] = {bv.x, bv.y, bv.z, bv.w};
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
            if (head < Q.H) {                                    // rotated query as two bf16 terms
              __nv_bfloat16* qd = Q.qbuf + ((size_t)tok * Q.H + head) * Q.Dh + i;
              __nv_bfloat16* ql = qd + (size_t)CS_MAX_ROWS * Q.H * Q.Dh;
              *reinterpret_cast<uint2*>(qd) = h0;
              *reinterpret_cast<uint2*>(qd + hd) = h1;
              *reinterpret_cast<uint2*>(ql) = l0;
              *reinterpret_cast<uint2*>(ql + hd) = l1;
            } else if (row_w) {                                  // new K (rotated) / V row of the cache, stored in bf16
              const int kvh = is_v ? head - Q.H - Q.Hkv : head - Q.H;
              __nv_bfloat16* dst = Q.kv + ((((size_t)Q.layer * 2 + (is_v ? 1 : 0)) * Q.max_batch + tok / Q.R) * Q.Hkv + kvh) *
                                              (size_t)Q.max_seq * Q.Dh + (size_t)row_p * Q.Dh + i;
              *reinterpret_cast<uint2*>(dst) = h0;
              *reinterpret_cast<uint2*>(dst + hd) = h1;
            }
          }
          continue;
        }
        const float2 g01 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&gain.x));
        const float2 g23 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&gain.y));
        for (int tok0 = lo + warp; tok0 < hi; tok0 += kBatch * kEpiWarps) {
          float4 y[kBatch];
          if (resid && vec && (tok0 != lo + warp || r != split)) {
#pragma unroll
            for (int u = 0; u < kBatch; ++u)
              x_pre[u] = *reinterpret_cast<const float4*>(a.out + (size_t)min(tok0 + u * kEpiWarps, a.rows - 1) * a.N + n0 + f);
          }
#pragma unroll
          for (int u = 0; u < kBatch; ++u) y[u] = zero;
#pragma unroll 1
          for (int q0 = 0; q0 < S; q0 += 4) {
            float4 v[kBatch][4];
#pragma unroll
            for (int u = 0; u < kBatch; ++u) ask(q0, min(tok0 + u * kEpiWarps, a.rows - 1), f, v[u]);
#pragma unroll
            for (int u = 0; u < kBatch; ++u) y[u] = add(y[u], v[u]);
          }
#pragma unroll
          for (int u = 0; u < kBatch; ++u) {
            const int tok = tok0 + u * kEpiWarps;                // (the same for the whole warp)
            if (tok >= hi) break;
            float* dst = a.out + (size_t)tok * a.N + n0 + f;
            float ss = 0.f;
            if (vec) {
              const float o[4] = {y[u].x + x_pre[u].x, y[u].y + x_pre[u].y, y[u].z + x_pre[u].z, y[u].w + x_pre[u].w};
              *reinterpret_cast<float4*>(dst) = make_float4(o[0], o[1], o[2], o[3]);
              if (feeds) {
                const float w[4] = {o[0] * g01.x, o[1] * g01.y, o[2] * g23.x, o[3] * g23.y};
                uint2 hi2, lo2;
                split4(w, hi2, lo2);
                __nv_bfloat16* xo = a.nf.xn_out + (size_t)tok * a.N + n0 + f;
                *reinterpret_cast<uint2*>(xo) = hi2;
                *reinterpret_cast<uint2*>(xo + (size_t)CS_MAX_ROWS * a.N) = lo2;
                ss = (o[0] * o[0] + o[1] * o[1]) + (o[2] * o[2] + o[3] * o[3]);
              }
            } else {
              const float yv[4] = {y[u].x, y[u].y, y[u].z, y[u].w};
#pragma unroll
              for (int e = 0; e < 4; ++e)
                if (n0 + f + e < a.N) dst[e] = resid ? dst[e] + yv[e] : yv[e];
            }
            if (feeds) {
#pragma unroll
              for (int off = 16; off > 0; off >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
              if (lane == 0 && n0 < a.N) a.nf.ssq_out[(size_t)tok * a.nf.slot_stride + tile] = ss;
            }
          }
        }
      }
      // the last of the tile's pairs to leave puts the word back to rest
      if (S > 1 && tid == 0 && ((atomicAdd(word, 1 << 16) >> 16) & 0xff) + 1 == S) atomicExch(word, 0);
    }
  }
  // ---------------------------------------------------------------- teardown: nobody leaves while a peer
  // still reads its shared memory, signals its barriers or uses the pair's tensor memory
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  cluster_sync();
  if (tid == 0) cs_stamp_end(a.stamp);
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
  }
}

typedef void (*PairKernel)(const CUtensorMap, const CUtensorMap, PairArgs);

// what one CTA needs behind the ring, and the ring's depth for a block height
int pair_fixed_bytes(int n_tok, bool stream) { return 1024 /*alignment slack*/ + kCtlBytes + n_tok * 4 + (stream ? 2 * 32 * CS_GEMM_BM * 4 : 0); }   // (G x C = 32)
int pair_stage_bytes(int n_tok, int terms) { return kABytes + terms * n_tok * 64; }
cs_status ensure_pair_attrs(cs_ctx* ctx) {
  if (!ctx->pair_attr_set) {
    for (PairKernel k : {(PairKernel)k_gemm_pair<false, 4, 8>, (PairKernel)k_gemm_pair<true, 4, 8>, (PairKernel)k_gemm_pair<true, 2, 16>})
      CS_CUDA_OK(ctx, cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
    ctx->pair_attr_set = true;
  }
  return CS_OK;
}

// How many pairs, one CTA per SM, the device runs at once (the two CTAs of a pair are a cluster).  Asked of the
// runtime once per context.
int pairs_at_once(const cs_ctx* cctx) {
  cs_ctx* ctx = const_cast<cs_ctx*>(cctx);
  if (ctx->pairs_at_once == 0) {
    int n = 0;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(2 * ctx->num_sms, 1, 1);
    lc.blockDim = dim3(pair_threads(4), 1, 1);
    lc.dynamicSmemBytes = 200 * 1024;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    lc.attrs = at;
    lc.numAttrs = 1;
    if (ensure_pair_attrs(ctx) != CS_OK || cudaOccupancyMaxActiveClusters(&n, k_gemm_pair<false, 4, 8>, &lc) != cudaSuccess || n < 1) {
      (void)cudaGetLastError();
      n = max(1, ctx->num_sms * 85 / 100 / 2);   // no answer: leave room
    }
    ctx->pairs_at_once = min(n, CS_MAX_PAIRS);
  }
  return ctx->pairs_at_once;
}

}  // namespace

// Split-K factor of the split form: K blocks per pair times the clocks of one (tensor pipe, issue, or the
// pair's share of HBM), plus the epilogue, times waves.  A split launch is a single wave.
static void pair_splits(const cs_ctx* ctx, const GemmPlan* g, int rows, bool two_terms, int* splits, int* kb_per_split) {
  const int n_tok = cs_ceil_div(rows, 16) * 16, terms = two_terms ? 2 : 1;
  const int tiles2 = cs_ceil_div(g->N, 2 * CS_GEMM_BM), kb = cs_ceil_div(g->K, CS_GEMM_BK), fit = pairs_at_once(ctx);
  long best = -1;
  for (int sp = 1; sp <= CS_PAIR_MAX_SPLITS && sp <= max(1, kb / 4); ++sp) {
    const int kps = cs_ceil_div(kb, sp), spl = cs_ceil_div(kb, kps);
    if (spl > 1 && tiles2 * spl > fit) break;
    const long waves = cs_ceil_div(tiles2, fit);
    const long active = 2L * min(tiles2 * spl, fit);
    const long per_kb = max(max(2L * terms * n_tok, 350L), kABytes * active / 3500);
    const long cost = waves * (kps * per_kb + 4000 + (spl > 1 ? 2500 : 0) + 20L * n_tok + 40L * n_tok / spl);
    if (best < 0 || cost < best) { best = cost; *splits = spl; *kb_per_split = kps; }
  }
}

// sums of squares a residual GEMM leaves per token: one per 128-feature tile, in the one-SM kernel times its split-K factor
int cs_norm_slots(const GemmPlan* g, int rows) {
  return cs_ceil_div(g->N, CS_GEMM_BM) * (cs_gemm_on_pairs(CS_EPI_RESIDUAL, rows) ? 1 : g->splits);
}

cs_status cs_launch_gemm_pair(cs_ctx* ctx, const GemmPlan* g, const CUtensorMap* tmX, int lo_row, int rows, int mode, float* out,
                              __nv_bfloat16* act, __nv_bfloat16* act_lo, int F, const QkvEpi* q, const NormFuse* nf,
                              cudaStream_t st) {
  const bool stream = mode == CS_EPI_SWIGLU || mode == CS_EPI_ARGMAX;
  if (nf != nullptr && nf->gain_out != nullptr && (mode != CS_EPI_RESIDUAL || (g->N & 3) != 0)) {
    snprintf(ctx->err, sizeof(ctx->err), "a norm can only be folded into a residual GEMM whose width is a multiple of 4");
    return CS_ERR_UNSUPPORTED;
  }
  PairArgs a = {};
  a.rows = rows;
  a.n_tok = cs_ceil_div(rows, 16) * 16;
  a.N = g->N;
  a.num_kb = cs_ceil_div(g->K, CS_GEMM_BK);
  a.terms = lo_row >= 0 ? 2 : 1;
  a.stacked = (a.terms == 2 && a.n_tok <= 128) ? 1 : 0;
  a.lo_row = lo_row;
  a.mode = mode;
  a.out = out;
  a.vec_out = (g->N & 3) == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0;
  a.act = act; a.act_lo = act_lo; a.F = F;
  if (q != nullptr) a.q = *q;
  if (nf != nullptr) a.nf = *nf;
  a.tile_max = ctx->tile_max; a.tile_idx = ctx->tile_idx; a.tile_stride = cs_ceil_div(g->N, CS_GEMM_BM);
  a.part = ctx->pair_part; a.part_flag = ctx->pair_flag;
  a.drop_kb = ctx->debug_drop_kb;
  ctx->debug_drop_kb = -1;            // the hook covers one launch
  a.status = ctx->d_status;
  a.wait_ns = ctx->wait_limit_ns;
  a.stamp = cs_next_stamp(ctx, mode == CS_EPI_ARGMAX ? CS_FAM_LMHEAD : CS_FAM_GEMM);
  // (up to 32 rows two groups of 16 columns read the tile out in one step; taller, four groups of eight)
  const bool narrow = stream && a.n_tok <= 32;
  const int groups = narrow ? 2 : 4, fixed = pair_fixed_bytes(a.n_tok, stream), stage = pair_stage_bytes(a.n_tok, a.terms);
  a.stages = min(kMaxStages, (227 * 1024 - fixed) / stage);
  const size_t smem = (size_t)fixed + (size_t)a.stages * stage;
  const int tiles2 = cs_ceil_div(g->N, 2 * CS_GEMM_BM);
  cs_status s = ensure_pair_attrs(ctx);
  if (s != CS_OK) return s;
  cudaLaunchConfig_t lc = {};
  a.splits = 1;
  if (stream) {
    const int pairs = min(pairs_at_once(ctx), tiles2);   // a run is never shorter than one tile
    a.units = tiles2 * a.num_kb;
    lc.gridDim = dim3(2 * pairs, 1, 1);
  } else {
    pair_splits(ctx, g, rows, lo_row >= 0, &a.splits, &a.kb_per_split);
    a.leave = ctx->debug_leave & ((1 << (a.splits - 1)) - 1);   // (the last K range's pair always waits for the others)
    lc.gridDim = dim3(2 * tiles2 * a.splits, 1, 1);
  }
  lc.blockDim = dim3(pair_threads(groups), 1, 1);
  lc.dynamicSmemBytes = smem;
  lc.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = 2; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
  lc.attrs = at;
  lc.numAttrs = 2;
  const PairKernel kernel = !stream ? k_gemm_pair<false, 4, 8> : narrow ? k_gemm_pair<true, 2, 16> : k_gemm_pair<true, 4, 8>;
  CS_CUDA_OK(ctx, cudaLaunchKernelEx(&lc, kernel, g->tmW, *tmX, a));
  return CS_OK;
}
