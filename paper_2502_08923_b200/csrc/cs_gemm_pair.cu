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
// Two launch forms share the pipeline (TMA producer warp, MMA warp on the even CTA, eight read-out
// warps):
//   cluster form (STORE, RESIDUAL, QKV: few feature tiles, long K): cluster of 2 x S CTAs = one
//     256-feature tile, K split S ways, parked tiles summed over distributed shared memory in
//     rank order, every rank finishing a slice of the features;
//   stream form (SWIGLU, ARGMAX: many feature tiles): one persistent pair per two SMs; the
//     (tile, K block) units of the whole matrix are dealt out in equal contiguous runs, so 112 tiles
//     on 74 pairs take 1.51 turns instead of two.  A tile cut by a run boundary is finished by the
//     pair that holds its first K blocks - it gets there last - while the other pair left its sums
//     in the workspace at the start of its run.  Two accumulators in TMEM: a tile is read out
//     while the next one is multiplied.
//
// Measured on the 8B shape (us per launch: QKV / attention output / gate/up / down / LM head), before
// (one-SM tiles, launch shapes by a cost model) and now:
//    88 rows  23.5 19.9 54.9 36.5 272 -> 18.7 18.6 48.6 33.4 179
//   176 rows  31.8 26.7 90.7 49.1 509 -> 23.8 25.6 61.7 45.7 244   (two-term tensor floor 10.6 7.1 49 25 222)
//   256 rows  42.2 36.4 114 70.7 791  -> 29.5 33.0 79.1 60.4 273 with 256 keys cached
// and the stream form at 11 rows: gate/up 41.0 -> 40.1, LM head 168 -> 153 us (6.9 TB/s).
//
// Every wait is bounded as in cs_gemm.cu; the wait for another pair's sums is a poll with the same
// limit, and its writer never waits for anyone before it writes.
#include <algorithm>

#include "cs_common.cuh"
#include "cs_tcgen.cuh"

using std::max;
using std::min;

namespace {

constexpr int kEpiWarps = 8, kEpiThreads = kEpiWarps * 32;   // read-out and epilogue: two groups of four warps (one per TMEM lane quarter)
constexpr int kProdWarp = 8, kMmaWarp = 9, kThreads = 320;
constexpr int kABytes = CS_GEMM_BM * CS_GEMM_BK * 2;         // 16 KB: this CTA's weight tile of one K block
constexpr int kMaxStages = 10;
constexpr int kChunk = 16;                                   // token columns per read-out step
constexpr int kChunkBytes = kChunk * CS_GEMM_BM * 4;
constexpr int kParkBytes = 4 * kChunkBytes;                  // stream form: two chunk buffers per group
constexpr int kCtlBytes = (2 * kMaxStages + 4) * 8 + 16;

struct PairArgs {
  int rows, n_tok, N, num_kb;
  int splits, kb_per_split;   // cluster form
  int units;                  // stream form: pair tiles x K blocks
  int stages, terms, stacked, mode;
  int lo_row;                 // row coordinate of the activations' second term
  float* out;
  __nv_bfloat16 *act, *act_lo;
  int F;
  QkvEpi q;
  NormFuse nf;
  float* tile_max;
  int* tile_idx;
  int tile_stride;
  float* part;                // stream form: sums of the tile a run starts inside of, [pair][half][256][128]
  int* part_flag;             // [pair][half], 0 between launches
  int* status;
  unsigned long long wait_ns;
  unsigned long long* stamp;
};

__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {   // barrier of any CTA of the cluster
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __noinline__ bool flag_wait(const int* flag, volatile int* abort_flag, unsigned long long limit_ns) {
  const unsigned long long t0 = globaltimer_ns();
  for (;;) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
    if (v != 0) return true;
    if (*abort_flag || globaltimer_ns() - t0 > limit_ns) return false;
  }
}
// a copy of the pair: it lands in this CTA's shared memory and counts on the even CTA's barrier
__device__ __forceinline__ void tma_load_pair(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(tm), "r"(bar), "r"(c0), "r"(c1) : "memory");
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
__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_landed(uint32_t (&v)[16]) {   // the registers are valid only behind the wait
  asm volatile("" : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]), "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]) :: "memory");
}
// like every barrier the cluster barrier counts warps: each executes both halves once, converged
__device__ __forceinline__ void cluster_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ float4 ld_cluster(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void epi_barrier() { asm volatile("bar.sync 1, 256;" ::: "memory"); }                      // the eight read-out warps
__device__ __forceinline__ void group_barrier(int g) { asm volatile("bar.sync %0, 128;" ::"r"(2 + g) : "memory"); }   // one group of four

// four values as two leading bf16 pairs and the pairs of what that rounding lost
__device__ __forceinline__ void split4(const float (&v)[4], uint2& hi, uint2& lo) {
  const __nv_bfloat162 h0 = __floats2bfloat162_rn(v[0], v[1]), h1 = __floats2bfloat162_rn(v[2], v[3]);
  const float2 f0 = __bfloat1622float2(h0), f1 = __bfloat1622float2(h1);
  const __nv_bfloat162 l0 = __floats2bfloat162_rn(v[0] - f0.x, v[1] - f0.y), l1 = __floats2bfloat162_rn(v[2] - f1.x, v[3] - f1.y);
  hi = make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1));
  lo = make_uint2(*reinterpret_cast<const uint32_t*>(&l0), *reinterpret_cast<const uint32_t*>(&l1));
}

// 16 token columns of this thread's feature (the two terms' halves added when they are stacked)
__device__ __forceinline__ void read_chunk(uint32_t taddr, const PairArgs& a, float (&v)[16]) {
  uint32_t r[16], w[16];
  tmem_ld16_nowait(taddr, r);
  if (a.stacked) tmem_ld16_nowait(taddr + (uint32_t)a.n_tok, w);
  tmem_ld_wait();
  tmem_landed(r);
#pragma unroll
  for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
  if (a.stacked) {
    tmem_landed(w);
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] += __uint_as_float(w[j]);
  }
}

// SwiGLU of one parked chunk ([16 tokens][64 gate, 64 up features]): thread = four features of two tokens
__device__ __forceinline__ void finish_swiglu(const PairArgs& a, const float* park, int tile, int c0, int t) {
  const int j = 4 * (t & 15), jj0 = tile * 64 + j;
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int lt = (t >> 4) + 8 * u, tok = c0 + lt;
    if (tok >= a.rows || jj0 >= a.F) continue;
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
}

// largest logit (lowest id on ties) of one parked chunk's tokens: eight threads per token, 16 features each
__device__ __forceinline__ void finish_argmax(const PairArgs& a, const float* park, int tile, int c0, int t) {
  const int lt = t >> 3, i = t & 7, tok = c0 + lt, n0 = tile * CS_GEMM_BM;
  float best = -INFINITY;
  int idx = INT32_MAX;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int f = 4 * i + 32 * q;
    const float4 y = *reinterpret_cast<const float4*>(park + lt * CS_GEMM_BM + f);
    const float v[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (n0 + f + e < a.N && v[e] > best) { best = v[e]; idx = n0 + f + e; }
    if (a.out != nullptr && tok < a.rows) {
      float* dst = a.out + (size_t)tok * a.N + n0 + f;
      if ((a.N & 3) == 0 && n0 + f < a.N) {
        *reinterpret_cast<float4*>(dst) = y;
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (n0 + f + e < a.N) dst[e] = v[e];
      }
    }
  }
#pragma unroll
  for (int off = 4; off > 0; off >>= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, best, off);
    const int oi = __shfl_xor_sync(0xffffffffu, idx, off);
    if (ov > best || (ov == best && oi < idx)) { best = ov; idx = oi; }
  }
  if (i == 0 && tok < a.rows && n0 < a.N) {
    a.tile_max[(size_t)tok * a.tile_stride + tile] = best;
    a.tile_idx[(size_t)tok * a.tile_stride + tile] = idx;
  }
}

template <bool STREAM>
__global__ void __launch_bounds__(kThreads, 1)
k_gemm_pair(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX, PairArgs a) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  uint8_t* smem = smem_raw + (((raw + 1023u) & ~1023u) - raw);   // operand tiles need 1024-byte alignment
  const int n_tok = a.n_tok, stages = a.stages;
  const int xbytes = a.terms * n_tok * 64;                       // this CTA's share of the activations of one K block
  const int stage_bytes = kABytes + xbytes;
  float* park = reinterpret_cast<float*>(smem + (size_t)stages * stage_bytes);   // stream form only
  uint8_t* ctl = smem + (size_t)stages * stage_bytes + (STREAM ? kParkBytes : 0);
  uint64_t* bars = reinterpret_cast<uint64_t*>(ctl);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kMaxStages + 4);
  volatile int* s_abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* s_never = reinterpret_cast<volatile int*>(tmem_slot + 2);   // stays 0: drains wait on time only
  float* rstd_s = reinterpret_cast<float*>(ctl + kCtlBytes);     // [n_tok]
  const uint32_t b_full = smem_u32(bars), b_empty = smem_u32(bars + kMaxStages), b_accf = smem_u32(bars + 2 * kMaxStages),
                 b_acce = b_accf + 16;

  const int tid = threadIdx.x, warp = (int)uniform(tid >> 5), lane = tid & 31;
  // cluster of (2, S, 1) CTAs, so the rank follows from the block index
  const uint32_t rank = (blockIdx.x & 1u) + 2u * (STREAM ? 0u : blockIdx.y), even = rank & ~1u;
  const int half = (int)(blockIdx.x & 1u);                       // which 128 features of the pair's 256, which half of the tokens
  // this pair's run of (tile, K block) units
  int u0, u1;
  if (STREAM) {
    const long long pairs = gridDim.x >> 1, p = blockIdx.x >> 1;
    u0 = (int)(p * a.units / pairs);
    u1 = (int)((p + 1) * a.units / pairs);
  } else {
    const int base = (int)(blockIdx.x >> 1) * a.num_kb, kb0 = (int)blockIdx.y * a.kb_per_split;
    u0 = base + kb0;
    u1 = base + min(a.num_kb, kb0 + a.kb_per_split);
  }
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
    const uint32_t full_even = uniform(map_rank(b_full, even)), ring = smem_u32(smem);
    const int xrow = a.stacked ? half * a.lo_row : half * (n_tok >> 1);
    const bool second = a.terms == 2 && !a.stacked;
    int tw = u0 / a.num_kb, kw = u0 - tw * a.num_kb;             // next weight tile and its K block
    int kx = kw;                                                 // next K block of the activations
    auto load_w = [&](int s) {                                   // (by the elected lane)
      if (half == 0) mbar_expect_tx(b_full + 8 * s, 2u * (uint32_t)stage_bytes);   // both CTAs' copies of the stage
      tma_load_pair(ring + (uint32_t)(s * stage_bytes), &tmW, full_even + 8 * s, kw * CS_GEMM_BK, (2 * tw + half) * CS_GEMM_BM);
    };
    auto load_x = [&](int s) {
      const uint32_t sx = ring + (uint32_t)(s * stage_bytes) + kABytes;
      tma_load_pair(sx, &tmX, full_even + 8 * s, kx * CS_GEMM_BK, xrow);
      if (second) tma_load_pair(sx + (uint32_t)n_tok * 64u, &tmX, full_even + 8 * s, kx * CS_GEMM_BK, a.lo_row + xrow);
    };
    auto next_w = [&]() { if (++kw == a.num_kb) { kw = 0; ++tw; } };
    auto next_x = [&]() { if (++kx == a.num_kb) kx = 0; };
    const int n = u1 - u0, npre = min(n, stages);
    bool ok = true;
    for (int i = 0; i < npre; ++i) {                             // weights depend on nothing
      if (elect_one()) load_w(i);
      next_w();
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int i = 0; i < npre; ++i) {
      if (elect_one()) load_x(i);
      next_x();
    }
    int i = npre, s = 0;
    uint32_t ph = 0;
    for (; i < n; ++i) {
      ok = mbar_wait_warp(b_empty + 8 * s, ph, s_abort, a.wait_ns);
      if (!ok) break;
      if (elect_one()) { load_w(s); load_x(s); }
      next_w();
      next_x();
      if (++s == stages) { s = 0; ph ^= 1u; }
    }
    if (!ok && lane == 0) { *s_abort = 1; atomicOr(a.status, CS_DEV_TIMEOUT); }
    __syncwarp();
    if (*s_abort && lane == 0) {
      // copies in flight land before this CTA's shared memory goes away: the even CTA sees them on its
      // barriers, the odd one gives them a thousand times their latency
      if (half == 0) {
        for (int j = max(0, i - stages); j < i; ++j) mbar_wait(b_full + 8 * (j % stages), (uint32_t)(j / stages) & 1u, s_never, a.wait_ns);
      } else {
        const unsigned long long t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 1000000ull) {}
      }
    }
  } else if (warp == kMmaWarp) {
    // ------------------------------------------------------------- MMA issuer (even CTA only)
    if (half == 0) {
      const uint16_t mask = (uint16_t)(3u << even);
      // bf16 x bf16 -> fp32, both operands K-major, M = 256 over the pair
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(accw >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
      const bool second = a.terms == 2 && !a.stacked;
      const uint64_t desc0 = desc_kmajor(smem_u32(smem));
      const uint64_t x_off = kABytes >> 4, lo_off = (uint64_t)(uint32_t)((kABytes + n_tok * 64) >> 4);
      bool ok = true;
      int j = 0, s = 0, kb = u0 % a.num_kb;
      uint32_t ph = 0;
      for (int u = u0; u < u1 && ok; ++j) {
        const int seg_end = min(u1, u + a.num_kb - kb);
        kb = 0;
        const int buf = STREAM ? (j & 1) : 0;
        const uint32_t acc = tmem_base + (uint32_t)(buf * accw);
        if (j >= 2) ok = mbar_wait_warp(b_acce + 8 * buf, (uint32_t)((j >> 1) - 1) & 1u, s_abort, a.wait_ns);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        uint32_t acc_on = 0;
        for (; u < seg_end && ok; ++u) {
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
        if (elect_one()) umma_commit_pair(b_accf + 8 * buf, mask);
        if (!ok) {
          if (lane == 0) {
            *s_abort = 1;
            atomicOr(a.status, CS_DEV_TIMEOUT);
          }
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
      epi_barrier();
    }
    const uint32_t lane_base = tmem_base + ((uint32_t)(wq * 32) << 16);
    const int feat = wq * 32 + lane;                             // this thread's feature within the CTA's tile
    const int nchunk = (min(n_tok, a.rows) + kChunk - 1) / kChunk;
    bool ok = true;
    if constexpr (STREAM) {
      const uint32_t acce_even = map_rank(b_acce, even);
      int j = 0, turn = 0;
      for (int u = u0; u < u1; ++j) {
        const int tp = u / a.num_kb, kb0 = u - tp * a.num_kb, tile = 2 * tp + half;
        const int seg_end = min(u1, (tp + 1) * a.num_kb);
        const bool whole_end = seg_end == (tp + 1) * a.num_kb;
        u = seg_end;
        const int buf = j & 1;
        ok = mbar_wait(b_accf + 8 * buf, (uint32_t)(j >> 1) & 1u, s_abort, a.wait_ns);
        const int pair = blockIdx.x >> 1;
        const int owner = kb0 > 0 ? pair : pair + 1;             // whose run starts inside this tile, if it is cut
        float* slot = a.part + (size_t)(2 * owner + half) * CS_GEMM_BM * CS_MAX_ROWS;
        int* flag = a.part_flag + 2 * owner + half;
        const bool take = kb0 == 0 && !whole_end;
        if (ok && take && lane == 0) ok = flag_wait(flag, s_abort, a.wait_ns);
        ok = __all_sync(0xffffffffu, ok) && *s_abort == 0;
        if (!ok) {
          *s_abort = 1;
          if (lane == 0) atomicOr(a.status, CS_DEV_TIMEOUT);
        }
        // the decision to go on is one for all eight warps: they meet at barriers below
        uint32_t go;
        asm volatile("{\n.reg .pred p, q;\nsetp.ne.b32 p, %1, 0;\nbar.red.and.pred q, 1, 256, p;\nselp.u32 %0, 1, 0, q;\n}"
                     : "=r"(go) : "r"((uint32_t)ok) : "memory");
        if (!go) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t acc = lane_base + (uint32_t)(buf * accw);
        for (int c = g; c < nchunk; c += 2, ++turn) {
          const int c0 = c * kChunk;
          float v[16];
          if (take) {
            float w[16];
#pragma unroll
            for (int q = 0; q < 16; ++q) w[q] = __ldcg(slot + (size_t)(c0 + q) * CS_GEMM_BM + feat);
            read_chunk(acc + (uint32_t)c0, a, v);
#pragma unroll
            for (int q = 0; q < 16; ++q) v[q] += w[q];
          } else {
            read_chunk(acc + (uint32_t)c0, a, v);
          }
          if (kb0 > 0) {
#pragma unroll
            for (int q = 0; q < 16; ++q) slot[(size_t)(c0 + q) * CS_GEMM_BM + feat] = v[q];
            continue;
          }
          float* pk = park + (size_t)(2 * g + (turn & 1)) * (kChunk * CS_GEMM_BM);
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            const float r = (scaled && c0 + q < a.rows) ? rstd_s[c0 + q] : 1.f;
            pk[q * CS_GEMM_BM + feat] = v[q] * r;
          }
          group_barrier(g);                                      // (two buffers: a thread that runs ahead fills the other one)
          if (a.mode == CS_EPI_SWIGLU) finish_swiglu(a, pk, tile, c0, t);
          else finish_argmax(a, pk, tile, c0, t);
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(acce_even + 8 * buf);
        if (kb0 > 0 || take) {
          epi_barrier();                                         // all of this CTA's sums are written, or read
          if (tid == 0) {
            __threadfence();
            asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(flag), "r"(kb0 > 0 ? 1 : 0) : "memory");
          }
        }
      }
    } else {
      ok = mbar_wait(b_accf, 0, s_abort, a.wait_ns);
      ok = __all_sync(0xffffffffu, ok) && *s_abort == 0;
      if (!ok && lane == 0) atomicOr(a.status, CS_DEV_TIMEOUT);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      // the MMAs have retired, so the ring is free: park the tile there, [token][128 features]
      float* dump = reinterpret_cast<float*>(smem);
      for (int c = g; c < nchunk; c += 2) {
        const int c0 = c * kChunk;
        float v[16];
        if (ok) {
          read_chunk(lane_base + (uint32_t)c0, a, v);
        } else {
#pragma unroll
          for (int q = 0; q < 16; ++q) v[q] = 0.f;
        }
#pragma unroll
        for (int q = 0; q < 16; ++q) {
          const float r = (scaled && c0 + q < a.rows) ? rstd_s[c0 + q] : 1.f;
          dump[(size_t)(c0 + q) * CS_GEMM_BM + feat] = v[q] * r;
        }
      }
    }
  }

  if constexpr (!STREAM) {
    cluster_sync();                                              // every rank's tile is parked
    if (warp < kEpiWarps) {
      const int tile = 2 * (int)(blockIdx.x >> 1) + half, n0 = tile * CS_GEMM_BM, split = (int)blockIdx.y, S = a.splits;
      const uint32_t dump = smem_u32(smem);
      uint32_t peer[CS_PAIR_MAX_SPLITS];
#pragma unroll
      for (int q = 0; q < CS_PAIR_MAX_SPLITS; ++q) peer[q] = map_rank(dump, (uint32_t)(2 * min(q, S - 1) + half));
      auto sum4 = [&](int tok, int f) {                          // four features of one token over the ranks, in rank order
        const uint32_t off = 4u * (uint32_t)(tok * CS_GEMM_BM + f);
        float4 v[CS_PAIR_MAX_SPLITS];
#pragma unroll
        for (int q = 0; q < CS_PAIR_MAX_SPLITS; ++q) v[q] = q < S ? ld_cluster(peer[q] + off) : make_float4(0.f, 0.f, 0.f, 0.f);
        float4 y = v[0];
#pragma unroll
        for (int q = 1; q < CS_PAIR_MAX_SPLITS; ++q) { y.x += v[q].x; y.y += v[q].y; y.z += v[q].z; y.w += v[q].w; }
        return y;
      };
      // this rank's slice of the features, in fours; a thread keeps its four features and walks the tokens
      const int width = a.mode == CS_EPI_QKV ? 64 : CS_GEMM_BM;
      const int per = ((width + S - 1) / S + 3) & ~3, lo = split * per;
      const int per_tok = max(0, min(width, lo + per) - lo) >> 2;
      const int tstep = per_tok > 0 ? kEpiThreads / per_tok : 1;
      const int jq = per_tok > 0 ? tid % per_tok : 0, tok_first = per_tok > 0 ? tid / per_tok : 0;
      const bool busy = per_tok > 0 && tok_first < tstep && n0 < a.N;
      const int f = lo + 4 * jq;
      if (a.mode == CS_EPI_QKV) {
        // RoPE pairs feature i of a head with i + Dh/2: both lie in this tile; f in [0, 64) walks the first halves
        const QkvEpi& Q = a.q;
        const int hd = Q.Dh >> 1, i = f % hd, f1 = (f / hd) * Q.Dh + i, f2 = f1 + hd;
        const int head = (n0 + f1) / Q.Dh;
        const bool live = busy && head < Q.H + 2 * Q.Hkv, is_v = head >= Q.H + Q.Hkv;
        for (int tok = tok_first; live && tok < a.rows; tok += tstep) {
          const float4* csp = reinterpret_cast<const float4*>(Q.rope_cs + 2 * ((size_t)tok * hd + i));
          const float4 cs01 = csp[0], cs23 = csp[1];             // (cos, sin) of dims i .. i + 3
          const int row_w = Q.row_write[tok], row_p = Q.row_pos[tok];
          const float4 av = sum4(tok, f1), bv = sum4(tok, f2);
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
          if (head < Q.H) {                                      // rotated query as two bf16 terms
            __nv_bfloat16* qd = Q.qbuf + ((size_t)tok * Q.H + head) * Q.Dh + i;
            __nv_bfloat16* ql = qd + (size_t)CS_MAX_ROWS * Q.H * Q.Dh;
            *reinterpret_cast<uint2*>(qd) = h0;
            *reinterpret_cast<uint2*>(qd + hd) = h1;
            *reinterpret_cast<uint2*>(ql) = l0;
            *reinterpret_cast<uint2*>(ql + hd) = l1;
          } else if (row_w) {                                    // new K (rotated) / V row of the cache, stored in bf16
            const int kvh = is_v ? head - Q.H - Q.Hkv : head - Q.H;
            __nv_bfloat16* dst = Q.kv + ((((size_t)Q.layer * 2 + (is_v ? 1 : 0)) * Q.max_batch + tok / Q.R) * Q.Hkv + kvh) *
                                            (size_t)Q.max_seq * Q.Dh + (size_t)row_p * Q.Dh + i;
            *reinterpret_cast<uint2*>(dst) = h0;
            *reinterpret_cast<uint2*>(dst + hd) = h1;
          }
        }
      } else {
        const bool feeds = a.nf.gain_out != nullptr, resid = a.mode == CS_EPI_RESIDUAL;
        const bool vec = (a.N & 3) == 0 && n0 + f + 3 < a.N;
        float* part = reinterpret_cast<float*>(smem) + (size_t)n_tok * CS_GEMM_BM;   // [rows][32] sums of squares, behind the parked tile
        float gn[4] = {0.f, 0.f, 0.f, 0.f};
        if (feeds && busy && vec) {
          const uint2 gw = *reinterpret_cast<const uint2*>(a.nf.gain_out + n0 + f);
          const float2 g01 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&gw.x));
          const float2 g23 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&gw.y));
          gn[0] = g01.x; gn[1] = g01.y; gn[2] = g23.x; gn[3] = g23.y;
        }
        if (busy) {
#pragma unroll 2
          for (int tok = tok_first; tok < a.rows; tok += tstep) {
            float* dst = a.out + (size_t)tok * a.N + n0 + f;
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
            if (resid && vec) x = *reinterpret_cast<const float4*>(dst);
            const float4 y = sum4(tok, f);
            if (vec) {
              const float o[4] = {y.x + x.x, y.y + x.y, y.z + x.z, y.w + x.w};
              *reinterpret_cast<float4*>(dst) = make_float4(o[0], o[1], o[2], o[3]);
              if (feeds) {
                const float w[4] = {o[0] * gn[0], o[1] * gn[1], o[2] * gn[2], o[3] * gn[3]};
                uint2 hi, lw;
                split4(w, hi, lw);
                __nv_bfloat16* xo = a.nf.xn_out + (size_t)tok * a.N + n0 + f;
                *reinterpret_cast<uint2*>(xo) = hi;
                *reinterpret_cast<uint2*>(xo + (size_t)CS_MAX_ROWS * a.N) = lw;
                part[tok * 32 + jq] = (o[0] * o[0] + o[1] * o[1]) + (o[2] * o[2] + o[3] * o[3]);
              }
            } else {
              const float yv[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
              for (int e = 0; e < 4; ++e)
                if (n0 + f + e < a.N) dst[e] = resid ? dst[e] + yv[e] : yv[e];
              if (feeds) part[tok * 32 + jq] = 0.f;
            }
          }
        }
        if (feeds) {
          epi_barrier();
          if (n0 < a.N)
            for (int tok = tid; tok < a.rows; tok += kEpiThreads) {
              float ss = 0.f;
              for (int q = 0; q < per_tok; ++q) ss += part[tok * 32 + q];
              a.nf.ssq_out[(size_t)tok * a.nf.slot_stride + tile * S + split] = ss;
            }
        }
      }
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
int pair_fixed_bytes(int n_tok, bool stream) { return 1024 /*alignment slack*/ + kCtlBytes + n_tok * 4 + (stream ? kParkBytes : 0); }
int pair_stage_bytes(int n_tok, int terms) { return kABytes + terms * n_tok * 64; }
int pair_stages(int n_tok, int terms, bool stream) {
  return min(kMaxStages, (227 * 1024 - pair_fixed_bytes(n_tok, stream)) / pair_stage_bytes(n_tok, terms));
}

cs_status ensure_pair_attrs(cs_ctx* ctx) {
  if (!ctx->pair_attr_set) {
    CS_CUDA_OK(ctx, cudaFuncSetAttribute(k_gemm_pair<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
    CS_CUDA_OK(ctx, cudaFuncSetAttribute(k_gemm_pair<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
    ctx->pair_attr_set = true;
  }
  return CS_OK;
}

// How many clusters of 2 x S CTAs, one per SM, the device runs at once: a cluster has to find all its
// CTAs inside one GPC.  Asked of the runtime once per context and size.
int pair_clusters_at_once(const cs_ctx* cctx, int S) {
  cs_ctx* ctx = const_cast<cs_ctx*>(cctx);
  int& slot = ctx->pair_clusters[S];
  if (slot == 0) {
    int n = 0;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(2 * ctx->num_sms, S, 1);
    lc.blockDim = dim3(kThreads, 1, 1);
    lc.dynamicSmemBytes = 200 * 1024;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2; at[0].val.clusterDim.y = S; at[0].val.clusterDim.z = 1;
    lc.attrs = at;
    lc.numAttrs = 1;
    if (ensure_pair_attrs(ctx) == CS_OK && cudaOccupancyMaxActiveClusters(&n, k_gemm_pair<false>, &lc) == cudaSuccess && n > 0) slot = n;
    else { (void)cudaGetLastError(); slot = max(1, ctx->num_sms * 85 / 100 / (2 * S)); }   // no answer: leave room for GPC borders
  }
  return slot;
}

}  // namespace

// Split-K factor of the cluster form: K blocks per CTA times the clocks of one (tensor pipe, issue, or
// this CTA's share of HBM), plus the epilogue, times waves.
static void pair_splits(const cs_ctx* ctx, const GemmPlan* g, int rows, bool two_terms, int* splits, int* kb_per_split) {
  const int n_tok = cs_ceil_div(rows, 16) * 16, terms = two_terms ? 2 : 1;
  const int pairs = cs_ceil_div(g->N, 2 * CS_GEMM_BM), kb = cs_ceil_div(g->K, CS_GEMM_BK);
  long best = -1;
  for (int sp = 1; sp <= CS_PAIR_MAX_SPLITS && sp <= max(1, kb / 4); ++sp) {
    const int kps = cs_ceil_div(kb, sp), spl = cs_ceil_div(kb, kps);
    const int fit = pair_clusters_at_once(ctx, spl);
    const long waves = cs_ceil_div(pairs, fit);
    const long active = 2L * spl * min(pairs, fit);
    const long per_kb = max(max(2L * terms * n_tok, 350L), kABytes * active / 3500);
    const long cost = waves * (kps * per_kb + 4000 + 30L * n_tok);
    if (best < 0 || cost < best) { best = cost; *splits = spl; *kb_per_split = kps; }
  }
}

int cs_gemm_splits(const cs_ctx* ctx, const GemmPlan* g, int mode, int rows, bool two_terms) {
  if (!cs_gemm_on_pairs(mode, rows)) return g->splits;
  int splits = 1, kps = 0;
  if (mode != CS_EPI_SWIGLU && mode != CS_EPI_ARGMAX) pair_splits(ctx, g, rows, two_terms, &splits, &kps);
  return splits;
}

cs_status cs_launch_gemm_pair(cs_ctx* ctx, const GemmPlan* g, const CUtensorMap* tmX, int lo_row, int rows, int mode, float* out,
                              __nv_bfloat16* act, __nv_bfloat16* act_lo, int F, const QkvEpi* q, const NormFuse* nf,
                              cudaStream_t st) {
  const bool stream = mode == CS_EPI_SWIGLU || mode == CS_EPI_ARGMAX;
  if (ctx->debug_drop_kb >= 0) {
    ctx->debug_drop_kb = -1;
    snprintf(ctx->err, sizeof(ctx->err), "the dropped-tile test hook is for blocks of at most 32 rows");
    return CS_ERR_UNSUPPORTED;
  }
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
  a.out = out; a.act = act; a.act_lo = act_lo; a.F = F;
  if (q != nullptr) a.q = *q;
  if (nf != nullptr) a.nf = *nf;
  a.tile_max = ctx->tile_max; a.tile_idx = ctx->tile_idx; a.tile_stride = cs_ceil_div(g->N, CS_GEMM_BM);
  a.part = ctx->pair_part; a.part_flag = ctx->pair_flag;
  a.status = ctx->d_status;
  a.wait_ns = ctx->wait_limit_ns;
  a.stamp = cs_next_stamp(ctx, mode == CS_EPI_ARGMAX ? CS_FAM_LMHEAD : CS_FAM_GEMM);
  a.stages = pair_stages(a.n_tok, a.terms, stream);
  const size_t smem = (size_t)pair_fixed_bytes(a.n_tok, stream) + (size_t)a.stages * pair_stage_bytes(a.n_tok, a.terms);
  const int tiles2 = cs_ceil_div(g->N, 2 * CS_GEMM_BM);
  cs_status s = ensure_pair_attrs(ctx);
  if (s != CS_OK) return s;
  cudaLaunchConfig_t lc = {};
  a.splits = 1;
  if (stream) {
    const int pairs = min(min(CS_MAX_PAIRS, pair_clusters_at_once(ctx, 1)), tiles2);   // a run is never shorter than one tile
    a.units = tiles2 * a.num_kb;
    lc.gridDim = dim3(2 * pairs, 1, 1);
  } else {
    pair_splits(ctx, g, rows, lo_row >= 0, &a.splits, &a.kb_per_split);
    lc.gridDim = dim3(2 * tiles2, a.splits, 1);
  }
  lc.blockDim = dim3(kThreads, 1, 1);
  lc.dynamicSmemBytes = smem;
  lc.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = 2; at[1].val.clusterDim.y = a.splits; at[1].val.clusterDim.z = 1;
  lc.attrs = at;
  lc.numAttrs = 2;
  const PairKernel kernel = stream ? k_gemm_pair<true> : k_gemm_pair<false>;
  CS_CUDA_OK(ctx, cudaLaunchKernelEx(&lc, kernel, g->tmW, *tmX, a));
  return CS_OK;
}
