// The whole generation loop of a small model in one launch (Sec. 3.1, 3.2; App. B.2, B.3): one thread-block
// cluster per sequence runs search, block assembly, forward, acceptance and append, step after step, until
// its sequence is finished.
//
// What bounds it: chains of latencies.  A step of the two-layer model (2 MB of weights a layer, 11 rows) has 1 us of bytes
// and of arithmetic; as 18 launches it takes 80 us, 2 - 5 us for each boundary with its release, its first loads and its
// restart.  Sequences do not depend on one another, weights of this size stay in L2, and the SMs of a cluster pass
// activations through distributed shared memory, so here a boundary is a wait on a shared-memory barrier.
//
// Layout: weights are the A operand of mma.sync, 16 rows of a matrix to a warp with all of its K (the first blocks of a phase are asked for
// ahead of the wait in front of it).  The K order within a block of 32 is permuted alike on both
// sides, so that a thread's fragments of four MMAs are 16 contiguous bytes.  (tcgen05 has no place here: a CTA's share of
// a projection is one to eight tiles of 16 rows, done in a few hundred clocks; M = 128 would leave fifteen of sixteen SMs idle.)
// QKV and gate/up are dealt out by rows: their operand, the normed residual stream, is in every CTA.  Attention output
// and down are dealt out by columns - a CTA multiplies what it made itself, its KV head's attention or its SwiGLU features - and
// their sums meet in the CTA that holds the feature of the residual stream: 11 KB a CTA sent and not 45, and shared memory of
// another SM takes 17 bytes a clock.
// What a CTA needs of another is written into its shared memory, in the layout in which it is read, by stores that count their
// bytes on the reader's mbarrier: no barrier of the cluster and no fence lies between two phases.  A new write into a buffer is
// sent only by a CTA that has heard, directly or through others, from everyone who read the old one.
// Blocks of 16 keys belong to the CTAs of a KV head in turn, and to their warps, by position: a CTA reads from the cache only rows that it
// wrote itself or that were there before the launch.  The block's own K/V rows reach it like the queries.  Every CTA holds
// the history in shared memory and searches all of it, and every CTA works out acceptance and append alike.
//
// What a phase costs is instructions in a row more than anything else: a warp alone on its scheduler issues one in about ten clocks.  The two-layer
// model, one sequence, 11 rows, us a call of 11 steps: launch by launch 876; with divisions in the index arithmetic, stores to sixteen CTAs one by one and
// cluster barriers 980 (11,400 instructions a warp and step); with hand-overs counted on mbarriers and K split over the warps 555; with the SwiGLU output
// multiplied where it was made, one turn of code for all projections and weights out of the registers 500; with weights by TMA and the
// statistics kept by a warp that nobody waits for 475; with what a warp does for a tile worked out once and fragment loads that meet every bank once
// 433; now 426, with softmax weights by exp2f (3 more) and nothing stored that nobody reads (4 less).  What is left of 38 us a step: 17 turns or hand-overs of
// 1.5 - 2 us.
//
// Arithmetic as in the other kernels: activations, queries and softmax weights enter products as two bf16 terms, sums, norms,
// rotation and softmax are fp32; every RMSNorm is folded into the projection behind it (1/rms scales the sums).
//
// Heads of 64 want more than the 128 registers that 512 threads leave each: 450 - 490 bytes of spill stores a thread, where heads of 32 have none.  They gain
// less than heads of 32 in the table at the launch.
//
// Waits are bounded as in the other kernels: after the limit a CTA raises the status bit, waits for nothing and sends nothing any
// more, gives its copies time to land and meets the others at the cluster barrier in front of the exit, which all of them reach.
#include <limits.h>

#include <algorithm>
#include <new>

#include "cs_common.cuh"
#include "cs_tcgen.cuh"

using std::max;
using std::min;

namespace {

constexpr int kThreads = 512, kWarps = kThreads / 32;
constexpr int kRing = 4;              // K blocks of 64 whose weights a warp has in flight
constexpr int kMaxLayers = 8;
constexpr int kMaxCluster = 16;
constexpr int kMaxRows = 16;          // of a block (shared memory holds no more beside the weights of a model of 256 features)
enum : int { kXQkv = 0, kXAttn = 1, kXOut = 2, kXNorm = 3, kXDown = 4, kXNext = 5, kXMax = 6, kExchanges = 8 };   // hand-overs, in their order
enum : int { kQkv = 0, kOut = 1, kGateUp = 2, kDown = 3, kLm = 4 };   // projections

// Activations as the MMAs' B operand lie in tiles of 16 features: the tile's sums of squares [Rp], then rows of a token's leading and second
// terms [Rp][2][16].  A term of a token is a column of its own, so four tokens make an MMA and the two terms' sums lie side by side in a
// thread.  The distance of two tiles is 64 mod 128 bytes, so that a fragment load meets every bank once.
__host__ __device__ constexpr int tile_bytes(int Rp) { return (68 * Rp + 63) / 128 * 128 + 64; }

// one operand map per turn: the four matrices of every layer, then the LM head; boxes of 64 K elements and a tile's 16 rows
struct SmallMaps {
  CUtensorMap w[4 * kMaxLayers + 1];
};
// What a warp does for a tile of a projection, worked out once for its first tile of each: the divisions and choices in it were 1,200 clocks a turn.
struct __align__(16) Job {
  int col, row, block, chunks;        // weights: coordinates of the first copy, how many (0 = the warp has no such job)
  int jobs, tile, quarter, rows;      // jobs of the CTA; this one's tile, the first of its tokens' quarters and its tokens
  int at, first, last, pieces;        // results: where they go in the CTAs first .. last - 1, and how many 16-byte pieces
  int op, kb, one, whole;             // operand, blocks of 32 K elements, whether the job has one quarter of the tokens only, whether both terms travel
};
// where things lie in shared memory (bytes); the same in every CTA
struct SmallSmem {
  int xn, at, act, sums, stage, norm, red, q, kv, xres, gain, gain0, rope, turn, jobs, ring, hist, misc, total;
};
struct SmallArgs {
  const __nv_bfloat16* norm[2 * kMaxLayers + 1];   // gains, in their order
  const __nv_bfloat16* embed;
  const double* inv_freq;
  int n_layers, d, H, Hkv, G, F, vocab, max_seq, max_batch;
  float inv_d, eps, scale_log2e;
  int *hist, *hist_len, *kv_len;
  const int* script;
  __nv_bfloat16* kv;
  int B, stride, gamma, k, policy, max_new, eos_id;
  int log_slices, log_rows, own_d, slice_bytes;   // CTAs per KV head and tiles of 16 query rows per KV head (powers of two), tiles of the residual stream per CTA at most, an attention result
  int *emitted, *done;
  unsigned long long* stats;
  int* status;
  unsigned long long *progress, *report;   // pinned: the word that the host waits for; status bits, then the image of cs_stats
  unsigned long long wait_ns;
  int drop;                           // test hook: kind of hand-over that the first CTA leaves out (-1 = none)
  SmallSmem at;
};

// (what branches and copies go by: see uniform())
__device__ __forceinline__ int uni(int v) { return (int)uniform((uint32_t)v); }
__device__ __forceinline__ uint32_t peer(uint32_t addr, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// 16 bytes into a CTA's shared memory, counted on its barrier
__device__ __forceinline__ void send16(uint32_t addr, uint4 v, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
               ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar) : "memory");
}
__device__ __forceinline__ void expect(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
               : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __noinline__ void wait_long(uint32_t bar, uint32_t parity, volatile int* abort_flag, unsigned long long limit_ns, int* status) {
  unsigned long long t0 = 0;
  for (uint32_t it = 0; !try_wait(bar, parity); ++it)
    if ((it & 63u) == 63u) {
      if (*abort_flag) return;
      const unsigned long long now = globaltimer_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > limit_ns) {
        *abort_flag = 1;
        atomicOr(status, CS_DEV_TIMEOUT);
        return;
      }
    }
}
__device__ __forceinline__ void cluster_meet() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}
// two values as a leading bf16 pair and the pair of what that rounding lost
__device__ __forceinline__ void split2(float a, float b, uint32_t& hi, uint32_t& lo) {
  hi = pack(a, b);
  const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&hi));
  lo = pack(a - f.x, b - f.y);
}
__device__ __forceinline__ void split1(float a, __nv_bfloat16* hi, __nv_bfloat16* lo) {
  const __nv_bfloat16 h = __float2bfloat16_rn(a);
  *hi = h;
  *lo = __float2bfloat16_rn(a - __bfloat162float(h));
}

// Weights travel by TMA, a warp's tile to a ring of the warp's own; its next tile, of whatever projection, is asked for once what others wait for is on
// its way.  (In registers the compiler put them aside, which waits for them; as cp.async of fragments, 8 rows of 64 bytes an instruction, they
// kept the load unit busy for 15 of 75 thousand clocks a step.)  K blocks i .. of a tile, as many as the ring holds:
__device__ __forceinline__ void ask(uint32_t ring, uint32_t bar, const CUtensorMap* tm, int i, int n, int col, int row, int block) {
  const int count = min(kRing, n - i);
  if (elect_one()) {
    mbar_expect_tx(bar, (uint32_t)count * 2048u);
#pragma unroll 1
    for (int u = 0; u < count; ++u)
      asm volatile(
          "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
          ::"r"(ring + 2048u * u), "l"(tm), "r"(bar), "r"(col + 64 * (i + u)), "r"(row), "r"(0), "r"(block) : "memory");
  }
  __syncwarp();
}
// 32 K elements: a tile's rows times all tokens, two chains of MMAs per sum (warps issue in order)
template <int NT>
__device__ __forceinline__ void multiply_block(float (&acc)[2][NT][4], const uint8_t* at, const uint8_t* op, bool one) {
  const uint4 a0 = *reinterpret_cast<const uint4*>(at), a1 = *reinterpret_cast<const uint4*>(at + 1024);
  const uint4 b = *reinterpret_cast<const uint4*>(op);
  mma_bf16(acc[0][0], a0.x, a1.x, a0.y, a1.y, b.x, b.y);
  mma_bf16(acc[1][0], a0.z, a1.z, a0.w, a1.w, b.z, b.w);
  if (!one) {
    uint4 c[NT];
#pragma unroll
    for (int q = 1; q < NT; ++q) c[q] = *reinterpret_cast<const uint4*>(op + q * 256);
#pragma unroll
    for (int q = 1; q < NT; ++q) {
      mma_bf16(acc[0][q], a0.x, a1.x, a0.y, a1.y, c[q].x, c[q].y);
      mma_bf16(acc[1][q], a0.z, a1.z, a0.w, a1.w, c[q].z, c[q].w);
    }
  }
}
// Keys first .. first + 15 and their values as B fragments: from the cache, of which rows up to kv - 1 are there, or the block's own R rows.  (What lies
// behind the rows must not reach the sums: 0 x NaN is NaN.)
template <int DH>
__device__ __forceinline__ void load_cached(uint4 (&kf)[2][DH / 32], uint32_t (&vf)[4][DH / 16], const __nv_bfloat16* Kg, const __nv_bfloat16* Vg,
                                            int first, int kv, int g, int t) {
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const __nv_bfloat16* p = Kg + (uint32_t)(min(first + 8 * q + g, kv - 1) * DH + 8 * t);
#pragma unroll
    for (int i = 0; i < DH / 32; ++i) kf[q][i] = __ldcg(reinterpret_cast<const uint4*>(p + 32 * i));
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int key = first + 2 * t + (q & 1) + 8 * (q >> 1);
    const __nv_bfloat16* p = Vg + (uint32_t)(min(key, kv - 1) * DH + DH / 8 * g);
    if (DH == 32) {
      const uint2 x = __ldcg(reinterpret_cast<const uint2*>(p));
      vf[q][0] = key < kv ? x.x : 0u; vf[q][1] = key < kv ? x.y : 0u;
    } else {
      const uint4 x = __ldcg(reinterpret_cast<const uint4*>(p));
      vf[q][0] = key < kv ? x.x : 0u; vf[q][1] = key < kv ? x.y : 0u;
      vf[q][DH / 16 - 2] = key < kv ? x.z : 0u; vf[q][DH / 16 - 1] = key < kv ? x.w : 0u;
    }
  }
}
template <int DH>
__device__ __forceinline__ void load_own(uint4 (&kf)[2][DH / 32], uint32_t (&vf)[4][DH / 16], const uint8_t* kn, int Rp, int first, int R, int g, int t) {
  constexpr int kParts = DH / 16;
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int i = 0; i < DH / 32; ++i) {
      const int ch = 4 * i + t;
      kf[q][i] = *reinterpret_cast<const uint4*>(kn + (ch % kParts * Rp + min(first + 8 * q + g, R - 1)) * 32 + ch / kParts * 16);
    }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int key = first + 2 * t + (q & 1) + 8 * (q >> 1), dim = DH / 8 * g;
    const uint8_t* p = kn + ((kParts + dim / 8 % kParts) * Rp + min(key, R - 1)) * 32 + dim / 8 / kParts * 16 + 2 * (dim % 8);
    if (DH == 32) {
      const uint2 x = *reinterpret_cast<const uint2*>(p);
      vf[q][0] = key < R ? x.x : 0u; vf[q][1] = key < R ? x.y : 0u;
    } else {
      const uint4 x = *reinterpret_cast<const uint4*>(p);
      vf[q][0] = key < R ? x.x : 0u; vf[q][1] = key < R ? x.y : 0u;
      vf[q][DH / 16 - 2] = key < R ? x.z : 0u; vf[q][DH / 16 - 1] = key < R ? x.w : 0u;
    }
  }
}

// NT: quarters of the tokens, four each
template <int NT, int DH>
__global__ void __launch_bounds__(kThreads, 1)
k_small_loop(const __grid_constant__ SmallMaps maps, const __grid_constant__ SmallArgs a) {
  constexpr int Rp = 4 * NT, TB = tile_bytes(Rp), kRows = 4 * Rp, kHalf = DH / 2, kParts = DH / 16, kDims = DH / 8;   // padded rows; where a tile's rows begin; tiles of a head; a V fragment's dims per thread
  extern __shared__ __align__(1024) uint8_t smem[];
  uint8_t* s_xn = smem + a.at.xn;                                               // gain * x, in tiles
  uint8_t* s_at = smem + a.at.at;                                               // this CTA's KV head's attention output, in tiles
  uint8_t* s_act = smem + a.at.act;                                             // this CTA's SwiGLU output, in tiles; shares its place with the
  uint8_t* s_po = s_act;                                                        // attention of the KV head's slices, each [rows][DH] and (max, sum) [rows]
  float* s_sums = reinterpret_cast<float*>(smem + a.at.sums);                   // sums of the residual stream by CTA that sent them, [sender][own tile][R][16]
  uint8_t* s_stage = smem + a.at.stage;                                         // results on their way to the others
  uint8_t* s_norm = smem + a.at.norm;                                           // the residual stream's next operand on its way to the others
  // attention of the warps, [16][DH] each, in the part of their rings that the attention output's weights leave free; rows begin 4 r columns on
  float* s_red = reinterpret_cast<float*>(smem + a.at.ring + kRing * 1024);
  constexpr int kRed = kRing * 512;                                             // from one warp's to the next
  static_assert(16 * DH <= kRing * 256, "half a ring");
  auto red_at = [](int r, int col) { return r * DH + ((col + 4 * r) & (DH - 1)); };
  float2* s_redml = reinterpret_cast<float2*>(smem + a.at.red);                 // and their (max, sum), [warp][16]
  uint8_t* s_q = smem + a.at.q;                                                 // this CTA's queries, in tiles (dims 8p .. and the partners half a head on)
  uint8_t* s_kn = smem + a.at.kv;                                               // the block's K rows of its KV head, [part][token][16], and V rows behind
  float* s_x = reinterpret_cast<float*>(smem + a.at.xres);                      // residual stream of this CTA's features, [own tile][Rp][16]
  float* s_gain = reinterpret_cast<float*>(smem + a.at.gain);                   // gains of the norms behind O and down, [2 * layers][own_d][16]
  __nv_bfloat16* s_gain0 = reinterpret_cast<__nv_bfloat16*>(smem + a.at.gain0); // gain of the first norm
  float2* s_rope = reinterpret_cast<float2*>(smem + a.at.rope);                 // rotation of the block's rows, [Rp][DH / 2]
  double2* s_turn = reinterpret_cast<double2*>(smem + a.at.turn);               // (cos, sin) of 0 .. R positions, [R + 1][DH / 2], then of the block's first row
  Job* s_job = reinterpret_cast<Job*>(smem + a.at.jobs) + (threadIdx.x >> 5) * 6;   // this warp's first job of every projection, and its present one behind
  int* s_hist = reinterpret_cast<int*>(smem + a.at.hist);                       // the history, [stride]
  uint2* s_max = reinterpret_cast<uint2*>(smem + a.at.misc);                    // largest logits and their ids by CTA, [kMaxCluster][Rp]
  uint2* s_wmax = reinterpret_cast<uint2*>(s_stage) + Rp;                       // by warp, [kWarps][Rp], behind this CTA's on their way to the others, [Rp]
  uint64_t* s_bar = reinterpret_cast<uint64_t*>(s_max + kMaxCluster * Rp);      // [kExchanges]
  uint64_t* s_wbar = s_bar + kExchanges;                                        // a warp's weights, [kWarps]
  int* s_script = reinterpret_cast<int*>(s_wbar + kWarps);                      // [Rp]
  int* s_tgt = s_script + Rp;                                                   // [Rp]
  float* s_rstd = reinterpret_cast<float*>(s_tgt + Rp);                         // [Rp]
  int* s_best = s_tgt + 2 * Rp;
  int* s_tau = s_best + 1;
  volatile int* s_abort = s_best + 2;

  uint32_t rank_u, nc_u;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank_u));
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(nc_u));
  const int c = (int)rank_u, NC = (int)nc_u, log_nc = NC == 16 ? 4 : 3, b = blockIdx.x >> log_nc;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int d = a.d, F = a.F, H = a.H, Hkv = a.Hkv, G = a.G, R = a.k + 1, S = 1 << a.log_slices, nq = G * R;
  const int dt = d / 16, qt = (H + 2 * Hkv) * kParts;          // tiles of the residual stream, of QKV
  const int d0 = c * dt >> log_nc, dn = ((c + 1) * dt >> log_nc) - d0;     // this CTA's: of the residual stream,
  const int q0 = c * qt >> log_nc, qn = ((c + 1) * qt >> log_nc) - q0;     // of QKV,
  const int f0 = c * (F / 32) >> log_nc, fn = ((c + 1) * (F / 32) >> log_nc) - f0;   // of SwiGLU (blocks of 32 features, four tiles of gate/up rows each),
  const int lt = (a.vocab + 15) / 16, l0 = c * lt >> log_nc, l1 = (c + 1) * lt >> log_nc;   // of the LM head
  const int kvh = c >> a.log_slices, slice = c & (S - 1);         // this CTA's share of the attention
  const bool attends = kvh < Hkv;
  const int o0 = slice * dt >> a.log_slices, on = attends ? ((slice + 1) * dt >> a.log_slices) - o0 : 0;   // and the rows of the attention output that it multiplies its KV head's result with
  const int MQ = 1 << a.log_rows, KG = kWarps >> a.log_rows, mq = warp & (MQ - 1), kg = warp >> a.log_rows;
  const int r_lo = min(16 * mq + g, nq - 1), r_hi = min(16 * mq + g + 8, nq - 1);   // query rows: head of the group * R + row of the block
  const int tok_lo = r_lo % R, tok_hi = r_hi % R, q_lo = kRows + r_lo / R * kParts * TB + tok_lo * 64, q_hi = kRows + r_hi / R * kParts * TB + tok_hi * 64;
  const int op_at = kRows + (t >> 1) * TB + g * 32 + (t & 1) * 16;   // this thread's piece of an operand
  // K of this CTA's KV head in the first layer, V behind it, the next layer
  const size_t k_half = (size_t)(a.max_batch * Hkv) * (uint32_t)(a.max_seq * DH), k_layer = 2 * k_half;
  __nv_bfloat16* K0 = a.kv + (size_t)(b * Hkv + (attends ? kvh : 0)) * (uint32_t)(a.max_seq * DH);
  constexpr int kClerk = kThreads - 32;                        // the thread that keeps the books in global memory
  const uint32_t base = smem_u32(smem), bars = smem_u32(s_bar) - base;
  const uint32_t to = peer(base, warp & (NC - 1));             // the CTA that this warp sends to
  const uint32_t ring = base + (uint32_t)(a.at.ring + warp * (kRing * 2048)), ring_bar = smem_u32(s_wbar + warp);
  // This thread's rows of its warp's tiles are row and row + 8, not g and g + 8: rows 4 apart lie in the two halves of the copies' swizzle, and a fragment load
  // of neighbouring lanes meets every bank once (with g, twice: the loads were what a projection took longest for).
  const int row = g >> 1 | (g & 1) << 2;
  const uint8_t* ring_at = smem + (ring - base) + row * 128;
  uint32_t ring_parity = 0;
  uint8_t* mine = s_stage + warp * (64 * Rp);                  // this warp's part of the stage

  if ((base & 1023u) != 0) {                                   // (alike in every CTA)
    if (tid == 0) atomicOr(a.status, CS_DEV_SMEM);
    return;
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  int n = __ldcg(a.hist_len + b), kv = __ldcg(a.kv_len + b), e = __ldcg(a.emitted + b);
  bool fin = __ldcg(a.done + b) != 0;
  int* h = a.hist + (size_t)b * a.stride;
  const bool latest = a.policy == CS_MATCH_LATEST;
  const int none = latest ? -1 : INT_MAX;
#pragma unroll 1
  for (int i = tid; i < min(n, a.stride) && !fin; i += kThreads) s_hist[i] = __ldcg(h + i);
#pragma unroll 1
  for (int i = tid; i < 2 * a.n_layers * 16 * a.own_d; i += kThreads) {
    const int norm = i / (16 * a.own_d), f = 16 * d0 + i % (16 * a.own_d);
    const __nv_bfloat16* gp = a.norm[norm + 1];
    s_gain[i] = f < 16 * (d0 + dn) ? __bfloat162float(gp[f]) : 0.f;
  }
#pragma unroll 1
  for (int i = tid; i < d; i += kThreads) s_gain0[i] = a.norm[0][i];
  // Rotation factors in double, as everywhere: those of a block's first row times those of the distance.  (sincos in the loop over the steps costs 2,000
  // clocks a step and room in the instruction cache; a product is right to 2e-16, and the steps' errors add up to 1e-13 over a thousand of them.)
#pragma unroll 1
  for (int i = tid; i < (R + 2) * kHalf; i += kThreads) {
    const int r = i / kHalf;
    double sn, co;
    sincos((double)(r <= R ? r : kv) * a.inv_freq[i % kHalf], &sn, &co);
    s_turn[i] = make_double2(co, sn);
  }
  double2* s_first = s_turn + (R + 1) * kHalf;
  // Few tiles: a warp for every quarter of the tokens.  Rows of a tile, of QKV: dims 8p .. and, half a head on, their partners in the rotation; of gate/up:
  // gate rows and, 64 on, their up rows; else 16 neighbours.  Results of QKV go to every CTA of their KV head (of keys and values the leading terms: what the
  // cache holds), of the attention output and down to the CTA that holds the tile.
  auto describe = [&](Job* j, int kind, int job) {
    const int tiles = kind == kQkv ? qn : kind == kOut ? on : kind == kGateUp ? 4 * fn : kind == kDown ? dt : l1 - l0;
    const bool one = NT > 1 && kind != kLm && tiles * NT <= kWarps;
    const int jobs = one ? tiles * NT : tiles, local = one ? job / NT : job, quarter = one ? job % NT : 0;
    const int tile = local + (kind == kQkv ? q0 : kind == kOut ? o0 : kind == kGateUp ? 4 * f0 : kind == kLm ? l0 : 0);
    const int kb = kind == kOut ? G * kParts / 2 : kind == kDown ? fn : d / 32;
    j->col = kind == kOut ? kvh * G * DH : kind == kDown ? 32 * f0 : 0;
    j->row = kind == kQkv ? tile % kParts * 8 : kind == kGateUp ? tile % 8 * 8 : 16 * tile;
    j->block = kind == kQkv ? tile / kParts : kind == kGateUp ? tile / 8 : 0;
    j->chunks = job < jobs ? (kb + 1) / 2 : 0;
    j->jobs = jobs;
    j->tile = kind == kGateUp ? local : tile;
    j->quarter = quarter;
    j->rows = min(R - 4 * quarter, one ? 4 : Rp);
    j->op = kind == kOut ? a.at.at : kind == kDown ? a.at.act : a.at.xn;
    j->kb = kb;
    j->one = one;
    const int head = tile / kParts, part = tile % kParts;
    const bool is_q = head < H;
    j->whole = kind != kQkv || is_q;
    j->pieces = (j->whole ? 4 : 2) * j->rows;
    if (kind == kQkv) {
      const int kh = is_q ? head / G : (head - H) % Hkv;
      j->first = kh * S;
      j->last = j->first + S;
      j->at = is_q ? a.at.q + kRows + ((head - kh * G) * kParts + part) * TB + quarter * 256 : a.at.kv + ((head - H) / Hkv * kParts + part) * 32 * Rp + quarter * 128;
    } else if (kind == kOut || kind == kDown) {
      const int p = ((tile + 1) * NC - 1) / dt, held = ((p + 1) * dt >> log_nc) - (p * dt >> log_nc);
      j->first = p;
      j->last = p + 1;
      j->at = a.at.sums + ((kind == kOut ? kvh : c) * held + tile - (p * dt >> log_nc)) * 64 * R + quarter * 256;
    }
  };
  if (lane <= kLm) describe(s_job + lane, lane, warp);
  // what a hand-over brings, in bytes
  auto arm = [&](int x) {
    expect(base + bars + 8 * x, (uint32_t)(x == kXQkv ? (G + 1) * kParts * 64 * R : x == kXAttn ? S * a.slice_bytes : x == kXOut ? Hkv * dn * 64 * R
                                           : x == kXDown ? NC * dn * 64 * R : x == kXMax ? NC * Rp * 8 : dt * (kRows + 64 * R)));
  };
  if (tid == 0) {
    for (int x = 0; x < kExchanges; ++x) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(base + bars + 8 * x));
    for (int x = 0; x < kWarps; ++x) mbar_init(smem_u32(s_wbar + x), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    for (int x = 0; x <= kXMax; ++x)
      if (x > kXAttn || attends) arm(x);
    *s_abort = 0;
    *s_best = none;
  }
  __syncthreads();

  uint32_t step_parity = 0;
  int layers_done = 0;                                         // (a hand-over of a layer is its barrier's phase number layers_done + l)
  auto wait = [&](int x, uint32_t parity) {
    if (!try_wait(base + bars + 8 * x, parity)) wait_long(base + bars + 8 * x, parity, s_abort, a.wait_ns, a.status);
    if (tid == 0 && *s_abort == 0) arm(x);                     // for the next time
    __syncwarp();
  };
  const int dropped = c == 0 ? a.drop : -1;
  auto silent = [&](int x) { return *s_abort != 0 || dropped == x; };
  // 1/rms of every token from one sum of squares per tile of the residual stream, by one warp
  auto rms = [&]() {
    constexpr int kLanes = Rp <= 8 ? 8 : Rp <= 16 ? 16 : 32;
    const float* p = reinterpret_cast<const float*>(s_xn + lane / kLanes * TB) + min(lane % kLanes, Rp - 1);
    float ss = 0.f;
#pragma unroll 4
    for (int i = lane / kLanes; i < dt; i += 32 / kLanes, p += 32 / kLanes * TB / 4) ss += *p;
#pragma unroll
    for (int off = kLanes; off < 32; off <<= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
    if (lane < Rp) s_rstd[lane] = rsqrtf(ss * a.inv_d + a.eps);
  };

  // asks for a job's weights (by a whole warp), from copy `first` on
  auto ask_for = [&](int turn, const Job* j, int first) {
    const int4 w = *reinterpret_cast<const int4*>(j);
    const int chunks = uni(w.w);
    if (chunks > 0) ask(ring, ring_bar, &maps.w[turn], first, chunks, uni(w.x), uni(w.y), uni(w.z));
    return chunks > 0;
  };
  auto ask_turn = [&](int turn) { return ask_for(turn, s_job + (turn == 4 * a.n_layers ? kLm : turn & 3), 0); };

  cluster_meet();                                              // every CTA of the cluster has its barriers set up
  bool asked = !fin && ask_turn(0);                      // the first weights of a step are asked for at the end of the one before
  while (!fin) {
    // ---------------------------------------------------------------- search (Sec. 3.1; App. B.3 step 1); half of the warps: rotation factors
    const int nn = max(0, min(n, a.stride)), n_cand = nn - 2 * a.gamma + 1;
    if (warp >= kWarps / 2) {
#pragma unroll 1
      for (int i = tid - kThreads / 2; i < R * kHalf; i += kThreads / 2) {
        const double2 x = s_first[i % kHalf], y = s_turn[i];
        s_rope[i] = make_float2((float)(x.x * y.x - x.y * y.y), (float)(x.y * y.x + x.x * y.y));
      }
    } else {
      int best = none;
      if (tid < n_cand) {
        const int k0 = s_hist[nn - a.gamma], k1 = s_hist[nn - 1];
#pragma unroll 1
        for (int p = tid; p < n_cand; p += kThreads / 2) {
          bool eq = s_hist[p] == k0 && s_hist[p + a.gamma - 1] == k1;
#pragma unroll 1
          for (int j = 1; eq && j < a.gamma - 1; ++j) eq = s_hist[p + j] == s_hist[nn - a.gamma + j];
          if (eq) best = latest ? max(best, p) : min(best, p);
        }
      }
      best = latest ? __reduce_max_sync(0xffffffffu, best) : __reduce_min_sync(0xffffffffu, best);
      if (lane == 0 && best != none) {
        if (latest) atomicMax(s_best, best); else atomicMin(s_best, best);
      }
      // this step's scripted targets, long before they are wanted
      if (tid < R) s_script[tid] = (a.script != nullptr && e + tid < a.max_new) ? __ldcg(a.script + (size_t)b * a.max_new + e + tid) : -1;
    }
    __syncthreads();
    const int p0 = *s_best == INT_MAX ? -1 : *s_best;
    const int from = p0 + a.gamma, dl = p0 < 0 ? 0 : min(a.k, nn - from);
    const bool fits = kv >= 0 && kv + dl + 1 <= a.max_seq;
    if (!fits) {                                               // no room for the block: the sequence stops here (none is let in that could come to this)
      if (c == 0 && tid == 0) atomicOr(a.status, CS_DEV_CAPACITY);
      break;
    }
    // ---------------------------------------------------------------- embedding and first norm, all rows in every CTA.  Row r: the last accepted
    // token, then the draft (rows past it are dead: nothing of theirs is accepted or cached)
#pragma unroll 1
    for (int r = warp; r < R; r += kWarps) {
      int tok = r == 0 || r > dl ? s_hist[nn - 1] : s_hist[from + r - 1];
      tok = tok < 0 ? 0 : (tok >= a.vocab ? a.vocab - 1 : tok);
      const __nv_bfloat16* er = a.embed + (size_t)tok * d;
      float ss = 0.f;
#pragma unroll 1
      for (int f = 8 * lane; f < d; f += 256) {
        const uint2 u0 = *reinterpret_cast<const uint2*>(er + f), u1 = *reinterpret_cast<const uint2*>(er + f + 4);
        const uint4 gn = *reinterpret_cast<const uint4*>(s_gain0 + f);
        const uint32_t u[4] = {u0.x, u0.y, u1.x, u1.y}, gg[4] = {gn.x, gn.y, gn.z, gn.w};
        uint32_t hi[4], lo[4];
        float x[8];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float2 v = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u[q]));
          const float2 gv = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&gg[q]));
          x[2 * q] = v.x; x[2 * q + 1] = v.y;
          ss += v.x * v.x + v.y * v.y;
          split2(v.x * gv.x, v.y * gv.y, hi[q], lo[q]);
        }
        uint8_t* dst = s_xn + (f >> 4) * TB + kRows + r * 64 + 2 * (f & 15);
        *reinterpret_cast<uint4*>(dst) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
        *reinterpret_cast<uint4*>(dst + 32) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        const int own = (f >> 4) - d0;
        if (own >= 0 && own < dn) {
          float* xd = s_x + (own * Rp + r) * 16 + (f & 15);
          *reinterpret_cast<float4*>(xd) = make_float4(x[0], x[1], x[2], x[3]);
          *reinterpret_cast<float4*>(xd + 4) = make_float4(x[4], x[5], x[6], x[7]);
        }
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
#pragma unroll 1
      for (int i = lane; i < dt; i += 32) *reinterpret_cast<float*>(s_xn + i * TB + 4 * r) = i == 0 ? ss : 0.f;
    }
    __syncthreads();
    if (tid == 0) *s_best = none;

    const int nold = (kv + 15) / 16, nblk = nold + (dl + 16) / 16;   // blocks of 16 keys: cached ones, then the block's own
    // One turn per projection: QKV, attention output, gate/up, down of every layer, then the LM head.  What they share is there
    // once: as five copies of it the kernel was 169 KB of instructions, more than the SM's caches hold.
    uint4 kf[2][DH / 32];                                      // attention: keys and values of this warp's next block
    uint32_t vf[4][kDims / 2];
    __nv_bfloat16 *Kg = K0, *Vg = K0;
    const float* gains = s_gain;
#pragma unroll 1
    for (int turn = 0; turn <= 4 * a.n_layers; ++turn) {
      const int l = min(turn >> 2, a.n_layers - 1), kind = turn == 4 * a.n_layers ? kLm : turn & 3;
      const Job* job = s_job + kind;
      const uint32_t parity = (uint32_t)(layers_done + l) & 1u;
      const int jobs = uni(job->jobs);
      int tl = warp;                                           // job
#pragma unroll 1
      do {
        if (tl == warp) {
          // ---------------------------------------------------------- what has to come first
          if (kind == kOut && attends) {
            wait(kXQkv, parity);
            // -------------------------------------------------------- attention: this warp's blocks of 16 keys, 16 query rows
            int blk = kg * S + slice;                          // the CTAs of a KV head, then their warps, in turn
            uint4 qf[2][DH / 32][2];
#pragma unroll
            for (int h2 = 0; h2 < 2; ++h2)
#pragma unroll
              for (int i = 0; i < DH / 32; ++i) {
                const int ch = 4 * i + t, at = ch % kParts * TB + h2 * 32 + ch / kParts * 16;
                qf[h2][i][0] = *reinterpret_cast<const uint4*>(s_q + q_lo + at);
                qf[h2][i][1] = *reinterpret_cast<const uint4*>(s_q + q_hi + at);
              }
            float m_lo = -INFINITY, m_hi = -INFINITY, s_lo = 0.f, s_hi = 0.f, o[kDims][4];
#pragma unroll
            for (int j = 0; j < kDims; ++j) { o[j][0] = 0.f; o[j][1] = 0.f; o[j][2] = 0.f; o[j][3] = 0.f; }
            bool have = blk < nold;                            // a cached first block has been asked for
#pragma unroll 1
            while (blk < nblk) {
              float s[2][2][4];                                // (by term)
              uint32_t v0[kDims], v1[kDims];                   // B fragments of the kDims column tiles: column g of tile j is dim kDims * g + j
              // keys of this block that a row attends to: all cached ones; of the block's own those up to the row
              const bool old = blk < nold;
              const int key0 = (old ? blk : blk - nold) * 16 + 2 * t, lim_lo = (old ? kv : tok_lo + 1) - key0, lim_hi = (old ? kv : tok_hi + 1) - key0;
              if (have) {
#pragma unroll
                for (int q = 0; q < 2; ++q)
#pragma unroll
                  for (int h2 = 0; h2 < 2; ++h2) { s[h2][q][0] = 0.f; s[h2][q][1] = 0.f; s[h2][q][2] = 0.f; s[h2][q][3] = 0.f; }
#pragma unroll
                for (int i = 0; i < DH / 32; ++i) {
#pragma unroll
                  for (int q = 0; q < 2; ++q)
#pragma unroll
                    for (int h2 = 0; h2 < 2; ++h2) mma_bf16(s[h2][q], qf[h2][i][0].x, qf[h2][i][1].x, qf[h2][i][0].y, qf[h2][i][1].y, kf[q][i].x, kf[q][i].y);
#pragma unroll
                  for (int q = 0; q < 2; ++q)
#pragma unroll
                    for (int h2 = 0; h2 < 2; ++h2) mma_bf16(s[h2][q], qf[h2][i][0].z, qf[h2][i][1].z, qf[h2][i][0].w, qf[h2][i][1].w, kf[q][i].z, kf[q][i].w);
                }
#pragma unroll
                for (int j = 0; j < kDims; ++j) {
                  v0[j] = __byte_perm(vf[0][j >> 1], vf[1][j >> 1], j & 1 ? 0x7632 : 0x5410);
                  v1[j] = __byte_perm(vf[2][j >> 1], vf[3][j >> 1], j & 1 ? 0x7632 : 0x5410);
                }
              }
              const int next = have ? blk + KG * S : blk;
              if (next < nold) load_cached<DH>(kf, vf, Kg, Vg, next * 16, kv, g, t);
              else if (next < nblk) load_own<DH>(kf, vf, s_kn, Rp, (next - nold) * 16, R, g, t);
              if (have) {
                float mx_lo = -INFINITY, mx_hi = -INFINITY;
#pragma unroll
                for (int q = 0; q < 2; ++q)
#pragma unroll
                  for (int i = 0; i < 2; ++i) {
                    s[0][q][i] = 8 * q + i < lim_lo ? s[0][q][i] + s[1][q][i] : -INFINITY;
                    s[0][q][2 + i] = 8 * q + i < lim_hi ? s[0][q][2 + i] + s[1][q][2 + i] : -INFINITY;
                    mx_lo = fmaxf(mx_lo, s[0][q][i]);
                    mx_hi = fmaxf(mx_hi, s[0][q][2 + i]);
                  }
                mx_lo = fmaxf(mx_lo, __shfl_xor_sync(0xffffffffu, mx_lo, 1));
                mx_hi = fmaxf(mx_hi, __shfl_xor_sync(0xffffffffu, mx_hi, 1));
                mx_lo = fmaxf(mx_lo, __shfl_xor_sync(0xffffffffu, mx_lo, 2));
                mx_hi = fmaxf(mx_hi, __shfl_xor_sync(0xffffffffu, mx_hi, 2));
                const float n_lo = fmaxf(m_lo, mx_lo * a.scale_log2e), n_hi = fmaxf(m_hi, mx_hi * a.scale_log2e);
                const float z_lo = n_lo == -INFINITY ? 0.f : n_lo, z_hi = n_hi == -INFINITY ? 0.f : n_hi;   // (a row may have no key here)
                const float c_lo = exp2f(m_lo - z_lo), c_hi = exp2f(m_hi - z_hi);
                m_lo = n_lo; m_hi = n_hi;
                s_lo *= c_lo; s_hi *= c_hi;
                uint32_t ph[4], pl[4];
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                  const float e0 = exp2f(fmaf(s[0][q][0], a.scale_log2e, -z_lo)), e1 = exp2f(fmaf(s[0][q][1], a.scale_log2e, -z_lo));
                  const float e2 = exp2f(fmaf(s[0][q][2], a.scale_log2e, -z_hi)), e3 = exp2f(fmaf(s[0][q][3], a.scale_log2e, -z_hi));
                  s_lo += e0 + e1;
                  s_hi += e2 + e3;
                  split2(e0, e1, ph[2 * q], pl[2 * q]);
                  split2(e2, e3, ph[2 * q + 1], pl[2 * q + 1]);
                }
#pragma unroll
                for (int j = 0; j < kDims; ++j) {
                  o[j][0] *= c_lo; o[j][1] *= c_lo; o[j][2] *= c_hi; o[j][3] *= c_hi;
                  mma_bf16(o[j], ph[0], ph[1], ph[2], ph[3], v0[j], v1[j]);
                }
#pragma unroll
                for (int j = 0; j < kDims; ++j) mma_bf16(o[j], pl[0], pl[1], pl[2], pl[3], v0[j], v1[j]);
              }
              blk = next;
              have = true;
            }
            s_lo += __shfl_xor_sync(0xffffffffu, s_lo, 1);
            s_hi += __shfl_xor_sync(0xffffffffu, s_hi, 1);
            s_lo += __shfl_xor_sync(0xffffffffu, s_lo, 2);
            s_hi += __shfl_xor_sync(0xffffffffu, s_hi, 2);
            ask_turn(turn);                                    // this projection's weights, beside the reduction (lower half of the ring)
            // a thread holds dims kDims * 2t .. and kDims * (2t + 1) .. of its two rows
            float* so = s_red + warp * kRed;
#pragma unroll
            for (int j = 0; j < kDims; j += 4) {
              *reinterpret_cast<float4*>(so + red_at(g, kDims * 2 * t + j)) = make_float4(o[j][0], o[j + 1][0], o[j + 2][0], o[j + 3][0]);
              *reinterpret_cast<float4*>(so + red_at(g, kDims * (2 * t + 1) + j)) = make_float4(o[j][1], o[j + 1][1], o[j + 2][1], o[j + 3][1]);
              *reinterpret_cast<float4*>(so + red_at(g + 8, kDims * 2 * t + j)) = make_float4(o[j][2], o[j + 1][2], o[j + 2][2], o[j + 3][2]);
              *reinterpret_cast<float4*>(so + red_at(g + 8, kDims * (2 * t + 1) + j)) = make_float4(o[j][3], o[j + 1][3], o[j + 2][3], o[j + 3][3]);
            }
            if (t == 0) {
              s_redml[warp * 16 + g] = make_float2(m_lo, s_lo);
              s_redml[warp * 16 + g + 8] = make_float2(m_hi, s_hi);
            }
            __syncthreads();
            // the warps' shares of a row meet, a warp per row: lane j weighs share j
            float* po = reinterpret_cast<float*>(s_stage);
#pragma unroll 1
            for (int q = warp; q < nq; q += kWarps) {
              const float2 ml = lane < KG ? s_redml[lane * MQ * 16 + q] : make_float2(-INFINITY, 0.f);
              float M = ml.x;
#pragma unroll
              for (int off = 8; off > 0; off >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, off));
              const float f = ml.x == -INFINITY ? 0.f : exp2f(ml.x - M);
              float sum = ml.y * f;
#pragma unroll
              for (int off = 8; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
              // half a warp per share, two (or four) dims a lane
              const float* r = s_red + ((lane >> 4) * MQ + (q >> 4)) * kRed;
              float y[kDims / 2];
#pragma unroll
              for (int x = 0; x < kDims / 2; ++x) y[x] = 0.f;
#pragma unroll 4
              for (int j = 0; j < KG; j += 2) {
                const float fj = __shfl_sync(0xffffffffu, f, j + (lane >> 4));
#pragma unroll
                for (int x = 0; x < kDims / 2; x += 2) {
                  const float2 v = *reinterpret_cast<const float2*>(r + j * MQ * kRed + red_at(q & 15, kDims / 2 * (lane & 15) + x));
                  y[x] = fmaf(v.x, fj, y[x]); y[x + 1] = fmaf(v.y, fj, y[x + 1]);
                }
              }
#pragma unroll
              for (int x = 0; x < kDims / 2; ++x) y[x] += __shfl_xor_sync(0xffffffffu, y[x], 16);
              if (lane < 16) {
#pragma unroll
                for (int x = 0; x < kDims / 2; x += 2) *reinterpret_cast<float2*>(po + q * DH + kDims / 2 * lane + x) = make_float2(y[x], y[x + 1]);
              }
              if (lane == 0) *reinterpret_cast<float2*>(po + nq * DH + 2 * q) = make_float2(M, sum);
            }
            __syncthreads();
            if (!silent(kXAttn))
#pragma unroll 1
              for (int s = 0; s < S; ++s) {
                const uint32_t dst = peer(base, kvh * S + s), at = dst + (uint32_t)(a.at.act + slice * a.slice_bytes);
#pragma unroll 1
                for (int i = 16 * tid; i < a.slice_bytes; i += 16 * kThreads) send16(at + i, *reinterpret_cast<const uint4*>(s_stage + i), dst + bars + 8 * kXAttn);
              }
            // the block's K/V rows into the cache, by the CTA that will read them
#pragma unroll 1
            for (int r = warp; r < 2 * (dl + 1); r += kWarps) {
              const int tok = r >> 1, is_v = r & 1;
              if ((((kv + tok) >> 4) & (S - 1)) == slice && lane < DH / 8)
                *reinterpret_cast<uint4*>((is_v ? Vg : Kg) + (uint32_t)((kv + tok) * DH + 8 * lane)) =
                    *reinterpret_cast<const uint4*>(s_kn + ((is_v * kParts + lane % kParts) * Rp + tok) * 32 + lane / kParts * 16);
            }
            wait(kXAttn, parity);
            // -------------------------------------------------------- the slices meet, a warp per query row
#pragma unroll 1
            for (int q = warp; q < nq; q += kWarps) {
              const uint8_t* r = s_po + 4 * nq * DH + 8 * q;
              float M = -INFINITY, sum = 0.f, y[DH / 32];
#pragma unroll 1
              for (int s = 0; s < S; ++s) M = fmaxf(M, *reinterpret_cast<const float*>(r + s * a.slice_bytes));
#pragma unroll
              for (int x = 0; x < DH / 32; ++x) y[x] = 0.f;
#pragma unroll 1
              for (int s = 0; s < S; ++s) {
                const float2 ml = *reinterpret_cast<const float2*>(r + s * a.slice_bytes);
                const float f = ml.x == -INFINITY ? 0.f : exp2f(ml.x - M);
                sum = fmaf(ml.y, f, sum);
#pragma unroll
                for (int x = 0; x < DH / 32; ++x) y[x] = fmaf(*reinterpret_cast<const float*>(s_po + s * a.slice_bytes + 4 * (q * DH + lane + 32 * x)), f, y[x]);
              }
              const float inv = sum > 0.f ? 1.f / sum : 0.f;
              const int hg = q / R, tok = q - hg * R;
#pragma unroll
              for (int x = 0; x < DH / 32; ++x) {
                const int f = hg * DH + lane + 32 * x;
                __nv_bfloat16* st = reinterpret_cast<__nv_bfloat16*>(s_at + (f >> 4) * TB + kRows + tok * 64) + (f & 15);
                split1(y[x] * inv, st, st + 16);
              }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // (the rings' second halves are copied into again)
            __syncthreads();
          }
          if (kind == kDown) __syncthreads();                  // (all of the SwiGLU output is there)
          if (kind != kOut && kind != kDown) {
            if (turn > 0) {
              // the residual stream's sums meet, and the next norm's operand goes to everyone; sixteen lanes per token
              const int xin = kind == kGateUp ? kXOut : kXDown, xout = xin + 1, senders = kind == kGateUp ? Hkv : NC;
              const uint32_t from_parity = kind == kQkv ? parity ^ 1u : parity;
              wait(xin, from_parity);
              __syncthreads();                                 // (s_norm is written again)
              const int tok = tid >> 4, f = tid & 15;
#pragma unroll 1
              for (int i = 0; i < dn; ++i) {
                float v = 0.f;
                if (tok < R) {
                  const float* p = s_sums + (i * R + tok) * 16 + f;
                  float* x = s_x + (i * Rp + tok) * 16 + f;
                  v = *x;
#pragma unroll 8
                  for (int q = 0; q < senders; ++q) v += p[q * dn * R * 16];
                  *x = v;
                  __nv_bfloat16* st = reinterpret_cast<__nv_bfloat16*>(s_norm + i * TB + kRows + tok * 64) + f;
                  split1(v * gains[i * 16 + f], st, st + 16);
                }
                float ss = v * v;
#pragma unroll
                for (int off = 8; off > 0; off >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
                if (f == 0 && tok < Rp) *reinterpret_cast<float*>(s_norm + i * TB + 4 * tok) = ss;
              }
              __syncthreads();
              if (!silent(xout))
#pragma unroll 1
                for (int i = 0; i < dn; ++i)
#pragma unroll 1
                  for (int q = 16 * (lane + 32 * (warp >> log_nc)); q < kRows + 64 * R; q += 512 * (kWarps >> log_nc))
                    send16(to + (uint32_t)(a.at.xn + (d0 + i) * TB + q), *reinterpret_cast<const uint4*>(s_norm + i * TB + q), to + bars + 8 * xout);
              gains += a.own_d * 16;
              wait(xout, from_parity);
            }
            if (kind != kLm && warp == kWarps - 1) rms();
          }
        }
        float acc[NT][2];
        if (tl < jobs) {
          // sums of this warp's tile: rows row and row + 8, tokens 4q + t; a thread's piece of a row of 128 bytes lies where the copy's swizzle put it
          float sum[2][NT][4];
#pragma unroll
          for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int q = 0; q < NT; ++q) { sum[h][q][0] = 0.f; sum[h][q][1] = 0.f; sum[h][q][2] = 0.f; sum[h][q][3] = 0.f; }
          const int4 what = *reinterpret_cast<const int4*>(&job->op);
          const int kb = uni(what.y);
          const bool one = uniform((uint32_t)what.z) != 0;
          const uint8_t* opq = smem + what.x + op_at + job->quarter * 256;
#pragma unroll 1
          for (int i0 = 0; i0 < kb; i0 += 2 * kRing) {
            if (!try_wait(ring_bar, ring_parity)) wait_long(ring_bar, ring_parity, s_abort, a.wait_ns, a.status);
            __syncwarp();
            ring_parity ^= 1u;
            const int here = min(2 * kRing, kb - i0);
            const int at0 = 16 * (t ^ row), at1 = 16 * ((t + 4) ^ row);
            int i = 0;
#pragma unroll 1
            for (; i + 4 <= here; i += 4)
#pragma unroll
              for (int u = 0; u < 4; ++u) multiply_block<NT>(sum, ring_at + 1024 * i + 2048 * (u >> 1) + (u & 1 ? at1 : at0), opq + 2 * TB * (i + u), one);
#pragma unroll 1
            for (; i < here; ++i) multiply_block<NT>(sum, ring_at + 2048 * (i >> 1) + (i & 1 ? at1 : at0), opq + 2 * TB * i, one);
            opq += 4 * TB * kRing;
            __syncwarp();                                      // (the ring is filled again)
            if (i0 + 2 * kRing < kb) ask_for(turn, job, i0 / 2 + kRing);
          }
#pragma unroll
          for (int q = 0; q < NT; ++q) {
            acc[q][0] = (sum[0][q][0] + sum[0][q][1]) + (sum[1][q][0] + sum[1][q][1]);
            acc[q][1] = (sum[0][q][2] + sum[0][q][3]) + (sum[1][q][2] + sum[1][q][3]);
          }
        }
        if (tl == warp && (kind == kQkv || kind == kGateUp)) __syncthreads();   // (1/rms is there)
        if (tl < jobs) {
          const int tile = job->tile, qb = job->quarter;
          const bool one = uniform((uint32_t)job->one) != 0;
          if (kind == kLm) {
            // a tile of 16 ids: the largest sum of each token, and of the warp's tiles (1/rms scales all of a token's sums alike; NaN and -inf are nobody's
            // choice, as launch by launch)
            const int r0 = 16 * tile + row;
#pragma unroll
            for (int q = 0; q < NT; ++q) {
              float v = -INFINITY;
              int id = INT_MAX;
              if (r0 < a.vocab && acc[q][0] > v) { v = acc[q][0]; id = r0; }
              if (r0 + 8 < a.vocab && acc[q][1] > v) { v = acc[q][1]; id = r0 + 8; }
#pragma unroll
              for (int off = 4; off < 32; off <<= 1) {
                const float ov = __shfl_xor_sync(0xffffffffu, v, off);
                const int oi = __shfl_xor_sync(0xffffffffu, id, off);
                if (ov > v || (ov == v && oi < id)) { v = ov; id = oi; }
              }
              uint2* best = s_wmax + warp * Rp + 4 * q + t;    // (ids grow: the first of equal sums stays)
              if (g == 0 && (tl == warp || v > __uint_as_float(best->x))) *best = make_uint2(__float_as_uint(v), (uint32_t)id);
            }
          } else if (kind == kGateUp) {
            __nv_bfloat16* st = reinterpret_cast<__nv_bfloat16*>(s_act + (tile >> 1) * TB + kRows) + (4 * qb + t) * 32 + (tile & 1) * 8 + row;
#pragma unroll
            for (int q = 0; q < NT; ++q)
              if (q == 0 || !one) {
                const float rt = s_rstd[4 * (qb + q) + t], gate = acc[q][0] * rt, up = acc[q][1] * rt;
                split1(__fdividef(gate, 1.f + __expf(-gate)) * up, st + q * 128, st + q * 128 + 16);
              }
          } else {
            const bool qkv = kind == kQkv;
            const int head = tile / kParts, part = tile % kParts;
            uint8_t* st = mine + (4 * qb + t) * 64;
            __syncwarp();
#pragma unroll
            for (int q = 0; q < NT; ++q)
              if (q == 0 || !one) {
                float x = acc[q][0], y = acc[q][1];
                if (qkv) {
                  const int tok = min(4 * (qb + q) + t, R - 1);
                  const float rt = s_rstd[tok];
                  const float2 r = head < H + Hkv ? s_rope[tok * kHalf + 8 * part + row] : make_float2(1.f, 0.f);
                  x *= rt;
                  y *= rt;
                  __nv_bfloat16* sb = reinterpret_cast<__nv_bfloat16*>(st + q * 256) + row;
                  split1(x * r.x - y * r.y, sb, sb + 16);
                  split1(y * r.x + x * r.y, sb + 8, sb + 24);
                } else {
                  float* sf = reinterpret_cast<float*>(st + q * 256) + row;
                  sf[0] = x;
                  sf[8] = y;
                }
              }
            __syncwarp();
            const int x = qkv ? kXQkv : kind == kOut ? kXOut : kXDown;
            if (!silent(x)) {
              const int4 to_at = *reinterpret_cast<const int4*>(&job->at);
              const bool whole = job->whole != 0;
              const uint8_t* from_st = mine + qb * 256;
#pragma unroll 1
              for (int p = to_at.y; p < to_at.z; ++p) {
                const uint32_t dst = peer(base, p);
#pragma unroll 1
                for (int i = lane; i < to_at.w; i += 32)
                  send16(dst + to_at.x + 16 * i, *reinterpret_cast<const uint4*>(from_st + (whole ? 16 * i : (i >> 1) * 64 + (i & 1) * 16)), dst + bars + 8 * x);
              }
            }
          }
        }
        // what comes next, once what others wait for is on its way
        tl += kWarps;
        if (tl < jobs) {
          __syncwarp();
          if (lane == 0) describe(s_job + kLm + 1, kind, tl);
          __syncwarp();
          job = s_job + kLm + 1;
          ask_for(turn, job, 0);
        }
      } while (tl < jobs);
      if (kind == kQkv && attends) {
        // this warp's first block of cached keys, while the queries travel (behind the cached rows there may be anything: 0 x NaN is NaN)
        Kg = turn == 0 ? K0 : Kg + k_layer;
        Vg = Kg + k_half;
        if (kg * S + slice < nold) load_cached<DH>(kf, vf, Kg, Vg, (kg * S + slice) * 16, kv, g, t);
      }
      if (kind != kLm && kind != kQkv) ask_turn(turn + 1);     // (behind QKV the keys come first)
    }
    layers_done += a.n_layers;
    // the largest of `count` lists for a token, by 16 lanes
    auto largest = [&](const uint2* list, int count, int tok) {
      const int i = lane & 15;
      uint2 v = make_uint2(__float_as_uint(-INFINITY), (uint32_t)INT_MAX);
      if (i < count && tok < Rp) v = list[i * Rp + tok];
#pragma unroll
      for (int off = 8; off > 0; off >>= 1) {
        const uint2 o = make_uint2(__shfl_xor_sync(0xffffffffu, v.x, off), __shfl_xor_sync(0xffffffffu, v.y, off));
        if (__uint_as_float(o.x) > __uint_as_float(v.x) || (__uint_as_float(o.x) == __uint_as_float(v.x) && (int)o.y < (int)v.y)) v = o;
      }
      return v;
    };
    __syncthreads();
    {
      const int tok = tid >> 4;                                // (as many groups of 16 lanes as a block has rows, at most)
      const uint2 v = largest(s_wmax, min(kWarps, l1 - l0), tok);
      if ((lane & 15) == 0 && tok < Rp) reinterpret_cast<uint2*>(s_stage)[tok] = v;
    }
    if (tid == 0) *s_tau = dl;
    __syncthreads();
    if (!silent(kXMax) && warp < NC && lane < Rp / 2)
      send16(to + (uint32_t)(a.at.misc + 8 * c * Rp + 16 * lane), *reinterpret_cast<const uint4*>(s_stage + 16 * lane), to + bars + 8 * kXMax);
    asked = ask_turn(0);
    wait(kXMax, step_parity);
    step_parity ^= 1u;
    // ------------------------------------------------------------------ acceptance (App. B.2) and append (App. B.3 step 4)
    {
      const int tok = tid >> 4;
      const uint2 v = largest(s_max, NC, tok);
      if ((lane & 15) == 0 && tok < R) {
        const int arg = tok <= dl && (int)v.y != INT_MAX ? (int)v.y : -1;
        const int tgt = tok > dl ? -1 : a.script != nullptr ? s_script[tok] : arg;
        s_tgt[tok] = tgt;
        if (tok < dl && s_hist[from + tok] != tgt) atomicMin(s_tau, tok);
      }
    }
    __syncthreads();
    if (*s_abort) break;
    const int tau = *s_tau;
    int cnt = min(tau + 1, a.max_new - e);
    if (a.script == nullptr && a.eos_id >= 0) {
#pragma unroll 1
      for (int i = 0; i < cnt; ++i)
        if (s_tgt[i] == a.eos_id) { cnt = i + 1; fin = true; break; }
    }
    if (tid < cnt) s_hist[n + tid] = s_tgt[tid];
    if (c == 0) {
      if (tid < cnt) h[n + tid] = s_tgt[tid];
      if (tid == kClerk) {
        cs_stats* st = reinterpret_cast<cs_stats*>(a.stats);
        a.hist_len[b] = n + cnt;
        a.kv_len[b] = n + cnt - 1;
        a.emitted[b] = e + cnt;
        atomicAdd((unsigned long long*)&st->steps, 1ull);
        atomicAdd((unsigned long long*)&st->emitted, (unsigned long long)cnt);
        if (p0 >= 0) {
          atomicAdd((unsigned long long*)&st->attempts, 1ull);
          atomicAdd((unsigned long long*)&st->accepted, (unsigned long long)(cnt - 1));
          atomicAdd((unsigned long long*)&st->tau_hist[min(cnt - 1, CS_TAU_HIST - 1)], 1ull);
        } else {
          atomicAdd((unsigned long long*)&st->no_match, 1ull);
        }
      }
    }
    if (tid < kHalf) {
      const double2 x = s_first[tid], y = s_turn[cnt * kHalf + tid];
      s_first[tid] = make_double2(x.x * y.x - x.y * y.y, x.y * y.x + x.x * y.y);
    }
    n += cnt;
    kv = n - 1;
    e += cnt;
    if (e >= a.max_new) fin = true;
    __syncthreads();                                           // (the next search reads what was appended)
  }
  if (asked && !try_wait(ring_bar, ring_parity)) wait_long(ring_bar, ring_parity, s_abort, a.wait_ns, a.status);   // (copies in flight land first)
  __syncthreads();
  if (*s_abort) {                                              // what was sent lands within microseconds
    const unsigned long long t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 1000000ull) {}
  }
  cluster_meet();
  // the last cluster to finish tells the host
  if (c == 0 && warp == 0) {
    int last = 0;
    if (lane == 0) {
      a.done[b] = 1;
      __threadfence();
      last = atomicAdd(a.done + a.max_batch + 1, 1) == a.B - 1;
    }
    if (__shfl_sync(0xffffffffu, last, 0)) {
      __threadfence();
      for (int i = lane; i < (int)(sizeof(cs_stats) / 8); i += 32) a.report[1 + i] = __ldcg(a.stats + i);
      if (lane == 0) a.report[0] = (unsigned long long)(unsigned)atomicExch(a.status, 0);
      __threadfence_system();
      __syncwarp();
      if (lane == 0) *reinterpret_cast<volatile unsigned long long*>(a.progress) = 1ull << 32;
    }
  }
}

typedef void (*SmallKernel)(const SmallMaps, const SmallArgs);
template <int DH>
SmallKernel small_kernel(int nt) {
  return nt == 1 ? k_small_loop<1, DH> : nt == 2 ? k_small_loop<2, DH> : nt == 3 ? k_small_loop<3, DH> : k_small_loop<4, DH>;
}

// A cluster of NC CTAs for blocks of R rows: what a launch needs, false = does not fit
struct SmallShape {
  int log_slices, log_rows, own_d, slice_bytes;
  SmallSmem at;
};
bool small_shape(const cs_model_config& c, int R, int NC, int stride, SmallShape* out) {
  const int d = c.d_model, F = c.d_ffn, Rp = 4 * cs_ceil_div(R, 4), G = c.n_heads / c.n_kv_heads, nq = G * R;
  const int parts = c.head_dim / 16;
  if ((c.head_dim != 32 && c.head_dim != 64) || d % 32 || F % 32 || c.n_layers > kMaxLayers || R > kMaxRows || c.n_kv_heads > NC || nq > 128) return false;
  if (G * c.head_dim > 32 * kRing) return false;      // (the attention output's weights take half of a ring)
  // every CTA has a tile of the residual stream, so that a layer never begins before all have finished the one before, and a block of SwiGLU
  if (d / 16 < NC || F / 32 < NC || d / 16 > 255) return false;
  out->log_slices = 0;
  while (c.n_kv_heads << (out->log_slices + 1) <= NC) ++out->log_slices;
  out->log_rows = 0;
  while (16 << out->log_rows < nq) ++out->log_rows;
  out->own_d = cs_ceil_div(d / 16, NC);
  out->slice_bytes = (nq * (4 * c.head_dim + 8) + 15) & ~15;
  const long long tile = tile_bytes(Rp);
  long long off = 0;
  auto take = [&](long long bytes) { const long long at = off; off += (bytes + 15) & ~15ll; return (int)min(at, 1ll << 30); };
  out->at.xn = take(d / 16 * tile);
  out->at.at = take(G * parts * tile);
  out->at.act = take(max(2 * cs_ceil_div(F / 32, NC) * tile, (long long)out->slice_bytes << out->log_slices));
  out->at.sums = take(64ll * NC * out->own_d * R);
  out->at.stage = take(max(64ll * Rp * kWarps, (long long)out->slice_bytes));
  out->at.norm = take(out->own_d * tile);
  out->at.red = take(8ll * kWarps * 16);
  out->at.q = take(G * parts * tile);
  out->at.kv = take(2ll * parts * 32 * Rp);
  out->at.xres = take(64ll * Rp * out->own_d);
  out->at.gain = take(128ll * c.n_layers * out->own_d);
  out->at.gain0 = take(2ll * d);
  out->at.rope = take(4ll * Rp * c.head_dim);
  out->at.turn = take(16ll * (R + 2) * (c.head_dim / 2));
  out->at.jobs = take((long long)sizeof(Job) * 6 * kWarps);
  off = (off + 1023) & ~1023ll;       // (the copies' swizzle goes by the address)
  out->at.ring = take(2048ll * kRing * kWarps);
  out->at.hist = take(4ll * stride);
  out->at.misc = take(8ll * kMaxCluster * Rp + 8ll * (kExchanges + kWarps) + 12ll * Rp + 16);
  out->at.total = (int)min(off, 1ll << 30);
  return off <= 227 * 1024;
}

}  // namespace

// Which loops: weights of a layer up to 3 MiB, an LM head up to 16 MiB, blocks of up to 16 rows, histories of up to 8,192 tokens (4,096 with
// heads of 64), and all sequences' clusters at once - of sixteen CTAs, or of eight where that is too many.  Calls of 6 to 8 steps, launch by
// launch / here, us (sequences x rows, tokens of history):
//                                        1 x 11, 512   1 x 1, 2000   1 x 11, 3500  4 x 11, 1000  8 x 4, 600   8 x 13, 600   14 x 7, 600   1 x 8, 8000
//   2 layers of 2.0 MiB, heads of 32        671/323       618/301       730/415       657/264       617/263      789/343       795/296
//   8 of them                              1865/1005     1727/940      2114/1349     1957/804      1784/783     2443/1040     2439/900
//   2 of 1.2 MiB, heads of 64               706/456       619/401       729/591       641/369       633/341      799/508       807/405       552/557
//   4 of 0.5 MiB (eight CTAs)              1089/593       923/486      1120/767       971/476       960/352     1298/482      1293/402       807/584
//   2 of 2.0 MiB, LM head of 16 MiB         702/501       657/409       743/594       692/395       638/417      832/645       842/502       578/529
// Sixteen CTAs stream a larger model from L2 slower than the chip does: 2 layers of 4.5 MiB with an LM head of 8 MiB 878/1352 for 16 x 7 rows, of 17 MiB
// 768/1122 for one row.  Clusters that do not all run at once wait for one another: 16 sequences of 7 rows with the 16 MiB LM head 857/1025.
cs_status cs_launch_small_loop(cs_ctx* ctx, bool* taken, cudaStream_t st) {
  const cs_model_config& c = ctx->cfg;
  const LoopState& L = ctx->loop;
  const int R = L.k + 1;
  *taken = false;
  if (ctx->small_force < 0 || ctx->attn_force != 0 || ctx->stamp_buf != nullptr || L.use_index || L.max_new < 1 || R > kMaxRows) return CS_OK;
  if (ctx->small_force == 0 && (cs_layer_bytes(c) > (3ll << 20) || 2ll * c.vocab * c.d_model > (16ll << 20) ||
                                (long long)L.stride * c.head_dim > (256 << 10))) return CS_OK;
  SmallShape shape;
  const int nt = cs_ceil_div(R, 4);
  SmallKernel kernel = c.head_dim == 32 ? small_kernel<32>(nt) : small_kernel<64>(nt);
  cudaLaunchConfig_t lc = {};
  cudaLaunchAttribute at[2];
  lc.blockDim = dim3(kThreads);
  lc.stream = st;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  int NC = 0;
  for (int big = 1; big >= 0 && NC == 0; --big) {
    const int nc = big ? kMaxCluster : kMaxCluster / 2;
    if (!small_shape(c, R, nc, L.stride, &shape)) continue;
    lc.gridDim = dim3(nc * L.B);
    lc.dynamicSmemBytes = (size_t)shape.at.total;
    at[0].val.clusterDim.x = nc;
    lc.numAttrs = 1;
    short& fit = ctx->small_fit[big][nt - 1];                  // clusters that run at once, + 1
    if (fit == 0) {
      CS_CUDA_OK(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
      CS_CUDA_OK(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, kernel, &lc) != cudaSuccess) { (void)cudaGetLastError(); n = 0; }
      fit = (short)(n + 1);
    }
    if (fit > L.B) NC = nc;
  }
  if (NC == 0) return CS_OK;
  SmallArgs a = {};
  SmallMaps* maps = static_cast<SmallMaps*>(ctx->small_maps);
  if (maps == nullptr) {
    // matrices as [blocks][halves][rows of a half][K], 128-byte swizzle
    maps = new (std::nothrow) SmallMaps;
    if (maps == nullptr) { snprintf(ctx->err, sizeof(ctx->err), "out of host memory"); return CS_ERR_ARG; }
    cs_status s = CS_OK;
    for (int i = 0; i <= 4 * c.n_layers && s == CS_OK; ++i) {
      const LayerPlan& P = ctx->layers[min(i >> 2, c.n_layers - 1)];
      const GemmPlan* g = i == 4 * c.n_layers ? &ctx->lm : (i & 3) == kQkv ? &P.qkv : (i & 3) == kOut ? &P.o : (i & 3) == kGateUp ? &P.gate_up : &P.down;
      const bool halves = i < 4 * c.n_layers && ((i & 3) == kQkv || (i & 3) == kGateUp);
      const unsigned long long K = g->K, half = !halves ? g->N : (i & 3) == kQkv ? c.head_dim / 2 : 64;
      const unsigned long long dims[4] = {K, half, halves ? 2ull : 1ull, halves ? g->N / (2 * half) : 1ull}, strides[3] = {2 * K, 2 * K * half, 4 * K * half};
      const unsigned box[4] = {64u, halves ? 8u : 16u, halves ? 2u : 1u, 1u};
      s = cs_encode_tiled(ctx, &maps->w[i], g->W, 4, dims, strides, box);
    }
    for (int i = 4 * c.n_layers + 1; i <= 4 * kMaxLayers; ++i) maps->w[i] = maps->w[0];
    if (s != CS_OK) { delete maps; return s; }
    ctx->small_maps = maps;
  }
  for (int l = 0; l < c.n_layers; ++l) { a.norm[2 * l] = ctx->layers[l].attn_norm; a.norm[2 * l + 1] = ctx->layers[l].ffn_norm; }
  a.norm[2 * c.n_layers] = ctx->final_norm;
  a.embed = ctx->embed; a.inv_freq = ctx->inv_freq;
  a.n_layers = c.n_layers; a.d = c.d_model; a.H = c.n_heads; a.Hkv = c.n_kv_heads; a.G = c.n_heads / c.n_kv_heads; a.F = c.d_ffn; a.vocab = c.vocab;
  a.max_seq = c.max_seq; a.max_batch = c.max_batch;
  a.inv_d = 1.f / (float)c.d_model; a.eps = c.rms_eps; a.scale_log2e = 1.4426950408889634f / sqrtf((float)c.head_dim);
  a.hist = L.hist; a.hist_len = L.hist_len; a.kv_len = L.kv_len; a.script = L.script; a.kv = static_cast<__nv_bfloat16*>(L.kv_cache);
  a.B = L.B; a.stride = L.stride; a.gamma = L.gamma; a.k = L.k; a.policy = L.policy; a.max_new = L.max_new; a.eos_id = L.eos_id;
  a.log_slices = shape.log_slices; a.log_rows = shape.log_rows; a.own_d = shape.own_d; a.slice_bytes = shape.slice_bytes; a.at = shape.at;
  a.emitted = ctx->loop_emitted; a.done = ctx->loop_done;
  a.stats = ctx->loop_stats; a.status = ctx->d_status;
  a.progress = ctx->progress_dev; a.report = reinterpret_cast<unsigned long long*>(ctx->step_out_dev);
  a.wait_ns = ctx->wait_limit_ns;
  a.drop = ctx->debug_drop_chain;
  ctx->debug_drop_chain = -1;         // the hook covers one launch
  lc.numAttrs = 2;
  CS_CUDA_OK(ctx, cudaLaunchKernelEx(&lc, kernel, (const SmallMaps)*maps, (const SmallArgs)a));
  *taken = true;
  return CS_OK;
}

void cs_small_free(cs_ctx* ctx) { delete static_cast<SmallMaps*>(ctx->small_maps); }
