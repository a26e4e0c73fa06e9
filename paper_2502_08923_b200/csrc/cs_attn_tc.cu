// Causal block attention over the bf16 KV cache on the 5th-generation tensor cores
// (Sec. 3.2; App. B.2), for head_dim 128.
//
// One CTA per SM = one (sequence, KV head), one slice of the key range and one group of at most 128 query
// rows (the (k+1) block rows of the G query heads sharing the KV head), which are the M dimension of
// both products, so that TMEM lane = query row:
//     S [128 x 128 keys]  = Q_hi K_tile^T + Q_lo K_tile^T   (A = Q in tensor memory, B = K tile)
//     O [128 x 128 dims] += P_hi V_tile   + P_lo V_tile     (A = P in tensor memory, B = V tile, MN-major
//                                                            straight from the cache layout)
// Queries and softmax weights enter as two bf16 terms each, so they are fp32-equivalent and only K and V -
// which the cache stores in bf16 - are rounded.  Both A operands live in TMEM: queries are put there once
// (they arrive by TMA in the ring's last slots; fetched by the softmax threads themselves, lane = row, they took up
// to 2 us at 11 rows and the layer 0.3 - 1 us longer),
// and a tile's weights overwrite its scores (128 fp32 columns = 64 columns of leading and 64 of second bf16
// terms), so shared memory holds nothing but the K and V tiles and the tensor cores read only those from it.
// Two S buffers: the scores of tile i + 1 are ready or under way while the softmax of tile i runs, and the MMA
// warp issues P V of tile i and the scores of tile i + 2 back to back.  Softmax: sixteen warps, four threads
// per query row (one per 32 keys).  Each row has a reference point for its exponentials that follows the true
// maximum only from afar: it moves when a score exceeds it by more than 2^8.  Softmax does not depend on the
// reference point, and weights up to 2^8 are as exact in two bf16 terms as weights up to 1; so on most tiles
// the threads of a lane quarter only vote (one predicate-reducing barrier, which also says that all of them
// have read their scores), and maxima are exchanged and O is rescaled on the few tiles where a point moves.
// K and V tiles come through one ring of six 32 KB slots in the order the MMAs use them: K0 K1 V0 K2 V1 K3 ...
// (A softmax thread that does not rescale runs up to two P V products ahead of the one that has retired, so
// "O holds tile i" has four barriers in turn, or a wait could be answered by the phase before.)  When the
// caller vouches for the cached lengths (kv_len_early), leading slots whose tiles lie wholly below the cached
// length are requested before the wait for the preceding kernel.  Lanes behind the last query row compute on
// zeroed or stale operands; nobody reads them.
//
// Each CTA writes its un-normalised (O, m, sum); k_attn_merge combines the key slices.
//
// Bound by the tensor cores for full tiles (two bf16 terms: 2,048 clocks of MMA per 128 x 128 tile at their
// peak rate, 2,400 - 2,500 measured) and by the key range's bytes or a chain of a few tiles otherwise.
// Attention plus merge per layer (8B shape; the kernel before, with P and Q in shared memory and one tile in
// flight -> this one; in brackets the kernel with the keys as M):
//   256 rows over 3,840+ keys 98.6 -> 51.0 us (117.2), 168 rows over 8 x 16,384 keys 234 -> 114 us (142),
//   11 rows over 4,096 keys 15.9 -> 14.6 us (17.7), 44 over 4 x 8,192 46.3 -> 36.1 us (37.2),
//   1 row over 2,048 keys 10.7 -> 11.1 us, 256 rows over one tile 13.6 -> 14.2 us.
// Taken back: handing O over through shared memory to store whole rows per warp, 9.4 -> 10.5 us at 11 rows over
// 4,096 keys.  Queries in TMEM instead of shared memory: 122 -> 112 us at 168 rows over 8 x 16,384 keys, six slots for all.
//
// Every wait is bounded (2 s by default): on expiry the CTA flags CS_DEV_TIMEOUT, drains its copies, frees
// its TMEM and returns; the softmax threads of a lane quarter decide together.
#include "cs_common.cuh"
#include "cs_tcgen.cuh"

namespace {

constexpr int kSoftWarps = 16, kProdWarp = 16, kMmaWarp = 17, kThreads = 576;
constexpr int kTileKeys = 128, kDh = 128, kNQMax = 128;
constexpr int kHalfBytes = kTileKeys * 128;      // one [128 keys x 64 dims] half tile
constexpr int kSlotBytes = 2 * kHalfBytes;
constexpr int kSlots = 6, kEarly = 3;               // ring; items asked for before the wait
constexpr uint32_t kOCol = 256, kQCol = 384, kTmemCols = 512;   // two S / P buffers of 128 columns, O, Q (64 columns per term)
constexpr int kCtlBytes = 256;                   // mbarriers, TMEM slot, flags

struct AttnArgs {
  const int* row_lim;
  const int* kv_len_early;   // cached lengths that no kernel in flight changes, or NULL
  int layer, R, Rg, G, H, Hkv, max_batch, max_seq, nsplit, rows;   // Rg = block rows per row group
  int smem_bytes;
  float scale_log2e;
  float* out_o;
  float* out_ml;
  __nv_bfloat16* whole;   // kWhole: the attention output, two bf16 terms
  int* status;
  unsigned long long wait_ns;
  unsigned long long* stamp;
};

// A from tensor memory: lane = row, a 32-bit column = two consecutive K elements
__device__ __forceinline__ void umma_bf16_ta(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}"
      ::"r"(tmem_d), "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(acc) : "memory");
}
// 32 accumulator columns of this thread's lane
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]),
        "=f"(v[8]), "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15]),
        "=f"(v[16]), "=f"(v[17]), "=f"(v[18]), "=f"(v[19]), "=f"(v[20]), "=f"(v[21]), "=f"(v[22]), "=f"(v[23]),
        "=f"(v[24]), "=f"(v[25]), "=f"(v[26]), "=f"(v[27]), "=f"(v[28]), "=f"(v[29]), "=f"(v[30]), "=f"(v[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
  // the registers are valid only from here on
  asm volatile("" : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]), "+f"(v[8]), "+f"(v[9]), "+f"(v[10]), "+f"(v[11]), "+f"(v[12]), "+f"(v[13]), "+f"(v[14]), "+f"(v[15]) :: "memory");
  asm volatile("" : "+f"(v[16]), "+f"(v[17]), "+f"(v[18]), "+f"(v[19]), "+f"(v[20]), "+f"(v[21]), "+f"(v[22]), "+f"(v[23]), "+f"(v[24]), "+f"(v[25]), "+f"(v[26]), "+f"(v[27]), "+f"(v[28]), "+f"(v[29]), "+f"(v[30]), "+f"(v[31]) :: "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
        "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
      : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// 2^x, hardware approximation (relative error about 2^-22; -inf gives 0)
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// two fp32 values in one 64-bit register and the packed fp32 arithmetic of this architecture
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 r, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(r)); }
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ void store8(float* dst, const float* v) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
               ::"l"(dst), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]) : "memory");
}
// barrier of the four warps of a lane quarter (ids 1 to 4) that also ORs a predicate
__device__ __forceinline__ bool quarter_any(int quarter, bool pred) {
  uint32_t out;
  asm volatile(
      "{\n.reg .pred p, q;\nsetp.ne.b32 p, %2, 0;\nbar.red.or.pred q, %1, 128, p;\nselp.u32 %0, 1, 0, q;\n}"
      : "=r"(out) : "r"(quarter + 1), "r"((uint32_t)pred) : "memory");
  return out != 0;
}

template <bool kWhole>   // one slice: what is written is the attention output itself, and there is nothing to merge
__global__ void __launch_bounds__(kThreads, 1)
k_attn_tc(const __grid_constant__ CUtensorMap tmKV, const __grid_constant__ CUtensorMap tmQ, AttnArgs a) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  uint8_t* smem = smem_raw + (((raw + 1023u) & ~1023u) - raw);
  // blockIdx.z picks a group of Rg consecutive block rows (blocks taller than 128 / G rows)
  const int G = a.G, R = a.R, r0 = blockIdx.z * a.Rg, Rcur = min(a.Rg, R - r0), nq = G * Rcur;
  uint8_t* ring = smem;                                // [slot][half][128 keys][128 B], K and V tiles in the order of use
  // the queries pass through the last slots on their way to tensor memory: [term][half][NQ rows][128 B]
  const uint32_t qpart = (uint32_t)((G * a.Rg + 7) & ~7) * 128u;
  const int qslot = kSlots - (int)((4 * qpart + kSlotBytes - 1) / kSlotBytes);
  uint8_t* sQ = ring + (size_t)qslot * kSlotBytes;
  uint8_t* ctl = ring + (size_t)kSlots * kSlotBytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(ctl);    // full, free per slot; 2 S, 2 P, 4 O, Q
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 24);
  volatile int* s_abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* s_never = reinterpret_cast<volatile int*>(tmem_slot + 2);   // stays 0: drains wait on time only
  int* s_lmax = reinterpret_cast<int*>(tmem_slot + 3);
  int* s_asked = reinterpret_cast<int*>(tmem_slot + 4);
  float* s_x = reinterpret_cast<float*>(ctl + kCtlBytes);   // [4 parts][128 rows]: row maxima, at the end row sums
  if ((size_t)(reinterpret_cast<uint8_t*>(s_x + 4 * 128) - smem_raw) > (size_t)a.smem_bytes) {
    if (threadIdx.x == 0) atomicOr(a.status, CS_DEV_SMEM);   // the launcher sizes the window for exactly this layout
    return;
  }
  const uint32_t b_full = smem_u32(bars), b_free = smem_u32(bars + kSlots), b_sready = smem_u32(bars + 2 * kSlots),
                 b_pready = smem_u32(bars + 2 * kSlots + 2), b_odone = smem_u32(bars + 2 * kSlots + 4),
                 b_qfull = smem_u32(bars + 2 * kSlots + 8), b_qland = smem_u32(bars + 2 * kSlots + 9);

  const int tid = threadIdx.x, warp = (int)uniform(tid >> 5), lane = tid & 31;
  const int b = blockIdx.x / a.Hkv, kvh = blockIdx.x % a.Hkv, split = blockIdx.y;
  const int nact = (nq + 31) >> 5;                     // lane quarters that hold real rows

  if (tid == kProdWarp * 32) {
    for (int s = 0; s < kSlots; ++s) { mbar_init(b_full + 8 * s, 1); mbar_init(b_free + 8 * s, 1); }
    for (int s = 0; s < 2; ++s) { mbar_init(b_sready + 8 * s, 1); mbar_init(b_pready + 8 * s, (uint32_t)nact * 4u); }
    for (int s = 0; s < 4; ++s) mbar_init(b_odone + 8 * s, 1);
    mbar_init(b_qfull, (uint32_t)nact * 4u);
    mbar_init(b_qland, 1);
    *s_abort = 0; *s_never = 0; *s_lmax = 0; *s_asked = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmKV) : "memory");
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_base = uniform(*tmem_slot);

  // Slice `split` works on key tiles split, split + nsplit, ...  Items of the ring: K0 K1 V0 K2 V1 ... (one tile: K0 V0)
  const long long krow = ((((long long)a.layer * 2 + 0) * a.max_batch + b) * a.Hkv + kvh) * (long long)a.max_seq;
  const long long vrow = ((((long long)a.layer * 2 + 1) * a.max_batch + b) * a.Hkv + kvh) * (long long)a.max_seq;
  // K and V leave L2 first, so that queries, sums and residual rows stay.  Blocks of at most 128 query rows per KV head read them
  // once; the row groups of taller ones run close enough together that the later ones still find them.  8 layers of the 8B shape
  // in turn, without / with, us: 11 rows over 30,000 keys 1,056 / 1,026, 8 x 21 over 4,096 1,699 / 1,685, over 16,384 2,364 / 2,356,
  // 256 rows (eight groups) behind 2,048 keys 2,063 / 2,059, behind 3,840 2,157 / 2,147
  const uint64_t policy = l2_evict_first();
  auto load_tile = [&](int s, long long first, int t) {          // tile t of this slice into slot s (by the elected lane)
    const uint32_t dst = smem_u32(ring) + (uint32_t)(s * kSlotBytes), bar = b_full + 8 * s;
    const int key0 = (split + t * a.nsplit) * kTileKeys;
    mbar_expect_tx(bar, (uint32_t)kSlotBytes);
    tma_load_2d_hint(dst, &tmKV, bar, 0, (int)(first + key0), policy);
    tma_load_2d_hint(dst + kHalfBytes, &tmKV, bar, 64, (int)(first + key0), policy);
  };
  // the first items are asked for before the preceding kernel is done while their tiles hold cached keys only
  int asked = 0;
  if (warp == kProdWarp && a.kv_len_early != nullptr) {
    const int cached = (int)uniform((uint32_t)min(a.kv_len_early[b], a.max_seq));
    for (; asked < kEarly; ++asked) {
      const bool is_k = asked < 2 || (asked & 1) != 0;
      const int t = asked < 2 ? asked : (is_k ? asked + 1 : asked - 2) >> 1;
      if ((split + t * a.nsplit + 1) * kTileKeys > cached) break;
      if (elect_one()) load_tile(asked, is_k ? krow : vrow, t);
    }
    if (lane == 0) *s_asked = asked < 2 ? asked : (asked + 2) >> 1;   // tiles
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");

  if (warp == kProdWarp && elect_one()) {
    mbar_expect_tx(b_qland, (uint32_t)(4 * G * a.Rg * 128));
    for (int term = 0; term < 2; ++term)
      for (int dh = 0; dh < 2; ++dh)
        tma_load_3d(smem_u32(sQ) + (uint32_t)(2 * term + dh) * qpart, &tmQ, b_qland, dh * 64, kvh * G,
                    term * CS_MAX_ROWS + b * R + r0);   // the box is always Rg rows tall; rows past the group are never used
  }
  const int quarter = warp & 3, part = warp >> 2, q = quarter * 32 + lane;   // of a softmax thread: query row = TMEM lane, quarter of the columns
  const uint32_t lane_base = tmem_base + ((uint32_t)(quarter * 32) << 16);
  const bool softmax = warp < kSoftWarps && quarter < nact, valid = softmax && q < nq;
  int lim = 0;                                         // keys this row attends to
  if (softmax) {
    // queries into tensor memory: this thread one half (64 dims) of one term of its row (swizzled rows: eight lanes
    // read eight different 16-byte columns)
    if (valid) lim = a.row_lim[b * R + r0 + q / G];
    const int lm = __reduce_max_sync(0xffffffffu, lim);
    if (lane == 0 && part == 0 && lm > 0) atomicMax(s_lmax, lm);
    if (!mbar_wait(b_qland, 0, s_abort, a.wait_ns)) *s_abort = 1;
    __syncwarp();
    uint32_t w[32];
    const uint8_t* src = sQ + (uint32_t)part * qpart + (uint32_t)q * 128u;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint4 t = valid ? *reinterpret_cast<const uint4*>(src + ((j ^ (q & 7)) << 4)) : make_uint4(0u, 0u, 0u, 0u);
      w[4 * j] = t.x; w[4 * j + 1] = t.y; w[4 * j + 2] = t.z; w[4 * j + 3] = t.w;
    }
    tmem_st16(lane_base + kQCol + 32u * (uint32_t)part, w);
    tmem_st16(lane_base + kQCol + 32u * (uint32_t)part + 16u, w + 16);
    tmem_st_wait();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncwarp();
    if (lane == 0) mbar_arrive(b_qfull);
  }
  __syncthreads();
  const int lmax = (int)uniform((uint32_t)*s_lmax);
  const int ntiles = (lmax + kTileKeys - 1) / kTileKeys;
  int ntl = (ntiles > split) ? (ntiles - split + a.nsplit - 1) / a.nsplit : 0;
  if (ntl > 0) ntl = max(ntl, (int)uniform((uint32_t)*s_asked));   // (tiles asked for lie in the range; were one beyond it, it would be masked)

  if (warp == kProdWarp) {
    // ------------------------------------------------------------------ TMA producer
    const int items = ntl > 0 ? 2 * ntl : asked;
    int j = 0, s = 0, tk = 0, tv = 0;
    uint32_t ph = 1;                                   // (the ring starts empty)
    bool ok = true;
    for (; j < items; ++j) {
      const bool is_k = tk < 2 ? (tk == 0 || (tk < ntl && tv == 0)) : (tk < ntl && tk < tv + 2);
      if (j >= kSlots) ok = mbar_wait_warp(b_free + 8 * s, ph, s_abort, a.wait_ns);
      if (j >= qslot && j < kSlots && ok) ok = mbar_wait_warp(b_qfull, 0, s_abort, a.wait_ns);   // (the queries have left the slot)
      if (!ok) break;
      if (j >= asked && elect_one()) load_tile(s, is_k ? krow : vrow, is_k ? tk : tv);
      if (is_k) ++tk; else ++tv;
      if (++s == kSlots) { s = 0; ph ^= 1u; }
    }
    if (!ok && lane == 0) { *s_abort = 1; atomicOr(a.status, CS_DEV_TIMEOUT); }
    __syncwarp();
    // copies that nobody will consume must land before the shared memory goes away
    if ((*s_abort || ntl == 0) && lane == 0) {
      mbar_wait(b_qland, 0, s_never, a.wait_ns);
      for (int i = max(0, j - kSlots); i < j; ++i) mbar_wait(b_full + 8 * (i % kSlots), (uint32_t)(i / kSlots) & 1u, s_never, a.wait_ns);
    }
  } else if (warp == kMmaWarp) {
    // ------------------------------------------------------------------ MMA issuer
    if (ntl > 0) {
      const uint32_t idesc1 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(128 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
      const uint32_t idesc2 = idesc1 | (1u << 16);     // B (= V) is MN-major
      const uint64_t dk0 = desc_kmajor(smem_u32(ring)), dv0 = desc_mnmajor(smem_u32(ring), kHalfBytes);
      int s = 0;
      uint32_t ph = 0;
      auto next_slot = [&]() { if (++s == kSlots) { s = 0; ph ^= 1u; } };
      auto issue_scores = [&](int t) -> bool {
        if (!mbar_wait_warp(b_full + 8 * s, ph, s_abort, a.wait_ns)) return false;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (elect_one()) {
          const uint64_t dk = dk0 + (uint64_t)(uint32_t)(s * (kSlotBytes >> 4));
          const uint32_t acc = tmem_base + (uint32_t)(t & 1) * 128u;
#pragma unroll
          for (int term = 0; term < 2; ++term)
#pragma unroll
            for (int dh = 0; dh < 2; ++dh)
#pragma unroll
              for (int kk = 0; kk < 4; ++kk)
                umma_bf16_ta(acc, tmem_base + kQCol + (uint32_t)(term * 64 + dh * 32 + kk * 8), dk + dh * (kHalfBytes >> 4) + 2 * kk,
                          idesc1, (term | dh | kk) ? 1u : 0u);
          umma_commit(b_free + 8 * s);
          umma_commit(b_sready + 8 * (t & 1));
        }
        next_slot();
        return true;
      };
      bool ok = mbar_wait_warp(b_qfull, 0, s_abort, a.wait_ns) && issue_scores(0);
      if (ok && ntl > 1) ok = issue_scores(1);
      for (int i = 0; i < ntl && ok; ++i) {
        ok = mbar_wait_warp(b_pready + 8 * (i & 1), (uint32_t)(i >> 1) & 1u, s_abort, a.wait_ns) &&
             mbar_wait_warp(b_full + 8 * s, ph, s_abort, a.wait_ns);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (elect_one()) {
          const uint64_t dv = dv0 + (uint64_t)(uint32_t)(s * (kSlotBytes >> 4));
          const uint32_t p = tmem_base + (uint32_t)(i & 1) * 128u;
#pragma unroll
          for (int term = 0; term < 2; ++term)
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)   // 16 keys per instruction
              umma_bf16_ta(tmem_base + kOCol, p + (uint32_t)(term * 64 + kk * 8), dv + kk * (2048 >> 4), idesc2,
                           (i > 0 || term > 0 || kk > 0) ? 1u : 0u);
          umma_commit(b_free + 8 * s);
          umma_commit(b_odone + 8 * (i & 3));
        }
        next_slot();
        if (i + 2 < ntl) {
          // its buffer is tile i's: the products run in the order of issue.  (The wait, long answered, is for the
          // softmax threads: whoever sees the scores of tile i + 2 knows that O holds tile i - 2.)
          if (i > 1) ok = mbar_wait_warp(b_odone + 8 * ((i - 2) & 3), (uint32_t)((i - 2) >> 2) & 1u, s_abort, a.wait_ns);
          if (ok) ok = issue_scores(i + 2);
        }
      }
      if (!ok && lane == 0) { *s_abort = 1; atomicOr(a.status, CS_DEV_TIMEOUT); }
    }
  } else if (softmax) {
    // ------------------------------------------------------------------ softmax + epilogue (four threads per query row)
    const float sc = a.scale_log2e;
    const f32x2 sc2 = pack2(sc, sc);
    float m = -INFINITY, thr = valid ? -INFINITY : INFINITY;   // reference point (log2 domain); raw score above which it moves
    f32x2 l2 = pack2(0.f, 0.f);                        // this thread's share of the row's sum
    bool have = ntl > 0;
    for (int i = 0; i < ntl; ++i) {
      const int tile0 = (split + i * a.nsplit) * kTileKeys, key0 = tile0 + 32 * part;   // first key of the tile, of this thread
      const uint32_t buf = lane_base + (uint32_t)(i & 1) * 128u;
      bool ok = mbar_wait(b_sready + 8 * (i & 1), (uint32_t)(i >> 1) & 1u, s_abort, a.wait_ns);
      ok = __all_sync(0xffffffffu, ok);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      float v[32];
      tmem_ld32(buf + 32u * (uint32_t)part, v);
      if (key0 + 32 > lim) {
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = key0 + j < lim ? v[j] : -INFINITY;
      }
      float mx4[4] = {v[0], v[1], v[2], v[3]};
#pragma unroll
      for (int j = 4; j < 32; ++j) mx4[j & 3] = fmaxf(mx4[j & 3], v[j]);
      const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
      const bool bad = !ok || *s_abort != 0;
      // (after this barrier every thread of the quarter has its scores in registers: the weights may overwrite them)
      if (quarter_any(quarter, mx > thr || bad)) {
        // ---- the rare path: the rows' true maxima, new reference points where needed
        s_x[part * 128 + q] = mx;
        if (quarter_any(quarter, bad)) { *s_abort = 1; have = false; break; }   // the same decision in every thread of the quarter
        const float t = fmaxf(fmaxf(s_x[q], s_x[128 + q]), fmaxf(s_x[256 + q], s_x[384 + q])) * sc;   // (sc > 0)
        const bool moves = valid && (m == -INFINITY ? t > m : t > m + 8.f);
        const float corr = moves ? (m == -INFINITY ? 0.f : ex2(m - t)) : 1.f;
        if (moves) { m = t; thr = (t + 8.f) / sc; }
        {
          float l0, l1;
          unpack2(l2, l0, l1);
          l2 = pack2(l0 * corr, l1 * corr);
        }
        if (i > 0 && __any_sync(0xffffffffu, moves)) {
          if (!mbar_wait(b_odone + 8 * ((i - 1) & 3), (uint32_t)((i - 1) >> 2) & 1u, s_abort, a.wait_ns)) *s_abort = 1;   // O holds all of tile i - 1
          __syncwarp();
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          float o[32];
          tmem_ld32(lane_base + kOCol + 32u * (uint32_t)part, o);
#pragma unroll
          for (int j = 0; j < 32; ++j) o[j] *= corr;
          tmem_st16(lane_base + kOCol + 32u * (uint32_t)part, reinterpret_cast<const uint32_t*>(o));
          tmem_st16(lane_base + kOCol + 32u * (uint32_t)part + 16u, reinterpret_cast<const uint32_t*>(o) + 16);
          tmem_st_wait();
        }
      }
      // ---- weights 2^(score * scale - m) as two bf16 terms, over the scores
      const float nm = m == -INFINITY ? -INFINITY : -m;
      const f32x2 nm2 = pack2(nm, nm);
      uint32_t hi[16], lo[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        float x0, x1;
        unpack2(fma2(pack2(v[2 * j], v[2 * j + 1]), sc2, nm2), x0, x1);
        const float w0 = ex2(x0), w1 = ex2(x1);        // masked scores are -inf: weight 0
        const f32x2 w2 = pack2(w0, w1);
        l2 = add2(l2, w2);
        const __nv_bfloat162 h = __floats2bfloat162_rn(w0, w1);
        hi[j] = *reinterpret_cast<const uint32_t*>(&h);
        float r0v, r1v;
        unpack2(sub2(w2, pack2(__uint_as_float(hi[j] << 16), __uint_as_float(hi[j] & 0xffff0000u))), r0v, r1v);
        const __nv_bfloat162 lw = __floats2bfloat162_rn(r0v, r1v);
        lo[j] = *reinterpret_cast<const uint32_t*>(&lw);
      }
      tmem_st16(buf + 16u * (uint32_t)part, hi);
      tmem_st16(buf + 64u + 16u * (uint32_t)part, lo);
      tmem_st_wait();
      // keys past the longest row of this sequence hold whatever the cache held: zero their V rows
      if (tile0 + kTileKeys > lmax) {
        // V of tile i is item 2 i + 2 of the ring, of the last tile the very last item
        const int item = i == ntl - 1 ? 2 * ntl - 1 : 2 * i + 2;
        const int s = item % kSlots;
        if (!mbar_wait(b_full + 8 * s, (uint32_t)(item / kSlots) & 1u, s_abort, a.wait_ns)) *s_abort = 1;
        uint8_t* vs = ring + (size_t)s * kSlotBytes;
        for (int rr = max(lmax - tile0, 0) + part * nact * 32 + q; rr < kTileKeys; rr += nact * 128) {
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            *reinterpret_cast<uint4*>(vs + (size_t)rr * 128 + c * 16) = make_uint4(0u, 0u, 0u, 0u);
            *reinterpret_cast<uint4*>(vs + kHalfBytes + (size_t)rr * 128 + c * 16) = make_uint4(0u, 0u, 0u, 0u);
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(b_pready + 8 * (i & 1));
    }
    // ---- un-normalised result of this key slice
    if (have) {
      bool ok = mbar_wait(b_odone + 8 * ((ntl - 1) & 3), (uint32_t)((ntl - 1) >> 2) & 1u, s_abort, a.wait_ns) && *s_abort == 0;
      if (quarter_any(quarter, !ok)) { *s_abort = 1; have = false; }
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    float o[32];
    if (have) {
      tmem_ld32(lane_base + kOCol + 32u * (uint32_t)part, o);
    } else {
#pragma unroll
      for (int j = 0; j < 32; ++j) o[j] = 0.f;
    }
    float l0, l1;
    unpack2(l2, l0, l1);
    s_x[part * 128 + q] = l0 + l1;
    quarter_any(quarter, false);
    if (valid) {
      const size_t obase = ((size_t)split * a.rows + (b * R + r0 + q / G)) * a.H + (kvh * G + q % G);
      auto sum = [&]() { return have ? (s_x[q] + s_x[128 + q]) + (s_x[256 + q] + s_x[384 + q]) : 0.f; };
      if constexpr (kWhole) {
        // nothing to merge: normalised, as the next projection's operand (what k_attn_merge makes of one slice)
        const float l = sum(), inv = l > 0.f ? 1.f / l : 0.f;
        __nv_bfloat16* dst = a.whole + obase * kDh + 32 * part;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          uint32_t h[4], w[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float y0 = o[8 * j + 2 * e] * inv, y1 = o[8 * j + 2 * e + 1] * inv;
            const __nv_bfloat162 hi = __floats2bfloat162_rn(y0, y1);
            const float2 f = __bfloat1622float2(hi);
            const __nv_bfloat162 lo = __floats2bfloat162_rn(y0 - f.x, y1 - f.y);
            h[e] = *reinterpret_cast<const uint32_t*>(&hi);
            w[e] = *reinterpret_cast<const uint32_t*>(&lo);
          }
          *reinterpret_cast<uint4*>(dst + 8 * j) = make_uint4(h[0], h[1], h[2], h[3]);
          *reinterpret_cast<uint4*>(dst + (size_t)CS_MAX_ROWS * a.H * kDh + 8 * j) = make_uint4(w[0], w[1], w[2], w[3]);
        }
      } else {
        float* dst = a.out_o + obase * kDh + 32 * part;
#pragma unroll
        for (int j = 0; j < 4; ++j) store8(dst + 8 * j, o + 8 * j);   // (whole 32-byte sectors)
        if (part == 0) {
          constexpr float kLn2 = 0.6931471805599453f;
          a.out_ml[obase * 2] = have ? m * kLn2 : -INFINITY;
          a.out_ml[obase * 2 + 1] = sum();
        }
      }
    }
    if (*s_abort && lane == 0) atomicOr(a.status, CS_DEV_TIMEOUT);
  }
  // ---------------------------------------------------------------------- teardown
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (tid == 0) cs_stamp_end(a.stamp);
  if (warp == kMmaWarp) {
    if (*s_abort && lane == 0 && ntl > 0) mbar_wait(b_odone + 8 * ((ntl - 1) & 3), (uint32_t)((ntl - 1) >> 2) & 1u, s_never, a.wait_ns);   // MMAs retired (bounded)
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
  }
}

}  // namespace

// Key tiles a CTA of this kernel walks at most for a block of B x R rows (same launch arithmetic as below).
int cs_attention_tc_tiles_per_cta(const cs_ctx* ctx, int B, int R) {
  const cs_model_config& c = ctx->cfg;
  const int G = c.n_heads / c.n_kv_heads;
  if (c.head_dim != kDh || G > kNQMax || R < 1) return 0;
  int nsplit = ctx->num_sms / (B * c.n_kv_heads * cs_ceil_div(G * R, kNQMax));
  if (nsplit > ctx->attn_splits) nsplit = ctx->attn_splits;
  if (nsplit < 1) nsplit = 1;
  return cs_ceil_div(cs_ceil_div(c.max_seq, kTileKeys), nsplit);
}

int cs_launch_attention_tc(cs_ctx* ctx, const void* kv_cache, int layer, int B, int R, bool* merge, cudaStream_t st) {
  const cs_model_config& c = ctx->cfg;
  const int G = c.n_heads / c.n_kv_heads;
  if (c.head_dim != kDh || G > kNQMax || R < 1 || R > 256) return 0;
  // blocks with more than 128 query rows per KV head are cut into groups of block rows
  const int ngroups = cs_ceil_div(G * R, kNQMax), Rg = cs_ceil_div(R, ngroups);
  if (G * Rg > kNQMax) return 0;
  if (ctx->tmKV_base != kv_cache) {
    const unsigned long long rows = (unsigned long long)c.n_layers * 2 * c.max_batch * c.n_kv_heads * c.max_seq;
    if (rows > 0x7fffffffull) return 0;
    const unsigned long long dims[2] = {(unsigned long long)kDh, rows}, strides[1] = {kDh * 2};
    const unsigned box[2] = {64, (unsigned)kTileKeys};
    if (cs_encode_tiled(ctx, &ctx->tmKV, kv_cache, 2, dims, strides, box) != CS_OK) return -1;
    ctx->tmKV_base = kv_cache;
  }
  if (ctx->tmQ_R != Rg) {
    const unsigned long long dims[3] = {(unsigned long long)kDh, (unsigned long long)c.n_heads, 2ull * CS_MAX_ROWS};
    const unsigned long long strides[2] = {kDh * 2, (unsigned long long)c.n_heads * kDh * 2};
    const unsigned box[3] = {64, (unsigned)G, (unsigned)Rg};
    if (cs_encode_tiled(ctx, &ctx->tmQ, ctx->qbuf, 3, dims, strides, box) != CS_OK) return -1;
    ctx->tmQ_R = Rg;
  }
  // one CTA per SM; 1 KB of slack for the 1024-byte alignment, then the ring, and barriers, flags and the exchange
  // rows of the softmax
  const size_t smem = 1024 + (size_t)kSlots * kSlotBytes + kCtlBytes + 4 * 128 * 4;
  int nsplit = ctx->num_sms / (B * c.n_kv_heads * ngroups);
  const bool whole = *merge && nsplit <= 1;            // (a cache of one tile is one slice too, but not worth a path of its own)
  if (nsplit > ctx->attn_splits) nsplit = ctx->attn_splits;
  if (nsplit < 1) nsplit = 1;
  if (smem > ctx->attn_tc_smem_set) {
    if (cudaFuncSetAttribute(k_attn_tc<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaFuncSetAttribute(k_attn_tc<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
      snprintf(ctx->err, sizeof(ctx->err), "attention needs %zu bytes of shared memory", smem);
      return -1;
    }
    ctx->attn_tc_smem_set = smem;
  }
  AttnArgs a;
  a.row_lim = ctx->row_lim;
  a.kv_len_early = ctx->kv_len_early;
  a.layer = layer; a.R = R; a.Rg = Rg; a.G = G; a.H = c.n_heads; a.Hkv = c.n_kv_heads;
  a.max_batch = c.max_batch; a.max_seq = c.max_seq; a.nsplit = nsplit; a.rows = B * R;
  a.smem_bytes = (int)smem;
  a.scale_log2e = 1.4426950408889634f / sqrtf((float)kDh);
  a.out_o = ctx->attn_o; a.out_ml = ctx->attn_ml; a.whole = ctx->attn_out; a.status = ctx->d_status;
  a.wait_ns = ctx->wait_limit_ns;
  a.stamp = cs_next_stamp(ctx, CS_FAM_ATTENTION);
  if (cs_launch_pdl(whole ? k_attn_tc<true> : k_attn_tc<false>, dim3(B * c.n_kv_heads, nsplit, ngroups), dim3(kThreads), smem, st, ctx->tmKV, ctx->tmQ, a) != cudaSuccess) {
    snprintf(ctx->err, sizeof(ctx->err), "attention launch failed");
    return -1;
  }
  if (whole) *merge = false;
  return nsplit;
}
