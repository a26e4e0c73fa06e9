// Causal block attention of the verification forward over the bf16 KV cache (Sec. 3.2;
// App. B.2): the (k+1) block rows of the G query heads that share one KV head form a small
// query tile (44 rows for k = 10, G = 4) that is multiplied against a slice of the cached
// keys/values.
//
// One CTA = one (sequence, KV head), one slice of the key range (split-KV) and up to 64
// query rows; its four warps run a register-resident flash-attention loop on bf16 tensor-core MMAs
// (m16n8k16, fp32 accumulation): S = Q K^T, running row max / sum, O += P V; Q and P enter the MMAs as two
// bf16 terms each (value = hi + lo), so only K and V - which the cache stores in bf16 - are rounded.
// K and V tiles of 64 keys stream through a double-buffered cp.async pipeline in shared memory (rows padded
// by 16 bytes so that fragment loads and ldmatrix are bank-conflict free).  Each warp owns 16 query rows;
// when at most 32 rows exist, two or four warps (KG) share the rows and divide the keys of every tile
// instead, and their results meet in shared memory at the end.  A slice's first tile is requested before
// the wait for the preceding kernel where it holds cached keys only, and queries and limits are requested
// together behind it.  Each slice writes its un-normalised output and (max, sum); k_attn_merge combines them.
//
// Bound by a chain of latencies at the sizes it serves (head_dim 32 and 64, small and draft models).
// Attention plus merge per layer, with one warp per 16 rows, queries loaded as fragments and nothing ahead of
// the wait -> now: 32 heads of 64 over 4,096 keys, 1 row 12.2 -> 9.1 us, 4 rows 13.2 -> 11.1, 11 rows 15.3 -> 14.4;
// 8 heads of 32 over 512 keys, 11 rows 8.4 -> 5.3.
#include <stdlib.h>

#include "cs_common.cuh"

namespace {

constexpr int kThreads = 128;
constexpr int kKeys = 64;      // keys per tile
constexpr int kStages = 2;
constexpr int kRowsPerCta = 64;   // / key groups

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem, int src_bytes) {
  const uint32_t s = (uint32_t)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(s), "l"(gmem), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], const void* smem) {
  const uint32_t s = (uint32_t)__cvta_generic_to_shared(smem);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(s));
}
// (lo, hi) as a leading bf16 pair plus the bf16 pair of what that rounding lost
__device__ __forceinline__ void pack_two(float lo, float hi, uint32_t& first, uint32_t& second) {
  const __nv_bfloat162 a = __floats2bfloat162_rn(lo, hi);
  const float2 af = __bfloat1622float2(a);
  const __nv_bfloat162 b = __floats2bfloat162_rn(lo - af.x, hi - af.y);
  first = *reinterpret_cast<const uint32_t*>(&a);
  second = *reinterpret_cast<const uint32_t*>(&b);
}

template <int DH, int KG>
__global__ void __launch_bounds__(kThreads)
k_attn_mma(const __nv_bfloat16* __restrict__ qbuf, const __nv_bfloat16* __restrict__ kv,
           const int* __restrict__ row_lim, const int* __restrict__ kv_len_early, int layer, int R, int H, int Hkv,
           int max_batch, int max_seq,
           int nsplit, float scale_log2e, float* __restrict__ out_o, float* __restrict__ out_ml, int rows,
           unsigned long long* stamp) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  constexpr int STRIDE = DH + 8;          // bf16 elements per shared-memory row
  constexpr int KSTEPS = DH / 16;         // MMA k-steps of the QK^T product
  constexpr int NB_S = kKeys / 8 / KG;    // 8-key column blocks of this warp's S
  constexpr int NB_O = DH / 8;            // 8-dim column blocks of O
  constexpr int CPR = DH / 8;             // 16-byte chunks per K/V row
  extern __shared__ __align__(16) uint8_t smem_raw[];
  __nv_bfloat16* Ks = reinterpret_cast<__nv_bfloat16*>(smem_raw);            // [stages][keys][STRIDE]
  __nv_bfloat16* Vs = Ks + kStages * kKeys * STRIDE;
  __shared__ int s_lmax;

  const int G = H / Hkv;
  const int b = blockIdx.x / Hkv, kvh = blockIdx.x % Hkv;
  const int split = blockIdx.y, rg = blockIdx.z;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;
  const int nq = G * R;
  const int kbase = warp % KG * (kKeys / KG);   // this warp's keys within a tile

  const __nv_bfloat16* Kg = kv + ((((size_t)layer * 2 + 0) * max_batch + b) * Hkv + kvh) * (size_t)max_seq * DH;
  const __nv_bfloat16* Vg = kv + ((((size_t)layer * 2 + 1) * max_batch + b) * Hkv + kvh) * (size_t)max_seq * DH;

  auto load_tile = [&](int tile, int stage, int keys) {   // keys from `keys` on are zero-filled
    const int key0 = tile * kKeys;
    __nv_bfloat16* kd = Ks + stage * kKeys * STRIDE;
    __nv_bfloat16* vd = Vs + stage * kKeys * STRIDE;
    for (int c = threadIdx.x; c < kKeys * CPR; c += kThreads) {
      const int j = c / CPR, cc = c % CPR;
      const int key = key0 + j;
      const int nbytes = key < keys ? 16 : 0;
      const size_t src = (size_t)min(key, max_seq - 1) * DH + cc * 8;
      cp_async16(kd + j * STRIDE + cc * 8, Kg + src, nbytes);
      cp_async16(vd + j * STRIDE + cc * 8, Vg + src, nbytes);
    }
  };
  // Slice `split` works on tiles split, split + nsplit, ...  Its first one is requested before the wait for the
  // preceding kernel when it holds cached keys only.
  bool early = false;
  if (kv_len_early != nullptr) {
    const int cached = min(__ldcg(kv_len_early + b), max_seq);
    early = (split + 1) * kKeys <= cached;
    if (early) load_tile(split, 0, cached);
    cp_async_commit();
  }
  if (threadIdx.x == 0) s_lmax = 0;
  __syncthreads();
  asm volatile("griddepcontrol.wait;" ::: "memory");

  // The queries, two bf16 terms each, pass through the second stage's buffers (K: leading, V: second terms).
  // They and the rows' limits are read through L2: L1 may hold what an earlier layer left there while this
  // kernel was already resident.
  constexpr int kRows = kRowsPerCta / KG;
  __nv_bfloat16* Qs = Ks + kKeys * STRIDE;
  __nv_bfloat16* Ql = Vs + kKeys * STRIDE;
  constexpr int kQIter = kRows * CPR * 2 / kThreads;   // 16-byte pieces per thread, all asked for at once
  static_assert(kRows * CPR * 2 % kThreads == 0 && kThreads % CPR == 0, "");
  uint4 qv[kQIter];
#pragma unroll
  for (int i = 0; i < kQIter; ++i) {
    const int tr = (i * kThreads + threadIdx.x) / CPR, term = tr / kRows, q = rg * kRows + tr % kRows;
    qv[i] = make_uint4(0u, 0u, 0u, 0u);
    if (q < nq)
      qv[i] = __ldcg(reinterpret_cast<const uint4*>(
          qbuf + (((size_t)term * CS_MAX_ROWS + b * R + q % R) * H + kvh * G + q / R) * DH + threadIdx.x % CPR * 8));
  }
  // the two query rows this thread holds fragments of
  const int r_lo = warp / KG * 16 + g, q_lo = rg * kRows + r_lo, q_hi = q_lo + 8;
  const bool v_lo = q_lo < nq, v_hi = q_hi < nq;
  const int grow_lo = v_lo ? b * R + q_lo % R : 0, grow_hi = v_hi ? b * R + q_hi % R : 0;
  const int head_lo = v_lo ? kvh * G + q_lo / R : 0, head_hi = v_hi ? kvh * G + q_hi / R : 0;
  const int lim_lo = v_lo ? __ldcg(row_lim + grow_lo) : 0, lim_hi = v_hi ? __ldcg(row_lim + grow_hi) : 0;
  // longest key range any row of this sequence's block attends to
  {
    int lm = 0;
    for (int r = threadIdx.x; r < R; r += kThreads) lm = max(lm, __ldcg(row_lim + b * R + r));
    lm = __reduce_max_sync(0xffffffffu, lm);
    if (lane == 0 && lm > 0) atomicMax(&s_lmax, lm);
  }
#pragma unroll
  for (int i = 0; i < kQIter; ++i) {
    const int tr = (i * kThreads + threadIdx.x) / CPR;
    *reinterpret_cast<uint4*>((tr < kRows ? Qs : Ql) + tr % kRows * STRIDE + threadIdx.x % CPR * 8) = qv[i];
  }
  __syncthreads();
  const int lmax = s_lmax;
  uint32_t qa[KSTEPS][4], qb[KSTEPS][4];   // (q = qa + qb: two MMAs give the product of the fp32 query)
#pragma unroll
  for (int ks = 0; ks < KSTEPS; ++ks)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int at = (r_lo + (i & 1) * 8) * STRIDE + ks * 16 + (i >> 1) * 8 + 2 * t;
      qa[ks][i] = *reinterpret_cast<const uint32_t*>(Qs + at);
      qb[ks][i] = *reinterpret_cast<const uint32_t*>(Ql + at);
    }
  __syncthreads();   // (their buffers are the second tile's)
  const int ntiles = (lmax + kKeys - 1) / kKeys;

  float m_lo = -INFINITY, m_hi = -INFINITY, l_lo = 0.f, l_hi = 0.f;
  float o[NB_O][4];
#pragma unroll
  for (int nd = 0; nd < NB_O; ++nd) { o[nd][0] = 0.f; o[nd][1] = 0.f; o[nd][2] = 0.f; o[nd][3] = 0.f; }

  if (!early && split < ntiles) load_tile(split, 0, lmax);
  cp_async_commit();
  int stage = 0;
  for (int tile = split; tile < ntiles; tile += nsplit, stage ^= 1) {
    if (tile + nsplit < ntiles) load_tile(tile + nsplit, stage ^ 1, lmax);
    cp_async_commit();
    cp_async_wait<1>();
    __syncthreads();
    const __nv_bfloat16* kt = Ks + stage * kKeys * STRIDE;
    const __nv_bfloat16* vt = Vs + stage * kKeys * STRIDE;
    const int key0 = tile * kKeys;

    // S = Q K^T for this warp's 16 rows and the tile's 64 keys
    float s[NB_S][4];
#pragma unroll
    for (int nb = 0; nb < NB_S; ++nb) {
      s[nb][0] = 0.f; s[nb][1] = 0.f; s[nb][2] = 0.f; s[nb][3] = 0.f;
#pragma unroll
      for (int ks = 0; ks < KSTEPS; ++ks) {
        const __nv_bfloat16* kp = kt + (kbase + nb * 8 + g) * STRIDE + ks * 16 + 2 * t;
        const uint32_t k0 = *reinterpret_cast<const uint32_t*>(kp), k1 = *reinterpret_cast<const uint32_t*>(kp + 8);
        mma_bf16(s[nb], qa[ks], k0, k1);
        mma_bf16(s[nb], qb[ks], k0, k1);
      }
    }
    // scale (log2 domain), causal mask, running max
    float mx_lo = -INFINITY, mx_hi = -INFINITY;
#pragma unroll
    for (int nb = 0; nb < NB_S; ++nb) {
      const int key = key0 + kbase + nb * 8 + 2 * t;
      s[nb][0] = (key < lim_lo) ? s[nb][0] * scale_log2e : -INFINITY;
      s[nb][1] = (key + 1 < lim_lo) ? s[nb][1] * scale_log2e : -INFINITY;
      s[nb][2] = (key < lim_hi) ? s[nb][2] * scale_log2e : -INFINITY;
      s[nb][3] = (key + 1 < lim_hi) ? s[nb][3] * scale_log2e : -INFINITY;
      mx_lo = fmaxf(mx_lo, fmaxf(s[nb][0], s[nb][1]));
      mx_hi = fmaxf(mx_hi, fmaxf(s[nb][2], s[nb][3]));
    }
    mx_lo = fmaxf(mx_lo, __shfl_xor_sync(0xffffffffu, mx_lo, 1));
    mx_lo = fmaxf(mx_lo, __shfl_xor_sync(0xffffffffu, mx_lo, 2));
    mx_hi = fmaxf(mx_hi, __shfl_xor_sync(0xffffffffu, mx_hi, 1));
    mx_hi = fmaxf(mx_hi, __shfl_xor_sync(0xffffffffu, mx_hi, 2));
    const float mn_lo = fmaxf(m_lo, mx_lo), mn_hi = fmaxf(m_hi, mx_hi);
    const float c_lo = (m_lo == -INFINITY) ? 0.f : exp2f(m_lo - mn_lo);
    const float c_hi = (m_hi == -INFINITY) ? 0.f : exp2f(m_hi - mn_hi);
    m_lo = mn_lo; m_hi = mn_hi;
    float ps_lo = 0.f, ps_hi = 0.f;
#pragma unroll
    for (int nb = 0; nb < NB_S; ++nb) {
      s[nb][0] = (s[nb][0] == -INFINITY) ? 0.f : exp2f(s[nb][0] - mn_lo);
      s[nb][1] = (s[nb][1] == -INFINITY) ? 0.f : exp2f(s[nb][1] - mn_lo);
      s[nb][2] = (s[nb][2] == -INFINITY) ? 0.f : exp2f(s[nb][2] - mn_hi);
      s[nb][3] = (s[nb][3] == -INFINITY) ? 0.f : exp2f(s[nb][3] - mn_hi);
      ps_lo += s[nb][0] + s[nb][1];
      ps_hi += s[nb][2] + s[nb][3];
    }
    l_lo = l_lo * c_lo + ps_lo;     // per-thread share of the row sum; the quad is summed at the end
    l_hi = l_hi * c_hi + ps_hi;
#pragma unroll
    for (int nd = 0; nd < NB_O; ++nd) { o[nd][0] *= c_lo; o[nd][1] *= c_lo; o[nd][2] *= c_hi; o[nd][3] *= c_hi; }

    // O += P V: the S accumulators are already laid out as the A fragments of the next MMA
#pragma unroll
    for (int j = 0; j < kKeys / 16 / KG; ++j) {
      // softmax weights as two bf16 terms as well
      uint32_t pa[4], pb[4];
      pack_two(s[2 * j][0], s[2 * j][1], pa[0], pb[0]);
      pack_two(s[2 * j][2], s[2 * j][3], pa[1], pb[1]);
      pack_two(s[2 * j + 1][0], s[2 * j + 1][1], pa[2], pb[2]);
      pack_two(s[2 * j + 1][2], s[2 * j + 1][3], pa[3], pb[3]);
#pragma unroll
      for (int nd = 0; nd < NB_O; nd += 2) {
        // four transposed 8x8 blocks of V: keys 16j..16j+15, dims nd*8 .. nd*8+15
        uint32_t vb[4];
        const int mi = lane >> 3, r8 = lane & 7;
        ldmatrix_x4_trans(vb, vt + (kbase + j * 16 + (mi & 1) * 8 + r8) * STRIDE + (nd + (mi >> 1)) * 8);
        mma_bf16(o[nd], pa, vb[0], vb[1]);
        mma_bf16(o[nd], pb, vb[0], vb[1]);
        mma_bf16(o[nd + 1], pa, vb[2], vb[3]);
        mma_bf16(o[nd + 1], pb, vb[2], vb[3]);
      }
    }
    __syncthreads();   // everyone is done with this stage before it is refilled
  }
  cp_async_wait<0>();

  l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 1);
  l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 2);
  l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 1);
  l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 2);
  // un-normalised partial result of this key slice; (max, sum) in the natural-log domain
  constexpr float kLn2 = 0.6931471805599453f;
  if (KG > 1) {
    // the key groups' shares meet in shared memory: [warp][16 rows][DH], then (max, sum) per warp and row
    float* so = reinterpret_cast<float*>(smem_raw);
    float2* sml = reinterpret_cast<float2*>(so + 4 * 16 * DH);
    __syncthreads();
#pragma unroll
    for (int nd = 0; nd < NB_O; ++nd) {
      *reinterpret_cast<float2*>(so + (warp * 16 + g) * DH + nd * 8 + 2 * t) = make_float2(o[nd][0], o[nd][1]);
      *reinterpret_cast<float2*>(so + (warp * 16 + g + 8) * DH + nd * 8 + 2 * t) = make_float2(o[nd][2], o[nd][3]);
    }
    if (t == 0) {
      sml[warp * 16 + g] = make_float2(m_lo, l_lo);
      sml[warp * 16 + g + 8] = make_float2(m_hi, l_hi);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 4 / KG * 16 * (DH / 4); e += kThreads) {
      const int row = e / (DH / 4), c = e % (DH / 4), q = rg * kRows + row;
      if (q >= nq) break;
      const int at0 = row / 16 * KG * 16 + row % 16;
      float M = -INFINITY;
#pragma unroll
      for (int w = 0; w < KG; ++w) M = fmaxf(M, sml[at0 + 16 * w].x);
      float L = 0.f;
      float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int w = 0; w < KG; ++w) {
        const float2 ml = sml[at0 + 16 * w];
        const float f = ml.x == -INFINITY ? 0.f : exp2f(ml.x - M);
        const float4 v = *reinterpret_cast<const float4*>(so + (at0 + 16 * w) * DH + 4 * c);
        L = fmaf(ml.y, f, L);
        y.x = fmaf(v.x, f, y.x); y.y = fmaf(v.y, f, y.y); y.z = fmaf(v.z, f, y.z); y.w = fmaf(v.w, f, y.w);
      }
      const size_t base = ((size_t)split * rows + b * R + q % R) * H + kvh * G + q / R;
      *reinterpret_cast<float4*>(out_o + base * DH + 4 * c) = y;
      if (c == 0) { out_ml[base * 2] = M * kLn2; out_ml[base * 2 + 1] = L; }
    }
  }
  if (KG == 1 && v_lo) {
    const size_t base = ((size_t)split * rows + grow_lo) * H + head_lo;
#pragma unroll
    for (int nd = 0; nd < NB_O; ++nd)
      *reinterpret_cast<float2*>(out_o + base * DH + nd * 8 + 2 * t) = make_float2(o[nd][0], o[nd][1]);
    if (t == 0) { out_ml[base * 2] = m_lo * kLn2; out_ml[base * 2 + 1] = l_lo; }
  }
  if (KG == 1 && v_hi) {
    const size_t base = ((size_t)split * rows + grow_hi) * H + head_hi;
#pragma unroll
    for (int nd = 0; nd < NB_O; ++nd)
      *reinterpret_cast<float2*>(out_o + base * DH + nd * 8 + 2 * t) = make_float2(o[nd][2], o[nd][3]);
    if (t == 0) { out_ml[base * 2] = m_hi * kLn2; out_ml[base * 2 + 1] = l_hi; }
  }
  if (stamp != nullptr) {
    __syncthreads();
    if (threadIdx.x == 0) cs_stamp_end(stamp);
  }
}

template <int DH, int KG>
int launch_groups(cs_ctx* ctx, const void* kv_cache, int layer, int B, int R, cudaStream_t st) {
  const cs_model_config& c = ctx->cfg;
  const int G = c.n_heads / c.n_kv_heads;
  const int rgs = cs_ceil_div(G * R, kRowsPerCta / KG);
  // enough key slices to give every SM about two CTAs (four of the shorter ones that share keys: 7.7 -> 5.9 us at
  // one row over 4,096 keys, the merge 2.8 -> 3.2; with all warps on rows of their own the merge costs what the
  // walk gains), never more than the workspace holds
  int nsplit = cs_ceil_div((KG > 1 ? 4 : 2) * ctx->num_sms, B * c.n_kv_heads * rgs);
  if (nsplit > ctx->attn_splits) nsplit = ctx->attn_splits;
  if (nsplit < 1) nsplit = 1;
  const size_t smem = (size_t)2 * kStages * kKeys * (DH + 8) * 2;
  constexpr unsigned kAttrBit = 1u << (DH / 32 * 3 + KG / 2);
  if (!(ctx->attn_mma_attr_set & kAttrBit)) {
    cudaFuncSetAttribute(k_attn_mma<DH, KG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    ctx->attn_mma_attr_set |= kAttrBit;
  }
  const float scale_log2e = 1.4426950408889634f / sqrtf((float)DH);
  cs_launch_pdl(k_attn_mma<DH, KG>, dim3(B * c.n_kv_heads, nsplit, rgs), dim3(kThreads), smem, st, ctx->qbuf,
                static_cast<const __nv_bfloat16*>(kv_cache), ctx->row_lim, ctx->kv_len_early, layer, R, c.n_heads, c.n_kv_heads,
                c.max_batch, c.max_seq, nsplit, scale_log2e, ctx->attn_o, ctx->attn_ml, B * R,
                cs_next_stamp(ctx, CS_FAM_ATTENTION));
  return nsplit;
}

// up to 32 query rows per KV head leave warps without rows: they share the keys of the tiles instead
template <int DH>
int launch(cs_ctx* ctx, const void* kv_cache, int layer, int B, int R, cudaStream_t st) {
  const int nq = ctx->cfg.n_heads / ctx->cfg.n_kv_heads * R;
  return nq <= 16 ? launch_groups<DH, 4>(ctx, kv_cache, layer, B, R, st)
       : nq <= 32 ? launch_groups<DH, 2>(ctx, kv_cache, layer, B, R, st) : launch_groups<DH, 1>(ctx, kv_cache, layer, B, R, st);
}

}  // namespace

int cs_launch_attention(cs_ctx* ctx, const void* kv_cache, int layer, int B, int R, bool merge, cudaStream_t st) {
  // head_dim 128 runs on the tcgen05 kernels.  The one with the query rows as M does a tile's work of
  // 128 rows whatever the block holds, but has the shorter chain; the one with keys and head dims as M does
  // only that of the real rows, and takes blocks of up to 48 rows per KV head whose CTAs walk many tiles.
  // Whole layers, rows as M / keys as M, us, with caches that are full - 44 rows: 9 tiles 139.8 / 140.2, 14 tiles 147.0 / 145.8, 20 tiles 155.8 /
  // 152.0 (4 sequences); 28 rows: 9 tiles 140.3 / 141.5, 20 tiles 155.5 / 153.2 (8); 16 rows: 5 tiles 115.2 / 114.5, 9 tiles 120.4 / 118.3, 20 tiles
  // 135.5 / 130.8 (4); 84 rows, 65 tiles, attention and merge alone: 120.2 / 173.9.  Full caches would gain from 7 tiles on with up to 16 rows
  // and from 13 with up to 48, by 1 - 2 %.  But tiles are counted from the cache's size, and where it is mostly empty the second
  // kernel's start, 2 - 4 us slower, is what counts: 44 rows over 500 or 4,000 keys in a cache of 40,000 106.6 / 110.5 and 108.4 / 112.5, 16 rows over
  // 300 of 4,600 117.3 / 118.6; so the line stays where the walk is long.  The register-resident mma.sync kernel takes the other head sizes.
  // CS_ATTN_KERNEL=tc|tcw|mma, read when the context is created, forces one of them (tests run
  // them on the same inputs).
  int nsplit = 0;
  if (ctx->attn_force != 1) {
    const bool wide = ctx->attn_force == 3 || (ctx->attn_force == 0 && cs_attention_tc_tiles_per_cta(ctx, B, R) > 20 &&
                                               ctx->cfg.n_heads / ctx->cfg.n_kv_heads * R <= 48);
    if (wide) nsplit = cs_launch_attention_tcw(ctx, kv_cache, layer, B, R, &merge, st);
    if (nsplit == 0) nsplit = cs_launch_attention_tc(ctx, kv_cache, layer, B, R, &merge, st);
  }
  if (nsplit <= 0)
    switch (ctx->cfg.head_dim) {
      case 32: nsplit = launch<32>(ctx, kv_cache, layer, B, R, st); break;
      case 64: nsplit = launch<64>(ctx, kv_cache, layer, B, R, st); break;
      default: nsplit = launch<128>(ctx, kv_cache, layer, B, R, st); break;
    }
  if (merge) cs_launch_attn_merge(ctx, nsplit, B * R, st);
  return nsplit;
}
