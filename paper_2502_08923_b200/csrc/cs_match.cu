// Suffix-match search and draft gather (Sec. 3.1, 3.2; App. B.3 step 1).
//
// One thread-block cluster per sequence.  The CTAs of a cluster split the candidate
// start positions [0, n - 2*gamma] between them; each thread tests four consecutive
// candidates at a time, four such groups from loads that are in flight together, the best position is reduced by
// warp vote / shared-memory atomics inside the CTA and sent to the first CTA of the cluster, which
// copies the draft.
// No global scratch memory, no global atomics, one launch, deterministic.
//
// Bound by a chain of latencies: length, tokens (through L2), cluster barrier, draft.  Launched back to back, us a search, with a load waited
// for per group of candidates, two barriers of the whole cluster behind them and rows off 16 bytes read token by token / now: 1 x 4,097 tokens 3.03 /
// 2.31, 1 x 32,768 3.76 / 2.81, 8 x 5,003 6.13 / 2.74, 64 x 1,003 3.77 / 2.86, 32 x 20,002 6.95 / 4.0, 64 x 30,001 10.0 / 5.1, 64 x 32,768
// 7.4 / 5.1, 64 x 131,072 18.2 / 10.6.  (The second four tokens of a thread from its neighbour by shuffles, half of the loads: 5.95 and
// 13.5 for the last two, where the present loads took 5.5 and 12.)
#include <limits.h>

#include "cs_common.cuh"

namespace {

constexpr int kThreads = 256, kMaxCluster = 8;

// The history is read through L2 only: this kernel may be resident while the step before still appends to
// it, and neither the read-only path nor L1 is coherent across that.
__device__ __forceinline__ int4 ld_int4(const int* p) { return __ldcg(reinterpret_cast<const int4*>(p)); }
// The cluster's barrier (warps arrive whole): a first phase, which everyone passes before anyone writes to another CTA's shared memory, says
// that all of them run; a second, at which only the first CTA waits, that the best positions are there.
__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
constexpr int kGroups = 4;             // groups of candidates whose tokens a thread has in flight

// Four CTAs an SM: 60 registers.  (72, as the compiler would have it, leave three: 64 x 32,768 tokens back to back 5.1 -> 6.7 us.  The keys are loaded where
// they are used; ahead of that branch all eight took the registers that the tokens in flight need: 5.5.)
__global__ void __launch_bounds__(kThreads, 4)
k_find_match(const int* hist, const int* hist_len, int stride, int gamma,
             int k, int policy, int* __restrict__ match_pos, int* __restrict__ draft,
             int* __restrict__ draft_len, int* __restrict__ last_tok,
             const int* skip, unsigned long long* stamp) {
  cluster_arrive();
  CS_PDL_PROLOGUE();
  uint32_t rank_u, nblk_u;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank_u));
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(nblk_u));
  const int b = blockIdx.y, rank = (int)rank_u, nblk = (int)nblk_u, tid = threadIdx.x, lane = tid & 31;
  __shared__ int s_best;
  __shared__ int s_all[kMaxCluster];   // first CTA: the best position of every CTA

  const int* h = hist + (size_t)b * stride;
  int n = __ldcg(hist_len + b);
  if (n > stride) n = stride;
  if (n < 0) n = 0;
  const bool dead = (skip != nullptr && __ldcg(skip + b) != 0);
  const int n_cand = dead ? 0 : n - 2 * gamma + 1;   // candidates p0 = 0 .. n - 2*gamma
  const bool latest = (policy == CS_MATCH_LATEST);
  const int none = latest ? -1 : INT_MAX;

  if (tid == 0) s_best = none;
  __syncthreads();

  int best = none;
  if (n_cand > 0) {
    // This CTA's candidates are lo .. hi - 1 (none where lo = hi; unsigned, as lo + per may pass 2^31 in the longest rows).  From here on positions count
    // from `first`, where the loads begin: c0 .. c1 - 1, and nothing that is added to them comes near 2^31.
    const int log_nblk = __ffs(nblk) - 1;                // (a power of two)
    const unsigned per = ((((unsigned)n_cand + nblk_u - 1) >> log_nblk) + 3) & ~3u;
    const unsigned lo = min(rank_u * per, (unsigned)n_cand), hi = min(lo + per, (unsigned)n_cand);
    // Four tokens at a time begin on 16 bytes, `off` tokens ahead of the row where a row does not.
    const bool vec_ok = gamma <= 5;
    const unsigned off = vec_ok ? (unsigned)(reinterpret_cast<uintptr_t>(h) >> 2 & 3) : 0u;
    const int first = (int)((lo + off) & ~3u) - (int)off, c0 = (int)lo - first, c1 = (int)hi - first;
    const int* hs = h + first;
    if (vec_ok) {
      int key[5];
#pragma unroll
      for (int j = 0; j < 5; ++j) key[j] = j < gamma ? __ldcg(h + n - gamma + j) : -1;
      // Candidates whose eight tokens lie in the caller's rows: w0 .. w1 - 1.  The others, at the rows' very ends, are looked at token by token.
      const int room = c1 + min(stride - (int)hi, 8) + (b + 1 < (int)gridDim.y ? min(stride, 8) : 0);   // tokens from `first` on, as far as they matter
      const int w0 = first < 0 && (b == 0 || stride < 3) ? min(4, c1) : c0, w1 = max(w0, min(c1, room < 8 ? 0 : (room - 4) & ~3));
      auto test = [&](const int4& u, const int4& v, int s) {
        // tokens s .. s+7 cover candidates s .. s+3 for gamma <= 5; what lies ahead of the row or past the
        // accepted length only feeds candidates that are masked off
        const int t[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          bool eq = (unsigned)(s + i - w0) < (unsigned)(w1 - w0);
#pragma unroll
          for (int j = 0; j < 5; ++j)
            if (j < gamma) eq = eq && (t[i + j] == key[j]);
          if (eq) best = latest ? max(best, s + i) : min(best, s + i);
        }
      };
      const int e = tid - (kThreads - 32), p = e < w0 - c0 ? c0 + e : w1 + e - (w0 - c0);   // (ten at most; the last warp has the least else to do)
      if (e >= 0 && p < c1) {
        bool eq = true;
#pragma unroll
        for (int j = 0; j < 5; ++j)
          if (j < gamma) eq = eq & (__ldcg(hs + p + j) == key[j]);
        if (eq) best = latest ? max(best, p) : min(best, p);
      }
      for (int base = w0 < w1 ? w0 & ~3 : w1; base < w1; base += kGroups * kThreads * 4) {
        int4 u[kGroups], v[kGroups];
#pragma unroll
        for (int q = 0; q < kGroups; ++q) {
          const int s = base + (q * kThreads + tid) * 4;
          if (s < w1) {
            u[q] = ld_int4(hs + s);
            v[q] = ld_int4(hs + s + 4);
          }
        }
#pragma unroll
        for (int q = 0; q < kGroups; ++q) {
          if (base + q * kThreads * 4 >= w1) break;      // (short shares end in the first group)
          test(u[q], v[q], base + (q * kThreads + tid) * 4);
        }
      }
    } else {
      int key[CS_MAX_GAMMA];
#pragma unroll
      for (int j = 0; j < CS_MAX_GAMMA; ++j) key[j] = j < gamma ? __ldcg(h + n - gamma + j) : -1;
      for (int s = tid * 4; s < c1; s += kThreads * 4)
        for (int i = 0; i < 4 && s + i < c1; ++i) {
          bool eq = true;
          for (int j = 0; j < gamma; ++j) eq = eq && (__ldcg(hs + s + i + j) == key[j]);
          if (eq) best = latest ? max(best, s + i) : min(best, s + i);
        }
    }
    if (best != none) best += first;
  }
  // warp vote, then one shared-memory atomic per warp
  best = latest ? __reduce_max_sync(0xffffffffu, best) : __reduce_min_sync(0xffffffffu, best);
  if (lane == 0 && best != none) {
    if (latest) atomicMax(&s_best, best); else atomicMin(&s_best, best);
  }
  __syncthreads();
  cluster_wait();
  if (tid == 0) {
    uint32_t to;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(to) : "r"((uint32_t)__cvta_generic_to_shared(s_all + rank)));
    asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(to), "r"(s_best) : "memory");
  }
  cluster_arrive();
  if (rank != 0) return;
  cluster_wait();
  int p0 = none;
  for (int r = 0; r < nblk; ++r) p0 = latest ? max(p0, s_all[r]) : min(p0, s_all[r]);
  if (p0 == INT_MAX) p0 = -1;
  const int start = p0 + gamma;
  const int len = (p0 < 0) ? 0 : min(k, n - start);
  if (tid == 0) {
    match_pos[b] = p0;
    draft_len[b] = len;
    if (last_tok != nullptr) last_tok[b] = (n > 0) ? __ldcg(h + n - 1) : 0;
  }
  for (int i = tid; i < k; i += kThreads) draft[(size_t)b * k + i] = (i < len) ? __ldcg(h + start + i) : -1;
  if (stamp != nullptr) {
    __syncthreads();
    if (tid == 0) cs_stamp_end(stamp);
  }
}

}  // namespace

cs_status cs_launch_find_match(const int32_t* hist, const int32_t* hist_len, int B, int stride,
                               int gamma, int k, int policy, int32_t* match_pos, int32_t* draft,
                               int32_t* draft_len, int32_t* last_tok, const int32_t* skip,
                               cudaStream_t st, unsigned long long* stamp) {
  // no entry point reaches the kernel with a key longer than its compare loop or an unknown policy
  if (gamma < 1 || gamma > CS_MAX_GAMMA || (policy != CS_MATCH_LATEST && policy != CS_MATCH_FIRST) || k < 0 || B < 0)
    return CS_ERR_ARG;
  if (B == 0) return CS_OK;
  // 4,096 candidates are one round of a CTA's loads in flight: short histories use a single CTA per
  // sequence, and only rows of more than 8 x 4,096 tokens take further rounds
  int cl = 1;
  while (cl < kMaxCluster && stride > cl * 4096) cl *= 2;
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(cl, B, 1);
  lc.blockDim = dim3(kThreads, 1, 1);
  lc.dynamicSmemBytes = 0;
  lc.stream = st;
  cudaLaunchAttribute at[2];
  // Launched early like the kernels behind it.  (When a call's host side took longer than the search: a search call 12.0 -> 10.9 us; a step of a small
  // model launch by launch 90 -> 87.)
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cl;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  lc.attrs = at;
  lc.numAttrs = 2;
  cudaError_t e = cudaLaunchKernelEx(&lc, k_find_match, (const int*)hist, (const int*)hist_len,
                                     stride, gamma, k, policy, (int*)match_pos, (int*)draft,
                                     (int*)draft_len, (int*)last_tok, (const int*)skip, stamp);
  return e == cudaSuccess ? CS_OK : CS_ERR_CUDA;
}
