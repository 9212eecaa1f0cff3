// C2R / Top-K routing, collaboration matrix, Top-T sets and dispatch volume; entry point of the gate logits, whose kernels are
// in gate_tc.cu and gemm_simt.cu.
// Integer outputs are exact and independent of scheduling (integer atomics only where the
// result does not depend on their order).
#include "c2r_common.cuh"
#include "gemm.h"

namespace c2r {

thread_local int g_last_cuda_error = 0;
unsigned long long g_launch_count = 0;

// ---------------------------------------------------------------------------------------------
// Routing (Sec. 3.3 step 2).  LANES threads per token hold its logits in registers, PER each, as order-preserving integer
// keys; K rounds, each a maximum and then the lowest index that has it under the total order (value desc, index asc), after
// the first among the experts of the top-1 expert's collaborator mask.  The number of blocks is fixed by the dispatch's blocking,
// at most one per SM up to 148 blocks, so up to there a block's latency is what the kernel takes: a thread per token over keys staged
// in shared memory waits for 60 dependent selects a round, here it is PER and two reductions of log2(LANES) shuffles.  With more
// blocks the kernel is bound by instructions, of which few threads with many experts each, and PER cut to E, need the fewest.
// us a call, a thread per token / always eight experts a thread / this: 16384 tokens of 60 experts, top-8 12.5 / 6.8 / 6.9; 40000, top-4
// 13.5 / 11.0 / 10.3; 65536 12.9 / 14.2 / 13.5; 262144 39.1 / 46.7 / 41.2; 48 experts, top-4, 131072 19.5 / 23.8 / 16.4; 24 experts
// 11.3 / 12.9 / 9.1; with p, 24000 tokens of 60, top-4 11.7 / 12.6 / 10.6, 131072 47 / 36 / 35.  Behind a pair GEMM (4096 tokens) 24 / 6, as its
// blocks spread.
// ---------------------------------------------------------------------------------------------
// Order-preserving map of a logit to an unsigned key above 0 (-0 and +0 share one, as they compare equal); 0 marks an
// expert that is not a candidate.
__device__ __forceinline__ uint32_t logit_key(float v) {
  const uint32_t u = __float_as_uint(v + 0.0f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_logit(uint32_t k) { return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k); }

// A block owns tokens_per_block consecutive tokens (the blocking of the dispatch's counting sort).  block_counts (optional):
// [blocks][E] experts' slot counts of the block's tokens -- the histogram the dispatch starts from, so it need not read
// idx again to build it.
//
// Lane l of a token's LANES holds experts 4 l .. 4 l + 3, as many from 4 LANES on, and so forth, PER in all: E <= PER LANES.  BITS:
// those that may not be chosen again are taken out by a bit each, ahead of the next round's maximum, and not by a compare of each with
// the choice (compares / bits, 262144 tokens: 60 experts, top-8 65.7 / 63.9, 24 experts 31.6 / 27.6; with eight a thread 16 experts
// 21.7 / 20.9 at top-8 but 16.1 / 17.1 at top-6).  FULL: the softmax over all experts is wanted, for p or for weights that are not renormalised.
template <int K, int LANES, int PER, bool FULL>
__global__ void __launch_bounds__(FULL ? 512 : 1024) route_kernel(const float* __restrict__ L, const uint64_t* __restrict__ mask,
                                                     int32_t* __restrict__ idx, float* __restrict__ w, float* __restrict__ p,
                                                     int32_t* __restrict__ status, int N, int E, int renorm, int tokens_per_block,
                                                     int32_t* __restrict__ block_counts) {
  chain_begin();
  __shared__ uint64_t s_mask[64];
  __shared__ int s_cnt[64];
  constexpr bool BITS = PER > 8;
  constexpr int OWN = (K + LANES - 1) / LANES;  // selections a lane keeps: j = sub, sub + LANES, ..
  const int tid = threadIdx.x, sub = tid & (LANES - 1);
  const int t_begin = blockIdx.x * tokens_per_block, tokens = min(N - t_begin, tokens_per_block);
  const bool vec = (E & 3) == 0 && ((uintptr_t)L & 15u) == 0;
  int flags = 0;
  auto expert = [&](int i) { return 4 * sub + (i & 3) + (i >> 2) * 4 * LANES; };
  auto load = [&](int t, float (&v)[PER]) {
    const float* row = L + (size_t)(t_begin + min(t, tokens - 1)) * E;
    if (vec) {
#pragma unroll
      for (int h = 0; h < PER / 4; ++h) {
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (expert(4 * h) < E) x = *reinterpret_cast<const float4*>(row + expert(4 * h));
        v[4 * h] = x.x; v[4 * h + 1] = x.y; v[4 * h + 2] = x.z; v[4 * h + 3] = x.w;
      }
    } else {
#pragma unroll
      for (int i = 0; i < PER; ++i) v[i] = expert(i) < E ? row[expert(i)] : 0.f;
    }
  };
  const int per_pass = blockDim.x / LANES, t_warp = tid / 32 * (32 / LANES), t_lane = (tid & 31) / LANES;
  float next[PER];
  load(t_warp + t_lane, next);
  if (tid < 64) {
    s_cnt[tid] = 0;
    s_mask[tid] = (tid < E && mask != nullptr) ? mask[tid] : ~0ull;
  }
  __syncthreads();
  for (int t0 = t_warp; t0 < tokens; t0 += per_pass) {  // warp-uniform
    const int t = t0 + t_lane;
    const bool live = t < tokens;
    uint32_t key[PER], avail = ~0u;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      float v = next[i];
      if (v != v) { v = -INFINITY; if (live) flags |= C2R_STATUS_NAN_LOGIT; }
      key[i] = expert(i) < E ? logit_key(v) : 0u;
    }
    if (t0 + per_pass < tokens) load(t + per_pass, next);
    float ex[FULL ? PER : 1], top = 0.f, lg[OWN];
    int own[OWN];
    uint64_t chosen = 0;
#pragma unroll
    for (int j = 0; j < K; ++j) {
      uint32_t best[4] = {0u, 0u, 0u, 0u};
#pragma unroll
      for (int i = 0; i < PER; ++i) {
        if (BITS && j > 0) key[i] = (avail >> i & 1u) ? key[i] : 0u;
        best[i & 3] = max(best[i & 3], key[i]);
      }
      uint32_t m = max(max(best[0], best[1]), max(best[2], best[3]));
#pragma unroll
      for (int o = LANES / 2; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
      int sel = 64;
#pragma unroll
      for (int i = PER - 1; i >= 0; --i) sel = key[i] == m ? expert(i) : sel;
#pragma unroll
      for (int o = LANES / 2; o > 0; o >>= 1) sel = min(sel, __shfl_xor_sync(0xffffffffu, sel, o));
      if (j == 0) {
        top = key_logit(m);
        if (FULL) {
#pragma unroll
          for (int i = 0; i < PER; ++i) ex[FULL ? i : 0] = expert(i) < E ? expf(key_logit(key[i]) - top) : 0.f;
        }
        const uint64_t set = s_mask[sel];
        avail = 0u;
#pragma unroll
        for (int h = 0; h < PER / 4; ++h) {
          const uint32_t bits = (uint32_t)(set >> ((4 * sub + h * 4 * LANES) & 63));
          if (BITS) avail |= (bits & 15u) << (4 * h);
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (!BITS) key[4 * h + i] = (bits >> i & 1u) ? key[4 * h + i] : 0u;
        }
      }
      if (BITS) {
        if ((sel >> 2 & (LANES - 1)) == sub) avail &= ~(1u << ((sel & 3) + 4 * (sel / (4 * LANES))));
      } else {
#pragma unroll
        for (int i = 0; i < PER; ++i) key[i] = expert(i) == sel ? 0u : key[i];
      }
      if (m == 0u) {  // candidate set exhausted: fall back to the lowest unselected expert
        if (live) flags |= C2R_STATUS_SET_TOO_SMALL;
        const uint64_t valid = (E == 64) ? ~0ull : ((1ull << E) - 1ull);
        sel = __ffsll((long long)(valid & ~chosen)) - 1;
      }
      chosen |= 1ull << sel;
      if ((j & (LANES - 1)) == sub) { own[j / LANES] = sel; lg[j / LANES] = m != 0u ? key_logit(m) : -INFINITY; }
    }
    // Eq. 1 weights.  The round-0 logit is the row maximum, so it is the softmax shift for both forms.  Sums are binary trees:
    // over the slot (distances 4, 2, 1), over the expert index (32, 16, 8, 4, 2, 1).
    float denom = 0.f;
    if (renorm) {
      float part[8 / LANES > 0 ? 8 / LANES : 1];
#pragma unroll
      for (int q = 0; q < 8 / LANES; ++q) part[q] = q < OWN && sub + q * LANES < K ? expf(lg[q < OWN ? q : 0] - top) : 0.f;
#pragma unroll
      for (int h = 4 / LANES; h > 0; h >>= 1)
#pragma unroll
        for (int q = 0; q < h; ++q) part[q] += part[q + h];
      denom = part[0];
#pragma unroll
      for (int o = LANES / 2; o > 0; o >>= 1) denom += __shfl_xor_sync(0xffffffffu, denom, o);
    }
    if (FULL) {
      constexpr int PARTS = PER <= 4 ? 1 : PER <= 8 ? 2 : 4;
      static_assert(!FULL || PER <= 16, "the sum's tree over a lane's groups of four");
      float u[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float part[PARTS];
#pragma unroll
        for (int h = 0; h < PARTS; ++h) part[h] = 4 * h < PER ? ex[FULL && 4 * h < PER ? 4 * h + i : 0] : 0.f;
#pragma unroll
        for (int x = PARTS / 2; x > 0; x >>= 1)
#pragma unroll
          for (int h = 0; h < x; ++h) part[h] += part[h + x];
        u[i] = part[0];
#pragma unroll
        for (int o = LANES / 2; o > 0; o >>= 1) u[i] += __shfl_xor_sync(0xffffffffu, u[i], o);
      }
      const float sum = (u[0] + u[2]) + (u[1] + u[3]);
      if (!renorm) denom = sum;
      if (p != nullptr && live) {
        float* out = p + (size_t)(t_begin + t) * E;
        if (vec && ((uintptr_t)p & 15u) == 0) {
#pragma unroll
          for (int h = 0; h < PER / 4; ++h)
            if (expert(4 * h) < E)
              *reinterpret_cast<float4*>(out + expert(4 * h)) =
                  make_float4(ex[FULL ? 4 * h : 0] / sum, ex[FULL ? 4 * h + 1 : 0] / sum, ex[FULL ? 4 * h + 2 : 0] / sum, ex[FULL ? 4 * h + 3 : 0] / sum);
        } else {
#pragma unroll
          for (int i = 0; i < PER; ++i)
            if (expert(i) < E) out[expert(i)] = ex[FULL ? i : 0] / sum;
        }
      }
    }
    if (live) {
      const size_t o = (size_t)(t_begin + t) * K;
#pragma unroll
      for (int q = 0; q < OWN; ++q) {
        const int j = sub + q * LANES;
        if (j < K) {
          idx[o + j] = own[q];
          w[o + j] = expf(lg[q] - top) / denom;
          if (block_counts != nullptr) atomicAdd(&s_cnt[own[q]], 1);  // integer counts: the order does not matter
        }
      }
    }
  }
  if (block_counts != nullptr) {
    __syncthreads();
    if (tid < E) block_counts[(size_t)blockIdx.x * E + tid] = s_cnt[tid];
  }
  if (status != nullptr) {
    flags = __reduce_or_sync(0xffffffffu, flags);
    if (flags && (tid & 31) == 0) atomicOr(status, flags);
  }
}

template <int K, int LANES, int PER, bool FULL>
static int route_launch(const c2r_config* cfg, const float* L, const uint64_t* mask, int32_t* idx, float* w, float* p,
                        int32_t* status, int32_t* block_counts, cudaStream_t s) {
  const int tpb = perm_tokens_per_block(K), most = (cfg->N < tpb ? cfg->N : tpb) * LANES;
  const int blocks = (cfg->N + tpb - 1) / tpb;
  // One block per SM with all its tokens at once; beyond, blocks that fit an SM together; far beyond, blocks that load their next
  // tokens while they rank these (60 experts, top-4, 512 / 256 threads: 65536 tokens 13.5 / 13.8, 90000 16.7 / 16.2, 262144 45.1 / 41.2;
  // with K > 4 a block has 320 threads or 256 anyway, and 320 are the better).
  const int limit = blocks <= SPREAD_SMS ? (FULL ? 512 : 1024) : FULL ? 256 : blocks > 4 * SPREAD_SMS && most > 384 ? 256 : 512;
  const int threads = most > limit ? limit : most < 64 ? 64 : (most + 31) / 32 * 32;  // at least the 64 that handle the mask and the counts
  static int done[64] = {};
  int own = 0;
  const int rc = allow_smem(route_kernel<K, LANES, PER, FULL>, done, SPREAD_SMEM, &own);
  if (rc) return rc;
  C2R_CUDA(launch_chained(route_kernel<K, LANES, PER, FULL>, blocks, threads, spread_smem(blocks, 0, own), s, L, mask, idx, w, p, status, cfg->N, cfg->E,
                          cfg->renorm, tpb, block_counts));
  C2R_LAUNCH_CHECK();
  return C2R_OK;
}
// Threads per token and experts per thread.  Where all of a block's tokens are ranked at once and no SM has a second block, latency
// counts: eight experts a thread (decode of one token 67.9 / 68.7 with sixteen).  Else two threads up to 24 experts and four beyond,
// with as few places as hold E (a place costs as much as an expert: 33 experts in 64 places 46.9 us, in 48 places 31.1, 262144
// tokens, top-4).  25 to 32 experts take four threads until instructions are all that counts (32 experts, four / two: top-4
// 65536 tokens 8.2 / 8.4, 90000 10.1 / 9.4, 262144 27.9 / 22.2, but top-2 131072 9.9 / 10.5; the full softmax is always better off
// with four, top-4 131072 tokens 19.0 / 20.5).
template <int K, bool FULL>
static int route_launch(const c2r_config* cfg, const float* L, const uint64_t* mask, int32_t* idx, float* w, float* p,
                        int32_t* status, int32_t* block_counts, cudaStream_t s) {
  const int tpb = perm_tokens_per_block(K), blocks = (cfg->N + tpb - 1) / tpb;
  const bool many = !FULL && cfg->N > 512 * SPREAD_SMS && blocks > 4 * SPREAD_SMS;
  auto at_once = [&](int lanes) { return blocks <= SPREAD_SMS && (cfg->N < tpb ? cfg->N : tpb) * lanes <= (FULL ? 512 : 1024); };
  const auto launch = cfg->E <= 8                   ? route_launch<K, 2, 4, FULL>
                      : cfg->E <= 16                ? route_launch<K, 2, 8, FULL>
                      : cfg->E <= 24 && !at_once(4) ? route_launch<K, 2, 12, FULL>
                      : cfg->E <= 32 && many        ? route_launch<K, 2, 16, FULL>
                      : cfg->E <= 32                ? route_launch<K, 4, 8, FULL>
                      : at_once(8)                  ? route_launch<K, 8, 8, FULL>
                      : cfg->E <= 48                ? route_launch<K, 4, 12, FULL>
                                                    : route_launch<K, 4, 16, FULL>;
  return launch(cfg, L, mask, idx, w, p, status, block_counts, s);
}
template <int K>
static int route_launch(const c2r_config* cfg, const float* L, const uint64_t* mask, int32_t* idx, float* w, float* p,
                        int32_t* status, int32_t* block_counts, cudaStream_t s) {
  return p != nullptr || !cfg->renorm ? route_launch<K, true>(cfg, L, mask, idx, w, p, status, block_counts, s)
                                      : route_launch<K, false>(cfg, L, mask, idx, w, p, status, block_counts, s);
}

__global__ void route_bwd_kernel(const float* __restrict__ w, const float* __restrict__ dw, float* __restrict__ dl,
                                 int N, int K) {
  chain_begin();
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= N) return;
  float s = 0.f;
  for (int k = 0; k < K; ++k) s = fmaf(w[(size_t)t * K + k], dw[(size_t)t * K + k], s);
  for (int k = 0; k < K; ++k) dl[(size_t)t * K + k] = w[(size_t)t * K + k] * (dw[(size_t)t * K + k] - s);
}

// Backward of the Eq. 1 weights when the experts applied them themselves (row-scaled SwiGLU): the backward
// GEMM left, per permuted row, partial dots whose sum is q = s_r <dH_r, H_r / s_r> = w dL/dw.  With
// S = sum_j q_j:  dl_k = w_k (dw_k - sum_j w_j dw_j) = q_k - w_k S  -- no division by a weight that may be 0.
// dw (optional, informational) = q_k / w_k where w_k > 0.  Shared expert: q_s = g dL/dg, dz = q_s (1 - g).
// Partials are added in index order.
constexpr int RBS_TOKENS = 64;  // tokens per block; one thread per slot
__global__ void __launch_bounds__(RBS_TOKENS * 8) route_bwd_scaled_kernel(const float* __restrict__ w,
                                                                          const int32_t* __restrict__ row_of_slot,
                                                                          const float* __restrict__ qpart, int nq,
                                                                          long long R, const float* __restrict__ z,
                                                                          const float* __restrict__ qspart, int nqs,
                                                                          float* __restrict__ dw, float* __restrict__ dl,
                                                                          float* __restrict__ dz, int N, int K) {
  chain_begin();
  __shared__ float s_q[RBS_TOKENS * 8];
  const int lt = threadIdx.x / K, k = threadIdx.x - lt * K;  // token of the block, slot of the token
  const int t = blockIdx.x * RBS_TOKENS + lt;
  float q = 0.f;
  if (t < N) {
    const long long row = row_of_slot[(size_t)t * K + k];
    for (int j = 0; j < nq; ++j) q += qpart[(long long)j * R + row];
  }
  s_q[threadIdx.x] = q;
  __syncthreads();
  if (t >= N) return;
  float S = 0.f;
  for (int j = 0; j < K; ++j) S += s_q[lt * K + j];  // slot order
  const float wk = w[(size_t)t * K + k];
  dl[(size_t)t * K + k] = q - wk * S;
  if (dw != nullptr) dw[(size_t)t * K + k] = wk > 0.f ? q / wk : 0.f;
  if (dz != nullptr && k == 0) {
    float acc = 0.f;
    for (int j = 0; j < nqs; ++j) acc += qspart[(long long)j * N + t];
    const float g = 1.0f / (1.0f + expf(-z[t]));
    dz[t] = acc * (1.0f - g);
  }
}

// Up to three arrays of 32-bit words set to a value: a kernel, because a memset between two kernels would end their chain
// (see launch_chained), and one launch instead of three memsets where the arrays are separate.
__global__ void __launch_bounds__(256) fill_words_kernel(uint32_t* __restrict__ a, long long na, uint32_t* __restrict__ b, long long nb,
                                                         uint32_t* __restrict__ c, long long nc, uint32_t value) {
  chain_begin();  // the arrays may still be in use by the kernel before, and the next one relies on this one having waited
  const long long first = (long long)blockIdx.x * blockDim.x + threadIdx.x, step = (long long)gridDim.x * blockDim.x;
  for (long long i = first; i < na; i += step) a[i] = value;
  for (long long i = first; i < nb; i += step) b[i] = value;
  for (long long i = first; i < nc; i += step) c[i] = value;
}

// ---------------------------------------------------------------------------------------------
// Collaboration matrix (Eq. 2): per-block table in shared memory, merged with integer adds.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) collab_count_kernel(const int32_t* __restrict__ idx, long long n_tokens,
                                                           int32_t* __restrict__ C, int E, int K) {
  chain_begin();
  extern __shared__ int32_t tab[];
  for (int i = threadIdx.x; i < E * E; i += blockDim.x) tab[i] = 0;
  __syncthreads();
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n_tokens;
       t += (long long)gridDim.x * blockDim.x) {
    int sel[8];
    for (int k = 0; k < K; ++k) {
      int e = idx[t * K + k];
      sel[k] = min(max(e, 0), E - 1);
    }
    for (int a = 0; a < K; ++a)
      for (int b = 0; b < K; ++b) atomicAdd(&tab[sel[a] * E + sel[b]], 1);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < E * E; i += blockDim.x)
    if (tab[i]) atomicAdd(&C[i], tab[i]);
}

// Top-T sets (Eq. 4): one warp per row; T rounds of arg-max under (count desc, index asc), self excluded.
__global__ void collab_sets_kernel(const int32_t* __restrict__ C, int32_t* __restrict__ I_T,
                                   uint64_t* __restrict__ mask, int E, int T) {
  chain_begin();
  const int lane = threadIdx.x & 31;
  const int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (i >= E) return;
  // key = count + 1, 0 marks "not a candidate" (itself, or a negative count, which cannot occur)
  const int n0 = (lane < E && lane != i) ? C[i * E + lane] : -1, n1 = (lane + 32 < E && lane + 32 != i) ? C[i * E + lane + 32] : -1;
  uint32_t c0 = n0 < 0 ? 0u : (uint32_t)n0 + 1u, c1 = n1 < 0 ? 0u : (uint32_t)n1 + 1u;
  uint64_t m = 0;
  int mine0 = 0, mine1 = 0;  // lane l keeps the members picked in rounds l and l + 32
  for (int r = 0; r < T; ++r) {
    const uint32_t best = __reduce_max_sync(0xffffffffu, max(c0, c1));
    const uint32_t at0 = __ballot_sync(0xffffffffu, c0 == best), at1 = __ballot_sync(0xffffffffu, c1 == best);
    const int bi = best == 0u ? 1 << 20 : at0 ? __ffs(at0) - 1 : 31 + __ffs(at1);
    if (bi == lane) c0 = 0u;
    if (bi == lane + 32) c1 = 0u;
    m |= 1ull << (bi & 63);
    if (r == lane) mine0 = bi;
    if (r == lane + 32) mine1 = bi;
  }
  if (lane < T) I_T[i * T + lane] = mine0;
  if (lane + 32 < T) I_T[i * T + lane + 32] = mine1;
  if (lane == 0) mask[i] = m;
}

// Collaboration degree (Eq. 3): P_i = - sum_{j != i} p_ij ln p_ij with p_ij = c_ij / sum_{j != i} c_ij
// (a row without co-activations gives 0; 0 ln 0 = 0).  One block; a warp per row, lanes over the
// columns, and a fixed-order sum over rows for the layer mean.
__global__ void __launch_bounds__(1024) collab_degree_kernel(const int32_t* __restrict__ C, float* __restrict__ degree,
                                                             float* __restrict__ mean, int E) {
  chain_begin();
  __shared__ float s_deg[64];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = warp; i < E; i += 32) {
    float c0 = (lane < E && lane != i) ? (float)max(C[i * E + lane], 0) : 0.f;
    float c1 = (lane + 32 < E && lane + 32 != i) ? (float)max(C[i * E + lane + 32], 0) : 0.f;
    float tot = c0 + c1;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, off);
    float h = 0.f;
    if (tot > 0.f) {
      const float p0 = c0 / tot, p1 = c1 / tot;
      if (p0 > 0.f) h -= p0 * logf(p0);
      if (p1 > 0.f) h -= p1 * logf(p1);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) h += __shfl_xor_sync(0xffffffffu, h, off);
    if (lane == 0) { s_deg[i] = h; degree[i] = h; }
  }
  __syncthreads();
  if (threadIdx.x == 0 && mean != nullptr) {
    float m = 0.f;
    for (int i = 0; i < E; ++i) m += s_deg[i];
    *mean = m / (float)E;
  }
}

// ---------------------------------------------------------------------------------------------
// Dispatch volume (Sec. 3.4 / 4.1): distinct (token, partition) pairs vs (token, expert) pairs.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) dispatch_volume_kernel(const int32_t* __restrict__ idx,
                                                              const int32_t* __restrict__ part,
                                                              unsigned long long* __restrict__ totals,
                                                              unsigned long long* __restrict__ send_naive,
                                                              unsigned long long* __restrict__ send_dedup, int N,
                                                              int E, int K, int P) {
  chain_begin();
  extern __shared__ uint32_t sm[];
  uint32_t* s_naive = sm;           // [P*P]
  uint32_t* s_dedup = sm + P * P;   // [P*P]
  uint32_t* s_part = sm + 2 * P * P;  // [E]
  for (int i = threadIdx.x; i < 2 * P * P; i += blockDim.x) sm[i] = 0;
  for (int i = threadIdx.x; i < E; i += blockDim.x) s_part[i] = (uint32_t)min(max(part[i], 0), P - 1);
  __syncthreads();
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < N; t += (long long)gridDim.x * blockDim.x) {
    const int home = (int)((t * P) / N);
    uint64_t seen = 0;
    for (int k = 0; k < K; ++k) {
      int e = min(max(idx[t * K + k], 0), E - 1);
      int q = s_part[e];
      atomicAdd(&s_naive[home * P + q], 1u);
      if (!((seen >> q) & 1ull)) {
        seen |= 1ull << q;
        atomicAdd(&s_dedup[home * P + q], 1u);
      }
    }
  }
  __syncthreads();
  unsigned long long tn = 0, td = 0, tnx = 0, tdx = 0;
  for (int i = threadIdx.x; i < P * P; i += blockDim.x) {
    uint32_t a = s_naive[i], b = s_dedup[i];
    if (a) atomicAdd(&send_naive[i], (unsigned long long)a);
    if (b) atomicAdd(&send_dedup[i], (unsigned long long)b);
    tn += a; td += b;
    if (i / P != i % P) { tnx += a; tdx += b; }
  }
  if (tn) atomicAdd(&totals[0], tn);
  if (td) atomicAdd(&totals[1], td);
  if (tnx) atomicAdd(&totals[2], tnx);
  if (tdx) atomicAdd(&totals[3], tdx);
}

}  // namespace c2r

using namespace c2r;

int c2r::fill_words(uint32_t* a, int64_t na, uint32_t* b, int64_t nb, uint32_t* c, int64_t nc, uint32_t value, cudaStream_t s) {
  const int64_t most = na > nb ? (na > nc ? na : nc) : (nb > nc ? nb : nc);
  if (most <= 0) return C2R_OK;
  const int blocks = (int)(most > 592 * 1024 ? 592 : (most + 1023) / 1024);
  C2R_CUDA(launch_chained(fill_words_kernel, blocks, 256, 0, s, a, na, b, nb, c, nc, value));
  C2R_LAUNCH_CHECK();
  return C2R_OK;
}

extern "C" int c2r_last_cuda_error(void) { return g_last_cuda_error; }

extern "C" uint64_t c2r_launch_count(void) { return __atomic_load_n(&g_launch_count, __ATOMIC_RELAXED); }

int c2r::gate_logits_impl(const c2r_config* cfg, const void* X, const void* Wg, const void* wsg, float* L, float* z,
                          int32_t* status, void* stream) {
  int rc = check_config(cfg);
  if (rc) return rc;
  C2R_REQUIRE(X && Wg && L, C2R_ERR_INVALID_ARG);
  C2R_REQUIRE(!wsg || z, C2R_ERR_INVALID_ARG);
  C2R_REQUIRE(cfg->E + (wsg ? 1 : 0) <= 64, C2R_ERR_UNSUPPORTED_SHAPE);
  if (cfg->N == 0) return C2R_OK;
  const bool aligned = (((uintptr_t)X | (uintptr_t)Wg | (uintptr_t)wsg | (uintptr_t)L) & 15u) == 0;
  if (aligned && gate_tc_supported(cfg)) return gate_tc_launch(cfg, X, Wg, wsg, L, z, status, as_stream(stream));
  return cfg->dtype == C2R_BF16 ? simt_gate_logits<__nv_bfloat16>(cfg, X, Wg, wsg, L, z, as_stream(stream))
                                : simt_gate_logits<float>(cfg, X, Wg, wsg, L, z, as_stream(stream));
}

extern "C" int c2r_gate_logits(const c2r_config* cfg, const void* X, const void* Wg, const void* wsg, float* L,
                               float* z, void* stream) {
  return gate_logits_impl(cfg, X, Wg, wsg, L, z, nullptr, stream);
}

int c2r::route_impl(const c2r_config* cfg, const float* L, const uint64_t* mask, int32_t* idx, float* w, float* p,
                    int32_t* status, int32_t* block_counts, void* stream) {
  int rc = check_config(cfg);
  if (rc) return rc;
  C2R_REQUIRE(L && idx && w, C2R_ERR_INVALID_ARG);
  if (mask) C2R_REQUIRE(cfg->T >= cfg->K - 1 && cfg->T <= cfg->E - 1, C2R_ERR_INVALID_ARG);
  if (cfg->N == 0) return C2R_OK;
  cudaStream_t s = as_stream(stream);
  switch (cfg->K) {
    case 1: return route_launch<1>(cfg, L, mask, idx, w, p, status, block_counts, s);
    case 2: return route_launch<2>(cfg, L, mask, idx, w, p, status, block_counts, s);
    case 3: return route_launch<3>(cfg, L, mask, idx, w, p, status, block_counts, s);
    case 4: return route_launch<4>(cfg, L, mask, idx, w, p, status, block_counts, s);
    case 5: return route_launch<5>(cfg, L, mask, idx, w, p, status, block_counts, s);
    case 6: return route_launch<6>(cfg, L, mask, idx, w, p, status, block_counts, s);
    case 7: return route_launch<7>(cfg, L, mask, idx, w, p, status, block_counts, s);
    default: return route_launch<8>(cfg, L, mask, idx, w, p, status, block_counts, s);
  }
}

extern "C" int c2r_route(const c2r_config* cfg, const float* L, const uint64_t* mask, int32_t* idx, float* w, float* p,
                         int32_t* status, void* permute_ws, void* stream) {
  return route_impl(cfg, L, mask, idx, w, p, status, (int32_t*)permute_ws, stream);
}

extern "C" int c2r_route_bwd_scaled(const c2r_config* cfg, const float* w, const int32_t* row_of_slot, const float* qpart,
                                    int nq, const float* z, const float* qspart, int nqs, float* dw, float* dl, float* dz,
                                    void* stream) {
  int rc = check_config(cfg);
  if (rc) return rc;
  C2R_REQUIRE(w && row_of_slot && qpart && dl && nq >= 0, C2R_ERR_INVALID_ARG);
  C2R_REQUIRE(!dz || (z && qspart && nqs >= 0), C2R_ERR_INVALID_ARG);
  C2R_REQUIRE(cfg->renorm == 1, C2R_ERR_UNSUPPORTED_SHAPE);
  if (cfg->N == 0) return C2R_OK;
  C2R_CUDA(launch_chained(route_bwd_scaled_kernel, (cfg->N + RBS_TOKENS - 1) / RBS_TOKENS, RBS_TOKENS * cfg->K, 0, as_stream(stream), w, row_of_slot, qpart, nq, permuted_rows(cfg),
                          z, qspart, nqs, dw, dl, dz, cfg->N, cfg->K));
  C2R_LAUNCH_CHECK();
  return C2R_OK;
}

extern "C" int c2r_route_bwd(const c2r_config* cfg, const float* w, const float* dw, float* dl, void* stream) {
  int rc = check_config(cfg);
  if (rc) return rc;
  C2R_REQUIRE(w && dw && dl, C2R_ERR_INVALID_ARG);
  C2R_REQUIRE(cfg->renorm == 1, C2R_ERR_UNSUPPORTED_SHAPE);
  if (cfg->N == 0) return C2R_OK;
  C2R_CUDA(launch_chained(route_bwd_kernel, (cfg->N + 255) / 256, 256, 0, as_stream(stream), w, dw, dl, cfg->N, cfg->K));
  C2R_LAUNCH_CHECK();
  return C2R_OK;
}

extern "C" int c2r_collab_count(const c2r_config* cfg, const int32_t* idx, int64_t n_tokens, int32_t* C,
                                int accumulate, void* stream) {
  int rc = check_config(cfg);
  if (rc) return rc;
  C2R_REQUIRE(idx && C && n_tokens >= 0, C2R_ERR_INVALID_ARG);
  const int E = cfg->E;
  if (!accumulate && (rc = fill_words((uint32_t*)C, E * E, nullptr, 0, nullptr, 0, 0u, as_stream(stream)))) return rc;
  if (n_tokens == 0) return C2R_OK;
  int blocks = (int)((n_tokens + 255) / 256);
  if (blocks > 296) blocks = 296;
  C2R_CUDA(launch_chained(collab_count_kernel, blocks, 256, sizeof(int32_t) * E * E, as_stream(stream), idx, (long long)n_tokens, C, E,
                          cfg->K));
  C2R_LAUNCH_CHECK();
  return C2R_OK;
}

extern "C" int c2r_collab_sets(const c2r_config* cfg, const int32_t* C, int32_t* I_T, uint64_t* mask, void* stream) {
  int rc = check_config(cfg);
  if (rc) return rc;
  C2R_REQUIRE(C && I_T && mask, C2R_ERR_INVALID_ARG);
  C2R_REQUIRE(cfg->T >= 0 && cfg->T <= cfg->E - 1, C2R_ERR_INVALID_ARG);
  const int warps = 4;
  C2R_CUDA(launch_chained(collab_sets_kernel, (cfg->E + warps - 1) / warps, warps * 32, 0, as_stream(stream), C, I_T, mask, cfg->E, cfg->T));
  C2R_LAUNCH_CHECK();
  return C2R_OK;
}

extern "C" int c2r_collab_degree(const c2r_config* cfg, const int32_t* C, float* degree, float* mean, void* stream) {
  int rc = check_config(cfg);
  if (rc) return rc;
  C2R_REQUIRE(C && degree, C2R_ERR_INVALID_ARG);
  C2R_CUDA(launch_chained(collab_degree_kernel, 1, 1024, 0, as_stream(stream), C, degree, mean, cfg->E));
  C2R_LAUNCH_CHECK();
  return C2R_OK;
}

extern "C" int c2r_dispatch_volume(const c2r_config* cfg, const int32_t* idx, const int32_t* part, uint64_t* totals,
                                   uint64_t* send_naive, uint64_t* send_dedup, void* stream) {
  int rc = check_config(cfg);
  if (rc) return rc;
  C2R_REQUIRE(idx && part && totals && send_naive && send_dedup, C2R_ERR_INVALID_ARG);
  const int P = cfg->P;
  C2R_REQUIRE(P >= 1 && P <= cfg->E, C2R_ERR_INVALID_ARG);
  cudaStream_t s = as_stream(stream);
  if ((rc = fill_words((uint32_t*)totals, 8, (uint32_t*)send_naive, 2 * P * P, (uint32_t*)send_dedup, 2 * P * P, 0u, s))) return rc;
  if (cfg->N == 0) return C2R_OK;
  int blocks = (cfg->N + 255) / 256;
  if (blocks > 296) blocks = 296;
  size_t smem = sizeof(uint32_t) * (2 * P * P + cfg->E);
  C2R_CUDA(launch_chained(dispatch_volume_kernel, blocks, 256, smem, s, idx, part, (unsigned long long*)totals,
                          (unsigned long long*)send_naive, (unsigned long long*)send_dedup,
                          cfg->N, cfg->E, cfg->K, P));
  C2R_LAUNCH_CHECK();
  return C2R_OK;
}
