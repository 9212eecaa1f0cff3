// Grouped SwiGLU forward (nothing kept for a backward pass) on CTA pairs with the tokens as the N operand, bf16, sm_100a.
//
// tc_gemm_kernel gives an expert whole 256-row tiles: 273 rows (4096 tokens of the Qwen-MoE-shaped layer, top-4 of 60) cost
// two of them, 1.9 times the products that are needed, and a pair MMA cannot do less.  Its N however goes in steps of 32.
// Here 256 weight rows are the M operand of tcgen05.mma.cta_group::2 and a chunk of an expert's tokens, rounded up to 32, is
// the N: the padding is at most 31 rows per expert.  A chunk may have up to RG_NB tokens (two MMAs per 16 k-elements share the
// A operand then), because what bounds a narrow tile is not the tensor core but the weights' way from the L2: per 64
// k-elements an SM fetches 16 KB of weights and 64 bytes per token of the chunk at about 64 bytes a cycle, against 2
// cycles of MMA per token.
//
// Tensor memory: the accumulators of successive units start at column 0 and end at column 511 in turn.  Where two
// neighbours need more than 512 columns together, the epilogue drains the columns that the next unit needs first and
// lets its MMAs begin then.  Units (expert, 256 weight rows, chunk) have unequal cost: experts are taken by falling chunk size and
// dealt out to the pairs forth and back, which evens out the sums without any communication.
//
// Up-projection: the tensor map interleaves 16 gate rows and the 16 up rows of the same channels, so the 32 TMEM lanes that a
// warp may read hold both operands of the SwiGLU, and loads of 16 lanes x 256 bits give a thread both at the same register
// index; 8 x 8 transposes in registers make the channels contiguous.  Down-projection: a lane is an output channel, a
// register a token, so a store writes 128 contiguous bytes.  Neither epilogue uses shared memory, whose bandwidth the MMAs need.
//
// Chunk sizes: one chunk per expert reads the weights once, but leaves pairs idle where units are few, so the blocks estimate the
// pass for eight largest sizes and take the best (us, one size of 384 / chosen: 8 experts of 512, d 1024, 300 rows each 29 / 24, single
// group of 1024 x 2048 with 384 rows 39 / 24; the estimate costs 0.5).  A ring stage is as large as the largest chunk needs.
//
// Measured against pair tiles of 256 tokens (csrc/gemm.h has the sizes at which the lines were drawn), us, whole forward passes: 4096
// tokens of the Qwen-MoE shape 686 -> 634, 1021 of the LLaMA-MoE shape 159 -> 146; the expert call with 273 rows each 405 -> 313.  What
// bounds it there: weights from HBM (1.04 GB, 160 us) and the power cap (SM clock 1.1 GHz in a loop).
//
// Warp roles (320 threads per CTA): warp 0 TMA producer, warp 1 MMA issuer (even CTA) and TMEM owner, warps 2..9 epilogue.
// Waits are bounded like in the other tensor-core kernels.
#include "gemm.h"
#include "tc_common.cuh"

namespace c2r {

constexpr int RG_THREADS = 320;
constexpr int RG_EPI_WARPS = 8;
constexpr int RG_NB = 384;                              // most tokens of a unit
constexpr int RG_A_BYTES = 128 * BK * 2;                // a CTA's share of the weight rows per stage
constexpr int RG_RING = 216 * 1024;                     // as many stages as fit: 5 with chunks of 384 tokens, 12 with 32
constexpr int RG_MAX_STAGES = RG_RING / (RG_A_BYTES + 16 * BK * 2);
constexpr int RG_SMEM = RG_RING + 1024;
constexpr int RG_TMEM = 512;

struct RaggedParams {
  const int32_t* counts;
  const int32_t* offsets;
  const float* row_scale;
  void* out;          // up: H [R, M] bf16; down: [R, M] float
  long long R;
  int scale_kind;
  int nE, M;          // M: output channels per expert (up: I, down: d)
  int kblocks;
  int slices;         // groups of 256 weight rows per expert
  int32_t* status;
};
// Weights: whole blocks of 128 channels and the partial last block (up), or plain rows; rows of X or H in boxes of 128, 64, 32, 16.
struct RaggedMaps {
  CUtensorMap w, w_last, x[4];
};

struct RaggedUnit {
  int expert, slice, row0, rows, nb;  // nb: MMA columns, rows <= nb of them are tokens
};

// Token of a unit that accumulator column c (a multiple of 16) holds.  A pair MMA takes the first half of its columns from the
// even CTA's rows and the second from the odd one's; the CTAs hold nb / 2 rows each, of which the first MMA takes n1 / 2.
__device__ __forceinline__ int ragged_first(int nb) { return nb <= 256 ? nb : (nb / 2 + 31) / 32 * 32; }
__device__ __forceinline__ int ragged_token(int c, int nb, int n1) {
  const int second = c >= n1;
  const int n = second ? nb - n1 : n1, x = second ? c - n1 : c, base = second ? n1 >> 1 : 0;
  return base + (x < (n >> 1) ? x : (nb >> 1) + x - (n >> 1));
}

// Largest chunk sizes the kernel chooses from, the chunk an expert of n rows then gets, and what a unit of it costs per 64
// k-elements in cycles (see the head of the file).
__device__ __forceinline__ int ragged_limit(int i) { return i == 0 ? RG_NB : 288 - 32 * i; }
__device__ __forceinline__ int ragged_chunk(int n, int limit, int& chunks) {
  // In groups of 32 rows.  Approximate quotients do: q = x / y with an error below 2^-21 q is floored, and x = integer - 1/2
  // keeps q at least 1 / (2 y) from an integer; y is at most 12 where q is at most 18750, and q at most 12 where y is that many.
  const float g = (n + 31) >> 5;
  const float by = (limit > 256 && n > limit ? 256 : limit) >> 5;
  const float k = floorf(__fdividef(g + by - 0.5f, by));
  const float nb = k > 0.f ? floorf(__fdividef(g + k - 0.5f, k)) : 0.f;
  chunks = nb > 0.f ? (int)__fdividef(g + nb - 0.5f, nb) : 0;
  return 32 * (int)nb;
}
__device__ __forceinline__ float ragged_cost(int nb) { return 48 + max(2 * nb, 256 + nb); }

__device__ __forceinline__ void ragged_ld_16x256(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
// 8 x 8 transpose of 16-bit elements held as an MMA fragment (thread: row lane / 4, columns 2 (lane % 4) and the next).
__device__ __forceinline__ uint32_t transpose8(uint32_t v) {
  uint32_t r;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(v));
  return r;
}
__device__ __forceinline__ void tma_pair_load_5d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y, int z, int w, int v) {
  asm volatile(
      "cp.async.bulk.tensor.5d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6, %7}], [%2];" ::"r"(
          dst),
      "l"(map), "r"(bar), "r"(x), "r"(y), "r"(z), "r"(w), "r"(v)
      : "memory");
}

template <bool UP>
__global__ void __launch_bounds__(RG_THREADS, 1)
ragged_kernel(const __grid_constant__ RaggedMaps maps, const RaggedParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  __shared__ uint64_t bars[2 * RG_MAX_STAGES + 4];
  __shared__ uint32_t tmem_slot;
  __shared__ int s_abort;
  __shared__ alignas(16) int s_nb[64], s_units[64];
  __shared__ int s_cnt[64], s_off[64], s_order[64], s_first[65];
  __shared__ alignas(16) float s_time[8];
  __shared__ alignas(16) float s_scale[UP ? RG_EPI_WARPS : 1][UP ? RG_NB / 2 : 1];

  const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();  // 0 = the CTA that issues the MMAs
  const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[RG_MAX_STAGES]);
  const uint32_t tfull0 = smem_u32(&bars[2 * RG_MAX_STAGES]), tfree0 = smem_u32(&bars[2 * RG_MAX_STAGES + 2]);
  if (warp == 0) {
    if (lane == 0) s_abort = 0;
    if (lane < RG_MAX_STAGES) { mbar_init(full0 + 8 * lane, 1); mbar_init(empty0 + 8 * lane, 1); }
    if (lane < 2) { mbar_init(tfull0 + 8 * lane, 1); mbar_init(tfree0 + 8 * lane, 2 * RG_EPI_WARPS); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(RG_TMEM)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    chain_release();  // not before: a block of the next kernel must not take the tensor memory this one waits for
  }
  chain_wait();  // before the first access to global memory
  const int pair_id = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  if (warp < 8) {  // each warp estimates the pass for one largest chunk size: whole rounds of units of the mean cost, or the longest unit
    float units = 0.f, cost = 0.f, worst = 0.f;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int e = lane + 32 * h;
      int n = 0, off = 0;
      if (e < p.nE) {
        off = p.offsets[e];
        n = (int)max(0ll, min((long long)p.counts[e], p.R - off));
      }
      if (warp == 0) { s_off[e] = off; s_cnt[e] = n; }
      int chunks;
      const float c = ragged_cost(ragged_chunk(n, ragged_limit(warp), chunks));
      units += chunks;
      cost += chunks * c;
      worst = fmaxf(worst, c);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      units += __shfl_xor_sync(0xffffffffu, units, o);
      cost += __shfl_xor_sync(0xffffffffu, cost, o);
      worst = fmaxf(worst, __shfl_xor_sync(0xffffffffu, worst, o));
    }
    if (lane == 0) s_time[warp] = units > 0.f ? fmaxf(worst, ceilf(__fdividef(units * p.slices, n_pairs)) * __fdividef(cost, units)) : 0.f;
  }
  __syncthreads();
  // from here four threads per expert
  const int my_e = threadIdx.x >> 2, my_sub = threadIdx.x & 3;
  int my_nb = 0, my_units = 0;
  if (my_e < 64) {
    const float4 t0 = *reinterpret_cast<const float4*>(&s_time[0]), t1 = *reinterpret_cast<const float4*>(&s_time[4]);
    const float ts[8] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w};
    int best = 0, chunks;
    float t = ts[0];
#pragma unroll
    for (int i = 1; i < 8; ++i)
      if (ts[i] < 0.95f * t) { t = ts[i]; best = i; }  // smaller chunks only for a clear gain
    my_nb = ragged_chunk(s_cnt[my_e], ragged_limit(best), chunks);
    my_units = chunks * p.slices;
    if (my_sub == 0) { s_nb[my_e] = my_nb; s_units[my_e] = my_units; }
  }
  __syncthreads();
  if (my_e < 64) {  // experts by falling chunk size, and the units before each of them
    int at = 0, first = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int e0 = 16 * i + 4 * my_sub;
      const int4 nb = *reinterpret_cast<const int4*>(&s_nb[e0]), k = *reinterpret_cast<const int4*>(&s_units[e0]);
      const int nbs[4] = {nb.x, nb.y, nb.z, nb.w}, ks[4] = {k.x, k.y, k.z, k.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const bool before = nbs[j] > my_nb || (nbs[j] == my_nb && e0 + j < my_e);
        at += before;
        first += before ? ks[j] : 0;
      }
    }
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
      at += __shfl_xor_sync(0xffffffffu, at, o);
      first += __shfl_xor_sync(0xffffffffu, first, o);
    }
    if (my_sub == 0) {
      s_order[at] = my_e;
      s_first[at] = first;
      if (at == 63) s_first[64] = first + my_units;
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // the peer's barriers are initialised before anything can arrive on them
  tc_fence_after();
  const uint32_t tmem_base = warp_uniform(tmem_slot);
  volatile int* abort_flag = &s_abort;
  const int total = s_first[64];
  const int stage_bytes = warp_uniform(RG_A_BYTES + (s_nb[s_order[0]] >> 1) * BK * 2);  // what the largest chunk needs
  const int stages = min(RG_MAX_STAGES, RG_RING / stage_bytes);

  // The pair's i-th unit.  Chunks of the same weight rows are neighbours: one of them fetches the rows, the others find them in the L2.
  auto unit_at = [&](int i, RaggedUnit& u, int& hint) -> bool {
    const int j = i * n_pairs + ((i & 1) ? n_pairs - 1 - pair_id : pair_id);
    if (j >= total) return false;
    int o = hint;
    while (s_first[o + 1] <= j) ++o;
    hint = o;
    const int e = s_order[o], n = s_cnt[e], nb = s_nb[e];
    const int chunks = (n + nb - 1) / nb, r = j - s_first[o];
    const int slice = r / chunks, c = r - slice * chunks;
    u.expert = warp_uniform(e);
    u.slice = warp_uniform(slice);
    u.row0 = warp_uniform(s_off[e] + c * nb);
    u.rows = warp_uniform(min(nb, n - c * nb));
    u.nb = warp_uniform(nb);
    return true;
  };

  if (warp == 0) {
    const uint32_t full_mma0 = map_to_cta(full0, 0);
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    int hint = 0;
    RaggedUnit u;
    for (int i = 0; ok && unit_at(i, u, hint); ++i) {
      const int half = u.nb >> 1, xrow = u.row0 + half * (int)rank;
      const bool last = UP && u.slice == (p.M >> 7);  // the partial block of 128 channels
      for (int kb = 0; kb < p.kblocks; ++kb) {
        if (!__all_sync(0xffffffffu, mbar_wait(empty0 + 8 * stage, phase ^ 1u, abort_flag))) { ok = false; break; }
        if (elect_one()) {
          if (rank == 0) mbar_expect_tx(full0 + 8 * stage, 2 * (RG_A_BYTES + half * BK * 2));
          const uint32_t fb = full_mma0 + 8 * stage;
          const uint32_t sa = smem_base + stage * stage_bytes;
          uint32_t sx = sa + RG_A_BYTES;
          if (UP)
            tma_pair_load_5d(sa, last ? &maps.w_last : &maps.w, fb, kb * BK, 0, 0, 16 * u.slice + 4 * (int)rank, u.expert);
          else
            tma_pair_load_3d(sa, &maps.w, fb, kb * BK, 256 * u.slice + 128 * (int)rank, u.expert);
          int row = xrow;
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            const int rows = 128 >> b;
            if (half & rows) {
              tma_pair_load_2d(sx, &maps.x[b], fb, kb * BK, row);
              sx += rows * BK * 2;
              row += rows;
            }
          }
        }
        __syncwarp();
        if (++stage == stages) { stage = 0; phase ^= 1u; }
      }
    }
    if (!ok && lane == 0) { *abort_flag = 1; if (p.status) atomicOr(p.status, C2R_STATUS_WAIT_TIMEOUT); }
  } else if (warp == 1) {
    if (rank == 0) {
      int stage = 0;
    uint32_t phase = 0;
      bool ok = true;
      int hint = 0;
      RaggedUnit u;
      for (int i = 0; ok && unit_at(i, u, hint); ++i) {
        if (i > 0 && !__all_sync(0xffffffffu, mbar_wait(tfree0 + 8 * ((i - 1) & 1), ((i - 1) >> 1) & 1, abort_flag))) { ok = false; break; }
        tc_fence_after();
        const int n1 = ragged_first(u.nb), n2 = u.nb - n1;
        const uint32_t d_tmem = tmem_base + ((i & 1) ? RG_TMEM - u.nb : 0);
        const uint32_t idesc1 = instr_desc_pair(n1, false, false), idesc2 = instr_desc_pair(n2, false, false);
        for (int kb = 0; kb < p.kblocks; ++kb) {
          if (!__all_sync(0xffffffffu, mbar_wait(full0 + 8 * stage, phase, abort_flag))) { ok = false; break; }
          tc_fence_after();
          const uint32_t sa = smem_base + stage * stage_bytes, sx = sa + RG_A_BYTES, sx2 = sx + (n1 >> 1) * BK * 2;
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < BK / UMMA_K; ++k) {
              const uint64_t dw = smem_desc(sa + k * 32, 16, 1024);
              const uint32_t acc = (kb > 0 || k > 0) ? 1u : 0u;
              tc_pair_mma(d_tmem, dw, smem_desc(sx + k * 32, 16, 1024), idesc1, acc);
              if (n2 > 0) tc_pair_mma(d_tmem + n1, dw, smem_desc(sx2 + k * 32, 16, 1024), idesc2, acc);
            }
            tc_pair_commit(empty0 + 8 * stage);
          }
          __syncwarp();
          if (++stage == stages) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        if (elect_one()) tc_pair_commit(tfull0 + 8 * (i & 1));
        __syncwarp();
      }
      if (!ok && lane == 0) { *abort_flag = 1; if (p.status) atomicOr(p.status, C2R_STATUS_WAIT_TIMEOUT); }
    }
  } else {
    const int q = warp & 3, hsel = (warp - 2) >> 2;
    const uint32_t tfree_mma0 = map_to_cta(tfree0, 0);
    bool ok = true;
    int hint = 0;
    RaggedUnit u, next;
    bool more = unit_at(0, u, hint);
    for (int i = 0; more; ++i) {
      more = unit_at(i + 1, next, hint);
      const int n1 = ragged_first(u.nb);
      const int steps = u.nb >> 5;                                         // 16-column groups per warp
      const int drain = more ? max(0, u.nb + next.nb - RG_TMEM) >> 5 : 0;  // of them before the next unit may begin
      auto group = [&](int it) { return (i & 1) ? 2 * it + hsel : 2 * (steps - 1 - it) + hsel; };  // the shared columns first
      if (UP) {
        for (int x = lane; x < steps * 16; x += 32) {
          const int tok = ragged_token(16 * group(x >> 4), u.nb, n1) + (x & 15);
          float sc = 1.f;
          if (p.scale_kind != 0 && tok < u.rows) {
            const float v = p.row_scale[u.row0 + tok];
            sc = p.scale_kind == 2 ? 1.0f / (1.0f + expf(-v)) : v;
          }
          s_scale[warp - 2][x] = sc;
        }
        __syncwarp();
      }
      if (drain == 0 && lane == 0) mbar_arrive_cluster(tfree_mma0 + 8 * (i & 1));  // the unit before is drained
      if (!__all_sync(0xffffffffu, mbar_wait(tfull0 + 8 * (i & 1), (i >> 1) & 1, abort_flag))) { ok = false; break; }
      tc_fence_after();
      const uint32_t taddr = tmem_base + ((i & 1) ? RG_TMEM - u.nb : 0) + ((uint32_t)(32 * q) << 16);
      for (int it = 0; it < steps; ++it) {
        const int c = 16 * group(it), tok0 = ragged_token(c, u.nb, n1), live = u.rows - tok0;
        if constexpr (UP) {
          const int ch0 = 128 * u.slice + 64 * (int)rank + 16 * q;
          uint32_t g[8], b[8];
          ragged_ld_16x256(taddr + c, g);
          ragged_ld_16x256(taddr + c + (16u << 16), b);
          tc_ld_wait();
          if (ch0 < p.M && live > 0) {
            const int col = 2 * (lane & 3);
#pragma unroll
            for (int blk = 0; blk < 2; ++blk) {  // 8 tokens
              const float2 sc = *reinterpret_cast<const float2*>(&s_scale[warp - 2][16 * it + 8 * blk + col]);
              uint32_t m[2];
#pragma unroll
              for (int h = 0; h < 2; ++h) {  // 8 channels
                const float a0 = __uint_as_float(g[4 * blk + 2 * h]), a1 = __uint_as_float(g[4 * blk + 2 * h + 1]);
                const float b0 = __uint_as_float(b[4 * blk + 2 * h]), b1 = __uint_as_float(b[4 * blk + 2 * h + 1]);
                const __nv_bfloat162 v = __floats2bfloat162_rn(sc.x * (a0 * sigmoid_fast(a0) * b0), sc.y * (a1 * sigmoid_fast(a1) * b1));
                m[h] = transpose8(*reinterpret_cast<const uint32_t*>(&v));
              }
              // thread: token lane / 4, channels col, col + 1 of both groups of 8; neighbours trade so that each has four in a row
              const bool odd = lane & 1;
              const uint32_t got = __shfl_xor_sync(0xffffffffu, odd ? m[0] : m[1], 1);
              const uint2 v = odd ? make_uint2(got, m[1]) : make_uint2(m[0], got);
              const int tok = 8 * blk + (lane >> 2);
              if (tok < live)
                *reinterpret_cast<uint2*>((__nv_bfloat16*)p.out + (long long)(u.row0 + tok0 + tok) * p.M + ch0 + (odd ? 8 : 0) +
                                          2 * (lane & 2)) = v;
            }
          }
        } else {
          const int ch = 256 * u.slice + 128 * (int)rank + 32 * q + lane;
          uint32_t r[16];
          tc_ld16(taddr + c, r);
          tc_ld_wait();
          if (ch < p.M) {
            float* o = (float*)p.out + (long long)(u.row0 + tok0) * p.M + ch;
#pragma unroll
            for (int n = 0; n < 16; ++n)
              if (n < live) o[(long long)n * p.M] = __uint_as_float(r[n]);
          }
        }
        if (it + 1 == drain) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(tfree_mma0 + 8 * (i & 1));
        }
      }
      tc_fence_before();
      __syncwarp();  // also: the scales are read before the next unit's are written
      u = next;
    }
    if (!ok && lane == 0) { *abort_flag = 1; if (p.status) atomicOr(p.status, C2R_STATUS_WAIT_TIMEOUT); }
  }

  // after a wait gave up, let TMA loads still in flight land before the CTA (and its shared memory) goes away
  __syncthreads();
  if (*abort_flag)
    for (int i = 0; i < 128; ++i) __nanosleep(2000);
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(RG_TMEM) : "memory");
  }
}

// Packed gate and up rows [expert][2 I][d] as [expert][group][gate, up][16 rows][d]: a box is 4 groups of 16 channels, each its gate
// rows and then its up rows.  Groups overlap in memory: the second 8 of a block of 128 channels are its up rows and are
// never asked for.  full: the blocks of 128 channels; else the partial last block, whose up rows follow its gate rows
// sooner and whose missing groups lie beyond the map and read zeros.
static int interleaved_map(CUtensorMap* m, const void* W13p, int64_t d, int64_t I, int64_t nE, bool full) {
  EncodeTiledFn enc = get_encode();
  if (!enc) return C2R_ERR_CUDA;
  const int64_t blocks = I / 128, rest = I % 128;
  cuuint64_t dims[5] = {(cuuint64_t)d, 16, 2, (cuuint64_t)(full ? 16 * blocks : 16 * blocks + rest / 16), (cuuint64_t)nE};
  cuuint64_t strides[4] = {(cuuint64_t)d * 2, (cuuint64_t)((full ? 128 : rest) * d) * 2, (cuuint64_t)(16 * d) * 2, (cuuint64_t)(2 * I * d) * 2};
  cuuint32_t box[5] = {BK, 16, 2, 4, 1};
  cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(W13p), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) { g_last_cuda_error = (int)cudaErrorInvalidValue; return C2R_ERR_CUDA; }
  return C2R_OK;
}

// R: the chunk arithmetic was checked up to 600000 rows.
bool ragged_supported(const c2r_config* cfg, const SwigluCall& a) {
  const uintptr_t bits = (uintptr_t)a.Xp | (uintptr_t)a.W13p | (uintptr_t)a.W2 | (uintptr_t)a.H | (uintptr_t)a.Yp;
  return a.AB == nullptr && a.X == nullptr && a.token_acc == nullptr && a.Xp != nullptr && a.Yp != nullptr && (bits & 15u) == 0 &&
         a.R <= 600000 && expected_rows(cfg, a) <= (a.nE == 1 ? RAGGED_ROWS_SINGLE : RAGGED_ROWS);
}

template <bool UP>
static int ragged_launch(const RaggedMaps& maps, const RaggedParams& p, cudaStream_t s) {
  constexpr int MAX_DEV = 64;
  static int grid_of_device[MAX_DEV] = {};  // CTAs of the persistent grid, per device
  int dev = 0;
  C2R_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= MAX_DEV) return C2R_ERR_UNSUPPORTED_SHAPE;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // see launch_chained
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.blockDim = dim3(RG_THREADS);
  cfg.dynamicSmemBytes = RG_SMEM;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int grid = __atomic_load_n(&grid_of_device[dev], __ATOMIC_ACQUIRE);
  if (grid == 0) {
    C2R_CUDA(cudaFuncSetAttribute(ragged_kernel<UP>, cudaFuncAttributeMaxDynamicSharedMemorySize, RG_SMEM));
    int sms = 0, pairs = 0;
    C2R_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    cfg.gridDim = dim3(sms / 2 * 2);
    C2R_CUDA(cudaOccupancyMaxActiveClusters(&pairs, ragged_kernel<UP>, &cfg));
    if (pairs < 1) return C2R_ERR_UNSUPPORTED_SHAPE;
    grid = 2 * (pairs < sms / 2 ? pairs : sms / 2);
    __atomic_store_n(&grid_of_device[dev], grid, __ATOMIC_RELEASE);
  }
  cfg.gridDim = dim3(grid);
  cfg.numAttrs = 2;
  C2R_CUDA(cudaLaunchKernelEx(&cfg, ragged_kernel<UP>, maps, p));
  C2R_LAUNCH_CHECK();
  return C2R_OK;
}

static int ragged_rows_maps(RaggedMaps& maps, const void* base, int64_t K, int64_t R) {
  for (int b = 0; b < 4; ++b) {
    const int rc = make_map(&maps.x[b], base, K, R, 0, BK, 128 >> b);
    if (rc) return rc;
  }
  return C2R_OK;
}

int ragged_swiglu_fwd(const c2r_config* cfg, const SwigluCall& a, cudaStream_t s) {
  RaggedMaps maps;
  RaggedParams p{};
  p.counts = a.counts; p.offsets = a.offsets; p.R = a.R; p.nE = a.nE; p.status = a.status;
  // H = s silu(Xp W1^T) (Xp W3^T)
  int rc = interleaved_map(&maps.w, a.W13p, cfg->d, a.I, a.nE, a.I >= 128);
  if (!rc) rc = interleaved_map(&maps.w_last, a.W13p, cfg->d, a.I, a.nE, a.I % 128 == 0);
  if (!rc) rc = ragged_rows_maps(maps, a.Xp, cfg->d, a.R);
  if (rc) return rc;
  p.M = a.I; p.kblocks = (cfg->d + BK - 1) / BK; p.slices = (a.I + 127) / 128; p.out = a.H;
  p.row_scale = a.row_scale; p.scale_kind = a.row_scale ? a.scale_kind : 0;
  if ((rc = ragged_launch<true>(maps, p, s))) return rc;
  // Yp = H W2^T (fp32)
  rc = make_map(&maps.w, a.W2, a.I, cfg->d, a.nE, BK, 128);
  if (!rc) rc = ragged_rows_maps(maps, a.H, a.I, a.R);
  if (rc) return rc;
  maps.w_last = maps.w;  // not read
  p.M = cfg->d; p.kblocks = (a.I + BK - 1) / BK; p.slices = (cfg->d + 255) / 256; p.out = a.Yp;
  p.row_scale = nullptr; p.scale_kind = 0;
  return ragged_launch<false>(maps, p, s);
}

}  // namespace c2r
