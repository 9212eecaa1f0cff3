// Grouped SwiGLU forward for a handful of rows per expert (decode steps, short prompts), bf16, sm_100a.
//
// With few rows the product is bound by reading every weight once: 138 MB for one token of the Qwen-MoE-shaped layer
// (d 2048, 60 experts of 1408, top-4, shared 5632), 1.1 GB for 64.  The 256 x 256 pair tiles of tc_gemm_kernel are the
// wrong shape for that: one token's output is 8 to 44 such tiles, so most SMs stay idle.  Here the weights are the M
// operand (128 accumulator lanes) and the tokens its N of 16..128 columns.  A unit of work is a slice of an expert's
// weight rows (CH gate and CH up rows, or 2 CH output channels) against one chunk of the expert's tokens over the
// whole contraction; CTAs are persistent and walk the units, the TMA ring (about 190 KB) runs across unit boundaries, so
// an SM always has its whole ring of weight bytes in flight.  A stage is several k-blocks that one TMA instruction
// brings (slab maps): with a stage per k-block of 6 to 18 KB the issuing thread, not the memory, set the pace (about
// 0.27 us per k-block).  CH is 64 unless that leaves half the SMs without a unit: narrow slices cost more
// instructions per byte than idle SMs do.  With fewer than 128 weight rows in a box the MMA still reads 128 shared-memory
// rows, and the lanes of the rows that are not the unit's hold garbage nobody reads.
//
// Two problems can share a launch (the routed experts and the shared expert), so one decode step has two expert
// launches, not four.
//
// Measured, Qwen shape, both products of the routed experts after an L2 flush: 64 tokens 237 -> 183 us (1.04 GB, 5.7 TB/s),
// 1 token 52 -> 36 us; a whole forward pass of 64 tokens, with the other kernels as they are now, 366 -> 221 us, of one token 172 -> 75 us.
//
// Warp roles (192 threads): warp 0 TMA producer, warp 1 MMA issuer and TMEM owner, warps 2..5 epilogue (TMEM -> shared
// memory -> coalesced stores).  Waits are bounded like in the other tensor-core kernels.
#include "gemm.h"
#include "tc_common.cuh"

namespace c2r {

constexpr int SK_THREADS = 192;
constexpr int SK_MAX_STAGES = 24;
constexpr int SK_RING = 190 * 1024;                // bytes of operands in flight per SM
constexpr int SK_STAGE = 40 * 1024;                // as many whole k-blocks per stage as fit this
constexpr int SK_OUT_PITCH = 132;                  // floats per token of the epilogue's staging tile
constexpr int SK_OUT_BYTES = 16 * SK_OUT_PITCH * 4;
constexpr int SK_SMEM = SK_RING + SK_OUT_BYTES + 16 * 1024 + 1024;  // + what the last stage's MMA reads past its rows

struct SkinnyProblem {
  const int32_t* counts;
  const int32_t* offsets;
  const float* row_scale;
  void* out;           // up: H [R, M] bf16; down: [R, M] float
  long long R;
  int scale_kind;
  int nE, M;           // M: output channels per expert (up: I, down: d)
  int kfull, tail;     // contraction: whole k-blocks, and whether a partial one follows
  int nb;              // tokens per chunk (MMA-N)
  int slices;          // weight slices per expert
};
struct SkinnyParams {
  SkinnyProblem pr[2];
  int n_problems;
  int up;              // 1: SwiGLU up-projection, 0: plain product
  int ch;              // see above
  int ks;              // k-blocks per stage
  int stages, stage_bytes;
  int32_t* status;
};
// Tensor maps of a problem: weights and rows, each as slabs of ks whole k-blocks ([k-block][row][64]) and, for the last
// partial k-block, plainly (zero fill beyond the contraction).
struct SkinnyMaps {
  CUtensorMap w, x, w_tail, x_tail;
};

struct SkinnyUnit {
  int problem, expert, slice, row0, rows;  // row0: first row of the chunk in the row-indexed operands
};

// Units: problem by problem, expert by expert, slice by slice, token chunks innermost (a slice's later chunks find its
// weights in the L2).  s_first[e] = units before expert e of its problem.  Warp-collective.
__device__ __forceinline__ bool skinny_unit(const SkinnyParams& p, const int (*s_first)[65], const int (*s_cnt)[64],
                                            const int (*s_off)[64], int u, SkinnyUnit& w, int& hint) {
  const int n0 = s_first[0][p.pr[0].nE];
  w.problem = u >= n0;
  if (w.problem) {
    u -= n0;
    if (p.n_problems < 2 || u >= s_first[1][p.pr[1].nE]) return false;
  }
  const int* first = s_first[w.problem];
  const int nE = p.pr[w.problem].nE;
  int e = (hint < nE && first[hint] <= u) ? hint : 0;
  while (e + 1 < nE && first[e + 1] <= u) ++e;
  hint = e;
  const int cnt = s_cnt[w.problem][e], nb = p.pr[w.problem].nb;
  const int chunks = (cnt + nb - 1) / nb;
  const int r = u - first[e];
  const int slice = r / chunks, c = r - slice * chunks;
  w.problem = warp_uniform(w.problem);
  w.expert = warp_uniform(e);
  w.slice = warp_uniform(slice);
  w.row0 = warp_uniform(s_off[w.problem][e] + c * nb);
  w.rows = warp_uniform(min(nb, cnt - c * nb));
  return true;
}

__device__ __forceinline__ void epilogue_sync() { asm volatile("bar.sync 1, 128;" ::: "memory"); }
// Barrier of the epilogue warps that also agrees on whether all of them may go on.
__device__ __forceinline__ bool epilogue_all(bool ok) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "bar.red.and.pred q, 1, 128, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)ok)
      : "memory");
  return r != 0;
}

__global__ void __launch_bounds__(SK_THREADS, 1)
skinny_kernel(const __grid_constant__ SkinnyMaps maps0, const __grid_constant__ SkinnyMaps maps1, const SkinnyParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  float* s_out = reinterpret_cast<float*>(smem_raw + (smem_base - smem_u32(smem_raw)) + SK_RING + 16 * 1024);
  __shared__ uint64_t bars[2 * SK_MAX_STAGES + 4];
  __shared__ uint32_t tmem_slot;
  __shared__ int s_abort;
  __shared__ int s_first[2][65], s_cnt[2][64], s_off[2][64];

  const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[SK_MAX_STAGES]);
  const uint32_t tfull0 = smem_u32(&bars[2 * SK_MAX_STAGES]), tempty0 = smem_u32(&bars[2 * SK_MAX_STAGES + 2]);
  if (threadIdx.x == 0) {
    s_abort = 0;
    for (int s = 0; s < p.stages; ++s) { mbar_init(full0 + 8 * s, 1); mbar_init(empty0 + 8 * s, 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(tfull0 + 8 * b, 1); mbar_init(tempty0 + 8 * b, 4); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    chain_release();  // not before: a block of the next kernel must not take the tensor memory this one waits for
  }
  chain_wait();  // before the first access to global memory
  for (int i = threadIdx.x; i < 64 * p.n_problems; i += blockDim.x) {
    const int q = i >> 6, e = i & 63;
    if (e < p.pr[q].nE) {
      const int off = p.pr[q].offsets[e];
      s_off[q][e] = off;
      s_cnt[q][e] = (int)max(0ll, min((long long)p.pr[q].counts[e], p.pr[q].R - off));
    }
  }
  __syncthreads();
  if (warp < p.n_problems) {  // a warp per problem: exclusive scan of the experts' unit counts
    const SkinnyProblem& pr = p.pr[warp];
    int run = 0;
    for (int e0 = 0; e0 < pr.nE; e0 += 32) {
      const int e = e0 + lane;
      const int v = e < pr.nE ? (s_cnt[warp][e] + pr.nb - 1) / pr.nb * pr.slices : 0;
      int incl = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
      }
      if (e < pr.nE) s_first[warp][e] = run + incl - v;
      run += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) s_first[warp][pr.nE] = run;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = warp_uniform(tmem_slot);
  volatile int* abort_flag = &s_abort;
  const int parts = p.up ? 2 : 1, wr = p.up ? p.ch : 2 * p.ch;  // weight boxes per stage and their rows
  const int kb_bytes = wr * BK * 2;                              // one k-block of a box

  if (warp == 0) {
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    int hint = 0;
    SkinnyUnit w;
    for (int u = blockIdx.x; ok && skinny_unit(p, s_first, s_cnt, s_off, u, w, hint); u += gridDim.x) {
      const SkinnyProblem& pr = p.pr[w.problem];
      const SkinnyMaps* m = w.problem ? &maps1 : &maps0;
      int y[2] = {wr * w.slice, 0};
      if (p.up) {  // CH gate rows and the up rows of the same channels inside the packed layout
        const int i0 = p.ch * w.slice, blk = i0 >> 7;
        y[0] = 256 * blk + (i0 & 127);
        y[1] = y[0] + min(128, pr.M - 128 * blk);
      }
      const int slabs = (pr.kfull + p.ks - 1) / p.ks;
      for (int j = 0; j < slabs + pr.tail; ++j) {
        if (!__all_sync(0xffffffffu, mbar_wait(empty0 + 8 * stage, phase ^ 1u, abort_flag))) { ok = false; break; }
        const uint32_t fb = full0 + 8 * stage;
        const uint32_t sa = smem_base + stage * p.stage_bytes, sx = sa + parts * p.ks * kb_bytes;
        if (elect_one()) {
          if (j < slabs) {
            mbar_expect_tx(fb, p.ks * (parts * kb_bytes + pr.nb * BK * 2));
            for (int q = 0; q < parts; ++q) tma_load_4d(sa + q * p.ks * kb_bytes, &m->w, fb, 0, y[q], j * p.ks, w.expert);
            tma_load_4d(sx, &m->x, fb, 0, w.row0, j * p.ks, 0);
          } else {
            mbar_expect_tx(fb, parts * kb_bytes + pr.nb * BK * 2);
            for (int q = 0; q < parts; ++q) tma_load_3d(sa + q * p.ks * kb_bytes, &m->w_tail, fb, pr.kfull * BK, y[q], w.expert);
            tma_load_2d(sx, &m->x_tail, fb, pr.kfull * BK, w.row0);
          }
        }
        __syncwarp();
        if (++stage == p.stages) { stage = 0; phase ^= 1u; }
      }
    }
    if (!ok && lane == 0) { *abort_flag = 1; if (p.status) atomicOr(p.status, C2R_STATUS_WAIT_TIMEOUT); }
  } else if (warp == 1) {
    int stage = 0;
    uint32_t phase = 0, acc = 0, acc_phase = 0;
    bool ok = true;
    int hint = 0;
    SkinnyUnit w;
    for (int u = blockIdx.x; ok && skinny_unit(p, s_first, s_cnt, s_off, u, w, hint); u += gridDim.x) {
      if (!__all_sync(0xffffffffu, mbar_wait(tempty0 + 8 * acc, acc_phase ^ 1u, abort_flag))) { ok = false; break; }
      tc_fence_after();
      const uint32_t d_tmem = tmem_base + acc * 256;
      const SkinnyProblem& pr = p.pr[w.problem];
      const uint32_t idesc = instr_desc(pr.nb, false, false);
      const int slabs = (pr.kfull + p.ks - 1) / p.ks;
      uint32_t accumulate = 0;
      for (int j = 0; j < slabs + pr.tail; ++j) {
        if (!__all_sync(0xffffffffu, mbar_wait(full0 + 8 * stage, phase, abort_flag))) { ok = false; break; }
        tc_fence_after();
        const int nk = j < slabs ? min(p.ks, pr.kfull - j * p.ks) : 1;
        uint32_t sa = smem_base + stage * p.stage_bytes, sx = sa + parts * p.ks * kb_bytes;
        if (elect_one()) {
          for (int kb = 0; kb < nk; ++kb) {
#pragma unroll
            for (int k = 0; k < BK / UMMA_K; ++k) {
              const uint64_t dx = smem_desc(sx + k * 32, 16, 1024);
              tc_mma(d_tmem, smem_desc(sa + k * 32, 16, 1024), dx, idesc, accumulate);
              if (parts == 2) tc_mma(d_tmem + 128, smem_desc(sa + p.ks * kb_bytes + k * 32, 16, 1024), dx, idesc, accumulate);
              accumulate = 1;
            }
            sa += kb_bytes;
            sx += pr.nb * BK * 2;
          }
          tc_commit(empty0 + 8 * stage);
        }
        __syncwarp();
        accumulate = 1;
        if (++stage == p.stages) { stage = 0; phase ^= 1u; }
      }
      if (!ok) break;
      if (elect_one()) tc_commit(tfull0 + 8 * acc);
      __syncwarp();
      if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
    }
    if (!ok && lane == 0) { *abort_flag = 1; if (p.status) atomicOr(p.status, C2R_STATUS_WAIT_TIMEOUT); }
  } else {
    const int q = warp & 3, tid = threadIdx.x - 64;
    uint32_t acc = 0, acc_phase = 0;
    bool ok = true;
    int hint = 0;
    SkinnyUnit w;
    for (int u = blockIdx.x; skinny_unit(p, s_first, s_cnt, s_off, u, w, hint); u += gridDim.x) {
      const SkinnyProblem& pr = p.pr[w.problem];
      ok = epilogue_all(mbar_wait(tfull0 + 8 * acc, acc_phase, abort_flag));  // all four warps leave together
      if (!ok) break;
      tc_fence_after();
      const uint32_t taddr = tmem_base + acc * 256 + ((uint32_t)(32 * q) << 16);
      for (int c = 0; c < w.rows; c += 16) {
        const int live = min(16, w.rows - c);
        if (32 * q < wr) {
          uint32_t r[16];
          tc_ld16(taddr + c, r);
          if (p.up) {
            uint32_t r2[16];
            tc_ld16(taddr + 128 + c, r2);
            tc_ld_wait();
#pragma unroll
            for (int n = 0; n < 16; ++n) {
              if (n >= live) break;
              float sc = 1.f;
              if (pr.scale_kind != 0) {
                const float v = pr.row_scale[w.row0 + c + n];
                sc = pr.scale_kind == 2 ? 1.0f / (1.0f + expf(-v)) : v;
              }
              const float a = __uint_as_float(r[n]), b = __uint_as_float(r2[n]);
              s_out[n * SK_OUT_PITCH + 32 * q + lane] = sc * (a * sigmoid_fast(a) * b);
            }
          } else {
            tc_ld_wait();
#pragma unroll
            for (int n = 0; n < 16; ++n) s_out[n * SK_OUT_PITCH + 32 * q + lane] = __uint_as_float(r[n]);
          }
        }
        epilogue_sync();
        const int quads = wr >> 2;  // groups of four output channels of the slice
        for (int x = tid; x < quads * live; x += 128) {
          const int n = x / quads, i = 4 * (x - n * quads), ch = wr * w.slice + i;
          if (ch >= pr.M) continue;
          const float4 v = *reinterpret_cast<const float4*>(&s_out[n * SK_OUT_PITCH + i]);
          const long long o = (long long)(w.row0 + c + n) * pr.M + ch;
          if (p.up) {
            const __nv_bfloat162 h0 = __floats2bfloat162_rn(v.x, v.y), h1 = __floats2bfloat162_rn(v.z, v.w);
            *reinterpret_cast<uint2*>((__nv_bfloat16*)pr.out + o) =
                make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1));
          } else {
            *reinterpret_cast<float4*>((float*)pr.out + o) = v;
          }
        }
        epilogue_sync();
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty0 + 8 * acc);
      if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
    }
    if (!ok && lane == 0) { *abort_flag = 1; if (p.status) atomicOr(p.status, C2R_STATUS_WAIT_TIMEOUT); }
  }

  // after a wait gave up, let TMA loads still in flight land before the CTA (and its shared memory) goes away
  __syncthreads();
  if (*abort_flag)
    for (int i = 0; i < 128; ++i) __nanosleep(2000);
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
  }
}

// Rows an expert is expected to have, as far as the host knows: all of R for a single group, else the batch's slots
// spread evenly.  Only a hint: the kernel takes any counts.
static int64_t expected_rows(const c2r_config* cfg, const SwigluCall& a) {
  return a.nE == 1 ? a.R : ((int64_t)cfg->N * cfg->K + a.nE - 1) / a.nE;
}

bool skinny_supported(const c2r_config* cfg, const SwigluCall& a, int max_rows) {
  const uintptr_t bits = (uintptr_t)a.Xp | (uintptr_t)a.W13p | (uintptr_t)a.W2 | (uintptr_t)a.H | (uintptr_t)a.Yp;
  return a.AB == nullptr && a.X == nullptr && a.token_acc == nullptr && a.Xp != nullptr && a.Yp != nullptr &&
         (bits & 15u) == 0 && expected_rows(cfg, a) <= max_rows;
}

static int skinny_launch(const c2r_config* cfg, const SwigluCall* calls, int n, bool up, cudaStream_t s) {
  constexpr int MAX_DEV = 64;
  static int sms_of_device[MAX_DEV] = {};  // SM count, also "the kernel's shared-memory limit is set on this device"
  int dev = 0;
  C2R_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= MAX_DEV) return C2R_ERR_UNSUPPORTED_SHAPE;
  int sms = __atomic_load_n(&sms_of_device[dev], __ATOMIC_ACQUIRE);
  if (sms == 0) {
    C2R_CUDA(cudaFuncSetAttribute(skinny_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SK_SMEM));
    C2R_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    __atomic_store_n(&sms_of_device[dev], sms, __ATOMIC_RELEASE);
  }
  SkinnyParams p{};
  p.n_problems = n; p.up = up; p.status = calls[0].status;
  // the widest slice that still gives half the SMs a unit (see the head of the file)
  for (p.ch = 64; p.ch > 16; p.ch >>= 1) {
    int64_t units = 0;
    for (int i = 0; i < n; ++i) {
      const int64_t slots = (int64_t)cfg->N * cfg->K, M = up ? calls[i].I : cfg->d, rows = up ? p.ch : 2 * p.ch;
      units += (M + rows - 1) / rows * (calls[i].nE == 1 ? 1 : slots < calls[i].nE ? slots : calls[i].nE);
    }
    if (units >= sms / 2) break;
  }
  const int wr = up ? p.ch : 2 * p.ch, parts = up ? 2 : 1;
  int nb_max = 16;
  for (int i = 0; i < n; ++i) {
    // Chunks of half as many tokens again as expected: most experts fit one, and few columns are empty.  In a shared launch
    // all stages have the size of the larger problem's, so the shared expert's tokens come in chunks of 32 at most, whose weights
    // the later chunks find in the L2 (64 tokens of the Qwen shape 235 us with one chunk of 64, 219 with two of 32; 128
    // tokens 263 / 247).
    const int64_t rows = expected_rows(cfg, calls[i]), want = calls[i].nE == 1 ? rows : rows + rows / 2;
    for (p.pr[i].nb = 16; p.pr[i].nb < want && p.pr[i].nb < (n > 1 ? 32 : 128); p.pr[i].nb <<= 1) {}
    if (p.pr[i].nb > nb_max) nb_max = p.pr[i].nb;
  }
  const int kb_bytes = (parts * wr + nb_max) * BK * 2;
  p.ks = SK_STAGE / kb_bytes > 1 ? SK_STAGE / kb_bytes : 1;
  p.stage_bytes = p.ks * kb_bytes;
  p.stages = SK_RING / p.stage_bytes < SK_MAX_STAGES ? SK_RING / p.stage_bytes : SK_MAX_STAGES;
  SkinnyMaps maps[2];
  for (int i = 0; i < n; ++i) {
    const SwigluCall& a = calls[i];
    SkinnyProblem& q = p.pr[i];
    const int K = up ? cfg->d : a.I;
    q.counts = a.counts; q.offsets = a.offsets; q.R = a.R; q.nE = a.nE;
    q.M = up ? a.I : cfg->d;
    q.kfull = K / BK; q.tail = K % BK != 0;
    q.slices = (q.M + wr - 1) / wr;
    q.out = up ? a.H : a.Yp;
    q.row_scale = up ? a.row_scale : nullptr;
    q.scale_kind = q.row_scale ? a.scale_kind : 0;
    const void* W = up ? a.W13p : a.W2;
    const void* X = up ? a.Xp : a.H;
    const int wrows = up ? 2 * a.I : cfg->d;
    int rc = make_map(&maps[i].w_tail, W, K, wrows, a.nE, BK, wr);
    if (!rc) rc = make_map(&maps[i].x_tail, X, K, a.R, 0, BK, q.nb);
    if (rc) return rc;
    if (q.kfull > 0) {
      rc = slab_map(&maps[i].w, W, K, wrows, q.kfull, a.nE, wr, p.ks);
      if (!rc) rc = slab_map(&maps[i].x, X, K, a.R, q.kfull, 1, q.nb, p.ks);
      if (rc) return rc;
    } else {
      maps[i].w = maps[i].w_tail; maps[i].x = maps[i].x_tail;  // not read
    }
  }
  if (n == 1) maps[1] = maps[0];
  C2R_CUDA(launch_chained(skinny_kernel, sms, SK_THREADS, SK_SMEM, s, maps[0], maps[1], p));
  C2R_LAUNCH_CHECK();
  return C2R_OK;
}

int skinny_swiglu_fwd(const c2r_config* cfg, const SwigluCall* calls, int n, cudaStream_t s) {
  const int rc = skinny_launch(cfg, calls, n, true, s);
  return rc ? rc : skinny_launch(cfg, calls, n, false, s);
}

}  // namespace c2r
