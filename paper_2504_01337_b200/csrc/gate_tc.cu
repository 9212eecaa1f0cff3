// Gate logits (Eq. 1) for bf16 hidden states on the tensor cores: L = X Wg^T and z = X wsg.
//
// The product is HBM-bound (X is read once, E <= 64 output columns), so the kernel is a streaming
// one: a CTA owns tiles of tm tokens x tw experts, TMA brings [tm x 64] blocks of X and the matching [tw x 64]
// block of Wg (rows >= E are zero-filled by the tensor map) and [16 x 64] block of wsg (row 0 is
// the vector, rows 1..15 zero fill) through a ring of 208 KB, one thread issues one tcgen05 MMA per
// 16 k-elements (N = tw, 16 more where the shared-expert gate's block rides along) into tensor
// memory, and four warps write the fp32 accumulators out.  Waits are bounded like in the grouped
// GEMM kernel.
//
// Few tokens are few tiles, and a CTA that streams 128 tokens alone is slow: a tile then has 64 or 32 tokens (the MMA still
// computes 128 rows, the rest is whatever the stage holds and is not stored), and where SMs are left over the experts are
// split into tiles of 32 or 16: a k-block is then as small as 6 KB, and a whole contraction of 2048 is in flight at once.  A split
// of the contraction over a cluster would add a token's products in another order, and logits that differ in their last bits
// route near-ties to other experts; every logit here is the same sum, bit for bit, in whatever tile.
// Where a k-block is small a stage holds up to four, brought by one instruction per operand (a k-block at a time took 175 ns of the
// issuing thread, however many were in flight).
// Whole tiles (128 tokens, all experts: more than 64 tokens for every SM) are bound by the memory and by the two issuing threads, so
// they have instances with everything known at compile time and plain maps (us a call, in the general form / so: 19000 tokens of 4096
// and 24 experts 40.0 / 37.0, 20000 of 2048 and 60 23.3 / 21.8, 25000 of 1024 and 48 15.0 / 13.8, 65536 of 512 and 12 15.5 / 14.1).
// (us by events after an L2 flush, all experts in a tile and a k-block per stage / this: 14.3 / 11.3 for 1 to 64 tokens of d = 2048 and
// 60 experts, 19.5 / 17.4 for 1021 and 24.6 / 23.4 for 8192 of d = 4096 and 16; 16384 and more take 128-token tiles as before.)
#include "gemm.h"
#include "tc_common.cuh"

namespace c2r {

constexpr int GT_RING = 208 * 1024;        // bytes of operands in flight: 8 to 11 stages of a whole tile; 4 to 8 of four k-blocks, or more of fewer, else
constexpr int GT_MAX_STAGES = 32;
constexpr int GT_S_BYTES = 16 * BK * 2;    // the shared gate's block, 2 KB
constexpr int GT_THREADS = 192;
constexpr int GT_TMEM_COLS = 256;          // two accumulators of 128 columns (64 logits | 16 shared gate | unused)

// X, Wg and wsg as slabs of ks whole k-blocks ([k-block][row][64]) and, for the last partial k-block, plainly.
struct GateMaps {
  CUtensorMap x, w, s, x_tail, w_tail, s_tail;
};

// TW > 0 (whole tiles): 128 tokens x all E <= TW experts, a k-block per stage, plain maps (the *_tail ones); tm, tw, ks are not read.
// S: with the shared gate's block in every stage.  TW = 0: everything as the arguments say.
template <int TW, bool S>
__global__ void __launch_bounds__(GT_THREADS, 1)
gate_tc_kernel(const __grid_constant__ GateMaps maps, float* __restrict__ L, float* __restrict__ z, int N, int d,
               int E, int has_shared, int tm_, int tw_, int ks_, int32_t* __restrict__ status) {
  constexpr bool WHOLE = TW > 0;
  const int tm = WHOLE ? BM : tm_, tw = WHOLE ? TW : tw_, ks = WHOLE ? 1 : ks_;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  __shared__ uint64_t bars[2 * GT_MAX_STAGES + 4];
  __shared__ uint32_t tmem_slot;
  __shared__ int s_abort;

  const int warp = warp_uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[GT_MAX_STAGES]);
  const uint32_t tfull0 = smem_u32(&bars[2 * GT_MAX_STAGES]), tempty0 = smem_u32(&bars[2 * GT_MAX_STAGES + 2]);
  if (warp == 0) {
    if (lane == 0) s_abort = 0;
    mbar_init(full0 + 8 * lane, 1);
    mbar_init(empty0 + 8 * lane, 1);
    if (lane < 2) { mbar_init(tfull0 + 8 * lane, 1); mbar_init(tempty0 + 8 * lane, 4); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(GT_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  chain_wait();  // before the first access to global memory
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = warp_uniform(tmem_slot);
  volatile int* abort_flag = &s_abort;

  // tiles of tm tokens x tw experts; the shared gate rides along with all experts, or is a tile of its own where they are split
  const bool with_s = WHOLE ? S : has_shared && E <= tw;
  const int e_parts = WHOLE ? 1 : (E + tw - 1) / tw, parts = WHOLE ? 1 : e_parts + (has_shared && !with_s), tiles = (N + tm - 1) / tm * parts;
  const int kfull = d / BK, slabs = WHOLE ? (d + BK - 1) / BK : (kfull + ks - 1) / ks, steps = WHOLE ? slabs : slabs + (d % BK != 0);
  // a stage holds ks k-blocks of X, then ks of Wg, each followed by wsg's if that rides along
  const uint32_t x_kb = tm * BK * 2, w_kb = tw * BK * 2 + (with_s ? GT_S_BYTES : 0), stage_bytes = ks * (x_kb + w_kb);
  const int stages = min(GT_MAX_STAGES, (int)(GT_RING / stage_bytes));

  if (warp == 0) {
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
      const int part = t % parts, row0 = t / parts * tm;
      const bool gate_s = part == e_parts;  // the shared gate's own tile: its map has one row, the others of a box read zeros
      for (int j = 0; j < steps; ++j) {
        if (!__all_sync(0xffffffffu, mbar_wait(empty0 + 8 * stage, phase ^ 1u, abort_flag))) { ok = false; break; }
        const uint32_t fb = full0 + 8 * stage;
        const uint32_t sx = smem_base + stage * stage_bytes, sw = sx + ks * x_kb;
        if (elect_one()) {
          if (WHOLE) {
            mbar_expect_tx(fb, stage_bytes);
            tma_load_2d(sx, &maps.x_tail, fb, j * BK, row0);
            tma_load_2d(sw, &maps.w_tail, fb, j * BK, 0);
            if (S) tma_load_2d(sw + tw * BK * 2, &maps.s_tail, fb, j * BK, 0);
          } else if (j < slabs) {
            mbar_expect_tx(fb, stage_bytes);
            tma_load_4d(sx, &maps.x, fb, 0, row0, j * ks, 0);
            if (with_s) {
              for (int i = 0; i < ks; ++i) {  // (a k-block past the last whole one reads zeros or is part of the last, and is not used)
                tma_load_2d(sw + i * w_kb, &maps.w, fb, (j * ks + i) * BK, 0);
                tma_load_2d(sw + i * w_kb + tw * BK * 2, &maps.s, fb, (j * ks + i) * BK, 0);
              }
            } else {
              tma_load_4d(sw, gate_s ? &maps.s : &maps.w, fb, 0, gate_s ? 0 : part * tw, j * ks, 0);
            }
          } else {
            mbar_expect_tx(fb, x_kb + w_kb);
            tma_load_2d(sx, &maps.x_tail, fb, kfull * BK, row0);
            tma_load_2d(sw, gate_s ? &maps.s_tail : &maps.w_tail, fb, kfull * BK, gate_s ? 0 : part * tw);
            if (with_s) tma_load_2d(sw + tw * BK * 2, &maps.s_tail, fb, kfull * BK, 0);
          }
        }
        __syncwarp();
        if (++stage == stages) { stage = 0; phase ^= 1u; }
      }
    }
    if (!ok && lane == 0) { *abort_flag = 1; if (status) atomicOr(status, C2R_STATUS_WAIT_TIMEOUT); }
  } else if (warp == 1) {
    int stage = 0;
    uint32_t phase = 0, acc = 0, acc_phase = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
      if (!__all_sync(0xffffffffu, mbar_wait(tempty0 + 8 * acc, acc_phase ^ 1u, abort_flag))) { ok = false; break; }
      tc_fence_after();
      const uint32_t d_tmem = tmem_base + acc * 128;
      // where the shared gate's [16 x 64] block follows the [tw x 64] block of Wg (same 128-byte swizzle rows) one MMA covers both:
      // accumulator columns 0 .. tw - 1 logits, tw the shared gate
      const uint32_t idesc_w = instr_desc(tw + (with_s ? 16 : 0), false, false);
      for (int j = 0; j < steps; ++j) {
        if (!__all_sync(0xffffffffu, mbar_wait(full0 + 8 * stage, phase, abort_flag))) { ok = false; break; }
        tc_fence_after();
        uint32_t sx = smem_base + stage * stage_bytes, sw = sx + ks * x_kb;
        const int nk = WHOLE ? 1 : j < slabs ? min(ks, kfull - j * ks) : 1;
        if (elect_one()) {
          for (int i = 0; i < nk; ++i, sx += x_kb, sw += w_kb) {
#pragma unroll
            for (int k = 0; k < BK / UMMA_K; ++k)
              tc_mma(d_tmem, smem_desc(sx + k * 32, 16, 1024), smem_desc(sw + k * 32, 16, 1024), idesc_w, (j > 0 || i > 0 || k > 0) ? 1u : 0u);
          }
          tc_commit(empty0 + 8 * stage);
        }
        __syncwarp();
        if (++stage == stages) { stage = 0; phase ^= 1u; }
      }
      if (!ok) break;
      if (elect_one()) tc_commit(tfull0 + 8 * acc);
      __syncwarp();
      if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
    }
    if (!ok && lane == 0) { *abort_flag = 1; if (status) atomicOr(status, C2R_STATUS_WAIT_TIMEOUT); }
    // Late: the routing kernel's blocks do not fit beside this kernel's, and released early all of them would be placed on
    // the few SMs without a token tile (calibration pass 43 us, released here 35).
    chain_release();
  } else {
    const int q = warp & 3;
    uint32_t acc = 0, acc_phase = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
      if (!__all_sync(0xffffffffu, mbar_wait(tfull0 + 8 * acc, acc_phase, abort_flag))) { ok = false; break; }
      tc_fence_after();
      const uint32_t taddr = tmem_base + acc * 128 + ((uint32_t)(32 * q) << 16);
      const int part = t % parts, e0 = part * tw;
      const long long tok = 32 * q < tm ? (long long)(t / parts) * tm + 32 * q + lane : N;
      for (int c = 0; c < tw && e0 + c < E && 32 * q < tm; c += 16) {
        uint32_t r[16];
        tc_ld16(taddr + c, r);
        tc_ld_wait();
        if (tok < N) {
          float* o = L + tok * E + e0 + c;
          if ((E & 3) == 0) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (e0 + c + 4 * i < E)
                reinterpret_cast<float4*>(o)[i] = make_float4(__uint_as_float(r[4 * i]), __uint_as_float(r[4 * i + 1]),
                                                              __uint_as_float(r[4 * i + 2]), __uint_as_float(r[4 * i + 3]));
          } else {
#pragma unroll
            for (int i = 0; i < 16; ++i)
              if (e0 + c + i < E) o[i] = __uint_as_float(r[i]);
          }
        }
      }
      if ((with_s || part == e_parts) && 32 * q < tm) {
        uint32_t r[16];
        tc_ld16(taddr + (with_s ? tw : 0), r);
        tc_ld_wait();
        if (tok < N) z[tok] = __uint_as_float(r[0]);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty0 + 8 * acc);
      if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
    }
    if (!ok && lane == 0) { *abort_flag = 1; if (status) atomicOr(status, C2R_STATUS_WAIT_TIMEOUT); }
  }

  // after a wait gave up, let TMA loads still in flight land before the CTA (and its shared memory) goes away
  __syncthreads();
  if (*abort_flag)
    for (int i = 0; i < 128; ++i) __nanosleep(2000);
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(GT_TMEM_COLS) : "memory");
  }
}

bool gate_tc_supported(const c2r_config* cfg) {
  return cfg->dtype == C2R_BF16 && cfg->E <= 64 && cfg->d % 8 == 0 && cfg->N > 0 && get_encode() != nullptr;
}

constexpr int GT_SMEM = GT_RING + BM * BK * 2 + 1024;  // + what the last stage's MMA reads past its rows

using GateKernel = void (*)(GateMaps, float*, float*, int, int, int, int, int, int, int, int32_t*);
// The kernel for whole tiles of tw experts, or (0) the general one.
static GateKernel gate_kernel(int tw, bool s) {
  switch (tw) {
    case 16: return s ? gate_tc_kernel<16, true> : gate_tc_kernel<16, false>;
    case 32: return s ? gate_tc_kernel<32, true> : gate_tc_kernel<32, false>;
    case 48: return s ? gate_tc_kernel<48, true> : gate_tc_kernel<48, false>;
    case 64: return s ? gate_tc_kernel<64, true> : gate_tc_kernel<64, false>;
    default: return gate_tc_kernel<0, false>;
  }
}

// SM count of the current device (a negative error code if that fails); the first call per device also sets the kernels'
// shared-memory limit.
static int gate_sms() {
  constexpr int MAX_DEV = 64;
  static int sms_of_device[MAX_DEV] = {};
  int dev = 0;
  C2R_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= MAX_DEV) return C2R_ERR_UNSUPPORTED_SHAPE;
  int sms = __atomic_load_n(&sms_of_device[dev], __ATOMIC_ACQUIRE);
  if (sms == 0) {
    for (int tw = 0; tw <= 64; tw += 16)
      for (int sh = 0; sh < 2; ++sh) C2R_CUDA(cudaFuncSetAttribute(gate_kernel(tw, sh), cudaFuncAttributeMaxDynamicSharedMemorySize, GT_SMEM));
    C2R_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    __atomic_store_n(&sms_of_device[dev], sms, __ATOMIC_RELEASE);
  }
  return sms;
}

int gate_tc_launch(const c2r_config* cfg, const void* X, const void* Wg, const void* wsg, float* L, float* z,
                   int32_t* status, cudaStream_t s) {
  const int sms = gate_sms();
  if (sms < 0) return sms;
  const int N = cfg->N, d = cfg->d, E = cfg->E, kfull = d / BK;
  int tm = BM, tw = (E + 15) / 16 * 16;  // halved while every tile still has an SM of its own
  while (tm > 32 && (N + tm / 2 - 1) / (tm / 2) <= sms) tm >>= 1;
  auto tiles_of = [&](int w) { return (int64_t)((N + tm - 1) / tm) * ((E + w - 1) / w + (wsg && w < E)); };
  if (tw > 32 && tiles_of(32) <= sms) tw = 32;
  if (tw > 16 && tiles_of(16) <= sms) tw = 16;
  const bool with_s = wsg != nullptr && E <= tw;
  // k-blocks per stage: one TMA instruction for several, as long as at least four stages are left; whole tiles are bound by their bytes
  const int kb_bytes = (tm + tw) * BK * 2 + (with_s ? GT_S_BYTES : 0);
  int ks = GT_RING / 4 / kb_bytes;
  ks = ks < 1 || tm == BM ? 1 : ks > 4 ? 4 : ks;
  if (ks > kfull) ks = kfull > 0 ? kfull : 1;
  GateMaps m;
  int rc = make_map(&m.x_tail, X, d, N, 0, BK, tm);
  if (!rc) rc = make_map(&m.w_tail, Wg, d, E, 0, BK, tw);
  if (!rc) rc = make_map(&m.s_tail, wsg ? wsg : Wg, d, 1, 0, BK, 16);
  if (rc) return rc;
  m.x = m.x_tail; m.w = m.w_tail; m.s = m.s_tail;  // without a whole k-block not read; W and wsg k-block by k-block where they alternate
  if (kfull > 0) {
    rc = slab_map(&m.x, X, d, N, kfull, 1, tm, ks);
    if (!rc && !with_s) rc = slab_map(&m.w, Wg, d, E, kfull, 1, tw, ks);
    if (!rc && !with_s && wsg) rc = slab_map(&m.s, wsg, d, 1, kfull, 1, tw, ks);
    if (rc) return rc;
  }
  if (!with_s && wsg && (rc = make_map(&m.s_tail, wsg, d, 1, 0, BK, tw))) return rc;
  const int grid = (int)(tiles_of(tw) < sms ? tiles_of(tw) : sms);
  const bool whole = tm == BM && E <= tw;
  C2R_CUDA(launch_chained(gate_kernel(whole ? tw : 0, wsg != nullptr), grid, GT_THREADS, GT_SMEM, s, m, L, z, N, d, E, wsg != nullptr, tm, tw, ks, status));
  C2R_LAUNCH_CHECK();
  return C2R_OK;
}

}  // namespace c2r
