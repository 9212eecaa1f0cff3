// Shared host/device helpers of the C2R library (internal; the public surface is include/c2r.h).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "c2r.h"

namespace c2r {

extern thread_local int g_last_cuda_error;
extern unsigned long long g_launch_count;  // kernels launched by this library in this process

inline int cuda_fail(cudaError_t e) {
  g_last_cuda_error = (int)e;
  return C2R_ERR_CUDA;
}

#define C2R_CUDA(expr)                                  \
  do {                                                  \
    cudaError_t _e = (expr);                            \
    if (_e != cudaSuccess) return ::c2r::cuda_fail(_e); \
  } while (0)

#define C2R_LAUNCH_CHECK()                                        \
  do {                                                            \
    __atomic_fetch_add(&::c2r::g_launch_count, 1ull, __ATOMIC_RELAXED); \
    C2R_CUDA(cudaGetLastError());                                 \
  } while (0)

#define C2R_REQUIRE(cond, code) \
  do {                          \
    if (!(cond)) return (code); \
  } while (0)

inline int check_config(const c2r_config* c) {
  if (!c) return C2R_ERR_INVALID_ARG;
  if (c->dtype != C2R_F32 && c->dtype != C2R_BF16) return C2R_ERR_INVALID_ARG;
  if (c->N < 0 || c->d <= 0 || c->E <= 0 || c->K <= 0 || c->row_align < 1) return C2R_ERR_INVALID_ARG;
  if (c->K > 8 || c->K > c->E) return C2R_ERR_UNSUPPORTED_SHAPE;
  if (c->E > 64 || (c->I_s > 0 && c->E > 63)) return C2R_ERR_UNSUPPORTED_SHAPE;
  if (c->d % 8 != 0) return C2R_ERR_UNSUPPORTED_SHAPE;
  if (c->I < 0 || c->I % 16 != 0 || c->I_s < 0 || c->I_s % 16 != 0) return C2R_ERR_UNSUPPORTED_SHAPE;
  if ((int64_t)c->N * c->K >= (1ll << 30)) return C2R_ERR_UNSUPPORTED_SHAPE;
  return C2R_OK;
}

inline int64_t round_up(int64_t x, int64_t a) { return (x + a - 1) / a * a; }

inline int64_t permuted_rows(const c2r_config* c) {
  return round_up((int64_t)c->N * c->K + (int64_t)c->E * (c->row_align - 1), c->row_align);
}

// Tokens owned by one block of the dispatch's counting sort: the largest count that keeps a block at no
// more than 512 slots and a whole number of 32-slot groups (K = 1, 2, 4, 8: exactly 512 slots).
__host__ __device__ inline int perm_tokens_per_block(int K) {
  const int m = 32 / (K & -K);  // tokens per whole number of 32-slot groups (K <= 8)
  return (512 / K) / m * m;
}

inline cudaStream_t as_stream(void* s) { return reinterpret_cast<cudaStream_t>(s); }

// Every kernel of the library is launched so that its blocks may start while the last blocks of the kernel before it on the
// stream still run (programmatic dependent launch), and begins with chain_begin(): let the next kernel do the same, then
// wait until the kernel before has completed and its writes are visible.  What overlaps is launch latency, block start-up,
// barrier and tensor-memory set-up -- a layer is 7 to 30 launches, most of them a few microseconds long (us without / with:
// forward pass of 1 token 88 / 74, of 64 tokens 233 / 221, fp32 training step of 1500 tokens 206 / 193; calibration, two-stage
// dispatch and passes past 0.5 ms move by no more than their spread).  No kernel may return, or touch what an earlier one
// reads or writes, before the wait: the next one relies on this one's completion to imply that of all earlier ones.
//
// MAX_SPLIT (the CUDA-core GEMMs): the largest split of the SM's L1 in favour of shared memory.  An SM must be empty to change the
// split, so a chain of kernels that each take the smallest one that holds them cannot overlap (smallest / largest: expert calls of
// a training step of 1500 fp32 tokens 111.4 / 106.4, whole training step of 300 173 / 149).  Routing and dispatch leave it alone: the row
// pass behind them reads through the L1 that they leave (two-stage dispatch of 25000 tokens of 1536, one expert each, 61.5 / 65.7).
template <bool MAX_SPLIT = false, typename... P, typename... A>
inline cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchConfig_t c = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
  attr[1].val.sharedMemCarveout = cudaSharedmemCarveoutMaxShared;
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = s;
  c.attrs = attr;
  c.numAttrs = MAX_SPLIT ? 2 : 1;
  return cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}

// Dynamic shared memory for a kernel of few blocks, `need` bytes each, that holds them at an even number per SM.  The blocks of a
// chained kernel become resident as the SMs of the kernel before it fall free, and the first SMs to do so take as many as fit:
// seven routing blocks on one SM, bound by its issue slots, while most of the chip waits (4096 tokens behind a pair GEMM: 24 us where
// the kernel alone takes 9).  A block counts with what it asks for, so it asks for its share of an SM.
// Its static shared memory and what the SM keeps for every block are part of the share: left out, with 22 KB of its own a block of the
// two-stage dispatch's ranking took a third of an SM where a fourth was meant (both stages' indices of 24000 tokens, top-4, 14.3 us; so, and
// with 14 KB, 12.5; 50000 tokens 22.5 / 19.2).
constexpr int SPREAD_SMS = 148, SPREAD_SMEM = 120 * 1024, SM_SMEM = 228 * 1024, SM_SMEM_PER_BLOCK = 1024;
constexpr int spread_share(int per_sm, int static_bytes) {
  const int dynamic = SM_SMEM / (per_sm + 1) + 512 - SM_SMEM_PER_BLOCK - static_bytes;
  return dynamic > 0 ? dynamic : 0;
}
constexpr bool spread_holds(int per_sm, int static_bytes) {  // so many blocks fit and one more does not
  const int block = (spread_share(per_sm, static_bytes) + static_bytes + 127) / 128 * 128 + SM_SMEM_PER_BLOCK;
  return per_sm * block <= SM_SMEM && (per_sm + 1) * block > SM_SMEM;
}
static_assert(spread_holds(1, 0) && spread_holds(2, 0) && spread_holds(3, 13824) && spread_holds(4, 13824) && spread_holds(8, 768) && spread_holds(8, 13824),
              "blocks per SM");
static_assert(spread_share(1, 0) <= SPREAD_SMEM, "within the kernels' limit");
inline int spread_smem(int64_t blocks, int need, int static_bytes) {
  const int64_t per_sm = (blocks + SPREAD_SMS - 1) / SPREAD_SMS;
  const int share = per_sm > 0 && per_sm <= 8 ? spread_share((int)per_sm, static_bytes) : 0;
  return share > need ? share : need;
}
// Raises a kernel's limit of dynamic shared memory, once per device (`done`: the kernel's static bytes and one more).
template <typename... P>
inline int allow_smem(void (*kernel)(P...), int (&done)[64], int bytes = SPREAD_SMEM, int* static_bytes = nullptr) {
  int dev = 0;
  C2R_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return C2R_ERR_UNSUPPORTED_SHAPE;
  int known = __atomic_load_n(&done[dev], __ATOMIC_ACQUIRE);
  if (known == 0) {
    cudaFuncAttributes a;
    C2R_CUDA(cudaFuncGetAttributes(&a, kernel));
    known = (int)a.sharedSizeBytes + 1;
    C2R_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    __atomic_store_n(&done[dev], known, __ATOMIC_RELEASE);
  }
  if (static_bytes != nullptr) *static_bytes = known - 1;
  return C2R_OK;
}

// ---- device helpers -------------------------------------------------------------------------

__device__ __forceinline__ void chain_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_begin() {
  chain_release();
  chain_wait();
}

template <typename T>
struct Vec16;  // 16-byte vector of T
template <>
struct Vec16<float> {
  static constexpr int N = 4;
  float4 v;
  __device__ void load(const float* p) { v = *reinterpret_cast<const float4*>(p); }
  __device__ void store(float* p) const { *reinterpret_cast<float4*>(p) = v; }
  __device__ void to_float(float* f) const { f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w; }
  __device__ void from_float(const float* f) { v = make_float4(f[0], f[1], f[2], f[3]); }
};
template <>
struct Vec16<__nv_bfloat16> {
  static constexpr int N = 8;
  uint4 v;
  __device__ void load(const __nv_bfloat16* p) { v = *reinterpret_cast<const uint4*>(p); }
  __device__ void store(__nv_bfloat16* p) const { *reinterpret_cast<uint4*>(p) = v; }
  __device__ void to_float(float* f) const {
    const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      f[2 * i] = __uint_as_float(u[i] << 16);
      f[2 * i + 1] = __uint_as_float(u[i] & 0xFFFF0000u);
    }
  }
  __device__ void from_float(const float* f) {
    uint32_t u[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      __nv_bfloat162 h = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
      u[i] = *reinterpret_cast<uint32_t*>(&h);
    }
    v = make_uint4(u[0], u[1], u[2], u[3]);
  }
};

__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 x) { return __bfloat162float(x); }
template <typename T>
__device__ __forceinline__ T from_f32(float x);
template <>
__device__ __forceinline__ float from_f32<float>(float x) { return x; }
template <>
__device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float x) { return __float2bfloat16_rn(x); }


}  // namespace c2r
