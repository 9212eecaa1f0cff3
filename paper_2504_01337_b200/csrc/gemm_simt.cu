// CUDA-core grouped GEMMs for the expert MLPs: the fp32 path (exact-arithmetic configurations)
// and any bf16 shape the tensor-core kernels do not cover.  Also the W1/W3 packing helpers.
#include "c2r_common.cuh"
#include "gemm.h"

namespace c2r {

__host__ __device__ inline int pack_col(int i, int I) {
  const int j = i >> 7;
  return (j << 8) + (i - (j << 7));
}
__host__ __device__ inline int pack_width(int i, int I) {
  const int j = i >> 7;
  const int rem = I - (j << 7);
  return rem < 128 ? rem : 128;
}

// rows of W1 / W3  <->  rows of W13p
template <typename T>
__global__ void pack_kernel(const T* __restrict__ W1, const T* __restrict__ W3, T* __restrict__ W13p, int I, int d,
                            int unpack, T* __restrict__ W1o, T* __restrict__ W3o) {
  chain_begin();
  using V = Vec16<T>;
  const int e = blockIdx.y;
  const int i = blockIdx.x;
  const int pg = pack_col(i, I), pu = pg + pack_width(i, I);
  const size_t src = ((size_t)e * I + i) * d;
  const size_t dg = ((size_t)e * 2 * I + pg) * d, du = ((size_t)e * 2 * I + pu) * d;
  for (int c = threadIdx.x * V::N; c < d; c += blockDim.x * V::N) {
    V a, b;
    if (!unpack) {
      a.load(W1 + src + c);
      b.load(W3 + src + c);
      a.store(W13p + dg + c);
      b.store(W13p + du + c);
    } else {
      a.load(W13p + dg + c);
      b.load(W13p + du + c);
      a.store(W1o + src + c);
      b.store(W3o + src + c);
    }
  }
}


// Four consecutive elements of a shared-memory tile as floats.
__device__ __forceinline__ float4 tile4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 tile4(const __nv_bfloat16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u), __uint_as_float(u.y << 16),
                     __uint_as_float(u.y & 0xFFFF0000u));
}

constexpr int SPAN = 32;  // k-elements of a tile

// A tile of W rows (columns of the output) x SPAN k of one operand on its way to shared memory by cp.async, in the order in which
// it lies in global memory: KM (k contiguous) as [W][SPAN] with rows padded against bank conflicts, else as [SPAN][W].
// Addresses are worked out once and advanced: the small problems are bound by instructions as much as by latency.
template <typename T, int W, bool KM, int THREADS>
struct TileLoad {
  static constexpr int EPC = 16 / sizeof(T);                                    // elements per 16-byte piece
  static constexpr int PITCH = KM ? SPAN + EPC : W;                             // elements per row of the tile
  static constexpr int ELEMS = KM ? W * PITCH : SPAN * W;
  static constexpr int PIECES = W * SPAN / EPC, PER = (PIECES + THREADS - 1) / THREADS;
  const T* src[PER];   // next piece; NULL where the tile has no such row
  int k_of[PER], at[PER];
  long long step;
  // row(m): address of element (m, 0); element (m, k) lies k * sk further, and without KM rows lie next to each other
  template <typename Row>
  __device__ __forceinline__ void init(Row row, long long sk, int m_left) {
    step = SPAN * sk;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const int x = threadIdx.x + i * THREADS;
      const int k = KM ? EPC * (x % (SPAN / EPC)) : x / (W / EPC), m = KM ? x / (SPAN / EPC) : EPC * (x % (W / EPC));
      k_of[i] = k;
      at[i] = KM ? m * PITCH + k : k * W + m;
      src[i] = (PIECES % THREADS == 0 || x < PIECES) && m < m_left ? row(m) + k * sk : nullptr;
    }
  }
  // any: an aligned address that may be named where nothing is read.  V16: pieces are aligned; else vec (simt_vec) says how far.
  template <bool V16>
  __device__ __forceinline__ void fetch(T* tile, int k_left, int vec, const T* any) {
    T plain[PER][EPC];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      if (PIECES % THREADS != 0 && (int)threadIdx.x + i * THREADS >= PIECES) continue;
      const bool live = src[i] != nullptr && k_of[i] < k_left;
      const T* from = live ? src[i] : any;
      const uint32_t to = (uint32_t)__cvta_generic_to_shared(tile + at[i]);
      const int n = live ? 16 : 0;
      if (V16) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to), "l"(from), "r"(n) : "memory");
      } else if (vec == 8) {
#pragma unroll
        for (int j = 0; j < 16; j += 8)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(to + j), "l"((const char*)from + (live ? j : 0)), "r"(n >> 1) : "memory");
      } else if (vec == 4) {
#pragma unroll
        for (int j = 0; j < 16; j += 4)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(to + j), "l"((const char*)from + (live ? j : 0)), "r"(n >> 2) : "memory");
      } else if (sizeof(T) == 2) {
#pragma unroll
        for (int j = 0; j < EPC; ++j) plain[i][j] = live ? src[i][j] : from_f32<T>(0.f);
      }
      if (src[i] != nullptr) src[i] += step;
    }
    if (!V16 && sizeof(T) == 2 && vec == 0) {
#pragma unroll
      for (int i = 0; i < PER; ++i) {
        if (PIECES % THREADS != 0 && (int)threadIdx.x + i * THREADS >= PIECES) continue;
#pragma unroll
        for (int j = 0; j < EPC; ++j) tile[at[i] + j] = plain[i][j];
      }
    }
  }
  // The four rows (columns of the output) that thread t of W / 4 has, and their elements k .. k + 3: v[row][k].
  static __device__ __forceinline__ int row_of(int t, int i) { return KM ? t + (W / 4) * i : 4 * t + i; }
  static __device__ __forceinline__ void read(const T* tile, int t, int k, float (&v)[4][4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 x = tile4(KM ? tile + row_of(t, i) * PITCH + k : tile + (k + i) * W + 4 * t);
      const float e[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (KM) v[i][j] = e[j];
        else v[j][i] = e[j];
      }
    }
  }
};

// Blocks per SM that the register limit has to allow.
template <bool DUAL, int TM, int TN>
constexpr int simt_min_blocks = DUAL || (TM == 64 && TN == 64) ? 2 : 1;

// C_g(m,n) = sum_k A_g(m,k) B_g(n,k) with arbitrary strides; see SimtGemm for the two modes.
//
// A block computes TM x TN outputs; (TM / 4)(TN / 4) threads hold a 4 x 4 share each.  A sum over k is kept as S partial sums,
// part j over the j-th of S equal pieces of every SPAN consecutive k, added in part order at the end.  Groups of threads keep
// a part each, or a thread keeps all: a result does not depend on the tile its batch was given, and is nearer to the
// exact sum than one chain is.  STAGES - 1 tiles of both operands are on their way (cp.async) while one is used.  The small
// configurations this serves are bound by latency and by the operands' way from shared memory (two 16-byte reads per 16 products;
// 8 x 8 outputs per thread halve those, but leave too few warps: training step of 1500 tokens 159 us, so 222).  Tiles that went
// through registers, one ahead, transposed on their way, took, in us before / after for expert calls (forward + backward): fp32, top-2 of 8
// experts of 128, d 256: 100 tokens 50.3 / 41.4, 512 70.7 / 57.0, 1500 120 / 99; 2600 tokens of 512, top-4 of 8 x 512 1767 / 1468; bf16 off
// the tensor-core shapes (8192 tokens of 264, top-2 of 8 x 512) 2406 / 1583; fp32 arrays on no 16-byte boundary (2600 tokens) 2179 / 1993,
// bf16 on an 8-byte one (512 tokens of 264) 87 / 65.  Left to itself the compiler holds the 32-wide forms to 60 registers, which costs the
// small launches a third (512 tokens 57.0 / 74.4), and gives the 64 x 64 ones more than half an SM's.
// 64 x 64 tiles where they fill the chip, else 32-wide ones; the two SwiGLU products always take 32 x 32, since at 64 x 64 their
// parts are 128 registers of a thread and one block per SM.
// Blocks: y = tile along N; x = tile along M -- SIMT_ROWS: over all groups' row tiles, found from the counts -- ; z = group
// (SIMT_WGRAD).
template <typename T, typename TC, int TM, int TN, bool DUAL, int S, bool AK, bool BN, int STAGES, bool V16, int SIMT_THREADS>
__global__ void __launch_bounds__(SIMT_THREADS, simt_min_blocks<DUAL, TM, TN>) simt_gemm_kernel(SimtGemm g) {
  chain_begin();
  using LA = TileLoad<T, TM, AK, SIMT_THREADS>;
  using LB = TileLoad<T, TN, BN, SIMT_THREADS>;
  constexpr int GROUP = (TM / 4) * (TN / 4), G = SIMT_THREADS / GROUP;  // threads per group, groups
  constexpr int PART = SPAN / S, O = S / G;                             // length of a part; a thread's parts per tile
  static_assert(!DUAL || G > 1, "two products keep their parts in groups");
  static_assert(PART % 4 == 0 && (G == 1 || O == 1), "a group of threads keeps one part, or a thread all of them");
  constexpr int MR = G == 1 ? 4 : TM * TN / (4 * SIMT_THREADS);         // output rows a thread finishes, four columns each
  constexpr int STAGE = LA::ELEMS + (DUAL ? 2 : 1) * LB::ELEMS;
  extern __shared__ __align__(16) uint8_t smem_raw[];
  T* const tiles = reinterpret_cast<T*>(smem_raw);
  float* const smem = reinterpret_cast<float*>(smem_raw);
  __shared__ float sred[TM][TN / 4 + 1];  // per-row partial dots of the SwiGLU backward, one column per thread column
  const int tid = threadIdx.x, lane = tid & 31;
  int grp, m0, M, Kd;
  long long a_off, b_off, c_off, r0 = 0;
  if (g.counts == nullptr) {  // one group whose size the host knows
    grp = 0; m0 = blockIdx.x * TM; M = g.Mdim; Kd = g.Kdim;
    a_off = b_off = c_off = 0;
  } else if (g.mode == SIMT_ROWS) {
    // row tiles are numbered through the groups; every warp finds the group of tile blockIdx.x by a scan over the counts
    const int n0 = lane < g.n_groups ? (max(g.counts[lane], 0) + TM - 1) / TM : 0;
    const int n1 = lane + 32 < g.n_groups ? (max(g.counts[lane + 32], 0) + TM - 1) / TM : 0;
    int s0 = n0, s1 = n1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int x0 = __shfl_up_sync(0xffffffffu, s0, o), x1 = __shfl_up_sync(0xffffffffu, s1, o);
      if (lane >= o) { s0 += x0; s1 += x1; }
    }
    s1 += __shfl_sync(0xffffffffu, s0, 31);
    const int y = blockIdx.x;
    const uint32_t in0 = __ballot_sync(0xffffffffu, y >= s0 - n0 && y < s0), in1 = __ballot_sync(0xffffffffu, y >= s1 - n1 && y < s1);
    if (!(in0 | in1)) return;
    const int src = in0 ? __ffs(in0) - 1 : __ffs(in1) - 1;
    grp = in0 ? src : 32 + src;
    m0 = (y - __shfl_sync(0xffffffffu, in0 ? s0 - n0 : s1 - n1, src)) * TM;
    M = g.counts[grp]; r0 = g.offsets[grp]; Kd = g.Kdim;
    a_off = r0 * g.sam; b_off = (long long)grp * g.sB; c_off = r0 * g.ldc;
  } else {
    grp = blockIdx.z; m0 = blockIdx.x * TM; M = g.Mdim;
    Kd = g.counts[grp]; r0 = g.offsets[grp];
    a_off = r0 * g.sak; b_off = r0 * g.sbk; c_off = (long long)grp * g.sC;
  }
  const int n0 = blockIdx.y * TN;
  if (m0 >= M || n0 >= g.Ndim) return;
  const T* A = (const T*)g.A + a_off + (long long)m0 * g.sam;
  const T* B = (const T*)g.B + b_off;
  const int vec = g.vec;
  auto rowA = [&](int m) { return A + (long long)m * g.sam; };
  auto rowB = [&](int n) {
    if (g.B_last != nullptr && n0 + n == g.Ndim - 1) return (const T*)g.B_last;
    return B + (long long)(DUAL ? pack_col(n0 + n, g.I) : n0 + n) * g.sbn;
  };
  auto rowB2 = [&](int n) { return B + (long long)(pack_col(n0 + n, g.I) + pack_width(n0 + n, g.I)) * g.sbn; };

  const int grp_k = tid / GROUP, tg = tid % GROUP;
  const int tx = tg % (TN / 4), ty = tg / (TN / 4);
  float sum[O][4][4] = {}, sum2[DUAL ? O : 1][4][4] = {};
  LA la;
  LB lb, lb2;
  la.init(rowA, g.sak, M - m0);
  lb.init(rowB, g.sbk, g.Ndim - n0);
  if (DUAL) lb2.init(rowB2, g.sbk, g.Ndim - n0);
  const int n_tiles = (Kd + SPAN - 1) / SPAN;
  auto fetch = [&](int t) {
    if (t < n_tiles) {
      T* sa = tiles + t % STAGES * STAGE;
      la.template fetch<V16>(sa, Kd - t * SPAN, vec, (const T*)g.A);
      lb.template fetch<V16>(sa + LA::ELEMS, Kd - t * SPAN, vec, (const T*)g.A);
      if (DUAL) lb2.template fetch<V16>(sa + LA::ELEMS + LB::ELEMS, Kd - t * SPAN, vec, (const T*)g.A);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int t = 0; t < STAGES - 1; ++t) fetch(t);
  for (int t = 0; t < n_tiles; ++t) {
    asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
    __syncthreads();  // tile t is there, and the one before it is no longer read
    fetch(t + STAGES - 1);
    const T* sa = tiles + t % STAGES * STAGE;
    const T* sb = sa + LA::ELEMS;
    const T* sb2 = sb + LB::ELEMS;
#pragma unroll
    for (int q = 0; q < O; ++q) {
#pragma unroll 4
      for (int k4 = 0; k4 < PART; k4 += 4) {
        const int k = (G == 1 ? q : grp_k) * PART + k4;
        float av[4][4], bv[4][4];
        LA::read(sa, ty, k, av);
        LB::read(sb, tx, k, bv);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) sum[q][i][j] = fmaf(av[i][kk], bv[j][kk], sum[q][i][j]);
        if (DUAL) {
          LB::read(sb2, tx, k, bv);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int j = 0; j < 4; ++j) sum2[DUAL ? q : 0][i][j] = fmaf(av[i][kk], bv[j][kk], sum2[DUAL ? q : 0][i][j]);
        }
      }
    }
  }
  // this thread's outputs: rows m_of(i), columns n_of(j) of the tile
  auto m_of = [&](int i) { return G == 1 ? LA::row_of(ty, i) : tid / (TN / 4) + i * (SIMT_THREADS / (TN / 4)); };
  auto n_of = [&](int j) { return G == 1 ? LB::row_of(tx, j) : 4 * (tid % (TN / 4)) + j; };
  float(&acc)[4][4] = sum[0];
  float(&acc2)[4][4] = sum2[0];
  // the parts added in part order: a thread's own, or all groups' through shared memory
  constexpr int P = TN + 4;
  if (G > 1) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float* row = &smem[(grp_k * TM + LA::row_of(ty, i)) * P];
      if constexpr (BN) {
#pragma unroll
        for (int j = 0; j < 4; ++j) row[LB::row_of(tx, j)] = acc[i][j];
      } else {  // four columns in a row
        *reinterpret_cast<float4*>(row + 4 * tx) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
      }
      if (DUAL) {
#pragma unroll
        for (int j = 0; j < 4; ++j) row[G * TM * P + LB::row_of(tx, j)] = acc2[i][j];
      }
    }
    __syncthreads();
  }
  if (S > 1) {
#pragma unroll
    for (int i = 0; i < MR; ++i) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float v = 0.f, v2 = 0.f;
#pragma unroll
        for (int q = 0; q < S; ++q) {
          v += G == 1 ? sum[q < O ? q : 0][i][j] : smem[(q * TM + m_of(i)) * P + n_of(j)];
          if (DUAL) v2 += smem[((G + q) * TM + m_of(i)) * P + n_of(j)];
        }
        acc[i][j] = v;
        if (DUAL) acc2[i][j] = v2;
      }
    }
  }
  TC* C = (TC*)g.C + c_off;
  const bool want_q = g.epi == SIMT_EPI_SWIGLU_BWD && g.qpart != nullptr;
#pragma unroll
  for (int i = 0; i < MR; ++i) {
    const int lm = m_of(i), m = m0 + lm;
    float qrow = 0.f;
    const int col4 = G == 1 ? tx : tid % (TN / 4);
    if (want_q) sred[lm][col4] = 0.f;
    if (m >= M) continue;
    float sc = 1.f;  // per-row scale of H (SwiGLU forms)
    if (g.scale_kind != 0 && g.row_scale != nullptr) {
      const float v = g.row_scale[r0 + m];
      sc = g.scale_kind == 2 ? 1.0f / (1.0f + expf(-v)) : v;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + n_of(j);
      if (n >= g.Ndim) continue;
      float v = acc[i][j];
      if (DUAL) {
        // v = A[r,n], acc2 = B[r,n]: H = silu(A) * B; the backward pass needs only the two local
        // derivatives dH/dA = B silu'(A) and dH/dB = silu(A), which are what is kept (packed columns)
        const int pg = pack_col(n, g.I), pu = pg + pack_width(n, g.I);
        const float b = acc2[i][j];
        const float sg = 1.0f / (1.0f + expf(-v));
        const float as = v * sg;
        if (g.C != nullptr) {  // inference: nothing is kept for a backward pass
          T* sv = (T*)g.C + (long long)(r0 + m) * 2 * g.I;
          sv[pg] = from_f32<T>(b * (sg + as - as * sg));
          sv[pu] = from_f32<T>(as);
        }
        ((T*)g.aux_out)[(long long)(r0 + m) * g.I + n] = from_f32<T>(sc * (as * b));
      } else if (g.epi == SIMT_EPI_STORE && g.token_acc != nullptr) {
        // fused combine: the row is added into its token's accumulator (fp32 atomics, order not fixed)
        const int sl = g.slot_of_row[r0 + m];
        if (sl >= 0) atomicAdd(g.token_acc + (long long)(sl / g.slots_per_token) * g.ldc + n, v);
      } else if (g.epi == SIMT_EPI_STORE) {
        TC* o = (g.C_last != nullptr && n == g.Ndim - 1) ? (TC*)g.C_last + m : C + (long long)m * g.ldc + n;
        if (g.accumulate) v += to_f32(*o);
        *o = from_f32<TC>(v);
      } else {  // SIMT_EPI_SWIGLU_BWD: v = dH[r, n]; dA = dH * (dH/dA), dB = dH * (dH/dB) at the packed columns
        const int pg = pack_col(n, g.I), pu = pg + pack_width(n, g.I);
        const T* sv = (const T*)g.aux + (long long)(r0 + m) * 2 * g.I;
        T* dab = (T*)g.C + (long long)(r0 + m) * 2 * g.I;
        dab[pg] = from_f32<T>(sc * v * to_f32(sv[pg]));
        dab[pu] = from_f32<T>(sc * v * to_f32(sv[pu]));
        if (want_q) qrow = fmaf(v, to_f32(((const T*)g.aux2)[(long long)(r0 + m) * g.I + n]), qrow);
      }
    }
    if (want_q) sred[lm][col4] = qrow;
  }
  if (want_q) {  // (uniform across the block) row dots <dH_r, H_r> over this block's 64 columns, in column order
    __syncthreads();
    if (tid < TM && m0 + tid < M) {
      float q = 0.f;
#pragma unroll
      for (int x = 0; x < TN / 4; ++x) q += sred[tid][x];
      g.qpart[(long long)blockIdx.y * g.R + r0 + m0 + tid] = q;
    }
  }
}

template <int STAGES, bool V16, typename T, typename TC, int TM, int TN, bool DUAL, int S, bool AK, bool BN, int SIMT_THREADS>
static int simt_launch_stages(const SimtGemm& g, dim3 grid, cudaStream_t s) {
  constexpr int G = SIMT_THREADS / ((TM / 4) * (TN / 4));
  constexpr int tiles = STAGES * (int)sizeof(T) * (TileLoad<T, TM, AK, SIMT_THREADS>::ELEMS + (DUAL ? 2 : 1) * TileLoad<T, TN, BN, SIMT_THREADS>::ELEMS);
  constexpr int red = G == 1 ? 0 : (DUAL ? 2 : 1) * G * TM * (TN + 4) * 4, smem = tiles > red ? tiles : red;
  static int done[64] = {};
  if (const int rc = allow_smem(simt_gemm_kernel<T, TC, TM, TN, DUAL, S, AK, BN, STAGES, V16, SIMT_THREADS>, done, smem)) return rc;
  C2R_CUDA(launch_chained<true>(simt_gemm_kernel<T, TC, TM, TN, DUAL, S, AK, BN, STAGES, V16, SIMT_THREADS>, grid, SIMT_THREADS, smem, s, g));
  C2R_LAUNCH_CHECK();
  return C2R_OK;
}
// Four stages, or two where they would be room taken for nothing: small launches, which begin beside the one before them if they fit, and
// weight gradients over at most two tiles of rows (us, expert calls, four everywhere / so: forward of 100 tokens, top-2 of 8 experts of
// 128, d 256, 19.8 / 17.6, of 512 23.1 / 21.6; backward of 100 tokens 35.5 / 29.7; two everywhere costs a training step of 1500
// 106 / 114).
template <typename T, typename TC, int TM, int TN, bool DUAL, int S, bool AK, bool BN, int SIMT_THREADS = 256>
static int simt_launch_tile(const SimtGemm& g, int m_tiles, int z, cudaStream_t s) {
  const dim3 grid(m_tiles, (g.Ndim + TN - 1) / TN, z);
  const bool two = g.mode == SIMT_ROWS ? (int64_t)grid.x * grid.y * z <= 3 * 148 : g.expect_k <= 2 * SPAN;
  if (g.vec != 16) return simt_launch_stages<4, false, T, TC, TM, TN, DUAL, S, AK, BN, SIMT_THREADS>(g, grid, s);
  return two ? simt_launch_stages<2, true, T, TC, TM, TN, DUAL, S, AK, BN, SIMT_THREADS>(g, grid, s)
             : simt_launch_stages<4, true, T, TC, TM, TN, DUAL, S, AK, BN, SIMT_THREADS>(g, grid, s);
}

// Bytes of a cp.async that every 16-byte piece the kernel loads is aligned to: 16, 8, 4, or 0 for elements of two bytes that lie on no
// 4-byte boundary.
template <typename T>
static int simt_vec(const SimtGemm& g) {
  const uint64_t bits = (uint64_t)(uintptr_t)g.A | (uintptr_t)g.B | (uintptr_t)g.B_last |
                        sizeof(T) * (uint64_t)((g.sak == 1 ? g.sam : g.sak) | (g.sbk == 1 ? g.sbn : g.sbk) | g.sB);
  return (bits & 15u) == 0 ? 16 : (bits & 7u) == 0 ? 8 : (bits & 3u) == 0 ? 4 : 0;
}

// max_m: rows (SIMT_ROWS: of all groups together) or Mdim.  AK / BN: the contraction index is the contiguous one of A / of B.
template <bool AK, bool BN, typename T, typename TC = T>
int simt_launch(SimtGemm g, int n_groups, int64_t max_m, cudaStream_t s) {
  if (n_groups == 0 || max_m == 0 || g.Ndim == 0) return C2R_OK;
  g.n_groups = n_groups;
  g.vec = simt_vec<T>(g);
  const bool rows = g.mode == SIMT_ROWS && g.counts != nullptr;
  const int z = rows ? 1 : n_groups;
  // SIMT_ROWS: whole tiles of all groups, and one more per group for its remainder
  auto m_tiles = [&](int tm) { return (int)((max_m + tm - 1) / tm) + (rows ? n_groups : 0); };
  const int64_t blocks64 = (int64_t)((max_m + 63) / 64) * ((g.Ndim + 63) / 64) * z;
  const bool large = blocks64 >= 2 * 148;
  // four partial sums; two in the backward of SwiGLU, whose partial row dots cover 64 columns each
  if constexpr (AK && BN) {
    if (g.epi == SIMT_EPI_SWIGLU_FWD) return simt_launch_tile<T, TC, 32, 32, true, 4, AK, BN>(g, m_tiles(32), z, s);
  }
  if constexpr (AK && !BN) {
    if (g.epi == SIMT_EPI_SWIGLU_BWD)
      return large ? simt_launch_tile<T, TC, 64, 64, false, 2, AK, BN>(g, m_tiles(64), z, s)
                   : simt_launch_tile<T, TC, 32, 64, false, 2, AK, BN>(g, m_tiles(32), z, s);
  }
  return large ? simt_launch_tile<T, TC, 64, 64, false, 4, AK, BN>(g, m_tiles(64), z, s)
               : simt_launch_tile<T, TC, 32, 32, false, 4, AK, BN>(g, m_tiles(32), z, s);
}

// Gate logits (Eq. 1) of fp32 layers: L = X Wg^T and, as one more row of the other operand, z = X wsg.  Every logit is one chain of
// products in k order, whatever the batch (near-ties must not move with it), so the time is that of a chain, 4 cycles a
// product, if nothing else is in its way: a block brings its tokens' rows and the whole gate in as few waits as shared memory
// allows, and batches are cut so that every SM has a block.  32 x 32 tiles whose k-tiles wait for one another took 25 us of a
// forward pass of 512 tokens and of a training step of 1500 (d 256, 8 experts), this takes 4 and less (whole passes 57 -> 40 and 194 -> 171).
// RT x RE outputs per thread: 1 x 1 where a block has few, 2 x 4 where the operands' way from shared memory would be the bound.
template <int RT, int RE>
__global__ void __launch_bounds__(RT == 1 ? 512 : 256) gate_simt_kernel(const float* __restrict__ X, const float* __restrict__ Wg,
                                                        const float* __restrict__ wsg, float* __restrict__ L, float* __restrict__ z,
                                                        int N, int d, int E, int cols, int tm, int kc, int vec) {
  chain_begin();
  extern __shared__ __align__(16) float s_gate[];  // [2][tm token rows, cols gate rows][kc + 4]
  const int t0 = blockIdx.x * tm, rows = min(tm, N - t0), pitch = kc + 4, buf_floats = (tm + cols) * pitch;
  auto fetch = [&](int k0, int buf) {  // rows of the tile that do not exist are neither loaded nor used
    const int kn = min(kc, d - k0), per = kn >> 2;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(s_gate + buf * buf_floats);
    for (int i = threadIdx.x; i < (rows + cols) * per; i += blockDim.x) {
      const int r = i / per, k = 4 * (i - r * per), c = r - rows;
      const float* src = (c < 0 ? X + (size_t)(t0 + r) * d : c < E ? Wg + (size_t)c * d : wsg) + k0 + k;
      const uint32_t dst = base + (uint32_t)((c < 0 ? r : tm + c) * pitch + k) * 4;
      if (vec) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + 4 * j), "l"(src + j) : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int groups = (cols + RE - 1) / RE;  // thread: tokens RT ty .. , gate rows tx, tx + groups, ..
  const int ty = threadIdx.x / groups, tx = threadIdx.x - ty * groups;
  const bool live = RT * ty < rows;
  float acc[RT][RE] = {};
  fetch(0, 0);
  for (int k0 = 0, buf = 0; k0 < d; k0 += kc, buf ^= 1) {
    if (k0 + kc < d) {
      fetch(k0 + kc, buf ^ 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    if (live) {
      const float* sx = s_gate + buf * buf_floats + RT * ty * pitch;
      const float* sw = s_gate + buf * buf_floats + (tm + tx) * pitch;
      const int kn = min(kc, d - k0);
#pragma unroll 4
      for (int k = 0; k < kn; k += 4) {
        float4 x[RT], w[RE];
#pragma unroll
        for (int i = 0; i < RT; ++i) x[i] = *reinterpret_cast<const float4*>(sx + i * pitch + k);
#pragma unroll
        for (int j = 0; j < RE; ++j)  // (a row past the last gate row is read inside the buffer and not used)
          w[j] = *reinterpret_cast<const float4*>(sw + (tx + j * groups < cols ? j * groups * pitch : 0) + k);
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
          for (int j = 0; j < RE; ++j)
            acc[i][j] = fmaf(x[i].w, w[j].w, fmaf(x[i].z, w[j].z, fmaf(x[i].y, w[j].y, fmaf(x[i].x, w[j].x, acc[i][j]))));
      }
    }
    __syncthreads();  // the buffer may be filled again
  }
  if (!live) return;
#pragma unroll
  for (int i = 0; i < RT; ++i) {
    const int t = RT * ty + i;
    if (t >= rows) break;
#pragma unroll
    for (int j = 0; j < RE; ++j) {
      const int c = tx + j * groups;
      if (c < E) L[(size_t)(t0 + t) * E + c] = acc[i][j];
      else if (c < cols) z[t0 + t] = acc[i][j];
    }
  }
}

static int gate_simt_launch(const c2r_config* cfg, const float* X, const float* Wg, const float* wsg, float* L, float* z, cudaStream_t s) {
  const int cols = cfg->E + (wsg ? 1 : 0), vec = (((uintptr_t)X | (uintptr_t)Wg | (uintptr_t)wsg) & 15u) == 0;
  // a block per SM, at most 32 tokens of it (16 thread rows of two tokens)
  int tm = (cfg->N + SPREAD_SMS - 1) / SPREAD_SMS;
  if (tm > 32) tm = 32;
  const bool wide = tm * cols > 512;
  if (wide) tm = (tm + 1) & ~1;
  const int blocks = (cfg->N + tm - 1) / tm;
  const int outputs = wide ? (tm / 2) * ((cols + 3) / 4) : tm * cols;
  const int threads = outputs < 128 ? 128 : (outputs + 31) / 32 * 32;
  // two buffers where the contraction does not fit one
  const int budget = (blocks <= SPREAD_SMS ? 200 : 100) * 1024;
  int kc = cfg->d;
  if ((tm + cols) * (kc + 4) * 4 > budget) kc = (budget / 2 / 4 / (tm + cols) - 4) / 32 * 32;
  const int need = (cfg->d > kc ? 2 : 1) * (tm + cols) * (kc + 4) * 4, smem = spread_smem(blocks, need, 0);
  static int done[2][64] = {};
  const int rc = wide ? allow_smem(gate_simt_kernel<2, 4>, done[1], 200 * 1024) : allow_smem(gate_simt_kernel<1, 1>, done[0], 200 * 1024);
  if (rc) return rc;
  C2R_CUDA(launch_chained<true>(wide ? gate_simt_kernel<2, 4> : gate_simt_kernel<1, 1>, blocks, threads, smem, s, X, Wg, wsg, L, z, cfg->N, cfg->d,
                          cfg->E, cols, tm, kc, vec));
  C2R_LAUNCH_CHECK();
  return C2R_OK;
}

// The same in fp32 arithmetic for bf16 inputs (the tensor-core kernel takes them wherever tensor maps can be made).
static int gate_simt_launch(const c2r_config* cfg, const __nv_bfloat16* X, const __nv_bfloat16* Wg, const __nv_bfloat16* wsg, float* L, float* z,
                            cudaStream_t s) {
  SimtGemm g{};
  g.mode = SIMT_ROWS; g.epi = SIMT_EPI_STORE;
  g.A = X; g.sam = cfg->d; g.sak = 1; g.B = Wg; g.sbn = cfg->d; g.sbk = 1; g.B_last = wsg;
  g.C = L; g.C_last = wsg ? z : nullptr; g.ldc = cfg->E;
  g.Mdim = cfg->N; g.Ndim = cfg->E + (wsg ? 1 : 0); g.Kdim = cfg->d;
  g.n_groups = 1;
  g.vec = simt_vec<__nv_bfloat16>(g);
  return simt_launch_tile<__nv_bfloat16, float, 32, 32, false, 1, true, true, 64>(g, (cfg->N + 31) / 32, 1, s);
}

template <typename T>
int simt_gate_logits(const c2r_config* cfg, const void* X, const void* Wg, const void* wsg, float* L, float* z, cudaStream_t s) {
  return gate_simt_launch(cfg, (const T*)X, (const T*)Wg, (const T*)wsg, L, z, s);
}
template int simt_gate_logits<float>(const c2r_config*, const void*, const void*, const void*, float*, float*, cudaStream_t);
template int simt_gate_logits<__nv_bfloat16>(const c2r_config*, const void*, const void*, const void*, float*, float*, cudaStream_t);

template <typename T>
int simt_swiglu_fwd(const c2r_config* cfg, const SwigluCall& a, cudaStream_t s) {
  const int d = cfg->d, I = a.I;
  const int64_t max_m = a.R;
  SimtGemm g{};
  g.counts = a.counts; g.offsets = a.offsets; g.mode = SIMT_ROWS; g.I = I; g.R = a.R;
  // A = Xp W1^T, B = Xp W3^T in one pass over Xp; epilogue stores H = s silu(A) * B and the two local derivatives
  g.epi = SIMT_EPI_SWIGLU_FWD; g.aux_out = a.H;
  g.row_scale = a.row_scale; g.scale_kind = a.row_scale ? a.scale_kind : 0;
  g.A = a.Xp; g.sam = d; g.sak = 1; g.B = a.W13p; g.sbn = d; g.sbk = 1; g.sB = (long long)2 * I * d;
  g.C = a.AB; g.ldc = 2 * I; g.Ndim = I; g.Kdim = d;
  int rc = simt_launch<true, true, T>(g, a.nE, max_m, s);
  if (rc) return rc;
  g.epi = SIMT_EPI_STORE; g.aux_out = nullptr; g.row_scale = nullptr; g.scale_kind = 0;
  // Yp = H W2^T  (fp32 partial result)
  g.A = a.H; g.sam = I; g.sak = 1; g.B = a.W2; g.sbn = I; g.sbk = 1; g.sB = (long long)d * I;
  g.C = a.Yp; g.ldc = d; g.Ndim = d; g.Kdim = I;
  g.token_acc = a.token_acc; g.slot_of_row = a.slot_of_row; g.slots_per_token = cfg->K;
  return simt_launch<true, true, T, float>(g, a.nE, max_m, s);
}

template <typename T>
int simt_swiglu_bwd(const c2r_config* cfg, const SwigluCall& a, cudaStream_t s) {
  const int d = cfg->d, I = a.I, nE = a.nE;
  const int64_t max_m = a.R;
  SimtGemm g{};
  g.counts = a.counts; g.offsets = a.offsets; g.I = I; g.R = a.R;
  // dH = dYp W2  (epilogue turns it into dA, dB at the packed columns, and the row dots with H)
  g.mode = SIMT_ROWS; g.epi = SIMT_EPI_SWIGLU_BWD; g.aux = a.AB; g.aux2 = a.H; g.qpart = a.qpart;
  g.row_scale = a.row_scale; g.scale_kind = a.row_scale ? a.scale_kind : 0;
  g.A = a.dYp; g.sam = d; g.sak = 1; g.B = a.W2; g.sbn = 1; g.sbk = I; g.sB = (long long)d * I;
  g.C = a.dAB; g.ldc = 2 * I; g.Ndim = I; g.Kdim = d;
  int rc = simt_launch<true, false, T>(g, nE, max_m, s);
  if (rc) return rc;
  // dXp = dAB W13p  (fp32 partial result)
  g.epi = SIMT_EPI_STORE; g.aux = nullptr; g.aux2 = nullptr; g.qpart = nullptr; g.row_scale = nullptr; g.scale_kind = 0;
  g.A = a.dAB; g.sam = 2 * I; g.sak = 1; g.B = a.W13p; g.sbn = 1; g.sbk = d; g.sB = (long long)2 * I * d;
  g.C = a.dXp; g.ldc = d; g.Ndim = d; g.Kdim = 2 * I;
  g.token_acc = a.token_acc; g.slot_of_row = a.slot_of_row; g.slots_per_token = cfg->K;
  rc = simt_launch<true, false, T, float>(g, nE, max_m, s);
  if (rc) return rc;
  g.token_acc = nullptr;
  // dW2_e = dYp_e^T H_e   [d, I]
  g.mode = SIMT_WGRAD; g.accumulate = a.accumulate; g.expect_k = nE == 1 ? max_m : (int64_t)cfg->N * cfg->K / nE;
  g.A = a.dYp; g.sam = 1; g.sak = d; g.B = a.H; g.sbn = 1; g.sbk = I;
  g.C = a.dW2; g.ldc = I; g.sC = (long long)d * I; g.Mdim = d; g.Ndim = I;
  rc = simt_launch<false, false, T>(g, nE, d, s);
  if (rc) return rc;
  // dW13p_e = dAB_e^T Xp_e   [2I, d]
  g.A = a.dAB; g.sam = 1; g.sak = 2 * I; g.B = a.Xp; g.sbn = 1; g.sbk = d;
  g.C = a.dW13p; g.ldc = d; g.sC = (long long)2 * I * d; g.Mdim = 2 * I; g.Ndim = d;
  return simt_launch<false, false, T>(g, nE, 2 * I, s);
}

template int simt_swiglu_fwd<float>(const c2r_config*, const SwigluCall&, cudaStream_t);
template int simt_swiglu_fwd<__nv_bfloat16>(const c2r_config*, const SwigluCall&, cudaStream_t);
template int simt_swiglu_bwd<float>(const c2r_config*, const SwigluCall&, cudaStream_t);
template int simt_swiglu_bwd<__nv_bfloat16>(const c2r_config*, const SwigluCall&, cudaStream_t);

}  // namespace c2r

using namespace c2r;

static int pack_common(const c2r_config* cfg, int nE, int I, const void* W1, const void* W3, void* W13p, int unpack,
                       void* W1o, void* W3o, void* stream) {
  int rc = check_config(cfg);
  if (rc) return rc;
  C2R_REQUIRE(nE >= 0 && I > 0 && I % 16 == 0, C2R_ERR_UNSUPPORTED_SHAPE);
  if (nE == 0) return C2R_OK;
  dim3 grid(I, nE);
  if (cfg->dtype == C2R_BF16)
    C2R_CUDA(launch_chained(pack_kernel<__nv_bfloat16>, grid, 128, 0, as_stream(stream), (const __nv_bfloat16*)W1, (const __nv_bfloat16*)W3,
                          (__nv_bfloat16*)W13p, I, cfg->d, unpack,
                          (__nv_bfloat16*)W1o, (__nv_bfloat16*)W3o));
  else
    C2R_CUDA(launch_chained(pack_kernel<float>, grid, 128, 0, as_stream(stream), (const float*)W1, (const float*)W3, (float*)W13p, I, cfg->d,
                          unpack, (float*)W1o, (float*)W3o));
  C2R_LAUNCH_CHECK();
  return C2R_OK;
}

extern "C" int c2r_pack_weights(const c2r_config* cfg, int n_experts, int I, const void* W1, const void* W3,
                                void* W13p, void* stream) {
  C2R_REQUIRE(W1 && W3 && W13p, C2R_ERR_INVALID_ARG);
  return pack_common(cfg, n_experts, I, W1, W3, W13p, 0, nullptr, nullptr, stream);
}

extern "C" int c2r_unpack_weights(const c2r_config* cfg, int n_experts, int I, const void* W13p, void* W1, void* W3,
                                  void* stream) {
  C2R_REQUIRE(W1 && W3 && W13p, C2R_ERR_INVALID_ARG);
  return pack_common(cfg, n_experts, I, nullptr, nullptr, (void*)W13p, 1, W1, W3, stream);
}
