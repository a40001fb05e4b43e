// FP32-FMA dense contraction with arbitrary operand strides: the contraction of the fp32 configuration (TF32 tensor-core math
// cannot hold a 1e-4 relative tolerance) and the fall-back for bf16 problems the tcgen05 kernels do not take.  Three kernels:
//   gemm_simt_small_kernel  float, rows aligned: tiles of 32 x 32;
//   gemm_simt_wide_kernel   the same sums in tiles of 64 x 64, many rows of a layer;
//   gemm_simt_kernel        bf16, and float with unaligned rows.
#include <cooperative_groups.h>

#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace bsr {

namespace cg = cooperative_groups;

// A CTA of 128 threads forms a 64 x 64 tile, 8 x 4 outputs per thread: per k step a warp reads 2 + 1 wavefronts of shared
// memory for 1024 multiply-adds, so the FMA pipe is the limit.  Slabs of 32 along k go through registers into two shared
// buffers, the loads of the next slab in flight during the arithmetic of this one.  Products of few tiles (520 x 576 x 192: 81 tiles
// on 148 SMs) leave SMs idle, so a tile's k range is split over the CTAs of a cluster (up to 8), whose
// partial tiles are summed through distributed shared memory in rank order before the epilogue: no second kernel, no
// workspace, the result does not depend on scheduling.  A step of 41 such products took 1310 us with 4 x 4 outputs per thread, no
// split and no loads in flight, 800 us so.
constexpr int SG_BM = 64, SG_BN = 64, SG_BK = 32, SG_THREADS = 128, SG_LD = SG_BM + 4, SG_MAXSPLIT = 8;

// One thread's share (16 values) of a 64 x 32 operand slab: contiguous along k (row r = t % 64, 16 k values) or along its
// own index (four k rows, 4 consecutive values each).  VEC: rows are aligned for four-element accesses.
template <typename T>
__device__ __forceinline__ void slab_load(const T* __restrict__ P, long ld, bool kmajor, bool vec, int r0, int k0, int R, int K, float* v) {
  const int t = threadIdx.x;
  if (kmajor) {
    const int r = r0 + (t & 63), k = k0 + (t >> 6) * 16;
    const T* src = P + (long)r * ld + k;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (vec && r < R && k + q * 4 + 3 < K) load4(src + q * 4, v + q * 4);
      else
#pragma unroll
        for (int j = 0; j < 4; ++j) v[q * 4 + j] = (r < R && k + q * 4 + j < K) ? to_f(src[q * 4 + j]) : 0.f;
    }
  } else {
    const int r = r0 + (t & 15) * 4;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int k = k0 + (t >> 4) + q * 8;
      const T* src = P + (long)k * ld + r;
      if (vec && k < K && r + 3 < R) load4(src, v + q * 4);
      else
#pragma unroll
        for (int j = 0; j < 4; ++j) v[q * 4 + j] = (k < K && r + j < R) ? to_f(src[j]) : 0.f;
    }
  }
}
__device__ __forceinline__ void slab_store(float (*S)[SG_LD], bool kmajor, const float* v) {
  const int t = threadIdx.x;
  if (kmajor) {
#pragma unroll
    for (int i = 0; i < 16; ++i) S[(t >> 6) * 16 + i][t & 63] = v[i];
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) *reinterpret_cast<float4*>(&S[(t >> 4) + q * 8][(t & 15) * 4]) = make_float4(v[q * 4], v[q * 4 + 1], v[q * 4 + 2], v[q * 4 + 3]);
  }
}

template <typename T, typename TC>
struct SimtEpi {
  TC* C;
  const float* bias;
  const TC* residual;
  TC* aux_out;
  const T* aux_in;
  int M, N, act;
  long res_ld;
  bool vec;                                  // all float, rows of whole aligned groups of four
  // four consecutive columns of one row
  __device__ __forceinline__ void operator()(int gm, int gn, const float* acc) const {
    if (gm >= M) return;
    if constexpr (sizeof(T) == 4) {
      if (vec) {
        if (gn >= N) return;
        const size_t o = (size_t)gm * N + gn;
        float v[4], x[4];
        if (bias != nullptr) load16(bias + gn, x);
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = bias != nullptr ? acc[j] + x[j] : acc[j];
        if (act == 1) {
          if (aux_out != nullptr) store16(aux_out + o, v);
#pragma unroll
          for (int j = 0; j < 4; ++j) v[j] = gelu_f(v[j]);
        } else if (act == 2) {
          load16(aux_in + o, x);
#pragma unroll
          for (int j = 0; j < 4; ++j) v[j] *= gelu_grad_f(x[j]);
          if (aux_out != nullptr) {
#pragma unroll
            for (int j = 0; j < 4; ++j) x[j] = gelu_f(x[j]);
            store16(aux_out + o, x);
          }
        }
        if (residual != nullptr) {
          load16(residual + (size_t)gm * res_ld + gn, x);
#pragma unroll
          for (int j = 0; j < 4; ++j) v[j] += x[j];
        }
        store16(C + o, v);
        return;
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (gn + j >= N) continue;
      size_t o = (size_t)gm * N + gn + j;
      float v = acc[j];
      if (bias != nullptr) v += bias[gn + j];
      if (act == 1) {
        if (aux_out != nullptr) aux_out[o] = from_f<TC>(v);
        v = gelu_f(v);
      } else if (act == 2) {
        float z = to_f(aux_in[o]);
        v *= gelu_grad_f(z);
        if (aux_out != nullptr) reinterpret_cast<T*>(aux_out)[o] = from_f<T>(gelu_f(z));     // GELU(z), storage type
      }
      if (residual != nullptr) v += to_f(residual[(size_t)gm * res_ld + gn + j]);
      C[o] = from_f<TC>(v);
    }
  }
};

template <typename T, typename TC>
__global__ void __launch_bounds__(SG_THREADS)
gemm_simt_kernel(const T* __restrict__ A, long lda, int a_kmajor, int a_vec, const T* __restrict__ B, long ldb, int b_kmajor, int b_vec,
                 int K, int k_per_split, SimtEpi<T, TC> epi) {
  __shared__ __align__(16) float As[2][SG_BK][SG_LD];
  __shared__ __align__(16) float Bs[2][SG_BK][SG_LD];
  if (leaves_sms_idle()) release_dependents();
  await_inputs();
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int m0 = blockIdx.y * SG_BM, n0 = blockIdx.x * SG_BN;
  const int splits = gridDim.z, rank = blockIdx.z;
  const int kb = rank * k_per_split, ke = min(K, kb + k_per_split);
  float acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  float va[16], vb[16];
  if (kb < ke) {
    slab_load(A, lda, a_kmajor, a_vec, m0, kb, epi.M, ke, va);
    slab_load(B, ldb, b_kmajor, b_vec, n0, kb, epi.N, ke, vb);
    slab_store(As[0], a_kmajor, va);
    slab_store(Bs[0], b_kmajor, vb);
  }
  __syncthreads();
  int buf = 0;
  for (int k0 = kb; k0 < ke; k0 += SG_BK) {
    const bool more = k0 + SG_BK < ke;
    if (more) {
      slab_load(A, lda, a_kmajor, a_vec, m0, k0 + SG_BK, epi.M, ke, va);
      slab_load(B, ldb, b_kmajor, b_vec, n0, k0 + SG_BK, epi.N, ke, vb);
    }
#pragma unroll 8
    for (int kk = 0; kk < SG_BK; ++kk) {
      float a[8], b[4];
      load16(&As[buf][kk][ty * 8], a);
      load16(&As[buf][kk][ty * 8 + 4], a + 4);
      load16(&Bs[buf][kk][tx * 4], b);
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    if (more) {
      slab_store(As[buf ^ 1], a_kmajor, va);
      slab_store(Bs[buf ^ 1], b_kmajor, vb);
    }
    __syncthreads();
    buf ^= 1;
  }
  if (splits == 1) {
#pragma unroll
    for (int i = 0; i < 8; ++i) epi(m0 + ty * 8 + i, n0 + tx * 4, acc[i]);
    return;
  }
  // partial tile [64][64] over the operand buffers; every rank sums and finishes its share of the tile
  float* part = &As[0][0][0];
  static_assert(sizeof(As) >= SG_BM * SG_BN * sizeof(float), "a partial tile fits the operand buffer");
  cg::cluster_group cluster = cg::this_cluster();
#pragma unroll
  for (int i = 0; i < 8; ++i) store16(part + (ty * 8 + i) * SG_BN + tx * 4, acc[i]);
  cluster.sync();
  constexpr int UNITS = SG_BM * SG_BN / 4;
  const int u1 = UNITS * (rank + 1) / splits;
  for (int u = UNITS * rank / splits + tid; u < u1; u += SG_THREADS) {
    float4 v[SG_MAXSPLIT];
#pragma unroll
    for (int s = 0; s < SG_MAXSPLIT; ++s)
      if (s < splits) v[s] = *reinterpret_cast<const float4*>(cluster.map_shared_rank(part, s) + u * 4);
    float4 t = v[0];
#pragma unroll
    for (int s = 1; s < SG_MAXSPLIT; ++s)
      if (s < splits) { t.x += v[s].x; t.y += v[s].y; t.z += v[s].z; t.w += v[s].w; }
    float o[4] = {t.x, t.y, t.z, t.w};
    epi(m0 + u / (SG_BN / 4), n0 + (u % (SG_BN / 4)) * 4, o);
  }
  cluster.sync();                          // no CTA leaves while another may still read its partial tile
}

__device__ __forceinline__ uint64_t simt_pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void simt_unpack2(uint64_t r, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r)); }
__device__ __forceinline__ uint64_t simt_fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
// The same for products of few tiles (the fp32 configuration's own: 520 x 192 x 192 is 27 tiles of 64).  Tiles of 32 x 32, a CTA of
// 256 threads in four groups of 64: every group forms the whole tile, 4 x 4 products a
// thread (two an instruction, fma.rn.f32x2), over a quarter of each slab of 64 along k, and the four sums are added in
// group order through shared memory.  So eight warps share the latency of a tile that two would otherwise work on.  Slabs
// arrive by cp.async, up to three in flight beside the one worked on: k is split over a cluster beyond 256, so these are most of them.
// us of a launch in a row of launches, tiles of 64 / this, forward and both products of the backward:
//   520 x 192 x 192   11.7 / 3.4   25.1 / 7.9    2080 x 576 x 192   24.1 / 17.4   62.0 / 42.4
//   520 x 576 x 192   12.8 / 7.3   28.9 / 16.7   2080 x 768 x 192   37.9 / 23.3   77.3 / 55.9
//   520 x 192 x 768   16.4 / 10.5  30.7 / 17.2   8192 x 768 x 768   361 / 368     860 / 632
// and the error against 64 bits falls, forward 1.8e-7 -> 1.0e-7, input gradients 1.8e-7 -> 1.3e-7, weight gradients over 2080 rows
// 4.1e-7 -> 2.2e-7.  A step of the fp32 configuration: batch 1 / 8 / 32 559 -> 367 / 749 -> 439 / 1162 -> 827 us.
// Rows of a slab lie where quarter-warps read them without bank conflicts: [row][64 + 4] where the operand is
// contiguous along k (fragments of four k), [k][32 + 4] where along its own index.
constexpr int SS_BM = 32, SS_BN = 32, SS_BK = 64, SS_THREADS = 256, SS_GROUPS = 4, SS_STAGES = 4;
constexpr int SS_KLD = SS_BK + 4, SS_MLD = SS_BM + 4;
constexpr int SS_OPERAND = SS_BK * SS_MLD;                    // floats of a slab of one operand, either layout (32 x 68 or 64 x 36)
static_assert(SS_OPERAND >= SS_BM * SS_KLD, "either layout fits");
constexpr size_t SS_SMEM = (size_t)SS_STAGES * 2 * SS_OPERAND * sizeof(float);

// Slab k0 .. k0 + 63 of ROWS rows from r0 on; what lies beyond R rows or K columns becomes zero.  Base and row pitch are multiples of 16 bytes.
template <bool KMAJOR, int ROWS = SS_BM>
__device__ __forceinline__ void ss_load(const float* __restrict__ P, long ld, int r0, int k0, int R, int K, float* S) {
  static_assert(KMAJOR || ROWS == SS_BM, "tiles of 64 are built for operands contiguous along k");
#pragma unroll
  for (int q = 0; q < ROWS / 16; ++q) {
    const int i = q * SS_THREADS + threadIdx.x;
    int left;
    const float* src;
    float* dst;
    if (KMAJOR) {
      const int r = i >> 4, k = (i & 15) * 4;
      left = r0 + r < R ? K - (k0 + k) : 0;
      src = P + (long)(r0 + r) * ld + k0 + k;
      dst = S + r * SS_KLD + k;
    } else {
      const int k = i >> 3, r = (i & 7) * 4;
      left = k0 + k < K ? R - (r0 + r) : 0;
      src = P + (long)(k0 + k) * ld + r0 + r;
      dst = S + k * SS_MLD + r;
    }
    const int bytes = left >= 4 ? 16 : left > 0 ? left * 4 : 0;
    copy16_async(dst, bytes > 0 ? src : P, bytes);
  }
}
// Four rows at k .. k + 3: v[row][k].  Rows r, r + 8, r + 16, r + 24 of an operand contiguous along k, r .. r + 3 of the other kind.
template <bool KMAJOR>
__device__ __forceinline__ void ss_frag(const float* S, int r, int k, float (&v)[4][4]) {
  if (KMAJOR) {
#pragma unroll
    for (int i = 0; i < 4; ++i) load16(S + (r + i * 8) * SS_KLD + k, v[i]);
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float t[4];
      load16(S + (k + j) * SS_MLD + r, t);
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i][j] = t[i];
    }
  }
}

template <bool A_K, bool B_K>
__global__ void __launch_bounds__(SS_THREADS)
gemm_simt_small_kernel(const float* __restrict__ A, long lda, const float* __restrict__ B, long ldb, int K, int k_per_split, SimtEpi<float, float> epi) {
  extern __shared__ __align__(16) float ss[];
  dependent_sync();                                          // (small CTAs, three to an SM: the next kernel may always be scheduled; 382 -> 377 us a step at batch 8)
  const int tid = threadIdx.x, grp = tid >> 6, ty = (tid & 63) >> 3, tx = tid & 7;
  const int m0 = blockIdx.y * SS_BM, n0 = blockIdx.x * SS_BN;
  const int splits = gridDim.z, rank = blockIdx.z;
  const int kb = rank * k_per_split, ke = min(K, kb + k_per_split), slabs = (ke - kb + SS_BK - 1) / SS_BK;
  auto stage = [&](int i) {
    if (i < slabs) {
      float* S = ss + (i % SS_STAGES) * 2 * SS_OPERAND;
      ss_load<A_K>(A, lda, m0, kb + i * SS_BK, epi.M, ke, S);
      ss_load<B_K>(B, ldb, n0, kb + i * SS_BK, epi.N, ke, S + SS_OPERAND);
    }
    copies_commit();
  };
#pragma unroll
  for (int i = 0; i < SS_STAGES - 1; ++i) stage(i);
  // Pairs of one instruction: where both operands come four k at a time, even and odd k (each a sum of its own), otherwise two columns.
  constexpr bool KP = A_K && B_K;
  constexpr int PAIRS = KP ? 4 : 2;
  uint64_t acc[4][PAIRS];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < PAIRS; ++j) acc[i][j] = 0ull;
  for (int s = 0; s < slabs; ++s) {
    copies_wait<SS_STAGES - 2>();
    __syncthreads();
    stage(s + SS_STAGES - 1);                                 // into the slab that every thread left before this barrier
    const float* As = ss + (s % SS_STAGES) * 2 * SS_OPERAND;
    const float* Bs = As + SS_OPERAND;
#pragma unroll
    for (int kk = 0; kk < SS_BK / SS_GROUPS; kk += 4) {
      const int k = grp * (SS_BK / SS_GROUPS) + kk;
      float a[4][4], b[4][4];
      ss_frag<A_K>(As, A_K ? ty : ty * 4, k, a);
      ss_frag<B_K>(Bs, B_K ? tx : tx * 4, k, b);
      if constexpr (KP) {
#pragma unroll
        for (int j = 0; j < 4; j += 2)
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int n = 0; n < 4; ++n) acc[i][n] = simt_fma2(simt_pack2(a[i][j], a[i][j + 1]), simt_pack2(b[n][j], b[n][j + 1]), acc[i][n]);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint64_t b0 = simt_pack2(b[0][j], b[1][j]), b1 = simt_pack2(b[2][j], b[3][j]);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const uint64_t av = simt_pack2(a[i][j], a[i][j]);
            acc[i][0] = simt_fma2(av, b0, acc[i][0]);
            acc[i][1] = simt_fma2(av, b1, acc[i][1]);
          }
        }
      }
    }
  }
  // the groups' tiles [4][32][32 + 4] over the operand buffers
  copies_wait<0>();
  __syncthreads();
  constexpr int TLD = SS_BN + 4;
  static_assert(SS_GROUPS * SS_BM * TLD <= SS_STAGES * 2 * SS_OPERAND, "the groups' tiles fit");
  float* tile = ss + grp * SS_BM * TLD;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = A_K ? ty + i * 8 : ty * 4 + i;
    float c[4];
    if constexpr (KP) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float even, odd;
        simt_unpack2(acc[i][j], even, odd);
        c[j] = even + odd;
      }
    } else {
      simt_unpack2(acc[i][0], c[0], c[1]);
      simt_unpack2(acc[i][1], c[2], c[3]);
    }
    if (B_K) {
#pragma unroll
      for (int j = 0; j < 4; ++j) tile[r * TLD + tx + j * 8] = c[j];
    } else {
      store16(tile + r * TLD + tx * 4, c);
    }
  }
  __syncthreads();
  const int r = tid >> 3, c4 = (tid & 7) * 4;                 // a thread has four columns of a row
  float v[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int g = 0; g < SS_GROUPS; ++g) {
    float t[4];
    load16(ss + (g * SS_BM + r) * TLD + c4, t);
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] += t[j];
  }
  if (splits == 1) {
    epi(m0 + r, n0 + c4, v);
    return;
  }
  // every rank finishes its share of the tile's rows, the others' sums read through distributed shared memory in rank order
  cg::cluster_group cluster = cg::this_cluster();
  store16(ss + r * TLD + c4, v);                              // (a thread rewrites what it alone has read)
  cluster.sync();
  const int share = (SS_BM + splits - 1) / splits;
  if (r < share && rank * share + r < SS_BM) {
    const int row = rank * share + r;
    float4 x[SG_MAXSPLIT];
#pragma unroll
    for (int q = 0; q < SG_MAXSPLIT; ++q)
      if (q < splits) x[q] = *reinterpret_cast<const float4*>(cluster.map_shared_rank(ss, q) + row * TLD + c4);
    float o[4] = {x[0].x, x[0].y, x[0].z, x[0].w};
#pragma unroll
    for (int q = 1; q < SG_MAXSPLIT; ++q)
      if (q < splits) { o[0] += x[q].x; o[1] += x[q].y; o[2] += x[q].z; o[3] += x[q].w; }
    epi(m0 + row, n0 + c4, o);
  }
  cluster.sync();                                             // no CTA leaves while another may still read its tile
}

// Tiles of 64 x 64 for many rows, both operands contiguous along k: 8 x 8 products a thread read shared memory half as often for a
// multiply-add, and that is what bounds the small tiles once nothing is idle.  The sum of an output is the one that
// gemm_simt_small_kernel forms, addition by addition -- four groups with even and odd k apart over each part of k, the groups in
// order, then the parts -- so the choice between the two may depend on the number of rows, and a row's result still does not.
// A CTA takes the parts of k one after the other; the next part's slabs arrive while this one's groups are added up, in memory of
// their own.  One CTA an SM: 255 registers a thread.
constexpr int SW_BM = 64, SW_BN = 64, SW_TLD = SW_BN + 4;
constexpr int SW_OPERAND = SW_BM * SS_KLD;
constexpr size_t SW_SMEM = ((size_t)SS_STAGES * 2 * SW_OPERAND + (size_t)SS_GROUPS * SW_BM * SW_TLD) * sizeof(float);

__global__ void __launch_bounds__(SS_THREADS, 1)
gemm_simt_wide_kernel(const float* __restrict__ A, long lda, const float* __restrict__ B, long ldb, int K, int k_per_split, SimtEpi<float, float> epi) {
  extern __shared__ __align__(16) float ss[];
  if (leaves_sms_idle()) release_dependents();
  await_inputs();
  const int tid = threadIdx.x, grp = tid >> 6, ty = (tid & 63) >> 3, tx = tid & 7;
  const int m0 = blockIdx.y * SW_BM, n0 = blockIdx.x * SW_BN;
  const int slabs = (K + SS_BK - 1) / SS_BK, per = k_per_split / SS_BK;      // per: slabs of a part
  float* tiles = ss + SS_STAGES * 2 * SW_OPERAND;
  auto stage = [&](int i) {
    if (i < slabs) {
      float* S = ss + (i % SS_STAGES) * 2 * SW_OPERAND;
      ss_load<true, SW_BM>(A, lda, m0, i * SS_BK, epi.M, K, S);
      ss_load<true, SW_BN>(B, ldb, n0, i * SS_BK, epi.N, K, S + SW_OPERAND);
    }
    copies_commit();
  };
#pragma unroll
  for (int i = 0; i < SS_STAGES - 1; ++i) stage(i);
  constexpr int MINE = SW_BM * SW_BN / 4 / SS_THREADS;       // of the finished tile: four columns of a row each
  uint64_t acc[8][8];
  float total[MINE][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0ull;
  int in_part = 0;
  bool first = true;
  for (int s = 0; s < slabs; ++s) {
    copies_wait<SS_STAGES - 2>();
    __syncthreads();
    stage(s + SS_STAGES - 1);                                 // into the slab that every thread left before this barrier
    const float* As = ss + (s % SS_STAGES) * 2 * SW_OPERAND;
    const float* Bs = As + SW_OPERAND;
#pragma unroll
    for (int kk = 0; kk < SS_BK / SS_GROUPS; kk += 4) {
      const int k = grp * (SS_BK / SS_GROUPS) + kk;
      float b[8][4];
#pragma unroll
      for (int n = 0; n < 8; ++n) load16(Bs + (tx + n * 8) * SS_KLD + k, b[n]);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        float a[4];
        load16(As + (ty + i * 8) * SS_KLD + k, a);
#pragma unroll
        for (int j = 0; j < 4; j += 2)
#pragma unroll
          for (int n = 0; n < 8; ++n) acc[i][n] = simt_fma2(simt_pack2(a[j], a[j + 1]), simt_pack2(b[n][j], b[n][j + 1]), acc[i][n]);
      }
    }
    if (++in_part < per && s + 1 < slabs) continue;
    // end of a part of k: its groups' tiles [4][64][64 + 4], added in order (the part before has been read: a slab's barrier lies between)
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int n = 0; n < 8; ++n) {
        float even, odd;
        simt_unpack2(acc[i][n], even, odd);
        tiles[(grp * SW_BM + ty + i * 8) * SW_TLD + tx + n * 8] = even + odd;
        acc[i][n] = 0ull;
      }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < MINE; ++q) {
      const int u = q * SS_THREADS + tid, r = u >> 4, c4 = (u & 15) * 4;
      float v[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int g = 0; g < SS_GROUPS; ++g) {
        float t[4];
        load16(tiles + (g * SW_BM + r) * SW_TLD + c4, t);
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] += t[j];
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) total[q][j] = first ? v[j] : total[q][j] + v[j];
    }
    in_part = 0;
    first = false;
  }
  copies_wait<0>();
#pragma unroll
  for (int q = 0; q < MINE; ++q) {
    const int u = q * SS_THREADS + tid;
    epi(m0 + (u >> 4), n0 + (u & 15) * 4, total[q]);
  }
}

// Wide tiles from the second part of k on (one part alone gains nothing: 25216 x 768 x 192 273 / 274 us) and where they fill at least two
// thirds of the waves they take.  us of a launch in a row of launches, small / wide:
//   520 x 768 x 768 (108 tiles on 148 SMs)   34.3 / 30.1   1576 x 768 x 768     89.6 / 85.8   788 x 1152 x 384  37.0 / 32.4
//   788 x 768 x 768 (156)                    48.0 / 57.3   6304 x 768 x 768     335  / 254    1576 x 384 x 1536 92.1 / 110
//   1576 x 768 x 3072 (300)                  331  / 317    2364 x 768 x 3072    486  / 321    3152 x 384 x 384  46.7 / 47.8
//   197 x 2304 x 768 (144)                   41.0 / 30.2   25216 x 768 x 768    1322 / 913    3152 x 384 x 1536 177  / 165
//   197 x 3072 x 768 (192)                   52.7 / 57.1   25216 x 768 x 3072   5110 / 3398   25216 x 384 x 384 338  / 257
// gemm_simt_kernel's tiles of 64, with sums in another order: 25216 x 768 x 768 1066, 25216 x 768 x 3072 4027, and, where the wide tiles' third
// wave is nearly empty, faster: 1576 x 768 x 3072 289.  An image's fp32 logits would then depend on the others of its batch.
static bool wide_tiles(int m, int n, int k, int sms) {
  const long tiles = (long)ceil_div(m, SW_BM) * ceil_div(n, SW_BN);
  return k > 256 && 3 * tiles >= 2 * ceil_div(tiles, sms) * (long)sms;
}

// Parts of the reduction: by its length alone for a layer's output or input gradient, so that an image's result does not
// depend on the batch; weight gradients by what fills the SMs.  Non-zero: not a product for these kernels -- by alignment, and more
// rows than a grid of small tiles has where the operands are not both contiguous along k.
static int launch_simt_small(const Ctx& c, const float* A, long lda, bool ak, const float* B, long ldb, bool bk, int m, int n, int k,
                             const SimtEpi<float, float>& epi) {
  if (lda % 4 != 0 || ldb % 4 != 0 || (uintptr_t)A % 16 != 0 || (uintptr_t)B % 16 != 0) return -1;
  const int sms = c.sm_count > 0 ? c.sm_count : B200_SMS;
  const long tiles = (long)ceil_div(m, SS_BM) * ceil_div(n, SS_BN);
  const bool tall = ceil_div(m, SS_BM) > 65535;
  int splits = ceil_div(k, 256) < SG_MAXSPLIT ? ceil_div(k, 256) : SG_MAXSPLIT;
  if (!ak)
    while (splits > 1 && tiles * splits > 4l * sms) --splits;
  const int per = ceil_div(ceil_div(k, splits), SS_BK) * SS_BK;
  splits = ceil_div(k, per) < 1 ? 1 : ceil_div(k, per);
  if (ak && bk && (tall || wide_tiles(m, n, k, sms))) {
    static SmemLimit lim;
    if (!ensure_smem(lim, gemm_simt_wide_kernel, SW_SMEM)) return -3;
    launch_k(gemm_simt_wide_kernel, dim3(ceil_div(n, SW_BN), ceil_div(m, SW_BM)), SS_THREADS, SW_SMEM, c.stream, A, lda, B, ldb, k, per, epi);
    return 0;
  }
  if (tall) return -1;
  auto go = [&](auto kern, SmemLimit& lim) {
    if (!ensure_smem(lim, kern, SS_SMEM)) return -3;
    launch_cluster(kern, dim3(ceil_div(n, SS_BN), ceil_div(m, SS_BM), splits), SS_THREADS, SS_SMEM, c.stream, dim3(1, 1, splits), A, lda, B, ldb, k, per, epi);
    return 0;
  };
  static SmemLimit l0, l1, l2, l3;
  return ak ? (bk ? go(gemm_simt_small_kernel<true, true>, l0) : go(gemm_simt_small_kernel<true, false>, l1))
            : (bk ? go(gemm_simt_small_kernel<false, true>, l2) : go(gemm_simt_small_kernel<false, false>, l3));
}

template <typename T, typename TC>
static void launch_simt(const Ctx& c, const void* A, long a_rs, long a_cs, const void* B, long b_rs, long b_cs, void* C, int m, int n, int k,
                        const GemmEpilogue& e) {
  const int tiles_n = ceil_div(n, SG_BN), tiles = tiles_n * ceil_div(m, SG_BM);
  const bool ak = a_cs == 1, bk = b_cs == 1;
  int splits;
  if (ak) {
    // A layer's output or input gradient: by the reduction length alone, so that an image's result does not depend on
    // how many others are in the batch.
    splits = ceil_div(k, 128) < SG_MAXSPLIT ? ceil_div(k, 128) : SG_MAXSPLIT;
  } else {
    // A weight gradient, reduced over the rows of the batch: the SM with the most CTAs sets the time, each CTA costing its
    // k range plus about 32 k steps of prologue and as much for the reduction.
    const int sms = c.sm_count > 0 ? c.sm_count : B200_SMS;
    int best = ceil_div(tiles, sms) * (k + 32);
    splits = 1;
    for (int s = 2; s <= SG_MAXSPLIT && k >= s * 2 * SG_BK; ++s) {
      int cost = ceil_div((long)tiles * s, sms) * (ceil_div(k, s) + 64);
      if (cost < best) { best = cost; splits = s; }
    }
  }
  const int per = ceil_div(ceil_div(k, splits), SG_BK) * SG_BK;
  splits = ceil_div(k, per) < 1 ? 1 : ceil_div(k, per);
  const long lda = ak ? a_rs : a_cs, ldb = bk ? b_rs : b_cs;
  const size_t quad = 4 * sizeof(T);
  SimtEpi<T, TC> epi = {(TC*)C, e.bias, (const TC*)e.residual, (TC*)e.aux_out, (const T*)e.aux_in, m, n, e.act, e.residual_ld ? e.residual_ld : n,
                         sizeof(T) == 4 && sizeof(TC) == 4 && n % 4 == 0 && e.residual_ld % 4 == 0 &&
                             (((uintptr_t)C | (uintptr_t)e.bias | (uintptr_t)e.residual | (uintptr_t)e.aux_out | (uintptr_t)e.aux_in) & 15) == 0};
  if constexpr (std::is_same<T, float>::value)
    if (launch_simt_small(c, (const float*)A, lda, ak, (const float*)B, ldb, bk, m, n, k, epi) == 0) return;
  launch_cluster(gemm_simt_kernel<T, TC>, dim3(tiles_n, ceil_div(m, SG_BM), splits), SG_THREADS, 0, c.stream, dim3(1, 1, splits), (const T*)A, lda, (int)ak,
                 (int)(lda % 4 == 0 && (uintptr_t)A % quad == 0), (const T*)B, ldb, (int)bk, (int)(ldb % 4 == 0 && (uintptr_t)B % quad == 0), k, per, epi);
}

// Strides: A(m, k) = A[m * a_rs + k * a_cs], B alike; one stride of each operand is 1.
void gemm(const Ctx& c, const void* A, long a_rs, long a_cs, const void* B, long b_rs, long b_cs, void* C,
          int out_is_float, int m, int n, int k, const GemmEpilogue& e) {
  if (m <= 0 || n <= 0) return;
  // The tensor-core kernels take any reduction length: what TMA wants aligned is the row pitch of each operand (checked
  // there), and slabs past the end arrive as zeros.  Weight gradients reduce over batch x tokens rows, which an odd batch
  // leaves odd: at batch 45 of ViT-B they took 515 us a launch on FP32 FMAs, 18 us on the tensor cores.
  if (c.dtype == 1 && c.use_tc && (n % 8) == 0) {
    // CTA pairs where a wide output over many rows keeps all of them busy (QKV and first FFN layer of ViT-B from batch 61).  us with
    // one CTA a tile / with pairs, launch after launch, at 12608, 16351 and 25216 rows:
    //   2304 columns, k = 768     52.6 / 49.7   56.4 / 55.2   82.7 / 82.2     (9000 and 11000 rows: 39.1 / 39.6, 44.8 / 45.0)
    //   3072 columns, k = 768     65.3 / 58.6   81.9 / 71.0   112  / 110      (with GELU 72.9 / 74.6, 97.6 / 97.8, 114 / 125)
    //   2048 columns, k = 768     43.4 / 43.3   50.0 / 49.7   79.3 / 77.0     (1536 columns 33.0 / 32.3, 37.8 / 37.0, 52.3 / 53.9)
    //   2304 columns, k = 640     42.6 / 42.0   48.4 / 50.2   71.2 / 75.3     (k = 512: 36.7 / 40.3, 42.2 / 48.4, 58.3 / 68.2)
    // A pair stages half of B on each SM, which also takes less power, and power is what limits a run of steps: there GELU's products
    // are as fast either way (with them on single CTAs a ViT-B step at batch 128 5.79 against 5.77 ms, inference 3.96 and 3.96).
    // Below k = 640 the set-up of a pair's tile shows more than that.  Float outputs and B read across k
    // lost on pairs (25216 x 768 x 3072: 92 -> 107 us; 159 -> 166 us) and are not built for them.
    const bool pairs = a_cs == 1 && b_cs == 1 && !out_is_float && (c.use_tc >= 2 ? m > 128 : (m >= 12000 && n >= 2048 && k >= 640));
    if (pairs && gemm_tc2(c, A, a_rs, B, b_rs, C, m, n, k, e) == 0) return;
    if (gemm_tc_strided(c, A, a_rs, a_cs, B, b_rs, b_cs, C, out_is_float, m, n, k, e, c.split_ws, c.split_ws_floats) == 0) return;
  }
  note_launch(1);
  if (c.dtype == 0) launch_simt<float, float>(c, A, a_rs, a_cs, B, b_rs, b_cs, C, m, n, k, e);
  else if (out_is_float) launch_simt<bf16, float>(c, A, a_rs, a_cs, B, b_rs, b_cs, C, m, n, k, e);
  else launch_simt<bf16, bf16>(c, A, a_rs, a_cs, B, b_rs, b_cs, C, m, n, k, e);
}

}  // namespace bsr
