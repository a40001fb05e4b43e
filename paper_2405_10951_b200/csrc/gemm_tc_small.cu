// bf16 dense contraction for products of few tiles (a batch of few images, the classification rows of the last block):
//
//   C[m, n] = epilogue( sum_k A(m, k) * B(n, k) ),   A contiguous along k, B along k or along n
//
// What bounds these is latency, not bytes or operations: 200 x 384 x 1536 is 12 tiles of 128 x 64 with 24 slabs of k each.
// So a tile's k range is split over the CTAs of a cluster (2 to 8), each of which has its whole share in flight at once.
// Every CTA finishes an equal share of the tile's rows: the others send it their partial sums of those rows straight from
// registers into its shared memory, and it adds them up in the order of k.  Nothing
// passes through global memory and no second kernel runs (DeiT-S, one image: a step 713 -> 661 us, inference 472 -> 437 us,
// against a split over partial sums in global memory).
//   all threads : set-up, then accumulators -> the rows' owners, then the sums and the epilogue of this CTA's rows, whose
//                 bias, residual and stored pre-activations were fetched while the products were formed
//   warp 0      : TMA producer (one lane)
//   warp 1      : tensor-memory allocation, MMA issue (one lane)
// The next kernel may always be scheduled early: one wave, and shared memory that two CTAs share when the slabs are few.
// Every wait is bounded as in gemm_tc.cu; a CTA that gave up still takes part in the cluster's barriers, so that none
// leaves while another may write to it.
#include <cuda.h>

#include "common.cuh"
#include "kernels.h"
#include "tc_epilogue.cuh"
#include "tc_ptx.cuh"

namespace bsr {
namespace tcs {
using namespace tc;

constexpr int BM = 128, BN = 64, BK = 64, UMMA_K = 16;
constexpr int A_BYTES = BM * BK * 2, B_BYTES = BN * BK * 2, STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int MAX_STAGES = 7, MIN_SPLITS = 2, MAX_SPLITS = 8;
constexpr int RECV_BYTES = (BM + MAX_SPLITS) * BN * 4;       // shares of the rows are rounded up
constexpr int THREADS = 256;
constexpr uint32_t TMEM_COLS = 64;
constexpr int PASSES = BM / MIN_SPLITS / 16;                  // a CTA finishes 16 rows a pass

template <bool B_MN, typename TOut, bool EXACT>
__global__ void __launch_bounds__(THREADS, 2)
gemm_tc_small_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, TOut* __restrict__ C,
                     int M, int N, int K, Epi ep, int stages, int* status) {
  extern __shared__ unsigned char smem_dyn[];
  __shared__ __align__(8) unsigned long long bar_mem[2 * MAX_STAGES + 1];
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag;
  const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
  const uint32_t recv = base + stages * STAGE_BYTES;
  const uint32_t bars = smem_u32(bar_mem);
  auto full_bar = [&](int s) { return bars + 8u * s; };
  auto empty_bar = [&](int s) { return bars + 8u * (MAX_STAGES + s); };
  const uint32_t done_bar = bars + 8u * (2 * MAX_STAGES);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nt = blockIdx.x, mt = blockIdx.y, rank = blockIdx.z, splits = gridDim.z;
  const int total_kb = (K + BK - 1) / BK;
  const int kb0 = rank * total_kb / splits, nkb = (rank + 1) * total_kb / splits - kb0;
  // rows of the tile, an equal share for every CTA of the cluster; this one's are r0 to r1 - 1
  const int rows = min(BM, M - mt * BM), share = (rows + splits - 1) / splits;
  const int r0 = rank * share, r1 = min(rows, r0 + share);

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < stages; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    mbar_init(done_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    prefetch_map(&map_a);
    prefetch_map(&map_b);
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&tmem_base_slot), TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  cluster_arrive();                        // this CTA has started: the others may write to its shared memory
  const uint32_t tmem_base = tmem_base_slot;
  release_dependents();
  await_inputs();
  volatile int* abortp = &abort_flag;

  if (threadIdx.x == 0) {
    int s = 0;
    uint32_t phase = 0;
    for (int i = 0; i < nkb; ++i) {
      const int kb = kb0 + i;
      if (!mbar_wait(empty_bar(s), phase ^ 1u, abortp)) break;
      mbar_expect_tx(full_bar(s), STAGE_BYTES);
      const uint32_t sa = base + s * STAGE_BYTES;
      tma_load_2d(sa, &map_a, full_bar(s), kb * BK, mt * BM);
      if (B_MN) tma_load_2d(sa + A_BYTES, &map_b, full_bar(s), nt * BN, kb * BK);
      else tma_load_2d(sa + A_BYTES, &map_b, full_bar(s), kb * BK, nt * BN);
      if (++s == stages) { s = 0; phase ^= 1u; }
    }
  } else if (threadIdx.x == 32) {
    constexpr uint32_t idesc = make_idesc_mn(BM, BN, false, B_MN);
    constexpr uint32_t A_KSTEP = (UMMA_K * 2) >> 4, B_KSTEP = (B_MN ? UMMA_K * 128 : UMMA_K * 2) >> 4;
    const uint64_t desc_a0 = make_desc(base, 16, 1024);
    const uint64_t desc_b0 = B_MN ? make_desc(base + A_BYTES, BK * 128, 1024) : make_desc(base + A_BYTES, 16, 1024);
    int s = 0;
    uint32_t phase = 0;
    for (int i = 0; i < nkb; ++i) {
      if (!mbar_wait(full_bar(s), phase, abortp)) break;
      tc_fence_after();
      const uint64_t da = desc_a0 + (uint64_t)((s * STAGE_BYTES) >> 4), db = desc_b0 + (uint64_t)((s * STAGE_BYTES) >> 4);
      umma_bf16(tmem_base, da, db, idesc, i > 0 ? 1u : 0u);
#pragma unroll
      for (int k = 1; k < BK / UMMA_K; ++k) umma_bf16_acc(tmem_base, da + (uint64_t)(k * A_KSTEP), db + (uint64_t)(k * B_KSTEP), idesc);
      umma_commit(empty_bar(s));
      if (++s == stages) { s = 0; phase ^= 1u; }
    }
    umma_commit(done_bar);                 // after a wait that gave up: of what was issued
  }
  __syncwarp();

  // epilogue operands of this CTA's rows, 16 a pass: a thread has four columns of a row
  const int unit = threadIdx.x & 15, sub = threadIdx.x >> 4, col = nt * BN + unit * 4;
  auto at = [&](int r) { return (size_t)(mt * BM + r) * N + col; };
  auto mine = [&](int p) { return r0 + p * 16 + sub < r1 && col < N; };
  float4 bias = make_float4(0.f, 0.f, 0.f, 0.f);
  float res[PASSES][4], z[PASSES][4];
  if (ep.bias != nullptr && col < N) bias = __ldg(reinterpret_cast<const float4*>(ep.bias + col));
#pragma unroll
  for (int p = 0; p < PASSES; ++p) {
    if (ep.residual != nullptr && mine(p)) load4(reinterpret_cast<const TOut*>(ep.residual) + (size_t)(mt * BM + r0 + p * 16 + sub) * ep.res_ld + col, res[p]);
    if (ep.act == 2 && mine(p)) load4(reinterpret_cast<const bf16*>(ep.aux_in) + at(r0 + p * 16 + sub), z[p]);
  }

  // accumulators -> their rows' owners: [splits][share][64], a row's 16-byte units permuted by the row (no bank conflicts)
  const bool ok = __all_sync(0xffffffffu, mbar_wait(done_bar, 0, abortp));
  tc_fence_after();
  cluster_wait();
  if (ok) {
    const int quarter = warp & 3, half = warp >> 2, row = quarter * 32 + lane;
    uint32_t r[32];
    tmem_ld32(tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(half * 32), r);
    tmem_ld_wait();
    if (row < rows) {
      const int owner = row / share, local = row - owner * share;
      const uint32_t dst = peer_addr(recv + (uint32_t)(rank * share + local) * (BN * 4), owner);
#pragma unroll
      for (int u = 0; u < 8; ++u) send16(dst + (((half * 8 + u) ^ (local & 7)) << 4), r + 4 * u);
    }
  }
  __syncwarp();
  tc_fence_before();
  cluster_arrive();
  cluster_wait();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }

  const float* got = reinterpret_cast<const float*>(smem_dyn + (recv - smem_u32(smem_dyn)));
#pragma unroll
  for (int p = 0; p < PASSES; ++p) {
    if (!mine(p) || !ok) continue;
    const int local = p * 16 + sub;
    const float* src = got + local * BN + ((unit ^ (local & 7)) << 2);
    float4 x[MAX_SPLITS];
#pragma unroll
    for (int q = 0; q < MAX_SPLITS; ++q)
      if (q < splits) x[q] = *reinterpret_cast<const float4*>(src + q * share * BN);
    float v[4] = {x[0].x, x[0].y, x[0].z, x[0].w};
#pragma unroll
    for (int q = 1; q < MAX_SPLITS; ++q)
      if (q < splits) { v[0] += x[q].x; v[1] += x[q].y; v[2] += x[q].z; v[3] += x[q].w; }
    v[0] += bias.x; v[1] += bias.y; v[2] += bias.z; v[3] += bias.w;
    if (ep.act == 1) {
      if (ep.aux_out != nullptr) store4(reinterpret_cast<TOut*>(ep.aux_out) + at(r0 + local), v);
      if (EXACT) {
        gelu_exact2(v[0], v[1]);
        gelu_exact2(v[2], v[3]);
      } else {
        gelu_fast2(v[0], v[1]);
        gelu_fast2(v[2], v[3]);
      }
    } else if (ep.act == 2) {
      if (EXACT) {
        gelu_grad_exact2(v[0], v[1], z[p][0], z[p][1]);
        gelu_grad_exact2(v[2], v[3], z[p][2], z[p][3]);
      } else {
        gelu_grad_mul2h(v[0], v[1], z[p][0], z[p][1], z[p][0], z[p][1]);
        gelu_grad_mul2h(v[2], v[3], z[p][2], z[p][3], z[p][2], z[p][3]);
      }
      if (ep.aux_out != nullptr) store4(reinterpret_cast<bf16*>(ep.aux_out) + at(r0 + local), z[p]);
    }
    if (ep.residual != nullptr) { v[0] += res[p][0]; v[1] += res[p][1]; v[2] += res[p][2]; v[3] += res[p][3]; }
    store4(C + at(r0 + local), v);
  }
  if (threadIdx.x == 0 && abort_flag) {
    unsigned long long t0 = global_ns();   // copies already issued still land in shared memory
    while (global_ns() - t0 < 1000000ull) {}
    if (status != nullptr) atomicOr(status, STATUS_TIMEOUT);
  }
}

template <bool B_MN, typename TOut, bool EXACT = false>
static int launch(const Ctx& c, const CUtensorMap& ma, const CUtensorMap& mb, void* C, int m, int n, int k, const Epi& ep, int splits) {
  auto kern = gemm_tc_small_kernel<B_MN, TOut, EXACT>;
  const int slabs = ceil_div(ceil_div(k, BK), splits), stages = slabs < MAX_STAGES ? slabs : MAX_STAGES;
  auto bytes = [](int st) { return (size_t)st * STAGE_BYTES + RECV_BYTES + 1024; };
  static SmemLimit lim;
  if (!ensure_smem(lim, kern, bytes(MAX_STAGES))) return -3;
  note_launch(1);
  launch_cluster(kern, dim3(ceil_div(n, BN), ceil_div(m, BM), splits), THREADS, bytes(stages), c.stream, dim3(1, 1, splits), ma, mb,
                 (TOut*)C, m, n, k, ep, stages, c.status);
  return 0;
}

// Splits of each tile's k range (a power of two), 0: not a product for this kernel.  As many as still fit the SMs in one wave
// and leave every CTA three slabs.  us of a launch in a row of launches, one CTA a tile (gemm_tc.cu) against this:
//   200 x 384 x 1536, 8 splits 8.7 / 5.9    64 x 384 x 1536, 8 splits 8.2 / 4.3    577 x 768 x 3072, 2 splits 14.9 / 11.3
//   200 x 768 x 768, 4 splits 5.65 / 5.4    7 x 768 x 768, 4 splits 5.4 / 3.6      200 x 384 x 1152, 2 splits 7.2 / 6.5
// A shorter k in two parts, or six slabs, is not worth the exchange:
//   577 x 768 x 768, 2 splits 5.9 / 6.15    128 x 3072 x 768, 2 splits 5.9 / 6.1    200 x 384 x 384, 2 splits 4.1 / 4.9
static int choose_splits(int m, int n, int k, int sms) {
  const long tiles = (long)ceil_div(m, BM) * ceil_div(n, BN);
  const int kb = ceil_div(k, BK);
  int s = 1;
  while (s < MAX_SPLITS && tiles * s * 2 <= sms && kb >= s * 2 * 3) s *= 2;
  return kb >= 12 && s >= (kb >= 18 ? 2 : 4) ? s : 0;
}

}  // namespace tcs

int gemm_tc_small(const Ctx& c, const void* A, long lda, const void* B, long ldb, int b_mn, void* C, int out_is_float, int m, int n, int k,
                  const GemmEpilogue& e) {
  using namespace tcs;
  const int splits = choose_splits(m, n, k, c.sm_count > 0 ? c.sm_count : B200_SMS);
  if (splits == 0) return -1;
  CUtensorMap ma, mb;
  if (!make_map(&ma, A, (uint64_t)k, (uint64_t)m, (uint64_t)lda, BM)) return -2;
  if (!(b_mn ? make_map(&mb, B, (uint64_t)n, (uint64_t)k, (uint64_t)ldb, BK) : make_map(&mb, B, (uint64_t)k, (uint64_t)n, (uint64_t)ldb, BN))) return -2;
  Epi ep;
  ep.bias = e.bias; ep.residual = e.residual; ep.res_ld = (int)(e.residual_ld ? e.residual_ld : n); ep.aux_out = e.aux_out; ep.aux_in = e.aux_in; ep.act = e.act;
  const bool timed = c.prof != nullptr && c.prof->on;
  if (timed) c.prof->begin(c.stream, 2.0 * m * n * (double)k);
  const bool exact = e.act != 0 && exact_gelu(m, k);
  auto go = [&](auto kern) { return kern(c, ma, mb, C, m, n, k, ep, splits); };
  int rc;
  if (out_is_float) rc = b_mn ? go(launch<true, float>) : go(launch<false, float>);
  else if (exact) rc = b_mn ? go(launch<true, bf16, true>) : go(launch<false, bf16, true>);
  else rc = b_mn ? go(launch<true, bf16>) : go(launch<false, bf16>);
  if (timed) c.prof->end(c.stream);
  return rc;
}

}  // namespace bsr
