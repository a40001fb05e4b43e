// bf16 GEMM on CTA pairs: tcgen05.mma cta_group::2 with a 256 x 256 accumulator tile spread over the tensor
// memory of two SMs.  Same contract as the single-CTA kernel for operands read along k and a bf16 output, but each SM stages
// only its own 128 rows of A and its own half of the columns of B per k-slab: 32 KB instead of 48 KB for the same number of
// multiply-accumulates.  That is what bounds the single-CTA kernel's main loop: four slabs of 48 KB in flight cover less
// than the 2000-odd clocks a slab takes to arrive; six slabs of 32 KB fit here.
//
// Cluster of two CTAs, persistent, one cluster per SM pair:
//   warp 0 (both CTAs) : TMA producer; every copy signals the full barrier of the leader CTA (rank 0)
//   warp 1 (leader)    : issues the MMAs; its commits arrive on the empty / accumulator-full barriers of both CTAs
//   warps 2..9 (both)  : epilogue of the CTA's own 128 rows; they release the accumulator on the leader's barrier
// Waits are bounded as in the single-CTA kernel.
#include <cuda.h>

#include "common.cuh"
#include "kernels.h"
#include "tc_ptx.cuh"
#include "tc_epilogue.cuh"

namespace bsr {
namespace tc2 {

using namespace tc;

constexpr int BM = 128;                   // rows per CTA (256 per pair)
constexpr int BN = 256;                   // columns per pair tile; each CTA stages BN/2 of B
constexpr int BK = 64;
constexpr int STAGES = 6;
constexpr int UMMA_K = 16;
constexpr int A_BYTES = BM * BK * 2, B_BYTES = (BN / 2) * BK * 2;
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;      // 32 KB
constexpr int EPI_WARPS = 8;
constexpr int STAGING_BYTES = 32 * 128;
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + EPI_WARPS * STAGING_BYTES + 1024 + 256;
constexpr int THREADS = 64 + EPI_WARPS * 32;
constexpr uint32_t TMEM_COLS = 512;
constexpr uint32_t PEER_MASK = 0xFEFFFFFFu;         // clears the CTA-rank bit of a shared address: the even CTA of the pair

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
      "l"(map), "r"(bar), "r"(c0), "r"(c1)
      : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t smem_dst, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(cols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
__device__ __forceinline__ void umma_bf16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrives (once the MMAs issued so far have completed) on the barrier at the same offset in both CTAs of the pair.
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
  uint16_t mask = 3;
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
               "h"(mask)
               : "memory");
}
// Arrive on the barrier at the same offset in the leader CTA's shared memory.
__device__ __forceinline__ void mbar_arrive_leader(uint32_t bar) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(remote) : "r"(bar));
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(remote) : "memory");
}


// The tiles of one pair.  Whole tiles go round in as many full waves as there are; the tiles of a last wave that would leave
// pairs idle are cut along n into as many parts as there are pairs for them (25216 rows are 98.5 tiles of 256: at 768 columns
// 297 tiles on 74 pairs, the last wave a single tile).  Parts are multiples of UNIT columns.  Stepping to the next whole tile
// takes no division.
struct Tile {
  int mt, n0, width;
};
constexpr int UNIT = 64, UNITS = BN / UNIT;
struct Walk {
  int i, row, nt, step, full, items, parts, workers;
  __device__ __forceinline__ static int part_units(int parts) { return (UNITS + parts - 1) / parts; }
  __device__ __forceinline__ Walk(int tiles_m, int tiles_n, int worker, int workers_) {
    const int total = tiles_m * tiles_n;
    workers = workers_;
    full = total - total % workers;
    const int rem = total - full;
    parts = rem > 0 ? min(UNITS, workers / rem) : 1;
    parts = (UNITS + part_units(parts) - 1) / part_units(parts);
    items = full + rem * parts;
    i = worker;
    row = i / tiles_n;
    nt = i - row * tiles_n;
    step = (workers / tiles_n) << 16 | (workers % tiles_n);
  }
  __device__ __forceinline__ bool next(int N, int tiles_n, Tile& t) {
    if (i >= items) return false;
    int off = 0, r = row, c = nt;
    t.width = BN;
    if (i >= full && parts > 1) {            // each pair comes here once at most
      const int j = i - full, q = j / parts, pu = part_units(parts), tile = full + q;
      r = tile / tiles_n;
      c = tile - r * tiles_n;
      off = (j - q * parts) * pu;
      t.width = min(pu, UNITS - off) * UNIT;
    }
    i += workers;
    row += step >> 16;
    nt += step & 0xffff;
    if (nt >= tiles_n) { nt -= tiles_n; ++row; }
    t.mt = r;
    t.n0 = c * BN + off * UNIT;
    return t.n0 < N;                         // false: a part past the last column, the last of this pair's items
  }
};

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
gemm_tc2_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, const __grid_constant__ CUtensorMap map_part,
                bf16* __restrict__ C, int M, int N, int K, Epi ep, int tiles_m, int tiles_n, int* status) {
  extern __shared__ unsigned char smem_dyn[];
  uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
  uint32_t staging0 = base + STAGES * STAGE_BYTES;
  uint32_t bars = staging0 + EPI_WARPS * STAGING_BYTES;   // full[STAGES], empty[STAGES], tfull[2], tempty[2]
  auto full_bar = [&](int s) { return bars + 8u * s; };
  auto empty_bar = [&](int s) { return bars + 8u * (STAGES + s); };
  auto tfull_bar = [&](int b) { return bars + 8u * (2 * STAGES + b); };
  auto tempty_bar = [&](int b) { return bars + 8u * (2 * STAGES + 2 + b); };
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const bool leader = rank == 0;
  const int total_kb = (K + BK - 1) / BK;

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(tfull_bar(b), 1); mbar_init(tempty_bar(b), 2 * EPI_WARPS); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    prefetch_map(&map_a);
    prefetch_map(&map_b);
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_u32(&tmem_base_slot), TMEM_COLS);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  cluster_sync_all();                       // barriers of both CTAs exist before anyone signals them
  tc_fence_after();
  uint32_t tmem_base = tmem_base_slot;
  await_inputs();                           // (fills the SMs: see release_dependents)
  volatile int* abortp = &abort_flag;
  Walk walk(tiles_m, tiles_n, blockIdx.x >> 1, gridDim.x >> 1);
  Tile t;

  if (warp == 0) {
    // ------------------------------- TMA producer (both CTAs) -------------------------------
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      int armed = 0;
      bool ok = true;
      while (ok && walk.next(N, tiles_n, t)) {
        const int m0 = t.mt * (2 * BM) + (int)rank * BM;        // this CTA's rows of A
        const int cols = t.width >> 1, n0 = t.n0 + (int)rank * cols;   // this CTA's share of B
        const uint32_t bytes = 2u * (uint32_t)(A_BYTES + cols * (BK * 2));
        for (int kb = 0; kb < total_kb; ++kb) {
          if (!mbar_wait(empty_bar(stage), phase ^ 1u, abortp)) { ok = false; break; }
          const uint32_t fb = full_bar(stage) & PEER_MASK;      // the leader's barrier collects both CTAs' bytes
          if (leader) mbar_expect_tx(full_bar(stage), bytes);
          const uint32_t sa = base + stage * STAGE_BYTES, sb = sa + A_BYTES;
          tma_load_2d_pair(sa, &map_a, fb, kb * BK, m0);
          if (t.width == BN) {
            tma_load_2d_pair(sb, &map_b, fb, kb * BK, n0);
          } else {
            for (int j = 0; j < cols; j += UNIT / 2) tma_load_2d_pair(sb + j * 128, &map_part, fb, kb * BK, n0 + j);
          }
          ++armed;
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
      }
      if (!ok && armed > 0) {
        unsigned long long t0 = global_ns();
        while (global_ns() - t0 < 1000000ull) {}
      }
    }
  } else if (warp == 1) {
    // ------------------------------- MMA issuer (leader CTA only) ---------------------------
    if (lane == 0 && leader) {
      constexpr uint32_t idesc0 = make_idesc_mn(2 * BM, 0, false, false);
      constexpr uint32_t KSTEP = (UMMA_K * 2) >> 4;
      const uint64_t desc_a0 = make_desc(base, 16, 1024);
      const uint64_t desc_b0 = make_desc(base + A_BYTES, 16, 1024);
      int stage = 0;
      uint32_t phase = 0;
      int local = 0;
      bool ok = true;
      for (; ok && walk.next(N, tiles_n, t); ++local) {
        const int buf = local & 1;
        const uint32_t idesc = idesc0 | ((uint32_t)(t.width >> 3) << 17);
        if (!mbar_wait(tempty_bar(buf), ((local >> 1) & 1) ^ 1u, abortp)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + buf * BN;
        for (int kb = 0; kb < total_kb; ++kb) {
          if (!mbar_wait(full_bar(stage), phase, abortp)) { ok = false; break; }
          tc_fence_after();
          const uint64_t off = (uint64_t)((stage * STAGE_BYTES) >> 4);
#pragma unroll
          for (int k = 0; k < BK / UMMA_K; ++k)
            umma_bf16_pair(d_tmem, desc_a0 + off + (uint64_t)(k * KSTEP), desc_b0 + off + (uint64_t)(k * KSTEP), idesc, (kb > 0 || k > 0) ? 1u : 0u);
          umma_commit_pair(empty_bar(stage));
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
        if (ok) umma_commit_pair(tfull_bar(buf));
      }
    }
  } else {
    // ------------------------------- epilogue (both CTAs, own rows) --------------------------
    const int ew = warp - 2, quarter = warp & 3, chalf = ew >> 2;
    unsigned char* st = smem_dyn + (staging0 - smem_u32(smem_dyn)) + ew * STAGING_BYTES;
    int local = 0;
    while (walk.next(N, tiles_n, t)) {
      const int buf = local & 1, nc = t.width >> 6;      // chunks of 32 columns for each half of the warps
      auto ready = [&]() {
        bool w = mbar_wait(tfull_bar(buf), (local >> 1) & 1, abortp);
        w = __all_sync(0xffffffffu, w);
        tc_fence_after();
        return w;
      };
      if (!epilogue_tile<bf16, false, false>(ready, ep, 0, C, M, N, t.mt * (2 * BM) + (int)rank * BM + quarter * 32, t.n0 + chalf * nc * 32, nc,
                                      tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * BN + chalf * nc * 32), st, lane))
        break;
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_leader(tempty_bar(buf));
      ++local;
    }
  }
  tc_fence_before();
  __syncwarp();
  cluster_sync_all();                       // neither CTA leaves while the other may still touch its memory
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, TMEM_COLS);
  }
  if (threadIdx.x == 0 && abort_flag && status != nullptr) atomicOr(status, STATUS_TIMEOUT);
}

}  // namespace tc2

// C[m, n] (bf16) = epilogue(A B^T) for operands contiguous along k, rows lda and ldb apart.  Returns non-zero when the problem is
// not taken.
int gemm_tc2(const Ctx& c, const void* A, long lda, const void* B, long ldb, void* C, int m, int n, int k, const GemmEpilogue& e) {
  using namespace tc2;
  if ((lda % 8) != 0 || (ldb % 8) != 0 || ((uintptr_t)A & 15) || ((uintptr_t)B & 15) || ((uintptr_t)C & 15)) return -1;
  if ((n % 8) != 0) return -1;
  CUtensorMap ma, mb, mp;
  if (!tc::make_map(&ma, A, (uint64_t)k, (uint64_t)m, (uint64_t)lda, BM) || !tc::make_map(&mb, B, (uint64_t)k, (uint64_t)n, (uint64_t)ldb, BN / 2) ||
      !tc::make_map(&mp, B, (uint64_t)k, (uint64_t)n, (uint64_t)ldb, UNIT / 2))
    return -2;
  static SmemLimit lim;
  if (!ensure_smem(lim, gemm_tc2_kernel, SMEM_BYTES)) return -3;
  const int tiles_m = ceil_div(m, 2 * BM), tiles_n = ceil_div(n, BN), pairs = (c.sm_count > 0 ? c.sm_count : B200_SMS) / 2;
  const long work = (long)tiles_m * tiles_n * UNITS;
  tc::Epi ep;
  ep.bias = e.bias; ep.residual = e.residual; ep.res_ld = (int)(e.residual_ld ? e.residual_ld : n); ep.aux_out = e.aux_out; ep.aux_in = e.aux_in; ep.act = e.act;
  if (c.prof != nullptr && c.prof->on) c.prof->begin(c.stream, 2.0 * m * n * (double)k);
  note_launch(1);
  launch_k(gemm_tc2_kernel, 2 * (int)(work < pairs ? work : pairs), THREADS, SMEM_BYTES, c.stream, ma, mb, mp, (bf16*)C, m, n, k, ep, tiles_m, tiles_n, c.status);
  if (c.prof != nullptr && c.prof->on) c.prof->end(c.stream);
  return 0;
}

}  // namespace bsr
