// Multi-head self-attention (paper Eq. 1) on the tcgen05 tensor cores for bf16, head dimension 64.
//
// Forward (T <= 256 keys): a persistent, warp-specialised kernel (see attn_fwd_ws_kernel): TMA loads Q, K, V tiles of
//   the packed projections [B*T, 3*H*64] into 128-byte-swizzled shared memory; S = Q K^T goes to tensor memory; a
//   thread owns (half of) a query row: row maximum, exp2, row sum in float from tcgen05.ld; the probabilities go back
//   into tensor memory as bf16 and O = P V reads them from there; the epilogue scales by 1 / row sum.
//   The classification token's row (query 0) is also written out as probabilities: these are the token
//   importance scores of Eq. 6.
// Rows and keys beyond T inside a tile belong to the next image (or are zero-filled past the tensor's end):
// keys are masked in the softmax, rows are computed and never stored.
#include "common.cuh"
#include "kernels.h"
#include "tc_ptx.cuh"

namespace bsr {
namespace tc {

constexpr int AT_D = 64;
constexpr int AT_BOX = 64;                       // rows per TMA box
constexpr int AT_BOX_BYTES = AT_BOX * AT_D * 2;  // 8 KB
constexpr int AT_QROWS = 128;
constexpr int AT_MAXKEYS = 256;
constexpr float AT_LONG_SLACK = 8.0f;             // binary orders the row maximum may exceed the reference before a rescale
constexpr int AT_LONG_MAXBLK = 64;                // key blocks of the longest sequence the kernel takes
constexpr int AT_LONG_KB = 64;                   // keys per block of the kernel for longer sequences (four CTAs per SM)

__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ float ex2_fast(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// ------------------------------------------------------------------------------------------------
// Forward for T <= 256, persistent and warp-specialised: one CTA per SM walks (image, head) pairs.
//   loader warp : TMA (one lane): K and V of a pair into a ring of slots, each 128-query tile of Q into another
//                 ring, running ahead of the tensor core as far as the slots allow;
//   NBUF softmax groups, one per accumulator buffer in tensor memory, each working on every NBUF-th tile.  A group's
//                 first thread also issues the group's MMAs: S = Q K^T for the group's next tile as soon as the
//                 previous O has been read, and O = P V as soon as the group has written P.  A thread owns (half
//                 of) a query row: row maximum and exp2 from tcgen05.ld, probabilities packed to bf16 and written
//                 back with tcgen05.st over the S columns already consumed (P never goes through shared memory,
//                 the second MMA reads it from tensor memory), then O scaled by the row sum and stored.
// NBUF is 4, 3 or 2 for up to 128, 160 or 256 keys; with two groups a group has eight warps, two per lane quarter
// splitting the keys (and the output columns).  Accumulator buffer layout (columns): S at 0 .. tpad-1 (fp32), P (bf16
// pairs) over S columns its writer has already consumed, O in the last 64 columns of the buffer, beyond P.
// ------------------------------------------------------------------------------------------------
constexpr int WS_QSLOTS = 3;
constexpr int WS_Q_BYTES = 2 * AT_BOX_BYTES;
constexpr int WS_MAXBUF = 4, WS_MAXKV = 6;

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&h);
}
// Two floats as a pair of bf16 plus the pair that the rounding left.
__device__ __forceinline__ void split_bf16x2(float a, float b, uint32_t& hi, uint32_t& lo) {
  hi = pack_bf16x2(a, b);
  lo = pack_bf16x2(a - __uint_as_float(hi << 16), b - __uint_as_float(hi & 0xffff0000u));
}
// Four neighbouring lanes hold a row of four 16-byte units each; afterwards lane j of them holds unit j of the four rows.
// Stored so, an instruction writes 64 bytes of 8 rows instead of 16 bytes of 32 rows (197 tokens, batch 128, 12 heads: 59.1
// -> 55.6 us).
__device__ __forceinline__ void transpose_units(uint4 (&u)[4], int lane) {
#pragma unroll
  for (int m = 1; m <= 2; m <<= 1)
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const int a = m == 1 ? 2 * p : p, b = a + m;
      const bool hi = (lane & m) != 0;
      uint32_t *ua = reinterpret_cast<uint32_t*>(&u[a]), *ub = reinterpret_cast<uint32_t*>(&u[b]);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t got = __shfl_xor_sync(0xffffffffu, hi ? ua[j] : ub[j], m);
        if (hi) ua[j] = got;
        else ub[j] = got;
      }
    }
}
__device__ __forceinline__ void group_sync(int id, int threads) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory"); }
// mbar_wait that gives up at once when another role already has: after a failure the groups keep walking their
// tiles (their named barriers need every thread) and every further wait must return quickly.
__device__ __forceinline__ bool mbar_wait_q(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  if (*abort_flag) return false;
  return mbar_wait(bar, parity, abort_flag);
}

template <int NBUF>
__global__ void __launch_bounds__((NBUF == 2 ? 19 : 4 * NBUF + 3) * 32, 1)
attn_fwd_ws_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_kv, bf16* __restrict__ out,
                   float* __restrict__ lse, float* __restrict__ cls_prob, int B, int T, int H, int kvslots, int* status) {
  constexpr int GW = NBUF == 2 ? 8 : 4;                         // warps per softmax group
  constexpr int GT = GW * 32;
  constexpr uint32_t BUF_COLS = NBUF == 2 ? 256u : (NBUF == 3 ? 160u : 128u);
  constexpr uint32_t O_COL = BUF_COLS - 64u;                                 // 192, 96, 64
  extern __shared__ unsigned char smem_dyn[];
  uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
  unsigned char* base_ptr = smem_dyn + (base - smem_u32(smem_dyn));
  const int tpad = (T + 15) & ~15;
  const int nqt = (T + AT_QROWS - 1) / AT_QROWS;
  const uint32_t kv_bytes = tpad * 128;                          // one of K, V: tpad rows of 64 bf16
  const uint32_t sQ = base, sKV = sQ + WS_QSLOTS * WS_Q_BYTES;
  const uint32_t tail = sKV + kvslots * 2 * kv_bytes;
  float* cls_buf = reinterpret_cast<float*>(base_ptr + (tail - base));     // [NBUF][AT_MAXKEYS]
  float* red = cls_buf + WS_MAXBUF * AT_MAXKEYS;                            // [NBUF][max, sum][2 halves][128 rows]
  const uint32_t bars = tail + (WS_MAXBUF * AT_MAXKEYS + WS_MAXBUF * 4 * AT_QROWS) * 4;
  auto q_full = [&](int s) { return bars + 8u * s; };
  auto q_empty = [&](int s) { return bars + 8u * (4 + s); };
  auto kv_full = [&](int s) { return bars + 8u * (8 + s); };
  auto kv_empty = [&](int s) { return bars + 8u * (16 + s); };
  auto s_full = [&](int b) { return bars + 8u * (24 + b); };
  auto o_full = [&](int b) { return bars + 8u * (28 + b); };
  auto p_full = [&](int b) { return bars + 8u * (32 + b); };
  auto t_empty = [&](int b) { return bars + 8u * (36 + b); };
  auto token = [&](int b) { return bars + 8u * (40 + b); };
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int pairs = B * H;
  constexpr int LOADER = NBUF * GW;                             // then the two MMA issuer warps

  if (tid == 0) {
    abort_flag = 0;
    for (int s = 0; s < WS_QSLOTS; ++s) { mbar_init(q_full(s), 1); mbar_init(q_empty(s), 1); }
    for (int s = 0; s < WS_MAXKV; ++s) { mbar_init(kv_full(s), 1); mbar_init(kv_empty(s), nqt); }
    for (int b = 0; b < WS_MAXBUF; ++b) {
      mbar_init(s_full(b), 1); mbar_init(o_full(b), 1); mbar_init(p_full(b), GW); mbar_init(t_empty(b), GW); mbar_init(token(b), 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    prefetch_map(&map_q);
    prefetch_map(&map_kv);
  }
  if (warp == LOADER) {
    tmem_alloc(smem_u32(&tmem_slot), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  if (leaves_sms_idle()) release_dependents();
  await_inputs();
  volatile int* abortp = &abort_flag;

  if (warp == LOADER) {
    // ------------------------------- TMA loader ---------------------------------
    if (lane == 0) {
      int i = 0, n = 0;
      bool ok = true;
      for (int bh = blockIdx.x; bh < pairs && ok; bh += gridDim.x, ++n) {
        int b = bh / H, h = bh % H, row0 = b * T;
        int ks = n % kvslots;
        if (!mbar_wait(kv_empty(ks), ((n / kvslots) & 1) ^ 1u, abortp)) { ok = false; break; }
        mbar_expect_tx(kv_full(ks), 2 * kv_bytes);
        uint32_t sK = sKV + ks * 2 * kv_bytes, sV = sK + kv_bytes;
        tma_load_2d(sK, &map_kv, kv_full(ks), (H + h) * AT_D, row0);
        tma_load_2d(sV, &map_kv, kv_full(ks), (2 * H + h) * AT_D, row0);
        for (int qt = 0; qt < nqt; ++qt, ++i) {
          int qs = i % WS_QSLOTS;
          if (!mbar_wait(q_empty(qs), ((i / WS_QSLOTS) & 1) ^ 1u, abortp)) { ok = false; break; }
          mbar_expect_tx(q_full(qs), WS_Q_BYTES);
          tma_load_2d(sQ + qs * WS_Q_BYTES, &map_q, q_full(qs), h * AT_D, row0 + qt * AT_QROWS);
        }
      }
      if (!ok) {                      // copies already issued still land: give them a bounded time before the CTA leaves
        unsigned long long t0 = global_ns();
        while (global_ns() - t0 < 1000000ull) {}
      }
    }
  } else if (warp == LOADER + 1) {
    // ------------------------------- S = Q K^T issuer ---------------------------
    if (lane == 0) {
      const uint32_t idesc_s = make_idesc_mn(AT_QROWS, tpad, false, false);
      int i = 0, n = 0;
      bool ok = true;
      for (int bh = blockIdx.x; bh < pairs && ok; bh += gridDim.x, ++n) {
        int ks = n % kvslots;
        for (int qt = 0; qt < nqt; ++qt, ++i) {
          int qs = i % WS_QSLOTS, buf = i % NBUF;
          if (qt == 0 && !mbar_wait(kv_full(ks), (n / kvslots) & 1, abortp)) { ok = false; break; }
          if (!mbar_wait(q_full(qs), (i / WS_QSLOTS) & 1, abortp)) { ok = false; break; }
          if (!mbar_wait(t_empty(buf), ((i / NBUF) & 1) ^ 1u, abortp)) { ok = false; break; }
          tc_fence_after();
          uint32_t sq = sQ + qs * WS_Q_BYTES, sK = sKV + ks * 2 * kv_bytes;
#pragma unroll
          for (int k = 0; k < AT_D / 16; ++k)
            umma_bf16(tmem + buf * BUF_COLS, make_desc(sq + k * 32, 16, 1024), make_desc(sK + k * 32, 16, 1024), idesc_s, k > 0 ? 1u : 0u);
          umma_commit(s_full(buf));
          umma_commit(q_empty(qs));
        }
      }
    }
  } else if (warp == LOADER + 2) {
    // ------------------------------- O = P V issuer -----------------------------
    if (lane == 0) {
      const uint32_t idesc_o = make_idesc_mn(AT_QROWS, AT_D, false, true);
      const int ksteps = tpad / 16;
      const int chs2 = ((((T + 31) >> 5) + 1) >> 1) * 2;       // first 16-key step of the second half's probabilities
      int i = 0, n = 0;
      bool ok = true;
      for (int bh = blockIdx.x; bh < pairs && ok; bh += gridDim.x, ++n) {
        int ks = n % kvslots;
        for (int qt = 0; qt < nqt; ++qt, ++i) {
          int pb = i % NBUF;
          if (!mbar_wait(p_full(pb), (i / NBUF) & 1, abortp)) { ok = false; break; }
          tc_fence_after();
          uint32_t tb = tmem + pb * BUF_COLS;
          uint32_t sV = sKV + ks * 2 * kv_bytes + kv_bytes;
          for (int k = 0; k < ksteps; ++k)
            umma_bf16_ts(tb + O_COL, tb + 8 * k + ((GW == 8 && k >= chs2) ? 8 * chs2 : 0), make_desc(sV + k * (16 * 128), 8192, 1024),
                         idesc_o, k > 0 ? 1u : 0u);
          umma_commit(o_full(pb));
          umma_commit(kv_empty(ks));
        }
      }
    }
  } else {
    // ------------------------------- softmax groups -----------------------------
    const int g = warp / GW, gw = warp % GW;
    const int quarter = gw & 3, half = gw >> 2;            // half: which part of the keys / output columns (eight-warp groups)
    const bool leader = (gw == 0 && lane == 0);
    const int row = quarter * 32 + lane;
    const float c = 0.125f * 1.4426950408889634f;          // 1/sqrt(64) * log2(e)
    const uint32_t tbuf = tmem + g * BUF_COLS;
    const uint32_t trow = tbuf + ((uint32_t)(quarter * 32) << 16);
    const int nchunk = (T + 31) >> 5;
    const int ch0 = (GW == 8 && half == 1) ? (nchunk + 1) >> 1 : 0;
    const int ch1 = (GW == 8 && half == 0) ? (nchunk + 1) >> 1 : nchunk;
    // An eight-warp group writes the second half's probabilities over the S columns that half itself has consumed
    // (the first half may still be reading its own): chunk ch >= chs lands 16 * chs columns further right.
    const int chs = (nchunk + 1) >> 1;
    const uint32_t p_shift = (GW == 8 && half == 1) ? 16u * chs : 0u;
    float* cbuf = cls_buf + g * AT_MAXKEYS;
    float* rmax = red + g * 4 * AT_QROWS;                  // [2][128]
    float* rsum = rmax + 2 * AT_QROWS;                     // [2][128]
    bool ok = true;
    // tile i of this CTA: pair n = i / nqt (bh = blockIdx.x + n * gridDim.x), query tile qt = i % nqt
    const int my_pairs = blockIdx.x < pairs ? (pairs - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    const int items = my_pairs * nqt;
    int use = 0;
    for (int i = g; i < items; i += NBUF, ++use) {
      const int n = i / nqt, qt = i - n * nqt;
      const int bh = blockIdx.x + n * gridDim.x;
      const int b = bh / H, h = bh - b * H;
      const uint32_t par = use & 1;
      const int q0 = qt * AT_QROWS;
      const bool live = q0 + quarter * 32 < T;           // warp-uniform: a quarter whose rows all lie past T does no work
      ok = mbar_wait_q(s_full(g), par, abortp) && ok;
      ok = __all_sync(0xffffffffu, ok);
      tc_fence_after();
      float mx = -INFINITY, sum = 0.f;
      const bool cls_row = (q0 == 0 && row == 0 && cls_prob != nullptr);
      if (live) {
        for (int ch = ch0; ch < ch1; ++ch) {
          uint32_t r[32];
          tmem_ld32(trow + ch * 32, r);
          tmem_ld_wait();
          if (ch * 32 + 32 <= T) {
#pragma unroll
            for (int j = 0; j < 32; j += 2) mx = fmax3(mx, __uint_as_float(r[j]), __uint_as_float(r[j + 1]));
          } else {
#pragma unroll
            for (int j = 0; j < 32; ++j)
              if (ch * 32 + j < T) mx = fmaxf(mx, __uint_as_float(r[j]));
          }
        }
      }
      if (GW == 8) {
        rmax[half * AT_QROWS + row] = mx;
        group_sync(1 + g, GT);
        mx = fmaxf(rmax[row], rmax[AT_QROWS + row]);
      }
      // With two groups the exponentials of successive tiles take turns (the special-function unit is shared), so
      // that one group's exponentials overlap the other's tensor-core and load/store phases instead of colliding
      // with its exponentials.  Three or four groups drift apart by themselves.
      if (NBUF == 2 && i > 0) {
        ok = mbar_wait_q(token(g), (g == 0 ? use - 1 : use) & 1, abortp) && ok;
        ok = __all_sync(0xffffffffu, ok);
      }
      if (live) {
        const float mc = mx * c;
        for (int ch = ch0; ch < ch1; ++ch) {
          uint32_t r[32];
          tmem_ld32(trow + ch * 32, r);
          tmem_ld_wait();
          float p[32];
          if (ch * 32 + 32 <= T) {
#pragma unroll
            for (int j = 0; j < 32; ++j) p[j] = ex2_fast(fmaf(__uint_as_float(r[j]), c, -mc));
          } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) p[j] = (ch * 32 + j < T) ? ex2_fast(fmaf(__uint_as_float(r[j]), c, -mc)) : 0.f;
          }
          float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll
          for (int j = 0; j < 32; j += 4) { s0 += p[j]; s1 += p[j + 1]; s2 += p[j + 2]; s3 += p[j + 3]; }
          sum += (s0 + s1) + (s2 + s3);
          if (cls_row) {
#pragma unroll
            for (int j = 0; j < 32; ++j) cbuf[ch * 32 + j] = p[j];
          }
          uint32_t pk[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) pk[j] = pack_bf16x2(p[2 * j], p[2 * j + 1]);
          tmem_st16(trow + ch * 16 + p_shift, pk);
        }
        tmem_st_wait();
      }
      if (GW == 8) rsum[half * AT_QROWS + row] = sum;
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(p_full(g));             // P of this warp's rows and keys is in tensor memory
      if (GW == 8) group_sync(1 + g, GT);                // partial sums and the classification row are in shared memory
      else __syncwarp();
      if (NBUF == 2 && leader) mbar_arrive(token((g + 1) % NBUF));
      if (GW == 8) sum = rsum[row] + rsum[AT_QROWS + row];
      const float inv = 1.0f / sum;
      const int q = q0 + row;
      if (live && q < T && half == 0 && lse != nullptr) lse[((size_t)b * H + h) * T + q] = mx * 0.125f + logf(sum);
      if (q0 == 0 && gw == 0 && cls_prob != nullptr) {        // this warp holds query 0 in lane 0
        float s_inv = __shfl_sync(0xffffffffu, inv, 0);
        float* cp = cls_prob + ((size_t)b * H + h) * (T - 1);
        for (int j = 1 + lane; j < T; j += 32) cp[j - 1] = cbuf[j] * s_inv;
      }
      ok = mbar_wait_q(o_full(g), par, abortp) && ok;
      ok = __all_sync(0xffffffffu, ok);
      tc_fence_after();
      constexpr int NH = GW == 8 ? 1 : 2;                // 32-column halves of O this thread reads
      if (live) {
#pragma unroll
        for (int hh = 0; hh < NH; ++hh) {
          uint32_t ro[32];
          tmem_ld32(trow + O_COL + (half + hh) * 32, ro);
          tmem_ld_wait();
          if (ok) {
            uint4 u[4];
#pragma unroll
            for (int gq = 0; gq < 4; ++gq) {
              uint32_t* w = reinterpret_cast<uint32_t*>(&u[gq]);
#pragma unroll
              for (int j = 0; j < 4; ++j)
                w[j] = pack_bf16x2(__uint_as_float(ro[gq * 8 + 2 * j]) * inv, __uint_as_float(ro[gq * 8 + 2 * j + 1]) * inv);
            }
            bf16* orow = out + ((size_t)b * T + q) * H * AT_D + (size_t)h * AT_D + (half + hh) * 32;
            if constexpr (GW == 8) {               // with four warps a group the exchange costs more than it saves (140 tokens: 38.1 -> 39.9 us)
              transpose_units(u, lane);
              const int j = lane & 3;
#pragma unroll
              for (int k = 0; k < 4; ++k)
                if (q - j + k < T) *reinterpret_cast<uint4*>(orow + (ptrdiff_t)(k - j) * H * AT_D + j * 8) = u[k];
            } else if (q < T) {
#pragma unroll
              for (int gq = 0; gq < 4; ++gq) *reinterpret_cast<uint4*>(orow + gq * 8) = u[gq];
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(t_empty(g));            // O has been read: the buffer may take the next S
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == LOADER) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
  if (tid == 0 && abort_flag && status != nullptr) atomicOr(status, STATUS_TIMEOUT);
}

// ------------------------------------------------------------------------------------------------
// Forward for T <= 256 where all (image, head, 128 queries) fit the SMs at once: a CTA each, nothing to overlap with, so what counts
// is the length of the chain.  Eight softmax warps, two threads a query row, and a warp whose first lane loads and issues.
// A thread has its half of the row's scores in registers (NC chunks of 32 keys): they are read from tensor memory once, in one
// go.  Columns of tensor memory as in attn_fwd_ws_kernel with two
// buffers: P of each half over the scores that half has read, O in the last 64.  Its sums are in that kernel's order and the outputs the
// same bit for bit: an image's result does not depend on how many others there are.
// us of a launch in a row of launches, attn_fwd_ws_kernel / this, 6 heads:
//   197 tokens, 1 / 8 images 8.0 / 5.4, 8.3 / 5.9   140 tokens 6.7 / 4.5, 7.0 / 5.1   100 tokens 5.3 / 3.9, 5.6 / 4.1   71 tokens 4.7 / 3.6, 4.9 / 3.7
// and where there are more tiles than SMs (12 heads) 197 tokens, 8 images 8.9 / 11.2; 100 tokens, 16 images 7.3 / 8.7.
// DeiT-S, one image: inference 430 -> 411 us, a step 642 -> 623.
// ------------------------------------------------------------------------------------------------
constexpr int WIDE_THREADS = 288;

template <int NC>
__global__ void __launch_bounds__(WIDE_THREADS, 1)
attn_fwd_wide_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_kv, bf16* __restrict__ out,
                     float* __restrict__ lse, float* __restrict__ cls_prob, int T, int H, int nqt, int* status) {
  constexpr uint32_t O_COL = 192;
  extern __shared__ unsigned char smem_dyn[];
  __shared__ __align__(8) unsigned long long bar_mem[5];
  __shared__ __align__(16) float cbuf[AT_MAXKEYS];
  __shared__ float rmax[2][AT_QROWS], csum[8][AT_QROWS];         // a half's maximum, a chunk's sum
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
  const int tpad = (T + 15) & ~15;
  const uint32_t kv_bytes = tpad * 128;
  const uint32_t sQ = base, sK = sQ + WS_Q_BYTES, sV = sK + kv_bytes;
  const uint32_t bars = smem_u32(bar_mem);
  const uint32_t qk_full = bars, v_full = bars + 8, s_full = bars + 16, p_full = bars + 24, o_full = bars + 32;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int bh = blockIdx.x / nqt, q0 = (blockIdx.x - bh * nqt) * AT_QROWS, b = bh / H, h = bh - b * H;
  const int nchunk = (T + 31) >> 5, chs = (nchunk + 1) >> 1;       // chunks of 32 keys; the first half's
  if (tid == 0) {
    abort_flag = 0;
    mbar_init(qk_full, 1); mbar_init(v_full, 1); mbar_init(s_full, 1); mbar_init(p_full, 8); mbar_init(o_full, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    prefetch_map(&map_q);
    prefetch_map(&map_kv);
  }
  if (warp == 8) {
    tmem_alloc(smem_u32(&tmem_slot), 256);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  if (leaves_sms_idle()) release_dependents();
  await_inputs();
  volatile int* abortp = &abort_flag;

  if (warp == 8) {
    if (lane == 0) {
      const int row0 = b * T;
      mbar_expect_tx(qk_full, WS_Q_BYTES + kv_bytes);
      tma_load_2d(sK, &map_kv, qk_full, (H + h) * AT_D, row0);
      tma_load_2d(sQ, &map_q, qk_full, h * AT_D, row0 + q0);
      mbar_expect_tx(v_full, kv_bytes);
      tma_load_2d(sV, &map_kv, v_full, (2 * H + h) * AT_D, row0);
      bool ok = mbar_wait(qk_full, 0, abortp);
      if (ok) {
        tc_fence_after();
        const uint32_t idesc = make_idesc_mn(AT_QROWS, tpad, false, false);
#pragma unroll
        for (int k = 0; k < AT_D / 16; ++k)
          umma_bf16(tmem, make_desc(sQ + k * 32, 16, 1024), make_desc(sK + k * 32, 16, 1024), idesc, k > 0 ? 1u : 0u);
        umma_commit(s_full);
        ok = mbar_wait(v_full, 0, abortp) && mbar_wait(p_full, 0, abortp);
      }
      if (ok) {
        tc_fence_after();
        const uint32_t idesc = make_idesc_mn(AT_QROWS, AT_D, false, true);
        for (int k = 0; k < tpad / 16; ++k)                          // 16 keys are 8 columns of P; the second half's start at its scores
          umma_bf16_ts(tmem + O_COL, tmem + 8 * k + (k >= 2 * chs ? 16 * chs : 0), make_desc(sV + k * (16 * 128), 8192, 1024), idesc, k > 0 ? 1u : 0u);
        umma_commit(o_full);
      } else {                        // copies already issued still land: give them a bounded time before the CTA leaves
        unsigned long long t0 = global_ns();
        while (global_ns() - t0 < 1000000ull) {}
      }
    }
  } else {
    const int quarter = warp & 3, half = warp >> 2, row = quarter * 32 + lane, q = q0 + row;
    const float c = 0.125f * 1.4426950408889634f;          // 1/sqrt(64) * log2(e)
    const uint32_t trow = tmem + ((uint32_t)(quarter * 32) << 16);
    const int ch0 = half == 0 ? 0 : chs, nch = (half == 0 ? chs : nchunk) - ch0;
    const bool live = q0 + quarter * 32 < T;             // warp-uniform: a quarter whose rows all lie past T does no work
    bool ok = __all_sync(0xffffffffu, mbar_wait(s_full, 0, abortp));
    tc_fence_after();
    uint32_t r[NC * 32];
    float mx = -INFINITY;
    if (live) {
#pragma unroll
      for (int i = 0; i < NC; ++i)
        if (i < nch) tmem_ld32(trow + (ch0 + i) * 32, r + i * 32);
      tmem_ld_wait();
#pragma unroll
      for (int i = 0; i < NC; ++i)
        if (i < nch) {
          if ((ch0 + i) * 32 + 32 > T) {
#pragma unroll
            for (int j = 0; j < 32; ++j)
              if ((ch0 + i) * 32 + j >= T) r[i * 32 + j] = 0xff800000u;        // -inf: probability zero
          }
#pragma unroll
          for (int j = 0; j < 32; j += 2) mx = fmax3(mx, __uint_as_float(r[i * 32 + j]), __uint_as_float(r[i * 32 + j + 1]));
        }
    }
    rmax[half][row] = mx;
    group_sync(1, 256);
    mx = fmaxf(rmax[0][row], rmax[1][row]);
    const bool cls_row = q == 0 && cls_prob != nullptr;
    if (live) {
      const float mc = mx * c;
#pragma unroll
      for (int i = 0; i < NC; ++i)
        if (i < nch) {
          float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
          uint32_t pk[16];
#pragma unroll
          for (int j = 0; j < 32; j += 4) {
            float p[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) p[e] = ex2_fast(fmaf(__uint_as_float(r[i * 32 + j + e]), c, -mc));
            s0 += p[0]; s1 += p[1]; s2 += p[2]; s3 += p[3];
            pk[j / 2] = pack_bf16x2(p[0], p[1]);
            pk[j / 2 + 1] = pack_bf16x2(p[2], p[3]);
            if (cls_row) *reinterpret_cast<float4*>(cbuf + (ch0 + i) * 32 + j) = make_float4(p[0], p[1], p[2], p[3]);
          }
          csum[ch0 + i][row] = (s0 + s1) + (s2 + s3);
          tmem_st16(trow + ch0 * 32 + i * 16, pk);
        }
      tmem_st_wait();
    }
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(p_full);                  // P of this warp's rows and keys is in tensor memory
    group_sync(1, 256);                                  // sums and the classification row are in shared memory
    // in the order of attn_fwd_ws_kernel: one sum up to 160 keys, a sum per half beyond
    const int cut = T > 160 ? chs : nchunk;
    float sum = 0.f, sum2 = 0.f;
    for (int i = 0; i < cut; ++i) sum += csum[i][row];
    for (int i = cut; i < nchunk; ++i) sum2 += csum[i][row];
    if (T > 160) sum += sum2;
    const float inv = 1.0f / sum;
    if (half == 0 && q < T && lse != nullptr) lse[(size_t)bh * T + q] = mx * 0.125f + logf(sum);
    if (q0 == 0 && cls_prob != nullptr && quarter == 0) {           // both warps that hold query 0 (in lane 0): a half of its row each
      const float s_inv = __shfl_sync(0xffffffffu, inv, 0);
      float* cp = cls_prob + (size_t)bh * (T - 1);
      for (int j = 1 + half * 32 + lane; j < T; j += 64) cp[j - 1] = cbuf[j] * s_inv;
    }
    ok = mbar_wait_q(o_full, 0, abortp) && ok;
    ok = __all_sync(0xffffffffu, ok);
    tc_fence_after();
    if (live && ok) {
      uint32_t ro[32];
      tmem_ld32(trow + O_COL + half * 32, ro);
      tmem_ld_wait();
      uint4 u[4];
#pragma unroll
      for (int gq = 0; gq < 4; ++gq) {
        uint32_t* w = reinterpret_cast<uint32_t*>(&u[gq]);
#pragma unroll
        for (int j = 0; j < 4; ++j)
          w[j] = pack_bf16x2(__uint_as_float(ro[gq * 8 + 2 * j]) * inv, __uint_as_float(ro[gq * 8 + 2 * j + 1]) * inv);
      }
      transpose_units(u, lane);
      const int j = lane & 3;
      bf16* orow = out + ((size_t)b * T + q) * H * AT_D + (size_t)h * AT_D + half * 32;
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (q - j + k < T) *reinterpret_cast<uint4*>(orow + (ptrdiff_t)(k - j) * H * AT_D + j * 8) = u[k];
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 8) {
    tc_fence_after();
    tmem_dealloc(tmem, 256);
  }
  if (tid == 0 && abort_flag && status != nullptr) atomicOr(status, STATUS_TIMEOUT);
}

// ------------------------------------------------------------------------------------------------
// Forward for longer sequences (T > 256): the keys are walked once in blocks of AT_LONG_KB.  One CTA per (image, head, 128
// queries), four of them on an SM to cover one another's waits: four softmax warps, a thread per query row, and a warp
// whose first lane loads (two slots of K and V) and issues.  Per block the row's 64 scores are read from tensor memory
// once, P = exp(S - m) against the row's reference maximum m goes back over them as bf16, and the issuer runs O += P V and
// the next block's S = Q K^T as one group: the softmax warps wait once a block.  m follows the running maximum only
// in jumps of more than AT_LONG_SLACK binary orders, at which the accumulator is rescaled in place (rare after the first
// block).  The classification row's probabilities are written out block by block against the m of the moment and brought
// onto the final scale by its warp at the end.
// 577 tokens, batch 32, 12 heads: 83 us (290 tokens: 31, was 47); with the scores read twice, P through shared memory, two waits a
// block and loads that waited for the block before, 143 us.  The exponentials alone take 28 us, the products 20.
// ------------------------------------------------------------------------------------------------
constexpr int AT_LONG_THREADS = 160;

__global__ void __launch_bounds__(AT_LONG_THREADS, 4)
attn_fwd_tc_long_kernel(const __grid_constant__ CUtensorMap map_qkv, bf16* __restrict__ out, float* __restrict__ lse,
                        float* __restrict__ cls_prob, int B, int T, int H, int* status) {
  extern __shared__ unsigned char smem_dyn[];
  const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
  unsigned char* base_ptr = smem_dyn + (base - smem_u32(smem_dyn));
  constexpr int KB = AT_LONG_KB;
  constexpr uint32_t KV_BYTES = KB * 128;
  const uint32_t sQ = base, sKV = sQ + 2 * AT_BOX_BYTES;                   // [2 slots][K, V]
  const uint32_t bars = sKV + 4 * KV_BYTES;
  auto full_bar = [&](int s) { return bars + 8u * s; };
  const uint32_t s_bar = bars + 16, p_bar = bars + 24;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  __shared__ float cls_m[AT_LONG_MAXBLK];               // reference maximum of the classification row, block by block
  __shared__ __align__(16) float cls_p[32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int bh = blockIdx.y, b = bh / H, h = bh - b * H;
  const int q0 = blockIdx.x * AT_QROWS, row0 = b * T;
  const int nblk = (T + KB - 1) / KB;
  if (tid == 0) {
    abort_flag = 0;
    mbar_init(full_bar(0), 1); mbar_init(full_bar(1), 1); mbar_init(s_bar, 1); mbar_init(p_bar, 4);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    prefetch_map(&map_qkv);
  }
  if (warp == 4) {
    tmem_alloc(smem_u32(&tmem_slot), 2 * KB);           // S (then P) in the first KB columns, O behind it
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  if (leaves_sms_idle()) release_dependents();
  await_inputs();
  constexpr uint32_t C_O = KB;
  volatile int* abortp = &abort_flag;

  if (warp == 4) {
    // ------------------------------- loads and products -------------------------
    if (lane == 0) {
      auto load = [&](int kb) {
        const uint32_t dst = sKV + (kb & 1) * 2 * KV_BYTES, bar = full_bar(kb & 1);
        tma_load_2d(dst, &map_qkv, bar, (H + h) * AT_D, row0 + kb * KB);
        tma_load_2d(dst + KV_BYTES, &map_qkv, bar, (2 * H + h) * AT_D, row0 + kb * KB);
      };
      auto scores = [&](int kb) {
        const int kpad = (min(KB, T - kb * KB) + 15) & ~15;
        const uint32_t sK = sKV + (kb & 1) * 2 * KV_BYTES, idesc = make_idesc_mn(AT_QROWS, kpad, false, false);
#pragma unroll
        for (int k = 0; k < AT_D / 16; ++k)
          umma_bf16(tmem, make_desc(sQ + k * 32, 16, 1024), make_desc(sK + k * 32, 16, 1024), idesc, k > 0 ? 1u : 0u);
      };
      mbar_expect_tx(full_bar(0), 2 * AT_BOX_BYTES + 2 * KV_BYTES);
      for (int j = 0; j < 2; ++j) tma_load_2d(sQ + j * AT_BOX_BYTES, &map_qkv, full_bar(0), h * AT_D, row0 + q0 + j * AT_BOX);
      load(0);
      if (nblk > 1) {
        mbar_expect_tx(full_bar(1), 2 * KV_BYTES);
        load(1);
      }
      bool ok = mbar_wait(full_bar(0), 0, abortp);
      if (ok) {
        tc_fence_after();
        scores(0);
        umma_commit(s_bar);
      }
      for (int kb = 0; kb < nblk && ok; ++kb) {
        ok = mbar_wait(p_bar, kb & 1, abortp);           // P of this block is in tensor memory
        if (!ok) break;
        tc_fence_after();
        const int kpad = (min(KB, T - kb * KB) + 15) & ~15;
        const uint32_t sV = sKV + (kb & 1) * 2 * KV_BYTES + KV_BYTES, idesc = make_idesc_mn(AT_QROWS, AT_D, false, true);
        for (int k = 0; k < kpad / 16; ++k)
          umma_bf16_ts(tmem + C_O, tmem + 8 * k, make_desc(sV + k * (16 * 128), 8192, 1024), idesc, (kb > 0 || k > 0) ? 1u : 0u);
        if (kb + 1 < nblk) {                             // products run in order: the next scores overwrite P once it has been read
          ok = mbar_wait(full_bar((kb + 1) & 1), ((kb + 1) >> 1) & 1, abortp);
          if (ok) {
            tc_fence_after();
            scores(kb + 1);
          }
        }
        umma_commit(s_bar);
        if (ok && kb + 2 < nblk) {
          ok = mbar_wait(s_bar, (kb + 1) & 1, abortp);   // this block's K and V have been read
          if (ok) {
            mbar_expect_tx(full_bar(kb & 1), 2 * KV_BYTES);
            load(kb + 2);
          }
        }
      }
      if (!ok) {                                         // copies already issued still land: a bounded time before the CTA leaves
        unsigned long long t0 = global_ns();
        while (global_ns() - t0 < 1000000ull) {}
      }
    }
  } else {
    // ------------------------------- softmax ------------------------------------
    const float c = 0.125f * 1.4426950408889634f;          // 1/sqrt(64) * log2(e)
    const uint32_t trow = tmem + ((uint32_t)(warp * 32) << 16);
    const bool cls_warp = (q0 == 0 && warp == 0 && cls_prob != nullptr);
    float* cp = cls_warp ? cls_prob + (size_t)bh * (T - 1) : nullptr;
    float mx = -INFINITY, sum = 0.f;
    bool ok = true;
    for (int kb = 0; kb < nblk && ok; ++kb) {
      const int keys = min(KB, T - kb * KB);
      ok = mbar_wait_q(s_bar, kb & 1, abortp);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      uint32_t r[KB];
      tmem_ld32(trow, r);
      tmem_ld32(trow + 32, r + 32);
      tmem_ld_wait();
      if (keys < KB) {
#pragma unroll
        for (int j = 0; j < KB; ++j)
          if (j >= keys) r[j] = 0xff800000u;               // -inf: probability zero
      }
      float bm = -INFINITY;
#pragma unroll
      for (int j = 0; j < KB; j += 2) bm = fmax3(bm, __uint_as_float(r[j]), __uint_as_float(r[j + 1]));
      // The reference maximum of a row moves only when the block's maximum exceeds it by more than AT_LONG_SLACK in the
      // exponent (the probabilities then stay below 2^AT_LONG_SLACK, harmless in bf16 and in the fp32 sum); when it
      // moves, the accumulated output and sum of that row are scaled down.  The decision is taken per warp, because the
      // accumulator is read and written with warp-wide instructions; rows that do not move scale by one.
      if (kb == 0) {
        mx = bm;
      } else {
        const bool grow = (bm - mx) * c > AT_LONG_SLACK;
        if (__any_sync(0xffffffffu, grow)) {
          const float nm = grow ? bm : mx, f = ex2_fast((mx - nm) * c);
#pragma unroll 1
          for (int q = 0; q < 4; ++q) {
            uint32_t o[16];
            tmem_ld16(trow + C_O + q * 16, o);
            tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < 16; ++j) o[j] = __float_as_uint(__uint_as_float(o[j]) * f);
            tmem_st16(trow + C_O + q * 16, o);
          }
          sum *= f;
          mx = nm;
        }
      }
      const float mc = mx * c;
      if (cls_warp && lane == 0) cls_m[kb] = mx;
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        float s0 = 0.f, s1 = 0.f;
#pragma unroll
        for (int j = half * 32; j < half * 32 + 32; j += 2) {
          const float e0 = ex2_fast(fmaf(__uint_as_float(r[j]), c, -mc)), e1 = ex2_fast(fmaf(__uint_as_float(r[j + 1]), c, -mc));
          s0 += e0; s1 += e1;
          r[j] = __float_as_uint(e0); r[j + 1] = __float_as_uint(e1);
        }
        sum += s0 + s1;
        if (cls_warp) {                 // relative to this block's reference maximum; put on the final scale below
          if (lane == 0) {
#pragma unroll
            for (int j = 0; j < 32; j += 4) *reinterpret_cast<uint4*>(cls_p + j) = make_uint4(r[half * 32 + j], r[half * 32 + j + 1], r[half * 32 + j + 2], r[half * 32 + j + 3]);
          }
          __syncwarp();
          const int key = kb * KB + half * 32 + lane;
          if (key >= 1 && key < T) cp[key - 1] = cls_p[lane];
          __syncwarp();
        }
        uint32_t pk[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) pk[j] = pack_bf16x2(__uint_as_float(r[half * 32 + 2 * j]), __uint_as_float(r[half * 32 + 2 * j + 1]));
        tmem_st16(trow + half * 16, pk);
      }
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(p_bar);
    }
    if (ok) ok = mbar_wait_q(s_bar, nblk & 1, abortp);     // the last P V
    ok = __all_sync(0xffffffffu, ok);
    tc_fence_after();
    if (ok && cls_warp) {
      // the classification row's probabilities: from each block's reference maximum to the final one, over the row sum
      const float fm = __shfl_sync(0xffffffffu, mx, 0), inv0 = 1.0f / __shfl_sync(0xffffffffu, sum, 0);
      for (int key = 1 + lane; key < T; key += 32) cp[key - 1] *= ex2_fast((cls_m[key / KB] - fm) * c) * inv0;
    }
    if (ok) {
      // the output rows go out through Q's space (read by now) so that a store instruction writes whole 128-byte rows
      const float inv = 1.0f / sum;
      unsigned char* st = base_ptr + warp * 32 * 128;
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        uint32_t r[32];
        tmem_ld32(trow + C_O + half * 32, r);
        tmem_ld_wait();
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          float v[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) v[j] = __uint_as_float(r[g * 8 + j]) * inv;
          store16(reinterpret_cast<bf16*>(st + lane * 128 + (((half * 4 + g) ^ (lane & 7)) << 4)), v);
        }
      }
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int rr = i * 4 + (lane >> 3), u = lane & 7, q = q0 + warp * 32 + rr;
        const uint4 x = *reinterpret_cast<const uint4*>(st + rr * 128 + ((u ^ (rr & 7)) << 4));
        if (q < T) *reinterpret_cast<uint4*>(out + ((size_t)row0 + q) * H * AT_D + (size_t)h * AT_D + u * 8) = x;
      }
      const int q = q0 + tid;
      if (q < T && lse != nullptr) lse[(size_t)bh * T + q] = mx * 0.125f + logf(sum);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 4) {
    tc_fence_after();
    tmem_dealloc(tmem, 2 * KB);
  }
  if (tid == 0 && abort_flag && status != nullptr) atomicOr(status, STATUS_TIMEOUT);
}

// Gradient rows leave through shared memory: a thread holds half of a row (lane = row of the accumulator), and stored from
// there each instruction touches 32 rows 16 bytes at a time; gathered first, 8 lanes write a row's 128 bytes.
// 16-byte units are permuted by the row, so that neither direction has bank conflicts.  Backward at batch 128, 12 heads: 100
// tokens 63.5 -> 51.4 us, 197 tokens 251 -> 228, 140 tokens 201 -> 184; batch 32, 577 tokens 444 -> 426.
__device__ __forceinline__ void stage_half_row(unsigned char* tile, uint32_t taddr, int row, int half) {
  uint32_t r[32];
  tmem_ld32(taddr + half * 32, r);
  tmem_ld_wait();
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    float v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = __uint_as_float(r[g * 8 + j]);
    store16(reinterpret_cast<bf16*>(tile + row * 128 + (((half * 4 + g) ^ (row & 7)) << 4)), v);
  }
}
// Rows 0 .. rows - 1 of a staged tile -> rows `pitch` elements apart (256 threads).
__device__ __forceinline__ void write_rows(const unsigned char* tile, bf16* dst, size_t pitch, int rows) {
  for (int i = threadIdx.x; i < rows * 8; i += 256) {
    const int r = i >> 3, u = i & 7;
    *reinterpret_cast<uint4*>(dst + r * pitch + u * 8) = *reinterpret_cast<const uint4*>(tile + r * 128 + ((u ^ (r & 7)) << 4));
  }
}

// ------------------------------------------------------------------------------------------------
// Backward (T <= 128): one CTA of 128 threads per (image, head).  With P = exp(S - lse):
//   dP = dO V^T;  delta_i = sum_j P_ij dP_ij;  dS = P * (dP - delta) / sqrt(d)
//   dQ = dS K;  dK = dS^T Q;  dV = P^T dO                      (chain rule through Eq. 1, cf. Eq. 3)
// S and dP are two MMA groups into tensor memory; each thread owns one query row and writes P and dS as
// bf16 operand tiles into shared memory; the three products then read those tiles K-major (dQ) or through
// transposing descriptors (dK, dV), so nothing is transposed by hand.  P stays in registers between the sum for delta and dS (formed again
// from S it took 51.6 instead of 50.0 us at 100 tokens, batch 128, 12 heads, 7.8 instead of 6.9 with 4 images).  A gradient arriving at the head-mean
// score of token j (cls_extra[b, j-1], from the fused token) is added to dP of the classification row.
// ------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256, 2)
attn_bwd_tc_kernel(const __grid_constant__ CUtensorMap map_qkv, const __grid_constant__ CUtensorMap map_do,
                   const float* __restrict__ lse, const float* __restrict__ cls_extra, bf16* __restrict__ dqkv,
                   int B, int T, int H, int* status) {
  extern __shared__ unsigned char smem_dyn[];
  uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
  unsigned char* base_ptr = smem_dyn + (base - smem_u32(smem_dyn));
  constexpr uint32_t TILE = 2 * AT_BOX_BYTES;            // 128 rows x 128 bytes
  int tpad = (T + 15) & ~15;
  // P and dS hold tpad query rows per 64-key chunk; dS starts in V's space (V is dead once dP = dO V^T is done).
  uint32_t CH = (uint32_t)tpad * 128u;
  uint32_t sQ = base, sK = sQ + TILE, sG = sK + TILE, sV = sG + TILE, sS = sV;
  uint32_t sP = sV + (2 * CH > TILE ? 2 * CH : TILE);
  uint32_t red_off = sP + 2 * CH + (3 * CH < 16384u ? 16384u - 3 * CH : 0u);   // slack: MMA row extent past tpad stays in bounds
  float* red = reinterpret_cast<float*>(base_ptr + (red_off - base));        // [2][128]: the halves' shares of delta
  float* exs = red + 2 * AT_QROWS;                                             // [128]: classification-row score gradients / H
  uint32_t bars = red_off + 3 * AT_QROWS * 4;
  unsigned char* pP = base_ptr + (sP - base);
  unsigned char* pS = base_ptr + (sS - base);
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  // 256 threads: warps w and w + 4 share the TMEM lane quarter w & 3 (query rows 32 * (w & 3) ..) and split the
  // keys (chunks 0-1 and 2-3 of 32) and later the output columns between them.
  int tid = threadIdx.x, warp = tid >> 5;
  int row = tid & 127, half = tid >> 7;
  int bh = blockIdx.x, b = bh / H, h = bh % H;
  uint32_t tma_bar = bars, mma_bar = bars + 8, mma2_bar = bars + 16;
  if (tid == 0) {
    abort_flag = 0;
    mbar_init(tma_bar, 1);
    mbar_init(mma_bar, 1);
    mbar_init(mma2_bar, 3);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    prefetch_map(&map_qkv);
    prefetch_map(&map_do);
  }
  if (warp == 0) {
    tmem_alloc(smem_u32(&tmem_slot), 256);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  uint32_t tmem = tmem_slot;
  if (leaves_sms_idle()) release_dependents();
  await_inputs();
  // dQ, dK, dV reuse the columns of S and dP, which are dead once P and dS sit in shared memory
  constexpr uint32_t C_S = 0, C_DP = 128, C_DQ = 0, C_DK = 64, C_DV = 128;
  volatile int* abortp = &abort_flag;
  bool ok = true;
  if (tid == 0) {
    mbar_expect_tx(tma_bar, 4 * TILE);
    int row0 = b * T;
    for (int j = 0; j < 2; ++j) {
      tma_load_2d(sQ + j * AT_BOX_BYTES, &map_qkv, tma_bar, h * AT_D, row0 + j * AT_BOX);
      tma_load_2d(sK + j * AT_BOX_BYTES, &map_qkv, tma_bar, (H + h) * AT_D, row0 + j * AT_BOX);
      tma_load_2d(sV + j * AT_BOX_BYTES, &map_qkv, tma_bar, (2 * H + h) * AT_D, row0 + j * AT_BOX);
      tma_load_2d(sG + j * AT_BOX_BYTES, &map_do, tma_bar, h * AT_D, row0 + j * AT_BOX);
    }
  }
  // inputs that do not come through TMA are fetched while the tiles are on their way
  const bool valid_row = row < T;
  const float l2 = valid_row ? lse[((size_t)b * H + h) * T + row] * 1.4426950408889634f : 0.f;
  const bool has_extra = cls_extra != nullptr;
  if (half == 0) exs[row] = (has_extra && row >= 1 && row < T) ? cls_extra[(size_t)b * (T - 1) + row - 1] * (1.0f / (float)H) : 0.f;
  __syncthreads();
  if (tid == 0) {
    ok = mbar_wait(tma_bar, 0, abortp);
    if (ok) {
      tc_fence_after();
      uint32_t idesc = make_idesc_mn(AT_QROWS, tpad, false, false);
#pragma unroll
      for (int k = 0; k < AT_D / 16; ++k)
        umma_bf16(tmem + C_S, make_desc(sQ + k * 32, 16, 1024), make_desc(sK + k * 32, 16, 1024), idesc, k > 0 ? 1u : 0u);
#pragma unroll
      for (int k = 0; k < AT_D / 16; ++k)
        umma_bf16(tmem + C_DP, make_desc(sG + k * 32, 16, 1024), make_desc(sV + k * 32, 16, 1024), idesc, k > 0 ? 1u : 0u);
      umma_commit(mma_bar);
    }
  }
  ok = mbar_wait(mma_bar, 0, abortp);
  ok = __all_sync(0xffffffffu, ok);
  tc_fence_after();

  const float c = 0.125f * 1.4426950408889634f;
  uint32_t trow = tmem + ((uint32_t)((warp & 3) * 32) << 16);
  const bool extra_row = (row == 0 && has_extra);
  float delta = 0.f;
  // tcgen05.ld is warp-collective: every lane issues it, rows past T only skip the arithmetic.  Keys are taken 16 at
  // a time (two loads of 16 columns); the probabilities of this thread's 64 keys stay in registers for dS.
  float p[4][16];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int kk = 4 * half + q;
#pragma unroll
    for (int j = 0; j < 16; ++j) p[q][j] = 0.f;
    if (!ok || kk * 16 >= T) continue;
    uint32_t rs[16], rp[16];
    tmem_ld16(trow + C_S + kk * 16, rs);
    tmem_ld16(trow + C_DP + kk * 16, rp);
    tmem_ld_wait();
    if (valid_row) {
      float d0 = 0.f, d1 = 0.f;
#pragma unroll
      for (int j = 0; j < 16; j += 2) {
        int key = kk * 16 + j;
        float p0 = key < T ? ex2_fast(fmaf(__uint_as_float(rs[j]), c, -l2)) : 0.f;
        float p1 = key + 1 < T ? ex2_fast(fmaf(__uint_as_float(rs[j + 1]), c, -l2)) : 0.f;
        float e0 = __uint_as_float(rp[j]), e1 = __uint_as_float(rp[j + 1]);
        if (extra_row) { e0 += exs[key]; e1 += exs[key + 1]; }
        d0 = fmaf(p0, e0, d0);
        d1 = fmaf(p1, e1, d1);
        p[q][j] = p0;
        p[q][j + 1] = p1;
      }
      delta += d0 + d1;
    }
  }
  red[half * AT_QROWS + row] = delta;          // every thread reaches this barrier, whatever the waits returned
  __syncthreads();
  delta = red[row] + red[AT_QROWS + row];
  if (ok) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int kk = 4 * half + q;
      float ds[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) ds[j] = 0.f;
      if (kk * 16 < T) {
        uint32_t rp[16];
        tmem_ld16(trow + C_DP + kk * 16, rp);
        tmem_ld_wait();
        if (valid_row) {
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            float dp = __uint_as_float(rp[j]);
            if (extra_row) dp += exs[kk * 16 + j];
            ds[j] = p[q][j] * (dp - delta) * 0.125f;
          }
        }
      }
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        uint4 vp, vs;
        __nv_bfloat162* hp = reinterpret_cast<__nv_bfloat162*>(&vp);
        __nv_bfloat162* hs = reinterpret_cast<__nv_bfloat162*>(&vs);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          hp[i] = __floats2bfloat162_rn(p[q][g * 8 + 2 * i], p[q][g * 8 + 2 * i + 1]);
          hs[i] = __floats2bfloat162_rn(ds[g * 8 + 2 * i], ds[g * 8 + 2 * i + 1]);
        }
        if (row < tpad) {
          int key8 = kk * 2 + g;
          uint32_t off = (uint32_t)(key8 >> 3) * CH + (uint32_t)row * 128u + (uint32_t)(((key8 & 7) ^ (row & 7)) << 4);
          *reinterpret_cast<uint4*>(pP + off) = vp;
          *reinterpret_cast<uint4*>(pS + off) = vs;
        }
      }
    }
  }
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  ok = ok && !abort_flag;
  // dQ, dK and dV are issued by three different threads (lane 0 of warps 0, 1, 2), each committing to the same barrier
  if (ok && (tid & 31) == 0 && warp < 3) {
    if (warp == 0) {
      // dQ = dS K: A = dS (contiguous along keys), B = K read with keys as the reduction index
      uint32_t id_q = make_idesc_mn(AT_QROWS, AT_D, false, true);
      for (int k = 0; k < tpad / 16; ++k)
        umma_bf16(tmem + C_DQ, make_desc(sS + (k >> 2) * CH + (k & 3) * 32, 16, 1024), make_desc(sK + k * 2048, 8192, 1024), id_q,
                  k > 0 ? 1u : 0u);
    } else {
      // dK = dS^T Q and dV = P^T dO: both operands read with queries as the reduction index
      uint32_t id_t = make_idesc_mn(AT_QROWS, AT_D, true, true);
      uint32_t sa = warp == 1 ? sS : sP, sb = warp == 1 ? sQ : sG, cd = warp == 1 ? C_DK : C_DV;
      for (int k = 0; k < tpad / 16; ++k)
        umma_bf16(tmem + cd, make_desc(sa + k * 2048, CH, 1024), make_desc(sb + k * 2048, 8192, 1024), id_t, k > 0 ? 1u : 0u);
    }
    umma_commit(mma2_bar);
  }
  if (ok) ok = mbar_wait(mma2_bar, 0, abortp);
  ok = __all_sync(0xffffffffu, ok);
  tc_fence_after();
  // every operand tile has been read: the first three hold the gradients' rows now
  if (ok && (warp & 3) * 32 < T) {
    stage_half_row(base_ptr, trow + C_DQ, row, half);
    stage_half_row(base_ptr + TILE, trow + C_DK, row, half);
    stage_half_row(base_ptr + 2 * TILE, trow + C_DV, row, half);
  }
  __syncthreads();
  if (ok)
    for (int which = 0; which < 3; ++which)
      write_rows(base_ptr + which * TILE, dqkv + ((size_t)b * T * 3 + which) * H * AT_D + (size_t)h * AT_D, (size_t)3 * H * AT_D, T);
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, 256);
  }
  if (tid == 0 && abort_flag && status != nullptr) atomicOr(status, STATUS_TIMEOUT);
}

// ------------------------------------------------------------------------------------------------
// Backward for 128 < T <= 256: one CTA of 256 threads per (image, head), queries and keys in two tiles of 128.
// The formulas are those of the kernel above; what changes is that delta_i = sum_j P_ij dP_ij runs over both key
// tiles, so a first sweep (one step per query tile, both key tiles at once) forms S and dP only to accumulate delta, and a
// second sweep (key tile outer, query tile inner) forms them again, writes P and dS as bf16 operand tiles and issues
// the three products: dQ_i accumulates over the key tiles, dK_j and dV_j over the query tiles, all in tensor memory
// (S 128 + dP 128 + dQ 2 x 64 + dK 64 + dV 64 = 512 columns: one CTA per SM).  No step leaves the loop early: after a
// wait that expired the remaining steps only keep the barriers in step.
// ------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256, 1)
attn_bwd_tc256_kernel(const __grid_constant__ CUtensorMap map_qkv, const __grid_constant__ CUtensorMap map_do,
                      const float* __restrict__ lse, const float* __restrict__ cls_extra, bf16* __restrict__ dqkv,
                      int B, int T, int H, int* status) {
  extern __shared__ unsigned char smem_dyn[];
  uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
  unsigned char* base_ptr = smem_dyn + (base - smem_u32(smem_dyn));
  constexpr uint32_t TILE = 2 * AT_BOX_BYTES;            // 128 rows x 128 bytes
  constexpr uint32_t CH = TILE;                          // one 64-key chunk of a P / dS tile: 128 query rows x 128 bytes
  uint32_t sQ = base, sK = sQ + 2 * TILE, sG = sK + 2 * TILE, sV = sG + 2 * TILE, sP = sV + 2 * TILE, sS = sP + 2 * TILE;
  uint32_t arrays = sS + 2 * TILE;
  float* sdelta = reinterpret_cast<float*>(base_ptr + (arrays - base));     // [256] delta of every query row
  float* sl2 = sdelta + 256;                                                 // [256] log-sum-exp in binary orders
  float* exs = sl2 + 256;                                                    // [256] classification-row score gradients / H
  float* red = exs + 256;                                                    // [2][128] the halves' shares of delta
  uint32_t bars = arrays + 4 * 256 * 4;
  unsigned char* pP = base_ptr + (sP - base);
  unsigned char* pS = base_ptr + (sS - base);
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  int tid = threadIdx.x, warp = tid >> 5;
  int rowl = tid & 127, half = tid >> 7;
  int bh = blockIdx.x, b = bh / H, h = bh % H;
  uint32_t tma_bar = bars, mma_bar = bars + 8, mma2_bar = bars + 16;
  if (tid == 0) {
    abort_flag = 0;
    mbar_init(tma_bar, 1);
    mbar_init(mma_bar, 1);
    mbar_init(mma2_bar, 3);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    prefetch_map(&map_qkv);
    prefetch_map(&map_do);
  }
  if (warp == 0) {
    tmem_alloc(smem_u32(&tmem_slot), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  uint32_t tmem = tmem_slot;
  if (leaves_sms_idle()) release_dependents();
  await_inputs();
  constexpr uint32_t C_S = 0, C_DP = 128, C_DQ = 256, C_DK = 384, C_DV = 448;
  volatile int* abortp = &abort_flag;
  const int tpad = (T + 15) & ~15;
  const int row0 = b * T;
  if (tid == 0) {
    mbar_expect_tx(tma_bar, 8 * TILE);
    for (int j = 0; j < 4; ++j) {                        // rows past the image: the next image's, or zero fill; never used
      tma_load_2d(sQ + j * AT_BOX_BYTES, &map_qkv, tma_bar, h * AT_D, row0 + j * AT_BOX);
      tma_load_2d(sK + j * AT_BOX_BYTES, &map_qkv, tma_bar, (H + h) * AT_D, row0 + j * AT_BOX);
      tma_load_2d(sV + j * AT_BOX_BYTES, &map_qkv, tma_bar, (2 * H + h) * AT_D, row0 + j * AT_BOX);
      tma_load_2d(sG + j * AT_BOX_BYTES, &map_do, tma_bar, h * AT_D, row0 + j * AT_BOX);
    }
  }
  const bool has_extra = cls_extra != nullptr;
  sl2[tid] = tid < T ? lse[((size_t)b * H + h) * T + tid] * 1.4426950408889634f : 0.f;
  exs[tid] = (has_extra && tid >= 1 && tid < T) ? cls_extra[(size_t)b * (T - 1) + tid - 1] * (1.0f / (float)H) : 0.f;
  __syncthreads();
  bool ok = true;
  if (tid == 0) ok = mbar_wait(tma_bar, 0, abortp);
  const float c = 0.125f * 1.4426950408889634f;
  const uint32_t trow = tmem + ((uint32_t)((warp & 3) * 32) << 16);
  uint32_t ph1 = 0, ph2 = 0;

  // S = Q_i K_j^T and dP = dO_i V_j^T into tensor memory; everyone waits for them
  auto scores = [&](int i, int j) {
    tc_fence_before();
    __syncthreads();                       // the previous step's reads of S / dP (and of the operand tiles) are over
    tc_fence_after();
    if (tid == 0 && ok && !abort_flag) {
      int kpad = min(128, tpad - 128 * j);
      uint32_t idesc = make_idesc_mn(AT_QROWS, kpad, false, false);
      uint32_t q = sQ + i * TILE, k_ = sK + j * TILE, g = sG + i * TILE, v = sV + j * TILE;
#pragma unroll
      for (int k = 0; k < AT_D / 16; ++k)
        umma_bf16(tmem + C_S, make_desc(q + k * 32, 16, 1024), make_desc(k_ + k * 32, 16, 1024), idesc, k > 0 ? 1u : 0u);
#pragma unroll
      for (int k = 0; k < AT_D / 16; ++k)
        umma_bf16(tmem + C_DP, make_desc(g + k * 32, 16, 1024), make_desc(v + k * 32, 16, 1024), idesc, k > 0 ? 1u : 0u);
      umma_commit(mma_bar);
    }
    bool w = mbar_wait(mma_bar, ph1, abortp);
    ph1 ^= 1u;
    ok = __all_sync(0xffffffffu, ok && w);
    tc_fence_after();
  };

  // S and dP of query tile i against BOTH key tiles at once: the second pair lands in the columns that hold dQ, dK, dV
  // later (free during the first sweep), so the sweep takes one product group and one wait per query tile
  auto scores_both = [&](int i) {
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid == 0 && ok && !abort_flag) {
      uint32_t q = sQ + i * TILE, g = sG + i * TILE;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        int kpad = min(128, tpad - 128 * j);
        uint32_t idesc = make_idesc_mn(AT_QROWS, kpad, false, false);
        uint32_t k_ = sK + j * TILE, v = sV + j * TILE;
#pragma unroll
        for (int k = 0; k < AT_D / 16; ++k)
          umma_bf16(tmem + 256 * j + C_S, make_desc(q + k * 32, 16, 1024), make_desc(k_ + k * 32, 16, 1024), idesc, k > 0 ? 1u : 0u);
#pragma unroll
        for (int k = 0; k < AT_D / 16; ++k)
          umma_bf16(tmem + 256 * j + C_DP, make_desc(g + k * 32, 16, 1024), make_desc(v + k * 32, 16, 1024), idesc, k > 0 ? 1u : 0u);
      }
      umma_commit(mma_bar);
    }
    bool w = mbar_wait(mma_bar, ph1, abortp);
    ph1 ^= 1u;
    ok = __all_sync(0xffffffffu, ok && w);
    tc_fence_after();
  };

  // ---- first sweep: delta of every query row ----
  for (int i = 0; i < 2; ++i) {
    const int row = i * 128 + rowl;
    const bool valid_row = row < T;
    const bool extra_row = (row == 0 && has_extra);
    const float l2 = sl2[row];
    float dacc = 0.f;
    scores_both(i);
    for (int j = 0; j < 2; ++j) {
      const int kbase = j * 128;
      const int kvalid = min(128, T - kbase);
      if (ok && i * 128 + (warp & 3) * 32 < T) {
        for (int kk = 4 * half; kk < 4 * half + 4 && kk * 16 < kvalid; ++kk) {
          uint32_t rs[16], rp[16];
          tmem_ld16(trow + 256 * j + C_S + kk * 16, rs);
          tmem_ld16(trow + 256 * j + C_DP + kk * 16, rp);
          tmem_ld_wait();
          if (valid_row) {
            float d0 = 0.f, d1 = 0.f;
#pragma unroll
            for (int jj = 0; jj < 16; jj += 2) {
              int key = kbase + kk * 16 + jj;
              float p0 = key < T ? ex2_fast(fmaf(__uint_as_float(rs[jj]), c, -l2)) : 0.f;
              float p1 = key + 1 < T ? ex2_fast(fmaf(__uint_as_float(rs[jj + 1]), c, -l2)) : 0.f;
              float e0 = __uint_as_float(rp[jj]), e1 = __uint_as_float(rp[jj + 1]);
              if (extra_row) { e0 += exs[key]; e1 += exs[key + 1]; }
              d0 = fmaf(p0, e0, d0);
              d1 = fmaf(p1, e1, d1);
            }
            dacc += d0 + d1;
          }
        }
      }
    }
    red[half * AT_QROWS + rowl] = dacc;
    __syncthreads();
    if (half == 0) sdelta[row] = red[rowl] + red[AT_QROWS + rowl];
  }

  // ---- second sweep: P and dS tiles, the three products ----
  // two accumulators of 128 rows -> rows row0 .. of dQ, dK or dV, through the P and dS tiles
  auto store_two = [&](uint32_t col_a, int which_a, int row_a, uint32_t col_b, int which_b, int row_b) {
    __syncthreads();                       // what was staged before has been written
    if (ok) {
      stage_half_row(pP, trow + col_a, rowl, half);
      stage_half_row(pS, trow + col_b, rowl, half);
    }
    __syncthreads();
    if (!ok) return;
    bf16* out = dqkv + (size_t)b * T * 3 * H * AT_D + (size_t)h * AT_D;
    const size_t pitch = (size_t)3 * H * AT_D;
    write_rows(pP, out + row_a * pitch + (size_t)which_a * H * AT_D, pitch, min(128, T - row_a));
    write_rows(pS, out + row_b * pitch + (size_t)which_b * H * AT_D, pitch, min(128, T - row_b));
  };
  for (int j = 0; j < 2; ++j) {
    const int kbase = j * 128;
    const int kvalid = min(128, T - kbase);
    const int kpad = min(128, tpad - kbase);
    for (int i = 0; i < 2; ++i) {
      scores(i, j);                          // its leading barrier also orders the delta written above before its use
      const int row = i * 128 + rowl;
      const bool valid_row = row < T;
      const bool extra_row = (row == 0 && has_extra);
      const float l2 = sl2[row];
      const float delta = sdelta[row];
      const int qpad = min(128, tpad - 128 * i);
      // rows past qpad and keys past kpad enter none of the products
      if (ok && (warp & 3) * 32 < qpad) {
        for (int kk = 4 * half; kk < 4 * half + 4 && kk * 16 < kpad; ++kk) {
          float p[16], ds[16];
#pragma unroll
          for (int jj = 0; jj < 16; ++jj) { p[jj] = 0.f; ds[jj] = 0.f; }
          if (kk * 16 < kvalid) {
            uint32_t rs[16], rp[16];
            tmem_ld16(trow + C_S + kk * 16, rs);
            tmem_ld16(trow + C_DP + kk * 16, rp);
            tmem_ld_wait();
            if (valid_row) {
#pragma unroll
              for (int jj = 0; jj < 16; ++jj) {
                int key = kbase + kk * 16 + jj;
                float pv = key < T ? ex2_fast(fmaf(__uint_as_float(rs[jj]), c, -l2)) : 0.f;
                float dp = __uint_as_float(rp[jj]);
                if (extra_row) dp += exs[key];
                p[jj] = pv;
                ds[jj] = pv * (dp - delta) * 0.125f;
              }
            }
          }
#pragma unroll
          for (int g = 0; g < 2; ++g) {
            uint4 vp, vs;
            __nv_bfloat162* hp = reinterpret_cast<__nv_bfloat162*>(&vp);
            __nv_bfloat162* hs = reinterpret_cast<__nv_bfloat162*>(&vs);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              hp[e] = __floats2bfloat162_rn(p[g * 8 + 2 * e], p[g * 8 + 2 * e + 1]);
              hs[e] = __floats2bfloat162_rn(ds[g * 8 + 2 * e], ds[g * 8 + 2 * e + 1]);
            }
            int key8 = kk * 2 + g;
            uint32_t off = (uint32_t)(key8 >> 3) * CH + (uint32_t)rowl * 128u + (uint32_t)(((key8 & 7) ^ (rowl & 7)) << 4);
            *reinterpret_cast<uint4*>(pP + off) = vp;
            *reinterpret_cast<uint4*>(pS + off) = vs;
          }
        }
      }
      fence_async_smem();
      tc_fence_before();
      __syncthreads();
      tc_fence_after();
      // dQ_i, dK_j and dV_j are issued by lane 0 of warps 0, 1, 2, each committing to the same barrier
      if ((tid & 31) == 0 && warp < 3) {
        if (ok && !abort_flag) {
          if (warp == 0) {
            uint32_t id_q = make_idesc_mn(AT_QROWS, AT_D, false, true);
            for (int k = 0; k < kpad / 16; ++k)
              umma_bf16(tmem + C_DQ + 64 * i, make_desc(sS + (k >> 2) * CH + (k & 3) * 32, 16, 1024),
                        make_desc(sK + j * TILE + k * 2048, 8192, 1024), id_q, (j > 0 || k > 0) ? 1u : 0u);
          } else {
            uint32_t id_t = make_idesc_mn(AT_QROWS, AT_D, true, true);
            uint32_t sa = warp == 1 ? sS : sP, sb = (warp == 1 ? sQ : sG) + i * TILE, cd = warp == 1 ? C_DK : C_DV;
            for (int k = 0; k < qpad / 16; ++k)
              umma_bf16(tmem + cd, make_desc(sa + k * 2048, CH, 1024), make_desc(sb + k * 2048, 8192, 1024), id_t,
                        (i > 0 || k > 0) ? 1u : 0u);
          }
          umma_commit(mma2_bar);
        }
      }
      bool w = ok && mbar_wait(mma2_bar, ph2, abortp);   // the products are done: P, dS, S and dP may be overwritten
      ph2 ^= 1u;
      ok = __all_sync(0xffffffffu, w);
      tc_fence_after();
    }
    store_two(C_DK, 1, kbase, C_DV, 2, kbase);
  }
  store_two(C_DQ, 0, 0, C_DQ + 64, 0, 128);
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
  if (tid == 0 && abort_flag && status != nullptr) atomicOr(status, STATUS_TIMEOUT);
}

// ------------------------------------------------------------------------------------------------
// The same range where two CTAs per (image, head) fit the SMs at once: a cluster of two CTAs of 256 threads, each with one tile of 128 keys
// and both tiles of queries.  delta_i = sum_j P_ij dP_ij and dQ_i = sum_j dS_ij K_j run
// over both CTAs' keys, which exchange their parts through distributed shared memory.  All scores of a CTA fit tensor memory at
// once (S and dP of two query tiles: 512 columns), so they are formed once: P stays in registers (128 values a thread) between the sum
// for delta and dS, dP in tensor memory, and the accumulators take the columns of S.
//   S, dP -> P (bf16 tiles in shared memory, dV = P^T dO under way) -> delta exchanged -> dS over the tiles of P -> dQ, dK -> the part of the
//   other CTA's query tile sent to it -> dQ, dK, dV of 128 rows each out.
// No step leaves early: after a wait that expired the remaining steps only keep the barriers in step.
// us of a launch in a row of launches, attn_bwd_tc256_kernel / this, 12 heads, 197 tokens: 1 image 19.5 / 11.4, 4 images 19.6 / 12.8, and beyond one
// wave 8 images 20.5 / 25.1, 128 images 229 / 270 (140 tokens: 15.8 / 10.5, 15.9 / 12.4, 16.9 / 24.4, 185 / 248).
// ------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256, 1)
attn_bwd_pair_kernel(const __grid_constant__ CUtensorMap map_qkv, const __grid_constant__ CUtensorMap map_do,
                     const float* __restrict__ lse, const float* __restrict__ cls_extra, bf16* __restrict__ dqkv,
                     int T, int H, int* status) {
  extern __shared__ unsigned char smem_dyn[];
  __shared__ __align__(8) unsigned long long bar_mem[4];
  __shared__ float red[2][256];                          // the halves' shares of delta of every query row, over this CTA's keys
  __shared__ float part[2][256];                         // ... summed, by key tile
  __shared__ float exs[AT_QROWS];                        // classification-row score gradients of this CTA's keys / H
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
  unsigned char* base_ptr = smem_dyn + (base - smem_u32(smem_dyn));
  constexpr uint32_t TILE = 2 * AT_BOX_BYTES;            // 128 rows x 128 bytes
  constexpr uint32_t CH = TILE;                          // one 64-key chunk of a P / dS tile: 128 query rows x 128 bytes
  const uint32_t sQ = base, sG = sQ + 2 * TILE, sK = sG + 2 * TILE, sV = sK + TILE, sP = sV + TILE, recv = sP + 4 * TILE;
  unsigned char* pP = base_ptr + (sP - base);
  const int tid = threadIdx.x, warp = tid >> 5, rowl = tid & 127, half = tid >> 7, quarter = warp & 3;
  const int bh = blockIdx.x >> 1, j = blockIdx.x & 1, b = bh / H, h = bh - b * H;
  const uint32_t bars = smem_u32(bar_mem), tma_bar = bars, s_bar = bars + 8, v_bar = bars + 16, m_bar = bars + 24;
  if (tid == 0) {
    abort_flag = 0;
    mbar_init(tma_bar, 1); mbar_init(s_bar, 1); mbar_init(v_bar, 1); mbar_init(m_bar, 2);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    prefetch_map(&map_qkv);
    prefetch_map(&map_do);
  }
  if (warp == 0) {
    tmem_alloc(smem_u32(&tmem_slot), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  cluster_arrive();                        // this CTA has started: the other may write to its shared memory
  const uint32_t tmem = tmem_slot;
  if (leaves_sms_idle()) release_dependents();
  await_inputs();
  constexpr uint32_t C_S = 0, C_DP = 256, C_DV = 0, C_DQ = 64, C_DK = 192;       // S, dP, dQ: one tile of queries after the other
  volatile int* abortp = &abort_flag;
  const int tpad = (T + 15) & ~15, row0 = b * T, kbase = 128 * j;
  const int kvalid = min(128, T - kbase), kpad = min(128, tpad - kbase);
  bool ok = true;
  if (tid == 0) {
    mbar_expect_tx(tma_bar, 6 * TILE);
    for (int q = 0; q < 2; ++q) {                        // rows past the image: the next image's, or zero fill; never used
      tma_load_2d(sK + q * AT_BOX_BYTES, &map_qkv, tma_bar, (H + h) * AT_D, row0 + kbase + q * AT_BOX);
      tma_load_2d(sV + q * AT_BOX_BYTES, &map_qkv, tma_bar, (2 * H + h) * AT_D, row0 + kbase + q * AT_BOX);
    }
    for (int q = 0; q < 4; ++q) {
      tma_load_2d(sQ + q * AT_BOX_BYTES, &map_qkv, tma_bar, h * AT_D, row0 + q * AT_BOX);
      tma_load_2d(sG + q * AT_BOX_BYTES, &map_do, tma_bar, h * AT_D, row0 + q * AT_BOX);
    }
  }
  const bool has_extra = cls_extra != nullptr;
  float l2[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) l2[i] = i * 128 + rowl < T ? lse[(size_t)bh * T + i * 128 + rowl] * 1.4426950408889634f : 0.f;
  if (tid < 128) exs[tid] = has_extra && kbase + tid >= 1 && tid < kvalid ? cls_extra[(size_t)b * (T - 1) + kbase + tid - 1] * (1.0f / (float)H) : 0.f;
  __syncthreads();
  if (tid == 0) {
    ok = mbar_wait(tma_bar, 0, abortp);
    if (ok) {
      tc_fence_after();
      const uint32_t idesc = make_idesc_mn(AT_QROWS, kpad, false, false);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
#pragma unroll
        for (int k = 0; k < AT_D / 16; ++k)
          umma_bf16(tmem + C_S + 128 * i, make_desc(sQ + i * TILE + k * 32, 16, 1024), make_desc(sK + k * 32, 16, 1024), idesc, k > 0 ? 1u : 0u);
#pragma unroll
        for (int k = 0; k < AT_D / 16; ++k)
          umma_bf16(tmem + C_DP + 128 * i, make_desc(sG + i * TILE + k * 32, 16, 1024), make_desc(sV + k * 32, 16, 1024), idesc, k > 0 ? 1u : 0u);
      }
      umma_commit(s_bar);
    }
  }
  __syncwarp();
  ok = mbar_wait_q(s_bar, 0, abortp) && ok;
  ok = __all_sync(0xffffffffu, ok);
  tc_fence_after();
  const float c = 0.125f * 1.4426950408889634f;
  const uint32_t trow = tmem + ((uint32_t)(quarter * 32) << 16);
  const int qpad1 = tpad - 128;                          // rows of the second query tile that enter products (the first: all)

  // 16-byte units of a P / dS tile: values of keys 8 g .. 8 g + 7 of this thread's row
  auto put = [&](int i, int kk, const float* v) {
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      uint4 x;
      __nv_bfloat162* hx = reinterpret_cast<__nv_bfloat162*>(&x);
#pragma unroll
      for (int e = 0; e < 4; ++e) hx[e] = __floats2bfloat162_rn(v[g * 8 + 2 * e], v[g * 8 + 2 * e + 1]);
      const int key8 = kk * 2 + g;
      *reinterpret_cast<uint4*>(pP + i * 2 * TILE + (uint32_t)(key8 >> 3) * CH + (uint32_t)rowl * 128u + (uint32_t)(((key8 & 7) ^ (rowl & 7)) << 4)) = x;
    }
  };
  // this thread's 64 keys in four groups of 16, of both query tiles; groups past kpad and rows past the tile's padding enter no product
  float p[2][4][16];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int row = i * 128 + rowl;
    const bool extra_row = row == 0 && has_extra;
    const bool enters = i == 0 || quarter * 32 < qpad1;
    float dacc = 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int kk = 4 * half + q;
#pragma unroll
      for (int e = 0; e < 16; ++e) p[i][q][e] = 0.f;
      if (!ok || !enters || kk * 16 >= kpad) continue;
      uint32_t rs[16], rp[16];
      tmem_ld16(trow + C_S + 128 * i + kk * 16, rs);
      tmem_ld16(trow + C_DP + 128 * i + kk * 16, rp);
      tmem_ld_wait();
      if (row < T) {
        float d0 = 0.f, d1 = 0.f;
#pragma unroll
        for (int e = 0; e < 16; e += 2) {
          const int key = kk * 16 + e;
          const float p0 = key < kvalid ? ex2_fast(fmaf(__uint_as_float(rs[e]), c, -l2[i])) : 0.f;
          const float p1 = key + 1 < kvalid ? ex2_fast(fmaf(__uint_as_float(rs[e + 1]), c, -l2[i])) : 0.f;
          float e0 = __uint_as_float(rp[e]), e1 = __uint_as_float(rp[e + 1]);
          if (extra_row) { e0 += exs[key]; e1 += exs[key + 1]; }
          d0 = key < kvalid ? fmaf(p0, e0, d0) : d0;
          d1 = key + 1 < kvalid ? fmaf(p1, e1, d1) : d1;
          p[i][q][e] = p0;
          p[i][q][e + 1] = p1;
        }
        dacc += d0 + d1;
      }
      put(i, kk, p[i][q]);
    }
    red[half][row] = dacc;
  }
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t id_t = make_idesc_mn(AT_QROWS, AT_D, true, true);
  // dV = P^T dO (over S, which every thread has read), and dK = dS^T Q: both operands read with queries as the reduction index
  auto by_queries = [&](uint32_t col, uint32_t sb) {
    for (int i = 0; i < 2; ++i)
      for (int k = 0; k < (i == 0 ? 128 : qpad1) / 16; ++k)
        umma_bf16(tmem + col, make_desc(sP + i * 2 * TILE + k * 2048, CH, 1024), make_desc(sb + i * TILE + k * 2048, 8192, 1024), id_t, (i > 0 || k > 0) ? 1u : 0u);
  };
  if (tid == 0 && ok && !abort_flag) {
    by_queries(C_DV, sG);
    umma_commit(v_bar);
  }
  __syncwarp();
  // delta: this CTA's part of every query row to both
  cluster_wait();
  {
    const float mine = red[0][tid] + red[1][tid];
    part[j][tid] = mine;
    st_cluster(peer_addr(smem_u32(&part[j][tid]), j ^ 1), mine);
  }
  cluster_arrive();
  cluster_wait();
  ok = mbar_wait_q(v_bar, 0, abortp) && ok;              // P has been read: dS takes its place
  ok = __all_sync(0xffffffffu, ok);
  tc_fence_after();
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int row = i * 128 + rowl;
    const bool extra_row = row == 0 && has_extra;
    const bool enters = i == 0 || quarter * 32 < qpad1;
    const float delta = part[0][row] + part[1][row];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int kk = 4 * half + q;
      if (!ok || !enters || kk * 16 >= kpad) continue;
      uint32_t rp[16];
      tmem_ld16(trow + C_DP + 128 * i + kk * 16, rp);
      tmem_ld_wait();
      float ds[16];
#pragma unroll
      for (int e = 0; e < 16; ++e) {
        float dp = __uint_as_float(rp[e]);
        if (extra_row) dp += exs[kk * 16 + e];
        ds[e] = row < T && kk * 16 + e < kvalid ? p[i][q][e] * (dp - delta) * 0.125f : 0.f;
      }
      put(i, kk, ds);
    }
  }
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if ((tid & 31) == 0 && warp < 2 && ok && !abort_flag) {
    if (warp == 0) {
      // dQ_i = dS_i K: A = dS (contiguous along keys), B = K read with keys as the reduction index
      const uint32_t id_q = make_idesc_mn(AT_QROWS, AT_D, false, true);
      for (int i = 0; i < 2; ++i)
        for (int k = 0; k < kpad / 16; ++k)
          umma_bf16(tmem + C_DQ + 64 * i, make_desc(sP + i * 2 * TILE + (k >> 2) * CH + (k & 3) * 32, 16, 1024), make_desc(sK + k * 2048, 8192, 1024), id_q,
                    k > 0 ? 1u : 0u);
    } else {
      by_queries(C_DK, sQ);
    }
    umma_commit(m_bar);
  }
  __syncwarp();
  ok = mbar_wait_q(m_bar, 0, abortp) && ok;
  ok = __all_sync(0xffffffffu, ok);
  tc_fence_after();
  // the other CTA's query tile: this CTA's part of its dQ, rows of 256 bytes, 16-byte units permuted by the row
  const int other = j ^ 1;
  if (ok && other * 128 + quarter * 32 < T) {
    uint32_t r[32];
    tmem_ld32(trow + C_DQ + 64 * other + half * 32, r);
    tmem_ld_wait();
    const uint32_t dst = peer_addr(recv + (uint32_t)rowl * 256u, other);
#pragma unroll
    for (int u = 0; u < 8; ++u) send16(dst + (((half * 8 + u) ^ (rowl & 7)) << 4), r + 4 * u);
  }
  __syncwarp();
  cluster_arrive();
  const size_t pitch = (size_t)3 * H * AT_D;
  bf16* rows_out = dqkv + ((size_t)b * T + kbase) * pitch + (size_t)h * AT_D;      // rows of this CTA's tile, Q's columns
  if (ok) {
    stage_half_row(pP, trow + C_DK, rowl, half);
    stage_half_row(pP + TILE, trow + C_DV, rowl, half);
  }
  __syncthreads();
  if (ok) {
    write_rows(pP, rows_out + (size_t)H * AT_D, pitch, kvalid);
    write_rows(pP + TILE, rows_out + 2 * (size_t)H * AT_D, pitch, kvalid);
  }
  __syncwarp();
  cluster_wait();
  if (ok && quarter * 32 < kvalid) {
    uint32_t r[32];
    tmem_ld32(trow + C_DQ + 64 * j + half * 32, r);
    tmem_ld_wait();
    const unsigned char* got = base_ptr + (recv - base) + (uint32_t)rowl * 256u;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      float v[8];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const float4 x = *reinterpret_cast<const float4*>(got + (((half * 8 + g * 2 + u) ^ (rowl & 7)) << 4));
        v[u * 4 + 0] = __uint_as_float(r[g * 8 + u * 4 + 0]) + x.x; v[u * 4 + 1] = __uint_as_float(r[g * 8 + u * 4 + 1]) + x.y;
        v[u * 4 + 2] = __uint_as_float(r[g * 8 + u * 4 + 2]) + x.z; v[u * 4 + 3] = __uint_as_float(r[g * 8 + u * 4 + 3]) + x.w;
      }
      store16(reinterpret_cast<bf16*>(pP + 2 * TILE + rowl * 128 + (((half * 4 + g) ^ (rowl & 7)) << 4)), v);
    }
  }
  __syncthreads();
  if (ok) write_rows(pP + 2 * TILE, rows_out, pitch, kvalid);
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
  if (tid == 0 && abort_flag) {
    unsigned long long t0 = global_ns();   // copies already issued still land in shared memory
    while (global_ns() - t0 < 1000000ull) {}
    if (status != nullptr) atomicOr(status, STATUS_TIMEOUT);
  }
}

// ------------------------------------------------------------------------------------------------
// Backward for longer sequences, in two launches of one kernel.  A CTA owns 128 rows of the attention map and walks the
// other side in blocks of BL_COLS:
//   KV = false: rows are queries.  S = Q K_j^T and dP = dO V_j^T; a first walk only accumulates delta_i = sum_j P_ij dP_ij
//               (the output O is not kept by frozen blocks, so dO . O is not available) and leaves it in `delta`, a second
//               walk forms dS and accumulates dQ += dS K_j.
//   KV = true : rows are keys.  S^T = K Q_i^T and dP^T = V dO_i^T, with lse and delta of the block's queries from shared
//               memory; dV += P^T dO_i and dK += dS^T Q_i.
// Either way the row operand of the second products is what the threads have just computed, so it goes back into tensor
// memory (over the score columns its writer has consumed) and is read from there: nothing is transposed and nothing passes
// through shared memory.  P and dS stay 32-bit values in effect: each goes back as two bf16 numbers, the value rounded and
// what the rounding left (2^-17 of the value is lost), in the columns that held the score, and both are multiplied: the
// error of dQ, dK and dV against 64 bits is that of their rounding to bf16, 1.66e-3, as with fp32 P and dS (rounded to bf16
// once they gave 2.35e-3).  What bounds it is the chain product -> read -> exponential -> write -> product of
// one block; 256 tensor-memory columns and 66 KB of shared memory let two CTAs share an SM and overlap their chains.
// 577 tokens, 12 heads: 495 us at batch 32 and 141 at batch 7, 290 tokens at batch 32 161 us (429, 121 and 141 us with P and dS
// rounded to bf16 once).
// No step leaves a loop early: after a wait that expired the remaining steps only keep the barriers in step.
// ------------------------------------------------------------------------------------------------
constexpr int BL_COLS = 64;

template <bool KV>
__global__ void __launch_bounds__(256, 2)
attn_bwd_long_kernel(const __grid_constant__ CUtensorMap map_qkv, const __grid_constant__ CUtensorMap map_do,
                     const float* __restrict__ lse, float* __restrict__ delta, const float* __restrict__ cls_extra,
                     bf16* __restrict__ dqkv, int B, int T, int H, int* status) {
  extern __shared__ unsigned char smem_dyn[];
  const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
  constexpr uint32_t ROWS = 2 * AT_BOX_BYTES, COLS = AT_BOX_BYTES;        // 128 rows, 64 rows of 128 bytes
  const uint32_t sR1 = base, sR2 = sR1 + ROWS, sC = sR2 + ROWS;           // column tiles: [2 slots][2 operands]
  const uint32_t bars = sC + 4 * COLS;
  const uint32_t s_bar = bars + 16, p_bar = bars + 24;
  auto full_bar = [&](int b) { return bars + 8u * b; };
  __shared__ float stats[2][2][BL_COLS];                                  // KV: lse (binary orders) and delta of the block's queries
  __shared__ float red[2][AT_QROWS];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int rowl = tid & 127, half = tid >> 7;                            // two warps per lane quarter split the block's columns
  const int bh = blockIdx.y, b = bh / H, h = bh - b * H;
  const int r0 = blockIdx.x * AT_QROWS, row = r0 + rowl, row0 = b * T;
  if (tid == 0) {
    abort_flag = 0;
    mbar_init(full_bar(0), 1); mbar_init(full_bar(1), 1); mbar_init(s_bar, 1); mbar_init(p_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    prefetch_map(&map_qkv);
    prefetch_map(&map_do);
  }
  if (warp == 0) {
    tmem_alloc(smem_u32(&tmem_slot), 256);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  if (leaves_sms_idle()) release_dependents();
  await_inputs();
  constexpr uint32_t C_S = 0, C_DP = 64, C_A1 = 128, C_A2 = 192;          // A1: dQ or dK, A2: dV
  volatile int* abortp = &abort_flag;
  const uint32_t trow = tmem + ((uint32_t)((warp & 3) * 32) << 16);
  const int nt = (T + BL_COLS - 1) / BL_COLS, steps = KV ? nt : 2 * nt;
  const float c = 0.125f * 1.4426950408889634f, invH = 1.0f / (float)H;
  const bool valid_row = row < T;
  const float* lse_bh = lse + (size_t)bh * T;
  float* delta_bh = delta + (size_t)bh * T;
  const float* extra = cls_extra != nullptr ? cls_extra + (size_t)b * (T - 1) : nullptr;
  auto load_cols = [&](int s) {                                           // thread 0: operands of step s into slot s & 1
    int k0 = row0 + (s % nt) * BL_COLS;
    uint32_t dst = sC + (s & 1) * 2 * COLS, bar = full_bar(s & 1);
    if (KV) {
      tma_load_2d(dst, &map_qkv, bar, h * AT_D, k0);
      tma_load_2d(dst + COLS, &map_do, bar, h * AT_D, k0);
    } else {
      tma_load_2d(dst, &map_qkv, bar, (H + h) * AT_D, k0);
      tma_load_2d(dst + COLS, &map_qkv, bar, (2 * H + h) * AT_D, k0);
    }
  };
  auto load_stats = [&](int s) {                                          // threads 0..127: lse and delta of step s's queries
    if (KV && tid < 2 * BL_COLS && s < steps) {
      int i = tid & (BL_COLS - 1), q = s * BL_COLS + i;
      stats[s & 1][tid >> 6][i] = q < T ? (tid < BL_COLS ? lse_bh[q] * 1.4426950408889634f : delta_bh[q]) : 0.f;
    }
  };
  if (tid == 0) {
    mbar_expect_tx(full_bar(0), 2 * ROWS + 2 * COLS);
    for (int j = 0; j < 2; ++j) {
      tma_load_2d(sR1 + j * AT_BOX_BYTES, &map_qkv, full_bar(0), ((KV ? H : 0) + h) * AT_D, row0 + r0 + j * AT_BOX);
      if (KV) tma_load_2d(sR2 + j * AT_BOX_BYTES, &map_qkv, full_bar(0), (2 * H + h) * AT_D, row0 + r0 + j * AT_BOX);
      else tma_load_2d(sR2 + j * AT_BOX_BYTES, &map_do, full_bar(0), h * AT_D, row0 + r0 + j * AT_BOX);
    }
    load_cols(0);
    if (steps > 1) {
      mbar_expect_tx(full_bar(1), 2 * COLS);
      load_cols(1);
    }
  }
  load_stats(0);
  const float l2 = (!KV && valid_row) ? lse_bh[row] * 1.4426950408889634f : 0.f;
  const bool row_extra = extra != nullptr && (KV ? (row >= 1 && valid_row) : row == 0);
  const float key_extra = (KV && row_extra) ? extra[row - 1] * invH : 0.f;      // KV: this key's share at the classification query
  float dsum = 0.f, dl = 0.f;
  bool ok = true;
  __syncthreads();

  for (int s = 0; s < steps; ++s) {
    const int tile = s % nt, k0 = tile * BL_COLS;
    const int cols = min(BL_COLS, T - k0), cpad = (cols + 15) & ~15;
    const uint32_t sC1 = sC + (s & 1) * 2 * COLS, sC2 = sC1 + COLS;
    if (tid == 0 && ok && !abort_flag) {
      // the previous step's products have read their operands (in tensor memory and in the other slot)
      if (s > 0 && (KV || s > nt)) ok = mbar_wait_q(p_bar, (KV ? s - 1 : s - nt - 1) & 1, abortp);
      if (ok && s >= 1 && s + 1 < steps) {
        mbar_expect_tx(full_bar((s + 1) & 1), 2 * COLS);
        load_cols(s + 1);
      }
      ok = ok && mbar_wait_q(full_bar(s & 1), (s >> 1) & 1, abortp);
      if (ok) {
        tc_fence_after();
        const uint32_t idesc = make_idesc_mn(AT_QROWS, cpad, false, false);
#pragma unroll
        for (int k = 0; k < AT_D / 16; ++k)
          umma_bf16(tmem + C_S, make_desc(sR1 + k * 32, 16, 1024), make_desc(sC1 + k * 32, 16, 1024), idesc, k > 0 ? 1u : 0u);
#pragma unroll
        for (int k = 0; k < AT_D / 16; ++k)
          umma_bf16(tmem + C_DP, make_desc(sR2 + k * 32, 16, 1024), make_desc(sC2 + k * 32, 16, 1024), idesc, k > 0 ? 1u : 0u);
        umma_commit(s_bar);
      }
    }
    load_stats(s + 1);
    ok = mbar_wait_q(s_bar, s & 1, abortp) && ok;
    ok = __all_sync(0xffffffffu, ok);
    tc_fence_after();
    const bool products = KV || s >= nt;
    if (ok) {
#pragma unroll
      for (int g = 0; g < 2; ++g) {                       // 16 columns at a time
        const int cc = half * 32 + g * 16;
        if (cc < cpad) {                                  // warp-uniform
          uint32_t rs[16], rp[16];
          tmem_ld16(trow + C_S + cc, rs);
          tmem_ld16(trow + C_DP + cc, rp);
          tmem_ld_wait();
          float p[16], dp[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const float l = KV ? stats[s & 1][0][cc + j] : l2;
            p[j] = cc + j < cols ? ex2_fast(fmaf(__uint_as_float(rs[j]), c, -l)) : 0.f;
            dp[j] = __uint_as_float(rp[j]);
          }
          if (row_extra) {
            if (KV) {
              if (k0 + cc == 0) dp[0] += key_extra;
            } else {
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                int key = k0 + cc + j;
                if (key >= 1 && key < T) dp[j] += extra[key - 1] * invH;
              }
            }
          }
          if (!products) {
#pragma unroll
            for (int j = 0; j < 16; ++j) dsum = fmaf(p[j], dp[j], dsum);
          } else {
            uint32_t pk[16];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const float d0 = KV ? stats[s & 1][1][cc + 2 * j] : dl, d1 = KV ? stats[s & 1][1][cc + 2 * j + 1] : dl;
              split_bf16x2(p[2 * j] * (dp[2 * j] - d0) * 0.125f, p[2 * j + 1] * (dp[2 * j + 1] - d1) * 0.125f, pk[j], pk[8 + j]);
            }
            tmem_st16(trow + C_DP + cc, pk);
            if (KV) {
#pragma unroll
              for (int j = 0; j < 8; ++j) split_bf16x2(p[2 * j], p[2 * j + 1], pk[j], pk[8 + j]);
              tmem_st16(trow + C_S + cc, pk);
            }
          }
        }
      }
      if (products) tmem_st_wait();
    }
    if (!KV && s == nt - 1) red[half][rowl] = dsum;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (!KV && s == nt - 1) {
      dl = red[0][rowl] + red[1][rowl];
      if (half == 0 && valid_row) delta_bh[row] = dl;
    }
    if (products && tid == 0 && ok && !abort_flag) {
      const uint32_t idesc = make_idesc_mn(AT_QROWS, AT_D, false, true);
      const bool first = KV ? s == 0 : s == nt;
      for (int i = 0; i < cpad / 8; ++i)                  // 16 columns of the block: their upper halves, then their lower ones
        umma_bf16_ts(tmem + C_A1, tmem + C_DP + i * 8, make_desc(sC1 + (i >> 1) * 2048, 8192, 1024), idesc, (first && i == 0) ? 0u : 1u);
      if (KV)
        for (int i = 0; i < cpad / 8; ++i)
          umma_bf16_ts(tmem + C_A2, tmem + C_S + i * 8, make_desc(sC2 + (i >> 1) * 2048, 8192, 1024), idesc, (first && i == 0) ? 0u : 1u);
      umma_commit(p_bar);
    }
  }
  ok = mbar_wait_q(p_bar, (nt - 1) & 1, abortp) && ok;
  ok = __all_sync(0xffffffffu, ok);
  tc_fence_after();
  // the products have read the row tiles: they hold the gradients' rows now
  unsigned char* out_tile = smem_dyn + (sR1 - smem_u32(smem_dyn));
  if (ok)
    for (int a = 0; a < (KV ? 2 : 1); ++a) stage_half_row(out_tile + a * ROWS, trow + C_A1 + 64 * a, rowl, half);
  __syncthreads();
  if (ok)
    for (int a = 0; a < (KV ? 2 : 1); ++a)
      write_rows(out_tile + a * ROWS, dqkv + (((size_t)row0 + r0) * 3 + (KV ? 1 + a : 0)) * H * AT_D + (size_t)h * AT_D, (size_t)3 * H * AT_D, min(AT_QROWS, T - r0));
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, 256);
  }
  if (tid == 0 && abort_flag && status != nullptr) atomicOr(status, STATUS_TIMEOUT);
}

}  // namespace tc

// Returns 0 when the tensor-core kernel took the problem, non-zero when the caller must use another kernel.
int attention_fwd_tc(const Ctx& c, const void* qkv, void* out, float* lse, float* cls_prob, int B, int T, int H, int d) {
  using namespace tc;
  if (c.dtype != 1 || d != AT_D || T < 1 || T > AT_LONG_KB * AT_LONG_MAXBLK) return -1;
  if (((uintptr_t)qkv & 15) || ((uintptr_t)out & 15)) return -1;
  CUtensorMap map;
  if (!make_map(&map, qkv, (uint64_t)3 * H * d, (uint64_t)B * T, (uint64_t)3 * H * d, AT_BOX)) return -2;
  // (up to 256 keys the kernel above, which holds a whole row of scores, is faster: 56 against 67 us at 197 tokens)
  if (T > AT_MAXKEYS) {
    size_t smem_l = 1024 + 2 * (size_t)AT_BOX_BYTES + 4 * (size_t)AT_LONG_KB * 128 + 64;
    static SmemLimit lim_l;
    if (!ensure_smem(lim_l, attn_fwd_tc_long_kernel, smem_l)) return -3;
    dim3 grid_l((T + AT_QROWS - 1) / AT_QROWS, B * H);
    note_launch(1);
    launch_k(attn_fwd_tc_long_kernel, grid_l, AT_LONG_THREADS, smem_l, c.stream, map, (bf16*)out, lse, cls_prob, B, T, H, c.status);
    return 0;
  }
  int tpad = (T + 15) & ~15;
  CUtensorMap map_q, map_kv;
  if (!make_map(&map_q, qkv, (uint64_t)3 * H * d, (uint64_t)B * T, (uint64_t)3 * H * d, AT_QROWS)) return -2;
  if (!make_map(&map_kv, qkv, (uint64_t)3 * H * d, (uint64_t)B * T, (uint64_t)3 * H * d, tpad)) return -2;
  int sms = c.sm_count > 0 ? c.sm_count : 148;
  const int nqt = ceil_div(T, AT_QROWS);
  if ((long)B * H * nqt <= sms) {
    const size_t smem_w = 1024 + WS_Q_BYTES + 2 * (size_t)tpad * 128;
    static SmemLimit lim_w[3];
    auto wide = [&](auto kern, SmemLimit& lim) -> int {
      if (!ensure_smem(lim, kern, smem_w)) return -3;
      note_launch(1);
      launch_k(kern, B * H * nqt, WIDE_THREADS, smem_w, c.stream, map_q, map_kv, (bf16*)out, lse, cls_prob, T, H, nqt, c.status);
      return 0;
    };
    if (T <= 128) return wide(attn_fwd_wide_kernel<2>, lim_w[0]);
    if (T <= 192) return wide(attn_fwd_wide_kernel<3>, lim_w[1]);
    return wide(attn_fwd_wide_kernel<4>, lim_w[2]);
  }
  int nbuf = tpad <= 128 ? 4 : (tpad <= 160 ? 3 : 2);
  size_t fixed = 1024 + (size_t)WS_QSLOTS * WS_Q_BYTES + (WS_MAXBUF * AT_MAXKEYS + WS_MAXBUF * 4 * AT_QROWS) * 4 + 44 * 8 + 64;
  size_t slot = (size_t)2 * tpad * 128;
  int kvslots = (int)((227 * 1024 - fixed) / slot);
  if (kvslots > WS_MAXKV) kvslots = WS_MAXKV;
  if (kvslots < 2) return -1;
  size_t smem = fixed + kvslots * slot;
  int grid = B * H < sms ? B * H : sms;
  static SmemLimit lim[5];
  auto launch = [&](auto kern, int threads) -> int {
    if (!ensure_smem(lim[nbuf], kern, smem)) return -3;
    note_launch(1);
    launch_k(kern, grid, threads, smem, c.stream, map_q, map_kv, (bf16*)out, lse, cls_prob, B, T, H, kvslots, c.status);
    return 0;
  };
  if (nbuf == 4) return launch(attn_fwd_ws_kernel<4>, 19 * 32);
  if (nbuf == 3) return launch(attn_fwd_ws_kernel<3>, 15 * 32);
  return launch(attn_fwd_ws_kernel<2>, 19 * 32);
}

}  // namespace bsr

namespace bsr {

int attention_bwd_tc(const Ctx& c, const void* qkv, const void* dout, const float* lse, const float* cls_extra, float* delta,
                     void* dqkv, int B, int T, int H, int d) {
  using namespace tc;
  if (c.dtype != 1 || d != AT_D || T < 1) return -1;
  if (T > 2 * AT_QROWS && (delta == nullptr || (long)B * H > 65535)) return -1;      // there (image, head) is the grid's second dimension
  if (((uintptr_t)qkv & 15) || ((uintptr_t)dout & 15) || ((uintptr_t)dqkv & 15)) return -1;
  CUtensorMap mq, mg;
  if (!make_map(&mq, qkv, (uint64_t)3 * H * d, (uint64_t)B * T, (uint64_t)3 * H * d, AT_BOX)) return -2;
  if (!make_map(&mg, dout, (uint64_t)H * d, (uint64_t)B * T, (uint64_t)H * d, AT_BOX)) return -2;
  // Up to 256 tokens the kernels below, which form every score once or twice instead of three times, are faster: 228 against
  // 318 us at 197 tokens, 51 against 118 us at 100 (batch 128, 12 heads; the longer kernels then still with P and dS rounded once).
  if (T > 2 * AT_QROWS) {
    size_t smem_l = 1024 + 4 * 2 * (size_t)AT_BOX_BYTES + 64;
    static SmemLimit lim_q, lim_kv;
    if (!ensure_smem(lim_q, attn_bwd_long_kernel<false>, smem_l) || !ensure_smem(lim_kv, attn_bwd_long_kernel<true>, smem_l)) return -3;
    dim3 grid((T + AT_QROWS - 1) / AT_QROWS, B * H);
    note_launch(2);
    launch_k(attn_bwd_long_kernel<false>, grid, 256, smem_l, c.stream, mq, mg, lse, delta, cls_extra, (bf16*)dqkv, B, T, H, c.status);
    launch_k(attn_bwd_long_kernel<true>, grid, 256, smem_l, c.stream, mq, mg, lse, delta, cls_extra, (bf16*)dqkv, B, T, H, c.status);
    return 0;
  }
  const int sms = c.sm_count > 0 ? c.sm_count : B200_SMS;
  if (T > AT_QROWS && 2l * B * H <= sms) { // a CTA per tile of keys
    const size_t smem_p = 1024 + 12 * 2 * (size_t)AT_BOX_BYTES;
    static SmemLimit lim_p;
    if (!ensure_smem(lim_p, attn_bwd_pair_kernel, smem_p)) return -3;
    note_launch(1);
    launch_cluster(attn_bwd_pair_kernel, dim3(2 * B * H), 256, smem_p, c.stream, dim3(2, 1, 1), mq, mg, lse, cls_extra, (bf16*)dqkv, T, H, c.status);
    return 0;
  }
  if (T > AT_QROWS) {                      // two tiles of queries and keys
    size_t smem2 = 1024 + 12 * 2 * (size_t)AT_BOX_BYTES + 4 * 256 * 4 + 64;
    static SmemLimit lim2;
    if (!ensure_smem(lim2, attn_bwd_tc256_kernel, smem2)) return -3;
    note_launch(1);
    launch_k(attn_bwd_tc256_kernel, B * H, 256, smem2, c.stream, mq, mg, lse, cls_extra, (bf16*)dqkv, B, T, H, c.status);
    return 0;
  }
  size_t tile = 2 * (size_t)AT_BOX_BYTES, ch = (size_t)((T + 15) & ~15) * 128;
  size_t smem = 1024 + 3 * tile + (2 * ch > tile ? 2 * ch : tile) + 2 * ch + (3 * ch < 16384 ? 16384 - 3 * ch : 0) + 3 * AT_QROWS * 4 + 64;
  static SmemLimit lim;
  if (!ensure_smem(lim, attn_bwd_tc_kernel, smem)) return -3;
  note_launch(1);
  launch_k(attn_bwd_tc_kernel, B * H, 256, smem, c.stream, mq, mg, lse, cls_extra, (bf16*)dqkv, B, T, H, c.status);
  return 0;
}

}  // namespace bsr
