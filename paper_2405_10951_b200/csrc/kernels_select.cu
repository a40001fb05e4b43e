// Token importance, per-image top-K and the compaction between MHSA and FFN (paper Section 4.1, Eq. 6).
#include <cooperative_groups.h>

#include <type_traits>

#include "common.cuh"
#include "kernels.h"
#include "layernorm.cuh"

namespace bsr {

// Monotone map float -> uint32 (larger float, larger key).
__device__ __forceinline__ uint32_t ordered_key(float f) {
  uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// The caller's copy of a drop location's kept positions, [B, k] (null: none).
__device__ __forceinline__ int* kept_copy_dst(const KeptCopy& c) {
  if (c.dst != nullptr) return c.dst;
  return c.eval != nullptr && c.eval->kept != nullptr ? c.eval->kept + c.off : nullptr;
}

// One warp per image.  Scores are the head mean of the classification token's attention row, summed in
// head order and divided by H in float.  The K-th largest key is found bit by bit (largest t with
// count(key >= t) >= K); ties at the threshold go to the lower index; both index lists come out ascending.
constexpr int SEL_WARPS = 4;

__global__ void token_select_kernel(const float* __restrict__ p, int B, int H, int M, int k,
                                    float* __restrict__ scores, int* __restrict__ kept, int* __restrict__ dropped, KeptCopy copy) {
  dependent_sync();
  extern __shared__ uint32_t keys_all[];
  int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int b = blockIdx.x * SEL_WARPS + warp;
  if (b >= B) return;
  uint32_t* keys = keys_all + (size_t)warp * M;
  const float* pb = p + (size_t)b * H * M;
  int* kcopy = kept_copy_dst(copy);
  for (int j = lane; j < M; j += 32) {
    float acc = pb[j];
    for (int h = 1; h < H; ++h) acc = acc + pb[(size_t)h * M + j];
    float s = acc / (float)H;
    scores[(size_t)b * M + j] = s;
    keys[j] = ordered_key(s);
  }
  __syncwarp();
  uint32_t t = 0;
  for (int bit = 31; bit >= 0; --bit) {
    uint32_t cand = t | (1u << bit);
    int cnt = 0;
    for (int j = lane; j < M; j += 32) cnt += (keys[j] >= cand) ? 1 : 0;
    cnt = warp_sum_int(cnt);
    if (cnt >= k) t = cand;
  }
  int gt = 0;
  for (int j = lane; j < M; j += 32) gt += (keys[j] > t) ? 1 : 0;
  gt = warp_sum_int(gt);
  int need_eq = k - gt;                 // how many of the keys equal to t are kept (lowest indices first)
  int n_kept = 0, n_drop = 0, eq_seen = 0;
  uint32_t lt_mask = (1u << lane) - 1u;
  for (int base = 0; base < M; base += 32) {
    int j = base + lane;
    bool valid = j < M;
    uint32_t key = valid ? keys[j] : 0u;
    bool is_eq = valid && key == t;
    uint32_t eq_mask = __ballot_sync(0xffffffffu, is_eq);
    int eq_rank = eq_seen + __popc(eq_mask & lt_mask);
    bool keep = valid && (key > t || (is_eq && eq_rank < need_eq));
    uint32_t keep_mask = __ballot_sync(0xffffffffu, keep);
    uint32_t drop_mask = __ballot_sync(0xffffffffu, valid && !keep);
    if (keep) {
      size_t at = (size_t)b * k + n_kept + __popc(keep_mask & lt_mask);
      kept[at] = j;
      if (kcopy != nullptr) kcopy[at] = j;
    } else if (valid) dropped[(size_t)b * (M - k) + n_drop + __popc(drop_mask & lt_mask)] = j;
    n_kept += __popc(keep_mask);
    n_drop += __popc(drop_mask);
    eq_seen += __popc(eq_mask);
  }
}

// Same selection with the keys of one image held in registers (IPL per lane, M <= 32 * IPL): the 32 threshold
// steps are register compares and one warp reduction each.  Element j lives in lane j % 32, slot j / 32, so a
// slot is a run of 32 consecutive tokens and ballots give positions in token order.
template <int IPL>
__global__ void __launch_bounds__(SEL_WARPS * 32)
token_select_reg_kernel(const float* __restrict__ p, int B, int H, int M, int k, float* __restrict__ scores,
                        int* __restrict__ kept, int* __restrict__ dropped, KeptCopy copy) {
  dependent_sync();
  int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int b = blockIdx.x * SEL_WARPS + warp;
  if (b >= B) return;
  const float* pb = p + (size_t)b * H * M;
  int* kcopy = kept_copy_dst(copy);
  uint32_t key[IPL];
  float acc[IPL];
  // head sum in head order per token; the IPL loads of one head are independent, so many are in flight
#pragma unroll
  for (int i = 0; i < IPL; ++i) acc[i] = (i * 32 + lane < M) ? pb[i * 32 + lane] : 0.f;
  // heads in groups of four: the loads of a group are all issued before its (ordered) additions
  int h = 1;
  for (; h + 4 <= H; h += 4) {
    float v[4][IPL];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float* ph = pb + (size_t)(h + u) * M;
#pragma unroll
      for (int i = 0; i < IPL; ++i) v[u][i] = (i * 32 + lane < M) ? ph[i * 32 + lane] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
#pragma unroll
      for (int i = 0; i < IPL; ++i) acc[i] = acc[i] + v[u][i];
    }
  }
  for (; h < H; ++h) {
    const float* ph = pb + (size_t)h * M;
#pragma unroll
    for (int i = 0; i < IPL; ++i)
      if (i * 32 + lane < M) acc[i] = acc[i] + ph[i * 32 + lane];
  }
#pragma unroll
  for (int i = 0; i < IPL; ++i) {
    int j = i * 32 + lane;
    key[i] = 0u;
    if (j < M) {
      float s = acc[i] / (float)H;
      scores[(size_t)b * M + j] = s;
      key[i] = ordered_key(s);
    }
  }
  // keys of absent elements are 0, below every real key (a real key has its top bit set unless the score is negative;
  // scores are probabilities), and they are excluded by index below anyway
  uint32_t t = 0;
  for (int bit = 31; bit >= 0; --bit) {
    uint32_t cand = t | (1u << bit);
    int cnt = 0;
#pragma unroll
    for (int i = 0; i < IPL; ++i) cnt += (i * 32 + lane < M && key[i] >= cand) ? 1 : 0;
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (cnt >= k) t = cand;
  }
  int gt = 0;
#pragma unroll
  for (int i = 0; i < IPL; ++i) gt += (i * 32 + lane < M && key[i] > t) ? 1 : 0;
  gt = __reduce_add_sync(0xffffffffu, gt);
  int need_eq = k - gt;
  int n_kept = 0, n_drop = 0, eq_seen = 0;
  uint32_t lt_mask = (1u << lane) - 1u;
#pragma unroll
  for (int i = 0; i < IPL; ++i) {
    int j = i * 32 + lane;
    if (i * 32 >= M) break;
    bool valid = j < M;
    bool is_eq = valid && key[i] == t;
    uint32_t eq_mask = __ballot_sync(0xffffffffu, is_eq);
    int eq_rank = eq_seen + __popc(eq_mask & lt_mask);
    bool keep = valid && (key[i] > t || (is_eq && eq_rank < need_eq));
    uint32_t keep_mask = __ballot_sync(0xffffffffu, keep);
    uint32_t drop_mask = __ballot_sync(0xffffffffu, valid && !keep);
    if (keep) {
      size_t at = (size_t)b * k + n_kept + __popc(keep_mask & lt_mask);
      kept[at] = j;
      if (kcopy != nullptr) kcopy[at] = j;
    } else if (valid) dropped[(size_t)b * (M - k) + n_drop + __popc(drop_mask & lt_mask)] = j;
    n_kept += __popc(keep_mask);
    n_drop += __popc(drop_mask);
    eq_seen += __popc(eq_mask);
  }
}

void token_select(cudaStream_t s, const float* p, int B, int H, int M, int k, float* scores, int* kept, int* dropped, KeptCopy copy) {
  note_launch(1);
  int blocks = ceil_div(B, SEL_WARPS), threads = SEL_WARPS * 32;
  if (M <= 256) { launch_k(token_select_reg_kernel<8>, blocks, threads, 0, s, p, B, H, M, k, scores, kept, dropped, copy); return; }
  if (M <= 640) { launch_k(token_select_reg_kernel<20>, blocks, threads, 0, s, p, B, H, M, k, scores, kept, dropped, copy); return; }
  size_t smem = (size_t)SEL_WARPS * M * sizeof(uint32_t);
  if (smem > 48 * 1024) cudaFuncSetAttribute(token_select_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  launch_k(token_select_kernel, blocks, threads, smem, s, p, B, H, M, k, scores, kept, dropped, copy);
}

// ------------------------------------------------------------------------------------------------
// Compaction.  grid = (B, copy_splits + fuse_slices), 256 threads.
//   blockIdx.y <  copy_splits : copies the classification row and a share of the kept rows (16-byte vectors);
//   blockIdx.y >= copy_splits : builds a column slice of the fused token, sum over dropped j of s_j * x_j,
//                               row lanes accumulate in float and are combined through shared memory in lane order.
// ------------------------------------------------------------------------------------------------
constexpr int GF_THREADS = 256;
constexpr int GF_SLICE_CHUNKS = 32;     // 16-byte chunks per fused-token column slice
constexpr int GF_ROWLANES = GF_THREADS / GF_SLICE_CHUNKS;

template <typename T>
__global__ void gather_fuse_kernel(const T* __restrict__ x, int M, int D, int k, const int* __restrict__ kept,
                                   const int* __restrict__ dropped, const float* __restrict__ scores, int fuse,
                                   T* __restrict__ out, int copy_splits, int* status) {
  dependent_sync();
  constexpr int N = Pack<T>::N;
  int b = blockIdx.x;
  int chunks = D / N;
  int t_out = 1 + k + (fuse ? 1 : 0);
  const T* xb = x + (size_t)b * (1 + M) * D;
  T* ob = out + (size_t)b * t_out * D;
  if ((int)blockIdx.y < copy_splits) {
    int rows = 1 + k;
    int per = (rows + copy_splits - 1) / copy_splits;
    int r0 = blockIdx.y * per, r1 = min(rows, r0 + per);
    int total = (r1 - r0) * chunks;
    for (int i = threadIdx.x; i < total; i += GF_THREADS) {
      int r = r0 + i / chunks, ch = i % chunks;
      int src = (r == 0) ? 0 : 1 + kept[(size_t)b * k + (r - 1)];
      if (!BSR_CHECK(src >= 0 && src <= M, status)) continue;
      uint4 v = *reinterpret_cast<const uint4*>(xb + (size_t)src * D + ch * N);
      *reinterpret_cast<uint4*>(ob + (size_t)r * D + ch * N) = v;
    }
    return;
  }
  __shared__ float sm[GF_ROWLANES][GF_SLICE_CHUNKS * N];
  __shared__ float weight_sum;
  int slice = blockIdx.y - copy_splits;
  int cs = threadIdx.x % GF_SLICE_CHUNKS, rl = threadIdx.x / GF_SLICE_CHUNKS;
  int ch = slice * GF_SLICE_CHUNKS + cs;
  float acc[N];
#pragma unroll
  for (int j = 0; j < N; ++j) acc[j] = 0.f;
  int nd = M - k;
  if (fuse == 2 && threadIdx.x < 32) {        // weighted mean: the sum of the dropped tokens' weights, in a fixed order
    float ws = 0.f;
    for (int i = threadIdx.x; i < nd; i += 32) ws += scores[(size_t)b * M + dropped[(size_t)b * nd + i]];
    ws = warp_sum(ws);
    if (threadIdx.x == 0) weight_sum = ws;
  }
  if (ch < chunks) {
    for (int i = rl; i < nd; i += GF_ROWLANES) {
      int j = dropped[(size_t)b * nd + i];
      if (!BSR_CHECK(j >= 0 && j < M, status)) continue;
      float w = scores[(size_t)b * M + j];
      float v[N];
      load16(xb + (size_t)(1 + j) * D + ch * N, v);
#pragma unroll
      for (int e = 0; e < N; ++e) acc[e] += w * v[e];
    }
  }
#pragma unroll
  for (int e = 0; e < N; ++e) sm[rl][cs * N + e] = acc[e];
  __syncthreads();
  if (rl == 0 && ch < chunks) {
    float o[N];
#pragma unroll
    for (int e = 0; e < N; ++e) {
      float s = 0.f;
#pragma unroll
      for (int r = 0; r < GF_ROWLANES; ++r) s += sm[r][cs * N + e];
      o[e] = fuse == 2 ? s / weight_sum : s;
    }
    store16(ob + (size_t)(1 + k) * D + ch * N, o);
  }
}

void gather_fuse(const Ctx& c, const void* x, int B, int M, int D, int k, const int* kept, const int* dropped,
                 const float* scores, int fuse, void* out) {
  note_launch(1);
  int n = (c.dtype == 0) ? 4 : 8;
  int chunks = D / n;
  int do_fuse = ((fuse == 1 || fuse == 2) && k < M) ? fuse : 0;          // 1: weighted sum, 2: weighted mean
  int fuse_slices = do_fuse ? ceil_div(chunks, GF_SLICE_CHUNKS) : 0;
  int sms = c.sm_count > 0 ? c.sm_count : 148;
  int copy_splits = ceil_div(4L * sms, B);            // about four blocks per SM in total
  if (copy_splits < 1) copy_splits = 1;
  if (copy_splits > 1 + k) copy_splits = 1 + k;
  dim3 grid(B, copy_splits + fuse_slices);
  if (c.dtype == 0)
    launch_k(gather_fuse_kernel<float>, grid, GF_THREADS, 0, c.stream, (const float*)x, M, D, k, kept, dropped, scores, do_fuse, (float*)out, copy_splits, c.status);
  else
    launch_k(gather_fuse_kernel<bf16>, grid, GF_THREADS, 0, c.stream, (const bf16*)x, M, D, k, kept, dropped, scores, do_fuse, (bf16*)out, copy_splits, c.status);
}

// Selection, compaction and the LayerNorm that follows, one image per cluster of eight CTAs.  As three launches each waited for the
// one before: the selection is one warp's work (9 us of inference with one image), and the compacted rows went out to be read again.
// Here every CTA selects for itself -- a thread has up to four tokens' keys, the K-th largest is found two bits at a time, three
// counts to a warp reduction and one barrier each -- and then takes every eighth row of each kind:
//   dropped rows : threads own four columns and add up s_j x_j; rank 0 combines the eight parts, read through distributed shared
//                  memory, in rank order (the order of gather_fuse_kernel, whatever the batch), and finishes the fused row;
//   kept rows    : a warp a row, taken from a counter; the row is in registers, so its LayerNorm costs no second pass.
// Scores, kept and dropped lists are those of token_select, ties at the K-th key going to the lower index.
// us a step, three launches -> one: ViT-B, 1 / 8 / 32 images 920 -> 884 / 1210 -> 1170 / 1951 -> 1916, DeiT-S, 8 / 24 images 772 -> 756 /
// 971 -> 956, ViT-B/384, 7 images 1691 -> 1666.  33 clusters are on the SMs at once (two of these CTAs on each; 119 registers a thread); more images
// wait for a second round, which costs more than the launches.  us of inference, three launches / one, around that: DeiT-S, 30 / 32 / 34 / 40
// images 630 / 623, 671 / 664, 673 / 680, 711 / 719; ViT-B, 32 / 34 / 40 images 1121 / 1110, 1134 / 1138, 1206 / 1215; 577 tokens, where rows outweigh
// launches, 32 / 34 / 64 images 2509 / 2484, 2748 / 2752, 4738 / 4761.
constexpr int SGA_MAXIMAGES = 32;
constexpr int SGA_THREADS = 256, SGA_RANKS = 8, SGA_MAXM = 1023;   // three counts of up to 1023 share one warp reduction
constexpr int SGA_MAXD = 1024;
// Kept rows are shared out over as many clusters an image as the SMs have room for; the first has the dropped ones.
constexpr int SGA_MAXCLUSTERS = 4;

template <int IPT, typename TY>
__global__ void __launch_bounds__(SGA_THREADS)
select_gather_kernel(const float* __restrict__ p, const float* __restrict__ x, int clusters, int H, int M, int D, int k, int fuse, float* __restrict__ scores,
                     int* __restrict__ kept, int* __restrict__ dropped, KeptCopy copy, float* __restrict__ out, const float* __restrict__ g,
                     const float* __restrict__ be, TY* __restrict__ y, float* __restrict__ mean, float* __restrict__ rstd, float eps, int* status) {
  dependent_sync();
  __shared__ float sc[SGA_MAXM + 1];
  __shared__ int list[SGA_MAXM + 1];                      // kept positions, then dropped ones, each ascending
  __shared__ __align__(16) float part[SGA_MAXD];
  __shared__ int next_row;
  constexpr int NCH = SGA_MAXD / 128;
  cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = blockIdx.x % SGA_RANKS, b = blockIdx.x / SGA_RANKS / clusters, share = blockIdx.x / SGA_RANKS - b * clusters;
  const bool first = share == 0, lead = first && rank == 0;
  const float* pb = p + (size_t)b * H * M;
  constexpr int WARPS = SGA_THREADS / 32;
  __shared__ __align__(16) uint32_t counts[2][WARPS];
  __shared__ int n_gt[IPT * WARPS], n_eq[IPT * WARPS], at_kept[IPT * WARPS], at_drop[IPT * WARPS], eq_left[IPT * WARPS];
  if (tid == 0) next_row = share * SGA_RANKS + rank;
  uint32_t key[IPT];                                       // token i * SGA_THREADS + tid; absent ones 0, below every candidate
#pragma unroll
  for (int i = 0; i < IPT; ++i) {
    const int j = i * SGA_THREADS + tid;
    key[i] = 0u;
    if (j < M) {
      float acc = 0.f;
      for (int h = 0; h < H; h += 12) {                    // the loads of twelve heads at once, the sum in head order
        float v[12];
#pragma unroll
        for (int u = 0; u < 12; ++u)
          if (h + u < H) v[u] = pb[(size_t)(h + u) * M + j];
#pragma unroll
        for (int u = 0; u < 12; ++u)
          if (h + u < H) acc = h + u == 0 ? v[u] : acc + v[u];
      }
      const float s = acc / (float)H;
      sc[j] = s;
      key[i] = ordered_key(s);
      if (lead) scores[(size_t)b * M + j] = s;
    }
  }
  uint32_t t = 0;
  for (int bit = 30; bit >= 0; bit -= 2) {
    const uint32_t c1 = t | (1u << bit), c2 = t | (2u << bit), c3 = t | (3u << bit);
    uint32_t cnt = 0;
#pragma unroll
    for (int i = 0; i < IPT; ++i) cnt += (key[i] >= c1 ? 1u : 0u) + (key[i] >= c2 ? 1u << 10 : 0u) + (key[i] >= c3 ? 1u << 20 : 0u);
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    uint32_t* row = counts[(bit >> 1) & 1];
    if (lane == 0) row[warp] = cnt;
    __syncthreads();
    const uint4 x = reinterpret_cast<const uint4*>(row)[0], z = reinterpret_cast<const uint4*>(row)[1];
    cnt = ((x.x + x.y) + (x.z + x.w)) + ((z.x + z.y) + (z.z + z.w));
    if ((cnt >> 20) >= (uint32_t)k) t = c3;
    else if (((cnt >> 10) & 1023u) >= (uint32_t)k) t = c2;
    else if ((cnt & 1023u) >= (uint32_t)k) t = c1;
  }
  // positions: groups of 32 tokens in token order (IPT * WARPS <= 32 of them, a lane of warp 0 each); of the keys equal to the K-th the
  // first ones are kept
  const uint32_t lt_mask = (1u << lane) - 1u;
  uint32_t gt_mask[IPT], eq_mask[IPT];
#pragma unroll
  for (int i = 0; i < IPT; ++i) {
    const bool valid = i * SGA_THREADS + tid < M;
    gt_mask[i] = __ballot_sync(0xffffffffu, valid && key[i] > t);
    eq_mask[i] = __ballot_sync(0xffffffffu, valid && key[i] == t);
    if (lane == 0) { n_gt[i * WARPS + warp] = __popc(gt_mask[i]); n_eq[i * WARPS + warp] = __popc(eq_mask[i]); }
  }
  __syncthreads();
  if (warp == 0) {
    const bool have = lane < IPT * WARPS;
    const int gt = have ? n_gt[lane] : 0, eq = have ? n_eq[lane] : 0;
    const int need_eq = k - __reduce_add_sync(0xffffffffu, gt);
    auto before = [&](int v) {                             // sum over the lanes below
      int s = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += u;
      }
      return s - v;
    };
    const int left = max(0, need_eq - before(eq)), kept_here = gt + min(eq, left), at = before(kept_here);
    if (have) { eq_left[lane] = left; at_kept[lane] = at; at_drop[lane] = k + min(lane * 32, M) - at; }
  }
  __syncthreads();
  int* kcopy = lead ? kept_copy_dst(copy) : nullptr;
#pragma unroll
  for (int i = 0; i < IPT; ++i) {
    const int j = i * SGA_THREADS + tid, w = i * WARPS + warp;
    const uint32_t bit = 1u << lane;
    const int eq_before = __popc(eq_mask[i] & lt_mask);
    const bool keep = (gt_mask[i] & bit) != 0 || ((eq_mask[i] & bit) != 0 && eq_before < eq_left[w]);
    const uint32_t keep_mask = __ballot_sync(0xffffffffu, keep);
    if (j >= M) continue;
    const int n = __popc(keep_mask & lt_mask), at = keep ? at_kept[w] + n : at_drop[w] + lane - n;
    if (!BSR_CHECK(keep ? at >= 0 && at < k : at >= k && at < M, status)) continue;
    list[at] = j;
    if (lead) {
      if (keep) {
        kept[(size_t)b * k + at] = j;
        if (kcopy != nullptr) kcopy[(size_t)b * k + at] = j;
      } else {
        dropped[(size_t)b * (M - k) + at - k] = j;
      }
    }
  }
  __syncthreads();
  const int nd = M - k, t_out = 1 + k + (fuse ? 1 : 0), col = tid * 4;
  const float* xb = x + (size_t)b * (1 + M) * D;
  const bool has = fuse && first && col < D;
  if (has) {
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    for (int i0 = rank; i0 < nd; i0 += 8 * SGA_RANKS) {    // eight rows at once, added in order
      float v[8][4];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (i0 + u * SGA_RANKS < nd && BSR_CHECK(list[k + i0 + u * SGA_RANKS] >= 0 && list[k + i0 + u * SGA_RANKS] < M, status))
          load16(xb + (size_t)(1 + list[k + i0 + u * SGA_RANKS]) * D + col, v[u]);
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (i0 + u * SGA_RANKS < nd && BSR_CHECK(list[k + i0 + u * SGA_RANKS] >= 0 && list[k + i0 + u * SGA_RANKS] < M, status)) {
          const float w = sc[list[k + i0 + u * SGA_RANKS]];
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[e] += w * v[u][e];
        }
    }
    store16(part + col, acc);
  }
  auto finish_row = [&](int r, const float* src) {         // row r of the image's output, by one warp
    const size_t ro = (size_t)b * t_out + r;
    float v[NCH * 4];
    ln_load_row<NCH>(src, D, v);
    float* dst = out + ro * D;
#pragma unroll
    for (int i = 0; i < NCH; ++i)
      if (lane + i * 32 < D / 4) store16(dst + (lane + i * 32) * 4, v + i * 4);
    if (y != nullptr) ln_write_row<TY, NCH>(v, g, be, y + ro * D, mean ? mean + ro : nullptr, rstd ? rstd + ro : nullptr, D, eps);
  };
  while (true) {
    int r = 0;
    if (lane == 0) r = atomicAdd(&next_row, clusters * SGA_RANKS);
    r = __shfl_sync(0xffffffffu, r, 0);
    if (r > k) break;
    const int src = r == 0 ? 0 : 1 + list[r - 1];
    if (!BSR_CHECK(src >= 0 && src <= M, status)) continue;
    finish_row(r, xb + (size_t)src * D);
  }
  if (!fuse || !first) return;
  cluster.sync();
  if (rank == 0 && has) {
    float o[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int r = 0; r < SGA_RANKS; ++r) {
      float v[4];
      load16(cluster.map_shared_rank(part, r) + col, v);
#pragma unroll
      for (int e = 0; e < 4; ++e) o[e] += v[e];
    }
    store16(part + col, o);                                // (a thread rewrites what it alone reads)
  }
  cluster.sync();                                          // no CTA leaves while rank 0 may still read its part
  if (rank == 0 && warp == 0) {
    if (fuse == 2) {                                       // weighted mean: by the sum of the dropped tokens' weights, in a fixed order
      float ws = 0.f;
      for (int i = lane; i < nd; i += 32)
        if (BSR_CHECK(list[k + i] >= 0 && list[k + i] < M, status)) ws += sc[list[k + i]];
      ws = warp_sum(ws);
      for (int c = lane; c < D; c += 32) part[c] = part[c] / ws;
      __syncwarp();
    }
    finish_row(1 + k, part);
  }
}

int select_gather(const Ctx& c, const float* p, const float* x, int B, int H, int M, int D, int k, int fuse, float* scores, int* kept, int* dropped,
                  KeptCopy copy, float* out, const float* g, const float* b, void* y, float* mean, float* rstd, float eps) {
  if (B > SGA_MAXIMAGES || M > SGA_MAXM || D > SGA_MAXD || D % 4 != 0 || k >= M) return -1;
  note_launch(1);
  const int sms = c.sm_count > 0 ? c.sm_count : B200_SMS;
  int clusters = sms / (B * SGA_RANKS);
  clusters = clusters < 1 ? 1 : clusters > SGA_MAXCLUSTERS ? SGA_MAXCLUSTERS : clusters;
  auto go = [&](auto kern, auto* yt) {
    launch_cluster(kern, dim3(B * clusters * SGA_RANKS), SGA_THREADS, 0, c.stream, dim3(SGA_RANKS, 1, 1), p, x, clusters, H, M, D, k, fuse, scores, kept, dropped, copy, out, g, b,
                   yt, mean, rstd, eps, c.status);
  };
  auto pick = [&](auto* yt) {
    using TY = std::remove_pointer_t<decltype(yt)>;
    if (M <= SGA_THREADS) go(select_gather_kernel<1, TY>, yt);
    else if (M <= 3 * SGA_THREADS) go(select_gather_kernel<3, TY>, yt);
    else go(select_gather_kernel<4, TY>, yt);
  };
  if (c.dtype == 0) pick((float*)y);
  else pick((bf16*)y);
  return 0;
}

// Backward of the compaction, one warp per input row (the index sets are constants, the fusion weights are
// differentiated):  dx_0 = g_0;  dx_{kept_i} = g_{1+i};  dx_j = s_j g_f and e_j = <g_f, x_j> for dropped j.
// Weighted mean (fuse == 2, f = sum_j s_j x_j / S, S = sum_j s_j): dx_j = (s_j / S) g_f, e_j = (<g_f, x_j> - <g_f, f>) / S
// with f read from the forward pass's compacted tensor `fwd_out`.
// Rows are float (residual stream); dx_copy optionally receives the same rows in bf16.
__global__ void gather_fuse_bwd_kernel(const float* __restrict__ dout, const float* __restrict__ x, int B, int M, int D, int k,
                                       const int* __restrict__ kept, const int* __restrict__ dropped,
                                       const float* __restrict__ scores, int fuse, float* __restrict__ dx,
                                       bf16* __restrict__ dx_copy, float* __restrict__ escore, const float* __restrict__ fwd_out,
                                       int* status) {
  dependent_sync();
  int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (warp >= B * (1 + M)) return;
  int b = warp / (1 + M), e = warp % (1 + M);
  int chunks = D / 4;
  int t_out = 1 + k + (fuse ? 1 : 0);
  const float* gb = dout + (size_t)b * t_out * D;
  size_t ob = (size_t)b * (1 + M) * D;
  if (e <= k) {                         // classification row or a kept row: plain copy
    int dst = (e == 0) ? 0 : 1 + kept[(size_t)b * k + (e - 1)];
    if (!BSR_CHECK(dst >= 0 && dst <= M, status)) return;
    for (int ch = lane; ch < chunks; ch += 32) {
      float v[4];
      load16(gb + (size_t)e * D + ch * 4, v);
      store16(dx + ob + (size_t)dst * D + ch * 4, v);
      if (dx_copy != nullptr) store4(dx_copy + ob + (size_t)dst * D + ch * 4, v);
    }
    if (e > 0 && lane == 0) escore[(size_t)b * M + (dst - 1)] = 0.f;
    return;
  }
  int j = dropped[(size_t)b * (M - k) + (e - 1 - k)];
  if (!BSR_CHECK(j >= 0 && j < M, status)) return;
  float w = fuse ? scores[(size_t)b * M + j] : 0.f;
  const float* gf = gb + (size_t)(1 + k) * D;
  const float* xr = x + ob + (size_t)(1 + j) * D;
  float inv_sum = 1.f, dot_f = 0.f;
  if (fuse == 2) {
    int nd = M - k;
    float ws = 0.f;
    for (int i = lane; i < nd; i += 32) ws += scores[(size_t)b * M + dropped[(size_t)b * nd + i]];
    inv_sum = 1.0f / warp_sum(ws);
    const float* fr = fwd_out + ((size_t)b * t_out + 1 + k) * D;
    for (int ch = lane; ch < chunks; ch += 32) {
      float g[4], fv[4];
      load16(gf + ch * 4, g);
      load16(fr + ch * 4, fv);
#pragma unroll
      for (int i = 0; i < 4; ++i) dot_f += g[i] * fv[i];
    }
    dot_f = warp_sum(dot_f);
    w *= inv_sum;
  }
  float dot = 0.f;
  for (int ch = lane; ch < chunks; ch += 32) {
    float g[4], o[4];
    if (fuse) {
      float xv[4];
      load16(gf + ch * 4, g);
      load16(xr + ch * 4, xv);
#pragma unroll
      for (int i = 0; i < 4; ++i) { dot += g[i] * xv[i]; o[i] = w * g[i]; }
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) o[i] = 0.f;
    }
    store16(dx + ob + (size_t)(1 + j) * D + ch * 4, o);
    if (dx_copy != nullptr) store4(dx_copy + ob + (size_t)(1 + j) * D + ch * 4, o);
  }
  dot = warp_sum(dot);
  if (lane == 0) escore[(size_t)b * M + j] = fuse == 2 ? (dot - dot_f) * inv_sum : dot;
}

void gather_fuse_bwd(const Ctx& c, const void* dout, const void* x, int B, int M, int D, int k, const int* kept,
                     const int* dropped, const float* scores, int fuse, void* dx, void* dx_copy, float* escore, const void* fwd_out) {
  note_launch(1);
  int do_fuse = ((fuse == 1 || fuse == 2) && k < M) ? fuse : 0;
  int threads = 256, blocks = ceil_div((long)B * (1 + M) * 32, threads);
  launch_k(gather_fuse_bwd_kernel, blocks, threads, 0, c.stream, (const float*)dout, (const float*)x, B, M, D, k, kept, dropped, scores,
                                                           do_fuse, (float*)dx, (bf16*)dx_copy, escore, (const float*)fwd_out, c.status);
}

}  // namespace bsr
