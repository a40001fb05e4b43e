// Classification head on the classification token: final LayerNorm, logits, cross-entropy and their backward.
#include <cooperative_groups.h>

#include "common.cuh"
#include "kernels.h"

namespace bsr {

namespace cg = cooperative_groups;

struct HeadDev {
  int num_tasks, cmax, D;
  int ncls[4];
  const void* w[4];
  const float* bias[4];
  float* dw[4];
  float* db[4];
};

static HeadDev to_dev(const HeadDesc& h) {
  HeadDev d;
  d.num_tasks = h.num_tasks; d.cmax = h.cmax; d.D = h.D;
  for (int i = 0; i < 4; ++i) { d.ncls[i] = h.ncls[i]; d.w[i] = h.w[i]; d.bias[i] = h.bias[i]; d.dw[i] = h.dw[i]; d.db[i] = h.db[i]; }
  return d;
}

constexpr int HC_THREADS = 256, HC_WARPS = HC_THREADS / 32;
constexpr int HC_MAXRANKS = 8;
constexpr int HC_SLICE = 1024;                   // classes of one CTA whose logits fit its shared memory; more go through global memory
constexpr int HC_MAXD = 1024;

// Sum (or maximum) over the block, combined in warp order; red holds HC_WARPS floats.
template <bool MAX>
__device__ __forceinline__ float hc_block(float v, float* red) {
  v = MAX ? warp_max(v) : warp_sum(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  float r = red[0];
#pragma unroll
  for (int w = 1; w < HC_WARPS; ++w) r = MAX ? fmaxf(r, red[w]) : r + red[w];
  return r;
}

// Everything between the last block's output and the gradient of it, one image per cluster: LayerNorm of the classification row,
// logits, loss and its gradient, back through the head's weights and the LayerNorm.  What bounds it is latency (100 classes x 768 are
// 154 KB that every image reads from L2), so an image's classes are split over the CTAs of a cluster (`ranks`, in
// training by the number of classes alone), which exchange the softmax's maximum and sum and their parts of the gradient through distributed
// shared memory in rank order.  Only what sums over images is left to head_grads_kernel, which runs beside the blocks' backward pass.
// In place of seven launches, and of the copies and zeroed tensors around the last block's classification rows, us a step:
//   DeiT-S, 1 / 8 images 659 -> 647 / 785 -> 772   ViT-B, 1 image 934 -> 920   ViT-B/384, 7 images 1719 -> 1691   two tasks, 4 images 1229 -> 1206
template <typename T, bool TRAIN>
__global__ void __launch_bounds__(HC_THREADS)
head_chain_kernel(HeadDev h, HeadRow io, const EvalIo* __restrict__ eval, const int* __restrict__ labels, const int* __restrict__ task_ids, T* dx_copy,
                  int ranks, int B, int* status) {
  dependent_sync();
  __shared__ __align__(16) float xs[HC_MAXD];                // the normalised row
  __shared__ __align__(16) float part[4 * HC_THREADS];       // this CTA's part of the gradient of it
  __shared__ float slice[HC_SLICE];
  __shared__ float red[HC_WARPS];
  __shared__ float ex[2];
  constexpr int N = Pack<T>::N;
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int b = blockIdx.x / ranks, rank = blockIdx.x - b * ranks;
  const int D = h.D, d4 = D / 4, col = tid * 4;
  const bool has = tid < d4;

  // LayerNorm of the row: four columns a thread
  float v[4] = {0.f, 0.f, 0.f, 0.f}, gam[4] = {0.f, 0.f, 0.f, 0.f}, bet[4] = {0.f, 0.f, 0.f, 0.f};
  if (has) {
    load16(io.x + (long)b * io.x_stride + col, v);
    load16(io.gamma + col, gam);
    load16(io.beta + col, bet);
  }
  const float mu = hc_block<false>((v[0] + v[1]) + (v[2] + v[3]), red) / (float)D;
#pragma unroll
  for (int j = 0; j < 4; ++j) v[j] = has ? v[j] - mu : 0.f;
  const float rs = rsqrtf(hc_block<false>((v[0] * v[0] + v[1] * v[1]) + (v[2] * v[2] + v[3] * v[3]), red) / (float)D + io.eps);
  if (has) {
    float o[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      v[j] *= rs;                                              // from here on the row without scale and shift
      o[j] = v[j] * gam[j] + bet[j];
    }
    store16(xs + col, o);
    if (TRAIN && rank == 0) {
      store16(io.xn + (long)b * D + col, o);
      store16(io.xhat + (long)b * D + col, v);
    }
  }
  int t = task_ids ? task_ids[b] : 0;
  // labels and task ids come from the caller: in every build a value outside its range raises STATUS_CHECK and is
  // clamped, instead of indexing outside the logits
  if (t < 0 || t >= h.num_tasks) {
    if (tid == 0 && status != nullptr) atomicOr(status, STATUS_CHECK);
    t = 0;
  }
  const int n = h.ncls[t];
  const int c0 = (int)((long)rank * h.cmax / ranks), c1 = (int)((long)(rank + 1) * h.cmax / ranks), cn = min(c1, n);
  const T* w = (const T*)h.w[t];
  float* lg = c1 - c0 <= HC_SLICE ? slice : io.dlogits + (size_t)b * h.cmax + c0;
  __syncthreads();

  // logits of this CTA's classes, a warp a class, two in flight
  float* lout = io.logits + (size_t)b * h.cmax;
  float* lcopy = eval != nullptr ? eval->logits + (size_t)b * h.cmax : nullptr;
  for (int c = c0 + warp; c < c1; c += 2 * HC_WARPS) {
    const int ca = c < n ? c : 0, cb = c + HC_WARPS < cn ? c + HC_WARPS : 0;
    float sa = 0.f, sb = 0.f;
#pragma unroll
    for (int it = 0; it < HC_MAXD / (32 * N); ++it) {          // (all loads of the two rows at once)
      const int e = (it * 32 + lane) * N;
      if (e < D) {
        float wa[N], wb[N];
        load16(w + (size_t)ca * D + e, wa);
        load16(w + (size_t)cb * D + e, wb);
#pragma unroll
        for (int j = 0; j < N; ++j) { sa = fmaf(xs[e + j], wa[j], sa); sb = fmaf(xs[e + j], wb[j], sb); }
      }
    }
    sa = warp_sum(sa);
    sb = warp_sum(sb);
    if (lane < 2) {
      const int cc = c + lane * HC_WARPS;
      if (cc < c1) {
        const float l = cc < n ? (lane == 0 ? sa : sb) + h.bias[t][cc] : -INFINITY;
        lg[cc - c0] = l;
        lout[cc] = l;
        if (lcopy != nullptr) lcopy[cc] = l;
      }
    }
  }
  if constexpr (TRAIN) {
    __syncthreads();
    // loss and its gradient: dlogits = (softmax - onehot) / B
    float mx = -INFINITY, se = 0.f;
    for (int c = c0 + tid; c < cn; c += HC_THREADS) mx = fmaxf(mx, lg[c - c0]);
    mx = hc_block<true>(mx, red);
    for (int c = c0 + tid; c < cn; c += HC_THREADS) {          // (a masked class adds nothing, even where all of this CTA's are masked)
      const float l = lg[c - c0];
      se += l == -INFINITY ? 0.f : expf(l - mx);
    }
    se = hc_block<false>(se, red);
    if (ranks > 1) {
      if (tid == 0) { ex[0] = mx; ex[1] = se; }
      cluster.sync();
      float m[HC_MAXRANKS], s[HC_MAXRANKS];
#pragma unroll
      for (int r = 0; r < HC_MAXRANKS; ++r)
        if (r < ranks) { const float* p = cluster.map_shared_rank(ex, r); m[r] = p[0]; s[r] = p[1]; }
      mx = m[0];
#pragma unroll
      for (int r = 1; r < HC_MAXRANKS; ++r)
        if (r < ranks) mx = fmaxf(mx, m[r]);
      se = 0.f;
#pragma unroll
      for (int r = 0; r < HC_MAXRANKS; ++r)
        if (r < ranks) se += s[r] > 0.f ? s[r] * expf(m[r] - mx) : s[r];       // (a CTA without classes of this task has sum 0)
    }
    int label = labels[b];
    if (label < 0 || label >= n) {
      if (tid == 0 && status != nullptr) atomicOr(status, STATUS_CHECK);
      label = 0;
    }
    const float inv = 1.0f / se, inv_b = 1.0f / (float)B;
    for (int c = c0 + tid; c < c1; c += HC_THREADS) {
      float gl = 0.f;
      if (c < n) {
        const float l = lg[c - c0];
        if (c == label) io.per_image[b] = logf(se) + mx - l;
        gl = (expf(l - mx) * inv - (c == label ? 1.f : 0.f)) * inv_b;
      }
      lg[c - c0] = gl;
      io.dlogits[(size_t)b * h.cmax + c] = gl;
    }
    __syncthreads();
    // this CTA's classes back through the head's weights: threads own four columns, groups of them take every groups-th class
    const int groups = HC_THREADS / d4, grp = tid / d4, gcol = (tid - grp * d4) * 4;
    if (grp < groups) {
      float a[4] = {0.f, 0.f, 0.f, 0.f};
      for (int c = c0 + grp; c < cn; c += 8 * groups) {
        float wv[8][4];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (c + u * groups < cn) load4(w + (size_t)(c + u * groups) * D + gcol, wv[u]);
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (c + u * groups < cn) {
            const float gl = lg[c + u * groups - c0];
#pragma unroll
            for (int j = 0; j < 4; ++j) a[j] = fmaf(gl, wv[u][j], a[j]);
          }
      }
      store16(part + grp * D + gcol, a);
    }
    __syncthreads();
    float dn[4] = {0.f, 0.f, 0.f, 0.f};
    if (has) {
      for (int q = 0; q < groups; ++q) {
        float pv[4];
        load16(part + q * D + col, pv);
#pragma unroll
        for (int j = 0; j < 4; ++j) dn[j] += pv[j];
      }
    }
    if (ranks > 1) {
      if (has) store16(part + col, dn);                      // (a thread rewrites what it alone has read)
      cluster.sync();
      if (rank == 0 && has) {
#pragma unroll
        for (int r = 1; r < HC_MAXRANKS; ++r)
          if (r < ranks) {
            float pv[4];
            load16(cluster.map_shared_rank(part, r) + col, pv);
#pragma unroll
            for (int j = 0; j < 4; ++j) dn[j] += pv[j];
          }
      }
      cluster.sync();                                        // no CTA leaves while another may still read its part
      if (rank != 0) return;
    }
    if (has) store16(io.dxn + (long)b * D + col, dn);
    if (io.dx == nullptr) return;
    // LayerNorm backward
    float s1 = 0.f, s2 = 0.f, dh[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      dh[j] = dn[j] * gam[j];
      s1 += dh[j];
      s2 += dh[j] * v[j];
    }
    s1 = hc_block<false>(s1, red) / (float)D;
    s2 = hc_block<false>(s2, red) / (float)D;
    if (has) {
      float o[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) o[j] = rs * (dh[j] - s1 - v[j] * s2);
      store16(io.dx + (long)b * io.x_stride + col, o);
      if (dx_copy != nullptr) store4(dx_copy + (long)b * io.x_stride + col, o);
    }
  }
}

// An image's CTAs: at least 16 classes each (10 classes 1, 40 classes 2, 100 classes 4, from 128 classes on 8, the most a cluster
// has).  In inference the CTAs exchange nothing and need no cluster: many classes of few images spread as far as eight CTAs fit an SM.  us of
// DeiT-S inference (two blocks), a cluster an image / so: 1000 classes, 1 / 64 images 86.1 / 80.6, 215 / 208; 10000 classes 144 / 82.7,
// 353 / 272; 21841 classes 219 / 84.6, 535 / 356 (to two CTAs an SM 91.0 and 516, to sixteen 84.6 and 351).
static int head_ranks(const Ctx& c, int cmax, int B, bool train) {
  int r = 1;
  while (r < HC_MAXRANKS && cmax >= r * 2 * 16) r *= 2;
  if (train || r < HC_MAXRANKS) return r;
  const int fill = 8 * (c.sm_count > 0 ? c.sm_count : B200_SMS) / B, most = ceil_div(cmax, 16);
  const int wide = fill < most ? fill : most;
  return wide > r ? wide : r;
}

void head_chain(const Ctx& c, const HeadDesc& h, const HeadRow& io, const EvalIo* eval, const int* labels, const int* task_ids, void* dx_copy, int B) {
  note_launch(1);
  const bool train = labels != nullptr;
  const int ranks = head_ranks(c, h.cmax, B, train);
  auto go = [&](auto kern, auto* copy) {
    launch_cluster(kern, dim3(B * ranks), HC_THREADS, 0, c.stream, dim3(train ? ranks : 1, 1, 1), to_dev(h), io, eval, labels, task_ids, copy, ranks, B, c.status);
  };
  if (c.dtype == 0) train ? go(head_chain_kernel<float, true>, (float*)nullptr) : go(head_chain_kernel<float, false>, (float*)nullptr);
  else train ? go(head_chain_kernel<bf16, true>, (bf16*)dx_copy) : go(head_chain_kernel<bf16, false>, (bf16*)nullptr);
}

// What the head's chain sums over the images, in image order where not said otherwise:
//   dW_t[c, d] = sum_b [task(b) = t] dlogits[b, c] xn[b, d],   db_t[c] = sum_b [..] dlogits[b, c]  (lanes stride the images)
//   dgamma[d] = sum_b dxn[b, d] xhat[b, d],   dbeta[d] = sum_b dxn[b, d]  (four warps stride the images), the mean loss (lanes stride them).
// A block forms 16 classes x 128 columns of one task, 4 x 4 sums a thread, the loads of eight images in flight (27 us for 128 images,
// 100 classes x 768, with a thread per element); the last blocks along the classes form the rest.
constexpr int HG_CLS = 16, HG_COLS = 128, HG_THREADS = 128;

__global__ void __launch_bounds__(HG_THREADS)
head_grads_kernel(HeadDev h, HeadRow io, const int* __restrict__ task_ids, float* __restrict__ dgamma, float* __restrict__ dbeta,
                  float* __restrict__ loss, float* __restrict__ loss_copy, int B, int* status) {
  dependent_sync();
  __shared__ float sm[2][HG_THREADS / 32][HG_COLS];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, D = h.D, t = blockIdx.z;
  const int col = blockIdx.y * HG_COLS + lane * 4, colr = col < D ? col : 0;
  if (blockIdx.x + 1 < gridDim.x) {
    const int n = h.ncls[t], c0 = blockIdx.x * HG_CLS + warp * 4;
    if (c0 >= n) return;
    float acc[4][4] = {};
#pragma unroll 8
    for (int b = 0; b < B; ++b) {
      const bool on = task_ids == nullptr || task_ids[b] == t;
      float x[4], gl[4];
      load16(io.xn + (size_t)b * D + colr, x);
#pragma unroll
      for (int i = 0; i < 4; ++i) gl[i] = on ? io.dlogits[(size_t)b * h.cmax + min(c0 + i, n - 1)] : 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(gl[i], x[j], acc[i][j]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (c0 + i >= n) break;
      if (col < D) store16(h.dw[t] + (size_t)(c0 + i) * D + col, acc[i]);
      if (blockIdx.y == 0) {
        float s = 0.f;
        for (int b = lane; b < B; b += 32) s += task_ids == nullptr || task_ids[b] == t ? io.dlogits[(size_t)b * h.cmax + c0 + i] : 0.f;
        s = warp_sum(s);
        if (lane == 0) h.db[t][c0 + i] = s;
      }
    }
    return;
  }
  if (t != 0) return;
  float sg[4] = {}, sb[4] = {};
#pragma unroll 8
  for (int b = warp; b < B; b += HG_THREADS / 32) {
    float dn[4], xh[4];
    load16(io.dxn + (size_t)b * D + colr, dn);
    load16(io.xhat + (size_t)b * D + colr, xh);
#pragma unroll
    for (int j = 0; j < 4; ++j) { sg[j] = fmaf(dn[j], xh[j], sg[j]); sb[j] += dn[j]; }
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) { sm[0][warp][lane * 4 + j] = sg[j]; sm[1][warp][lane * 4 + j] = sb[j]; }
  __syncthreads();
  const int out = blockIdx.y * HG_COLS + threadIdx.x;
  if (out < D) {
    float a = 0.f, s = 0.f;
#pragma unroll
    for (int q = 0; q < HG_THREADS / 32; ++q) { a += sm[0][q][threadIdx.x]; s += sm[1][q][threadIdx.x]; }
    dgamma[out] = a;
    dbeta[out] = s;
  }
  if (blockIdx.y == 0 && warp == 0) {
    float s = 0.f;
    for (int b = lane; b < B; b += 32) s += io.per_image[b];
    s = warp_sum(s);
    if (lane == 0) {
      const float l = s / (float)B;
      *loss = l;
      if (loss_copy != nullptr) *loss_copy = l;
      if (status != nullptr && !isfinite(l)) atomicOr(status, STATUS_NONFINITE);
    }
  }
}

void head_grads(const Ctx& c, const HeadDesc& h, const HeadRow& io, const int* task_ids, float* dgamma, float* dbeta, float* loss, float* loss_copy, int B) {
  note_launch(1);
  launch_k(head_grads_kernel, dim3(ceil_div(h.cmax, HG_CLS) + 1, ceil_div(h.D, HG_COLS), h.num_tasks), HG_THREADS, 0, c.stream, to_dev(h), io, task_ids,
           dgamma, dbeta, loss, loss_copy, B, c.status);
}

}  // namespace bsr
