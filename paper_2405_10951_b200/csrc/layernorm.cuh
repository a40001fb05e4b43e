// A LayerNorm row held by one warp (D <= 128 NCH, D % 4 == 0): lane l has the 16-byte chunks l, l + 32, ...
#pragma once

#include "common.cuh"

namespace bsr {

template <int NCH>
__device__ __forceinline__ void ln_load_row(const float* __restrict__ x, int D, float* v) {
  const int lane = threadIdx.x & 31, chunks = D / 4;
#pragma unroll
  for (int i = 0; i < NCH; ++i) {
    int ch = lane + i * 32;
    if (ch < chunks) load16(x + ch * 4, v + i * 4);
  }
}

// y = (x - mean) rstd g + b; mean and rstd (optional) receive the row's statistics.
template <typename TY, int NCH>
__device__ __forceinline__ void ln_write_row(const float* v, const float* __restrict__ g, const float* __restrict__ b, TY* __restrict__ y,
                                             float* mean, float* rstd, int D, float eps) {
  const int lane = threadIdx.x & 31, chunks = D / 4;
  float sum = 0.f;
#pragma unroll
  for (int i = 0; i < NCH; ++i) {
    if (lane + i * 32 < chunks) {
#pragma unroll
      for (int j = 0; j < 4; ++j) sum += v[i * 4 + j];
    }
  }
  float mu = warp_sum(sum) / (float)D;
  float sq = 0.f;
#pragma unroll
  for (int i = 0; i < NCH; ++i) {
    if (lane + i * 32 < chunks) {
#pragma unroll
      for (int j = 0; j < 4; ++j) { float t = v[i * 4 + j] - mu; sq += t * t; }
    }
  }
  float rs = rsqrtf(warp_sum(sq) / (float)D + eps);
  if (lane == 0) {
    if (mean) *mean = mu;
    if (rstd) *rstd = rs;
  }
#pragma unroll
  for (int i = 0; i < NCH; ++i) {
    int ch = lane + i * 32;
    if (ch < chunks) {
      float4 gg = *reinterpret_cast<const float4*>(g + ch * 4), bb = *reinterpret_cast<const float4*>(b + ch * 4);
      float o[4];
      o[0] = (v[i * 4 + 0] - mu) * rs * gg.x + bb.x;
      o[1] = (v[i * 4 + 1] - mu) * rs * gg.y + bb.y;
      o[2] = (v[i * 4 + 2] - mu) * rs * gg.z + bb.z;
      o[3] = (v[i * 4 + 3] - mu) * rs * gg.w + bb.w;
      store4(y + ch * 4, o);
    }
  }
}

}  // namespace bsr
