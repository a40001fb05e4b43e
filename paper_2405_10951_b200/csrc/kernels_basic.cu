// Bandwidth-bound kernels of the BSR step: patch extraction, token assembly, LayerNorm forward and
// backward, column sums, AdamW, conversions.  All reductions run in a fixed order.
#include "common.cuh"
#include "kernels.h"
#include "layernorm.cuh"

namespace bsr {

long g_kernel_launches = 0;

// ------------------------------------------------------------------------------------------------
// Patch extraction (Section 3.1: the image is partitioned into N patches).  Output row = one patch
// flattened as (channel, row in patch, column in patch).
// ------------------------------------------------------------------------------------------------
// img_offset (optional): element offset of this step's images from `img`, read from device memory (multi-step loop).
template <typename T>
__global__ void patchify_kernel(const T* __restrict__ img, T* __restrict__ out, int B, int C, int S, int P, long total,
                                const long long* __restrict__ img_offset) {
  dependent_sync();
  long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total) return;
  if (img_offset != nullptr) img += *img_offset;
  int g = S / P;
  int px = (int)(i % P); long r = i / P;
  int py = (int)(r % P); r /= P;
  int ch = (int)(r % C); r /= C;
  int gx = (int)(r % g); r /= g;
  int gy = (int)(r % g); r /= g;
  int b = (int)r;
  out[i] = img[(((long)b * C + ch) * S + (gy * P + py)) * S + gx * P + px];
}

// Same copy in 16-byte units (P * sizeof(T) a multiple of 16): a patch row is P/E units.
template <typename T>
__global__ void patchify_vec_kernel(const T* __restrict__ img, T* __restrict__ out, int B, int C, int S, int P, long units,
                                    const long long* __restrict__ img_offset) {
  dependent_sync();
  constexpr int E = 16 / sizeof(T);
  long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= units) return;
  if (img_offset != nullptr) img += *img_offset;
  int g = S / P, upr = P / E;
  int ux = (int)(i % upr); long r = i / upr;
  int py = (int)(r % P); r /= P;
  int ch = (int)(r % C); r /= C;
  int gx = (int)(r % g); r /= g;
  int gy = (int)(r % g); r /= g;
  int b = (int)r;
  const T* src = img + (((long)b * C + ch) * S + (gy * P + py)) * S + gx * P + ux * E;
  *reinterpret_cast<uint4*>(out + i * E) = *reinterpret_cast<const uint4*>(src);
}

void patchify(const Ctx& c, const void* images, void* patches, int B, int C, int S, int P, const long long* img_offset) {
  note_launch(1);
  int g = S / P;
  long total = (long)B * g * g * C * P * P;
  int threads = 256;
  size_t es = dtype_size(c.dtype);
  // with an offset read on the device, every step's images must be 16-byte aligned: one image holds C*S*S elements
  bool vec = (P * es) % 16 == 0 && (((uintptr_t)images | (uintptr_t)patches) & 15) == 0 &&
             (img_offset == nullptr || ((long)C * S * S * (long)es) % 16 == 0);
  if (vec) {
    long units = total * (long)es / 16;
    int blocks = ceil_div(units, threads);
    if (c.dtype == 0) launch_k(patchify_vec_kernel<float>, blocks, threads, 0, c.stream, (const float*)images, (float*)patches, B, C, S, P, units, img_offset);
    else launch_k(patchify_vec_kernel<bf16>, blocks, threads, 0, c.stream, (const bf16*)images, (bf16*)patches, B, C, S, P, units, img_offset);
    return;
  }
  int blocks = ceil_div(total, threads);
  if (c.dtype == 0)
    launch_k(patchify_kernel<float>, blocks, threads, 0, c.stream, (const float*)images, (float*)patches, B, C, S, P, total, img_offset);
  else
    launch_k(patchify_kernel<bf16>, blocks, threads, 0, c.stream, (const bf16*)images, (bf16*)patches, B, C, S, P, total, img_offset);
}

// x[b, 0] = cls + pos[0];  x[b, 1 + n] = emb[b, n] + pos[1 + n]   (classification token and positional embedding);
// four columns per thread (D % 4 == 0).
template <typename T>
__global__ void assemble_kernel(const T* __restrict__ emb, const float* __restrict__ cls, const float* __restrict__ pos,
                                float* __restrict__ x, int B, int N, int D, long total4) {
  dependent_sync();
  long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total4) return;
  int d4 = D / 4;
  int d = (int)(i % d4) * 4; long r = i / d4;
  int t = (int)(r % (N + 1));
  int b = (int)(r / (N + 1));
  float v[4], p[4];
  if (t == 0) load16(cls + d, v);
  else load4(emb + ((long)b * N + (t - 1)) * D + d, v);
  load16(pos + (long)t * D + d, p);
#pragma unroll
  for (int j = 0; j < 4; ++j) v[j] += p[j];
  store16(x + i * 4, v);
}

void assemble_tokens(const Ctx& c, const void* emb, const float* cls, const float* pos, float* x, int B, int N, int D) {
  note_launch(1);
  long total4 = (long)B * (N + 1) * D / 4;
  int threads = 256, blocks = ceil_div(total4, threads);
  if (c.dtype == 0)
    launch_k(assemble_kernel<float>, blocks, threads, 0, c.stream, (const float*)emb, cls, pos, x, B, N, D, total4);
  else
    launch_k(assemble_kernel<bf16>, blocks, threads, 0, c.stream, (const bf16*)emb, cls, pos, x, B, N, D, total4);
}

// ------------------------------------------------------------------------------------------------
// LayerNorm.  The residual stream x is float in every configuration (only the small block updates
// would survive bf16 rounding of the stream poorly); the normalised output feeds a GEMM and takes
// the storage dtype.  One warp per row, the row held in registers (D <= 1024, D % 4 == 0).
// ------------------------------------------------------------------------------------------------
// NCH = 16-byte chunks of the row each lane holds (D <= 128 * NCH); instantiated for 2, 3, 4, 6 and 8.

template <typename TY, int NCH>
__global__ void layernorm_fwd_kernel(const float* __restrict__ x, const float* __restrict__ g,
                                     const float* __restrict__ b, TY* __restrict__ y, float* __restrict__ mean,
                                     float* __restrict__ rstd, int rows, int D, float eps) {
  dependent_sync();
  int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (warp >= rows) return;
  float v[NCH * 4];
  ln_load_row<NCH>(x + (long)warp * D, D, v);
  ln_write_row<TY, NCH>(v, g, b, y + (long)warp * D, mean ? mean + warp : nullptr, rstd ? rstd + warp : nullptr, D, eps);
}

template <typename TY>
static void launch_ln_fwd(const Ctx& c, const float* x, const float* g, const float* b, TY* y, float* mean,
                          float* rstd, int rows, int D, float eps) {
  int threads = 256;
  int blocks = ceil_div((long)rows * 32, threads);
  int nch = ceil_div(D, 128);
#define BSR_LN_FWD(N) launch_k(layernorm_fwd_kernel<TY, N>, blocks, threads, 0, c.stream, x, g, b, y, mean, rstd, rows, D, eps)
  if (nch <= 2) BSR_LN_FWD(2); else if (nch == 3) BSR_LN_FWD(3); else if (nch == 4) BSR_LN_FWD(4); else if (nch <= 6) BSR_LN_FWD(6); else BSR_LN_FWD(8);
#undef BSR_LN_FWD
}

void layernorm_fwd(const Ctx& c, const float* x, const float* g, const float* b, void* y, float* mean, float* rstd, int rows, int D,
                   float eps) {
  note_launch(1);
  if (c.dtype == 0) launch_ln_fwd<float>(c, x, g, b, (float*)y, mean, rstd, rows, D, eps);
  else launch_ln_fwd<bf16>(c, x, g, b, (bf16*)y, mean, rstd, rows, D, eps);
}

// ------------------------------------------------------------------------------------------------
// E4M3 (8-bit floating point: 1 sign, 4 exponent, 3 mantissa bits, largest magnitude 448) rows with one scale each.
// ------------------------------------------------------------------------------------------------
// Two floats to two E4M3 bytes, round to nearest even, saturating; a in the low byte.
__device__ __forceinline__ uint16_t to_e4m3x2(float a, float b) {
  uint16_t r;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(b), "f"(a));
  return r;
}
__device__ __forceinline__ uint32_t to_e4m3x4(const float* v, float s) {
  return (uint32_t)to_e4m3x2(__fdiv_rn(v[0], s), __fdiv_rn(v[1], s)) | ((uint32_t)to_e4m3x2(__fdiv_rn(v[2], s), __fdiv_rn(v[3], s)) << 16);
}
__device__ __forceinline__ float e4m3_scale(float amax) { return amax > 0.f ? __fdiv_rn(amax, 448.0f) : 1.0f; }

// One warp per row (cols % 4 == 0): scale = max|row| / 448, q = round(x / scale).
__global__ void quantize_rows_e4m3_kernel(const bf16* __restrict__ x, int rows, int cols, uint8_t* __restrict__ q, float* __restrict__ scale) {
  dependent_sync();
  int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (warp >= rows) return;
  const bf16* xr = x + (size_t)warp * cols;
  float amax = 0.f;
  for (int ch = lane; ch < cols / 4; ch += 32) {
    float v[4];
    load4(xr + ch * 4, v);
#pragma unroll
    for (int j = 0; j < 4; ++j) amax = fmaxf(amax, fabsf(v[j]));
  }
  amax = warp_max(amax);
  float s = e4m3_scale(amax);
  if (lane == 0) scale[warp] = s;
  uint32_t* qr = reinterpret_cast<uint32_t*>(q + (size_t)warp * cols);
  for (int ch = lane; ch < cols / 4; ch += 32) {
    float v[4];
    load4(xr + ch * 4, v);
    qr[ch] = to_e4m3x4(v, s);
  }
}
void quantize_rows_e4m3(const Ctx& c, const void* x, int rows, int cols, void* q, float* scale) {
  note_launch(1);
  launch_k(quantize_rows_e4m3_kernel, ceil_div((long)rows * 32, 256), 256, 0, c.stream, (const bf16*)x, rows, cols, (uint8_t*)q, scale);
}

// E4M3 byte to float: sign, exponent (bias 7) and mantissa unpacked by hand (subnormals: exponent field 0).
__device__ __forceinline__ float from_e4m3(uint8_t b) {
  int e = (b >> 3) & 15, m = b & 7;
  float v = e == 0 ? (float)m * 0.001953125f : ldexpf(1.0f + (float)m * 0.125f, e - 7);
  return (b & 0x80) ? -v : v;
}
__global__ void dequantize_rows_e4m3_kernel(const uint8_t* __restrict__ q, const float* __restrict__ scale, int rows, int cols,
                                            float* __restrict__ out) {
  dependent_sync();
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (size_t)rows * cols) return;
  out[i] = from_e4m3(q[i]) * scale[i / cols];
}
void dequantize_rows_e4m3(const Ctx& c, const void* q, const float* scale, int rows, int cols, float* out) {
  note_launch(1);
  launch_k(dequantize_rows_e4m3_kernel, ceil_div((long)rows * cols, 256), 256, 0, c.stream, (const uint8_t*)q, scale, rows, cols, out);
}

// LayerNorm forward whose output row goes out as E4M3 with scale max|y| / 448: the row is already in the warp's
// registers, so the quantisation costs one more warp reduction and halves the bytes written.
template <int NCH>
__global__ void layernorm_fwd_e4m3_kernel(const float* __restrict__ x, long x_stride, const float* __restrict__ g,
                                          const float* __restrict__ b, uint8_t* __restrict__ yq, float* __restrict__ y_scale,
                                          int rows, int D, float eps) {
  dependent_sync();
  int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int lane = threadIdx.x & 31;
  if (warp >= rows) return;
  const float* xr = x + (long)warp * x_stride;
  int chunks = D / 4;
  float v[(NCH * 4)];
  float sum = 0.f;
#pragma unroll
  for (int i = 0; i < NCH; ++i) {
    int ch = lane + i * 32;
    if (ch < chunks) {
      load16(xr + ch * 4, v + i * 4);
#pragma unroll
      for (int j = 0; j < 4; ++j) sum += v[i * 4 + j];
    }
  }
  float mu = warp_sum(sum) / (float)D;
  float sq = 0.f;
#pragma unroll
  for (int i = 0; i < NCH; ++i) {
    int ch = lane + i * 32;
    if (ch < chunks) {
#pragma unroll
      for (int j = 0; j < 4; ++j) { float t = v[i * 4 + j] - mu; sq += t * t; }
    }
  }
  float rs = rsqrtf(warp_sum(sq) / (float)D + eps);
  float amax = 0.f;
#pragma unroll
  for (int i = 0; i < NCH; ++i) {
    int ch = lane + i * 32;
    if (ch < chunks) {
      float4 gg = *reinterpret_cast<const float4*>(g + ch * 4), bb = *reinterpret_cast<const float4*>(b + ch * 4);
      v[i * 4 + 0] = (v[i * 4 + 0] - mu) * rs * gg.x + bb.x;
      v[i * 4 + 1] = (v[i * 4 + 1] - mu) * rs * gg.y + bb.y;
      v[i * 4 + 2] = (v[i * 4 + 2] - mu) * rs * gg.z + bb.z;
      v[i * 4 + 3] = (v[i * 4 + 3] - mu) * rs * gg.w + bb.w;
#pragma unroll
      for (int j = 0; j < 4; ++j) amax = fmaxf(amax, fabsf(v[i * 4 + j]));
    }
  }
  amax = warp_max(amax);
  float s = e4m3_scale(amax);
  if (lane == 0) y_scale[warp] = s;
  uint32_t* qr = reinterpret_cast<uint32_t*>(yq + (size_t)warp * D);
#pragma unroll
  for (int i = 0; i < NCH; ++i) {
    int ch = lane + i * 32;
    if (ch < chunks) qr[ch] = to_e4m3x4(v + i * 4, s);
  }
}
void layernorm_fwd_e4m3(const Ctx& c, const float* x, long x_stride, const float* g, const float* b, void* yq, float* y_scale,
                        int rows, int D, float eps) {
  note_launch(1);
  int threads = 256;
  int blocks = ceil_div((long)rows * 32, threads);
  int nch = ceil_div(D, 128);
#define BSR_LN_Q(N) launch_k(layernorm_fwd_e4m3_kernel<N>, blocks, threads, 0, c.stream, x, x_stride, g, b, (uint8_t*)yq, y_scale, rows, D, eps)
  if (nch <= 2) BSR_LN_Q(2); else if (nch == 3) BSR_LN_Q(3); else if (nch == 4) BSR_LN_Q(4); else if (nch <= 6) BSR_LN_Q(6); else BSR_LN_Q(8);
#undef BSR_LN_Q
}

// Backward.  Each block owns rows blockIdx.x*8 + warp, stepping by gridDim.x*8; every lane accumulates the
// dgamma/dbeta contributions of its columns, warps are combined through shared memory in warp order, and the
// block's sums go to partials[0][block][col] (dgamma) and partials[1][block][col] (dbeta).
// dx (float, the gradient of the residual stream) = dres + LN'(dy); dx_copy receives the same values in the
// storage dtype for the GEMMs that consume them.
constexpr int LNB_WARPS = 8;

template <typename T, int NCH>
__global__ void __launch_bounds__(256, 2) layernorm_bwd_kernel(const T* __restrict__ dy, const float* __restrict__ x,
                                     const float* __restrict__ mean, const float* __restrict__ rstd,
                                     const float* __restrict__ g, const float* __restrict__ dres, int dres_period, float* __restrict__ dx,
                                     T* __restrict__ dx_copy, float* __restrict__ partials, int rows, int D, int nsum) {
  dependent_sync();
  extern __shared__ float sm[];   // [LNB_WARPS][nsum][D]: dgamma, dbeta and (nsum == 3) the column sums of dx
  int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int chunks = D / 4;
  // The warp's partial sums for the scale and shift gradients live in its slice of shared memory (each lane owns
  // its columns), which leaves the registers for a whole row of x, dy and the residual gradient in flight at once.
  float* mine = sm + (size_t)warp * nsum * D;
#pragma unroll
  for (int i = 0; i < NCH; ++i) {
    int ch = lane + i * 32;
    if (ch < chunks) {
      *reinterpret_cast<float4*>(mine + ch * 4) = make_float4(0.f, 0.f, 0.f, 0.f);
      *reinterpret_cast<float4*>(mine + D + ch * 4) = make_float4(0.f, 0.f, 0.f, 0.f);
      if (nsum == 3) *reinterpret_cast<float4*>(mine + 2 * D + ch * 4) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  for (int r = blockIdx.x * LNB_WARPS + warp; r < rows; r += gridDim.x * LNB_WARPS) {
    const float* xr = x + (long)r * D;
    const T* dyr = dy + (long)r * D;
    const int rr = r / dres_period;
    const float* res = dx != nullptr && dres != nullptr && rr * dres_period == r ? dres + (long)rr * D : nullptr;
    float mu = mean[r], rs = rstd[r];
    float xh[(NCH * 4)], dh[(NCH * 4)], o[(NCH * 4)];
#pragma unroll
    for (int i = 0; i < NCH; ++i) {                      // all loads of the row first
      int ch = lane + i * 32;
      if (ch < chunks) {
        load16(xr + ch * 4, xh + i * 4);
        load4(dyr + ch * 4, dh + i * 4);
        if (res != nullptr) load16(res + ch * 4, o + i * 4);
        else {
#pragma unroll
          for (int j = 0; j < 4; ++j) o[i * 4 + j] = 0.f;
        }
      }
    }
    float s1 = 0.f, s2 = 0.f;
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
      int ch = lane + i * 32;
      if (ch < chunks) {
        float4 gg = *reinterpret_cast<const float4*>(g + ch * 4);
        float gv[4] = {gg.x, gg.y, gg.z, gg.w};
        float4 pg = *reinterpret_cast<const float4*>(mine + ch * 4);
        float4 pb = *reinterpret_cast<const float4*>(mine + D + ch * 4);
        float pgv[4] = {pg.x, pg.y, pg.z, pg.w}, pbv[4] = {pb.x, pb.y, pb.z, pb.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float d = dh[i * 4 + j];
          float h = (xh[i * 4 + j] - mu) * rs;
          xh[i * 4 + j] = h;
          pgv[j] += d * h;
          pbv[j] += d;
          float dxh = d * gv[j];
          dh[i * 4 + j] = dxh;
          s1 += dxh;
          s2 += dxh * h;
        }
        *reinterpret_cast<float4*>(mine + ch * 4) = make_float4(pgv[0], pgv[1], pgv[2], pgv[3]);
        *reinterpret_cast<float4*>(mine + D + ch * 4) = make_float4(pbv[0], pbv[1], pbv[2], pbv[3]);
      }
    }
    s1 = warp_sum(s1) / (float)D;
    s2 = warp_sum(s2) / (float)D;
    if (dx != nullptr) {
      float* dxr = dx + (long)r * D;
#pragma unroll
      for (int i = 0; i < NCH; ++i) {
        int ch = lane + i * 32;
        if (ch < chunks) {
#pragma unroll
          for (int j = 0; j < 4; ++j) o[i * 4 + j] += rs * (dh[i * 4 + j] - s1 - xh[i * 4 + j] * s2);
          store16(dxr + ch * 4, o + i * 4);
          if (dx_copy != nullptr) store4(dx_copy + (long)r * D + ch * 4, o + i * 4);
          if (nsum == 3) {
            float4 ps = *reinterpret_cast<const float4*>(mine + 2 * D + ch * 4);
            ps.x += o[i * 4]; ps.y += o[i * 4 + 1]; ps.z += o[i * 4 + 2]; ps.w += o[i * 4 + 3];
            *reinterpret_cast<float4*>(mine + 2 * D + ch * 4) = ps;
          }
        }
      }
    }
  }
  __syncthreads();
  for (int col = threadIdx.x; col < nsum * D; col += blockDim.x) {
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < LNB_WARPS; ++w) s += sm[(size_t)w * nsum * D + col];
    int which = col / D, cc = col % D;
    partials[((size_t)which * gridDim.x + blockIdx.x) * D + cc] = s;
  }
}

// out_y[col] = sum over groups of partials[y][group][col] for y = blockIdx.y (one or two outputs per launch).
// 16 lanes stride the groups and are combined through shared memory in lane order: the result is deterministic.
__global__ void reduce_partials_kernel(const float* __restrict__ partials, int groups, int cols, float* __restrict__ out0,
                                       float* __restrict__ out1, float* __restrict__ out2) {
  dependent_sync();
  __shared__ float sm[16][17];
  int cx = threadIdx.x & 15, gy = threadIdx.x >> 4;
  int col = blockIdx.x * 16 + cx;
  const float* p = partials + (size_t)blockIdx.y * groups * cols;
  float s = 0.f;
  if (col < cols)
    for (int g = gy; g < groups; g += 16) s += p[(size_t)g * cols + col];
  sm[gy][cx] = s;
  __syncthreads();
  if (gy == 0 && col < cols) {
    float t = 0.f;
#pragma unroll
    for (int i = 0; i < 16; ++i) t += sm[i][cx];
    float* out = blockIdx.y == 0 ? out0 : (blockIdx.y == 1 ? out1 : out2);
    if (out != nullptr) out[col] = t;
  }
}

int layernorm_bwd_groups(const Ctx& c, int rows) {
  int want = ceil_div(rows, LNB_WARPS);
  int cap = c.sm_count > 0 ? 2 * c.sm_count : 296;
  return want < cap ? (want < 1 ? 1 : want) : cap;
}

template <typename T>
static void launch_ln_bwd(const Ctx& c, int groups, size_t smem, const void* dy, const float* x, const float* mean, const float* rstd,
                          const float* g, const float* dres, int dres_period, float* dx, void* dx_copy, float* partials, int rows, int D, int nsum) {
  int nch = ceil_div(D, 128);
#define BSR_LN_BWD(N)                                                                                                   \
  do {                                                                                                                  \
    static SmemLimit lim;                                                                                               \
    ensure_smem(lim, layernorm_bwd_kernel<T, N>, smem);                                                                 \
    launch_k(layernorm_bwd_kernel<T, N>, groups, LNB_WARPS * 32, smem, c.stream, (const T*)dy, x, mean, rstd, g, dres, dres_period, \
                                                                           dx, (T*)dx_copy, partials, rows, D, nsum);   \
  } while (0)
  if (nch <= 2) BSR_LN_BWD(2); else if (nch == 3) BSR_LN_BWD(3); else if (nch == 4) BSR_LN_BWD(4); else if (nch <= 6) BSR_LN_BWD(6); else BSR_LN_BWD(8);
#undef BSR_LN_BWD
}

void layernorm_bwd(const Ctx& c, const void* dy, const float* x, const float* mean, const float* rstd, const float* g, const float* dres,
                   int dres_period, float* dx, void* dx_copy, float* partials, float* dgamma, float* dbeta, int rows, int D, float* dx_colsum) {
  note_launch(2);
  int groups = layernorm_bwd_groups(c, rows);
  int nsum = (dx_colsum != nullptr && dx != nullptr) ? 3 : 2;
  size_t smem = (size_t)LNB_WARPS * nsum * D * sizeof(float);
  side_join(c, 0);                                                     // the previous reduction has read the partials
  if (c.dtype == 0) launch_ln_bwd<float>(c, groups, smem, dy, x, mean, rstd, g, dres, dres_period, dx, nullptr, partials, rows, D, nsum);
  else launch_ln_bwd<bf16>(c, groups, smem, dy, x, mean, rstd, g, dres, dres_period, dx, dx_copy, partials, rows, D, nsum);
  if (dgamma == nullptr && nsum == 2) return;                          // a frozen block in the gradient path: only dx is wanted
  dim3 grid(ceil_div(D, 16), nsum);
  cudaStream_t rs = side_begin(c);                                     // only the optimiser reads these sums
  launch_k(reduce_partials_kernel, grid, 256, 0, rs, partials, groups, D, dgamma, dbeta, nsum == 3 ? dx_colsum : nullptr);
  side_end(c, 0);
}

// ------------------------------------------------------------------------------------------------
// Column sums (bias gradients): two stages, fixed order.
// ------------------------------------------------------------------------------------------------
constexpr int CS_ROWLANES = 8;
constexpr int CS_GROUPS = 64;

template <typename T>
__global__ void colsum_kernel(const T* __restrict__ x, int rows, int cols, float* __restrict__ partials) {
  dependent_sync();
  constexpr int N = Pack<T>::N;
  __shared__ float sm[CS_ROWLANES][32 * N];
  int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  int col0 = (blockIdx.x * 32 + tx) * N;
  float acc[N];
#pragma unroll
  for (int j = 0; j < N; ++j) acc[j] = 0.f;
  if (col0 < cols) {
    // four rows per trip: their loads are independent and issued together, the additions keep the row order
    const int step = gridDim.y * CS_ROWLANES;
    int r = blockIdx.y * CS_ROWLANES + ty;
    for (; r + 3 * step < rows; r += 4 * step) {
      float v[4][N];
#pragma unroll
      for (int u = 0; u < 4; ++u) load16(x + (long)(r + u * step) * cols + col0, v[u]);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
#pragma unroll
        for (int j = 0; j < N; ++j) acc[j] += v[u][j];
      }
    }
    for (; r < rows; r += step) {
      float v[N];
      load16(x + (long)r * cols + col0, v);
#pragma unroll
      for (int j = 0; j < N; ++j) acc[j] += v[j];
    }
  }
#pragma unroll
  for (int j = 0; j < N; ++j) sm[ty][tx * N + j] = acc[j];
  __syncthreads();
  for (int cidx = threadIdx.x; cidx < 32 * N; cidx += blockDim.x) {
    int col = blockIdx.x * 32 * N + cidx;
    if (col < cols) {
      float s = 0.f;
#pragma unroll
      for (int w = 0; w < CS_ROWLANES; ++w) s += sm[w][cidx];
      partials[(size_t)blockIdx.y * cols + col] = s;
    }
  }
}

int colsum_groups(int rows) {
  int want = ceil_div(rows, CS_ROWLANES);
  return want < CS_GROUPS ? (want < 1 ? 1 : want) : CS_GROUPS;
}

void colsum(const Ctx& c, const void* x, int rows, int cols, float* partials, float* out) {
  note_launch(2);
  int groups = colsum_groups(rows);
  int threads = CS_ROWLANES * 32;
  side_join(c, 1);
  if (c.dtype == 0) {
    dim3 grid(ceil_div(cols, 32 * 4), groups);
    launch_k(colsum_kernel<float>, grid, threads, 0, c.stream, (const float*)x, rows, cols, partials);
  } else {
    dim3 grid(ceil_div(cols, 32 * 8), groups);
    launch_k(colsum_kernel<bf16>, grid, threads, 0, c.stream, (const bf16*)x, rows, cols, partials);
  }
  cudaStream_t rs = side_begin(c);
  launch_k(reduce_partials_kernel, dim3(ceil_div(cols, 16), 1), 256, 0, rs, partials, groups, cols, out, out, nullptr);
  side_end(c, 1);
}

// ------------------------------------------------------------------------------------------------
// AdamW over the flat trainable-parameter buffers (Section 5: DeiT-S is trained with AdamW).
//   m <- b1 m + (1-b1) g;  v <- b2 v + (1-b2) g^2;  p <- p - lr * (m/bc1) / (sqrt(v/bc2) + eps) - lr * wd * p
// One block per chunk; a chunk never straddles two tensors.
// ------------------------------------------------------------------------------------------------
// Bound by DRAM: 26 bytes an element with a float copy only, 30 with a bf16 one.  16-byte accesses, the loads of two groups
// before the first store, and evict-first hints: the optimiser's state is not read again before the next update, and the
// weights and activations of a small batch stay in L2 (DeiT-S, one image: 732 -> 722 us a step).  Blocks walk the chunk
// table, so that a launch of UPDATE_BESIDE blocks an SM moves data without taking the slots of the kernels it runs beside
// (one block an SM leaves the update behind: ViT-B, 128 images 5826 -> 5926 us against 5860 with three);
// alone the update gets UPDATE_ALONE blocks an SM.
constexpr int UPDATE_BESIDE = 3, UPDATE_ALONE = 6;

// A rule reads N values an element: parameter, gradient, and the optimiser's state, which it replaces.
struct AdamRule {
  static constexpr int N = 4;
  float *p, *s0, *s1;
  const float* g;
  float lr, bc1, bc2, b1, b2, eps, wd;
  __device__ __forceinline__ void operator()(float* x, bool decays) const {
    x[2] = b1 * x[2] + (1.f - b1) * x[1];
    x[3] = b2 * x[3] + (1.f - b2) * x[1] * x[1];
    x[0] = x[0] - lr * (x[2] / bc1) / (sqrtf(x[3] / bc2) + eps) - (decays ? lr * wd : 0.f) * x[0];
  }
};

// SGD with momentum: buf <- mu buf + (g + wd p), p <- p - lr buf.
struct SgdRule {
  static constexpr int N = 3;
  float *p, *s0, *s1;
  const float* g;
  float lr, mu, wd;
  __device__ __forceinline__ void operator()(float* x, bool decays) const {
    x[2] = mu * x[2] + (x[1] + (decays ? wd : 0.f) * x[0]);
    x[0] = x[0] - lr * x[2];
  }
};

template <typename T, typename Rule>
__device__ __forceinline__ void update_chunks(const AdamChunk* __restrict__ chunks, int nchunks, const Rule& rule, T* __restrict__ shadow_base) {
  constexpr int U = 2;
  float* const arr[4] = {rule.p, const_cast<float*>(rule.g), rule.s0, rule.s1};
  for (int c = blockIdx.x; c < nchunks; c += gridDim.x) {
    const AdamChunk ch = chunks[c];
    const uint32_t full = ch.count & ~3u, pitch = blockDim.x * 4;
    for (uint32_t i0 = threadIdx.x * 4; i0 < full; i0 += U * pitch) {
      float4 x[U][Rule::N];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (i0 + u * pitch < full)
#pragma unroll
          for (int a = 0; a < Rule::N; ++a) x[u][a] = __ldcs(reinterpret_cast<const float4*>(arr[a] + ch.offset + i0 + u * pitch));
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint32_t i = i0 + u * pitch;
        if (i >= full) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float e[4];
#pragma unroll
          for (int a = 0; a < Rule::N; ++a) e[a] = reinterpret_cast<const float*>(&x[u][a])[j];
          rule(e, ch.decay != 0);
#pragma unroll
          for (int a = 0; a < Rule::N; ++a) reinterpret_cast<float*>(&x[u][a])[j] = e[a];
        }
#pragma unroll
        for (int a = 0; a < Rule::N; ++a)
          if (a != 1) __stcs(reinterpret_cast<float4*>(arr[a] + ch.offset + i), x[u][a]);
        if (ch.shadow >= 0) store4(shadow_base + ch.shadow + i, reinterpret_cast<const float*>(&x[u][0]));
      }
    }
    for (uint32_t i = full + threadIdx.x; i < ch.count; i += blockDim.x) {
      float e[4];
#pragma unroll
      for (int a = 0; a < Rule::N; ++a) e[a] = arr[a][(size_t)ch.offset + i];
      rule(e, ch.decay != 0);
#pragma unroll
      for (int a = 0; a < Rule::N; ++a)
        if (a != 1) arr[a][(size_t)ch.offset + i] = e[a];
      if (ch.shadow >= 0) shadow_base[ch.shadow + i] = from_f<T>(e[0]);
    }
  }
}

// Step-dependent scalars live in device memory so that a captured graph of the step stays valid: lr, 1-b1^t, 1-b2^t.
template <typename T>
__global__ void __launch_bounds__(256)
adamw_kernel(const AdamChunk* chunks, int nchunks, AdamRule rule, T* shadow_base, const float* scalars) {
  dependent_sync();
  rule.lr = scalars[0];
  rule.bc1 = scalars[1];
  rule.bc2 = scalars[2];
  update_chunks(chunks, nchunks, rule, shadow_base);
}

template <typename T>
__global__ void __launch_bounds__(256)
sgd_kernel(const AdamChunk* chunks, int nchunks, SgdRule rule, T* shadow_base, const float* scalars) {
  dependent_sync();
  rule.lr = scalars[0];
  update_chunks(chunks, nchunks, rule, shadow_base);
}

static int update_blocks(const Ctx& c, int nchunks, bool beside) {
  const int cap = (c.sm_count > 0 ? c.sm_count : B200_SMS) * (beside ? UPDATE_BESIDE : UPDATE_ALONE);
  return nchunks < cap ? nchunks : cap;
}

void sgd_momentum(const Ctx& c, const AdamChunk* chunks, int nchunks, bool beside, float* master, const float* grad, float* buf,
                  void* shadow_base, const float* scalars, float mu, float wd) {
  if (nchunks <= 0) return;
  note_launch(1);
  const int blocks = update_blocks(c, nchunks, beside);
  const SgdRule rule = {master, buf, nullptr, grad, 0.f, mu, wd};
  if (c.dtype == 0) launch_k(sgd_kernel<float>, blocks, 256, 0, c.stream, chunks, nchunks, rule, (float*)shadow_base, scalars);
  else launch_k(sgd_kernel<bf16>, blocks, 256, 0, c.stream, chunks, nchunks, rule, (bf16*)shadow_base, scalars);
}

// ------------------------------------------------------------------------------------------------
// Multi-step loop (Section 5: cosine learning-rate decay).  The state lives in device memory; each step's graph reads
// it, so a run of steps needs no host scalars: lr(t) = lr_min + (lr_max - lr_min) (1 + cos(pi t / total)) / 2 for the
// t-th step overall (t from 0, held at lr_min from t = total on), bias corrections 1 - beta^(t+1).
// ------------------------------------------------------------------------------------------------
__global__ void loop_init_kernel(LoopState* st, long long step_done, long long total, long long image_stride, float lr_max,
                                 float lr_min, float b1, float b2, int n) {
  dependent_sync();
  st->step_done = step_done; st->total_steps = total; st->image_stride = image_stride; st->image_offset = 0;
  st->lr_max = lr_max; st->lr_min = lr_min; st->beta1 = b1; st->beta2 = b2; st->i = 0; st->n = n;
}
__global__ void loop_begin_kernel(LoopState* st, float* scalars, const int* __restrict__ labels, const int* __restrict__ tasks,
                                  int* __restrict__ lab_stage, int* __restrict__ task_stage, int batch) {
  dependent_sync();
  int i = st->i;
  for (int j = threadIdx.x; j < batch; j += blockDim.x) {
    lab_stage[j] = labels[(long)i * batch + j];
    if (tasks != nullptr) task_stage[j] = tasks[(long)i * batch + j];
  }
  if (threadIdx.x == 0) {
    long long t = st->step_done;
    double frac = st->total_steps > 0 ? (double)(t < st->total_steps ? t : st->total_steps) / (double)st->total_steps : 1.0;
    double lr = (double)st->lr_min + 0.5 * ((double)st->lr_max - (double)st->lr_min) * (1.0 + cos(3.14159265358979323846 * frac));
    scalars[0] = (float)lr;
    scalars[1] = (float)(1.0 - pow((double)st->beta1, (double)(t + 1)));
    scalars[2] = (float)(1.0 - pow((double)st->beta2, (double)(t + 1)));
    st->image_offset = (long long)i * st->image_stride;
  }
}
__global__ void loop_end_kernel(LoopState* st, const float* __restrict__ loss, float* __restrict__ loss_out) {
  dependent_sync();
  loss_out[st->i] = *loss;
  st->i += 1;
  st->step_done += 1;
}
void loop_init(cudaStream_t s, LoopState* st, long long step_done, long long total, long long image_stride, float lr_max, float lr_min,
               float b1, float b2, int n) {
  note_launch(1);
  launch_k(loop_init_kernel, 1, 1, 0, s, st, step_done, total, image_stride, lr_max, lr_min, b1, b2, n);
}
void loop_begin(cudaStream_t s, LoopState* st, float* scalars, const int* labels, const int* tasks, int* lab_stage, int* task_stage, int batch) {
  note_launch(1);
  launch_k(loop_begin_kernel, 1, 256, 0, s, st, scalars, labels, tasks, lab_stage, task_stage, batch);
}
void loop_end(cudaStream_t s, LoopState* st, const float* loss, float* loss_out) {
  note_launch(1);
  launch_k(loop_end_kernel, 1, 1, 0, s, st, loss, loss_out);
}

__global__ void eval_begin_kernel(EvalIo* io, EvalIo value, const int* __restrict__ tasks, int* __restrict__ task_stage, int batch) {
  dependent_sync();
  if (threadIdx.x == 0) *io = value;
  if (tasks != nullptr)
    for (int j = threadIdx.x; j < batch; j += blockDim.x) task_stage[j] = tasks[j];
}
void eval_begin(cudaStream_t s, EvalIo* io, const EvalIo& value, const int* tasks, int* task_stage, int batch) {
  note_launch(1);
  launch_k(eval_begin_kernel, 1, 128, 0, s, io, value, tasks, task_stage, batch);
}
// Guard words after every workspace slice: one warp per guard.
__global__ void guards_write_kernel(char* base, const unsigned long long* __restrict__ table, int n, int words, uint32_t word) {
  dependent_sync();
  int g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (g >= n) return;
  uint32_t* p = reinterpret_cast<uint32_t*>(base + table[g]);
  for (int i = lane; i < words; i += 32) p[i] = word;
}
__global__ void guards_check_kernel(const char* base, const unsigned long long* __restrict__ table, int n, int words, uint32_t word,
                                    int* status) {
  dependent_sync();
  int g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (g >= n) return;
  const uint32_t* p = reinterpret_cast<const uint32_t*>(base + table[g]);
  bool bad = false;
  for (int i = lane; i < words; i += 32) bad |= p[i] != word;
  if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(status, STATUS_GUARD);
}
void guards_write(cudaStream_t s, char* base, const unsigned long long* table, int n, int words, uint32_t word) {
  note_launch(1);
  launch_k(guards_write_kernel, ceil_div((long)n * 32, 256), 256, 0, s, base, table, n, words, word);
}
void guards_check(cudaStream_t s, const char* base, const unsigned long long* table, int n, int words, uint32_t word, int* status) {
  note_launch(1);
  launch_k(guards_check_kernel, ceil_div((long)n * 32, 256), 256, 0, s, base, table, n, words, word, status);
}

__global__ void set_scalars_kernel(float* dst, float a, float b, float c3) {
  dependent_sync();
  dst[0] = a; dst[1] = b; dst[2] = c3;
}
void set_scalars(cudaStream_t s, float* dst, float a, float b, float c3) {
  note_launch(1);
  launch_k(set_scalars_kernel, 1, 1, 0, s, dst, a, b, c3);
}

void adamw(const Ctx& c, const AdamChunk* chunks, int nchunks, bool beside, float* master, const float* grad, float* m, float* v,
           void* shadow_base, const float* scalars, float b1, float b2, float eps, float wd) {
  if (nchunks <= 0) return;
  note_launch(1);
  const int blocks = update_blocks(c, nchunks, beside);
  const AdamRule rule = {master, m, v, grad, 0.f, 1.f, 1.f, b1, b2, eps, wd};
  if (c.dtype == 0) launch_k(adamw_kernel<float>, blocks, 256, 0, c.stream, chunks, nchunks, rule, (float*)shadow_base, scalars);
  else launch_k(adamw_kernel<bf16>, blocks, 256, 0, c.stream, chunks, nchunks, rule, (bf16*)shadow_base, scalars);
}

// ------------------------------------------------------------------------------------------------
// Strided row copy in 16-byte units: dst[r] = src[r] for rows of row_bytes, each side with its own row pitch.
// Gathers the classification rows of a [B, T, D] tensor into [B, D] and scatters them back.
// ------------------------------------------------------------------------------------------------
__global__ void copy_rows_kernel(const char* __restrict__ src, long src_pitch, char* __restrict__ dst, long dst_pitch, int rows,
                                 int units) {
  dependent_sync();
  long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long)rows * units) return;
  int r = (int)(i / units), u = (int)(i % units);
  *reinterpret_cast<uint4*>(dst + (long)r * dst_pitch + u * 16L) = *reinterpret_cast<const uint4*>(src + (long)r * src_pitch + u * 16L);
}

void copy_rows(cudaStream_t st, const void* src, long src_pitch_bytes, void* dst, long dst_pitch_bytes, int rows, int row_bytes) {
  note_launch(1);
  int units = row_bytes / 16;
  long total = (long)rows * units;
  launch_k(copy_rows_kernel, ceil_div(total, 256), 256, 0, st, (const char*)src, src_pitch_bytes, (char*)dst, dst_pitch_bytes, rows, units);
}

// ------------------------------------------------------------------------------------------------
// Conversions
// ------------------------------------------------------------------------------------------------
template <typename T>
__global__ void from_float_kernel(const float* __restrict__ s, T* __restrict__ d, size_t n) {
  dependent_sync();
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) d[i] = from_f<T>(s[i]);
}
template <typename T>
__global__ void to_float_kernel(const T* __restrict__ s, float* __restrict__ d, size_t n) {
  dependent_sync();
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) d[i] = to_f(s[i]);
}
__global__ void fill_kernel(float* d, float v, size_t n) {
  dependent_sync();
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) d[i] = v;
}

void convert_from_float(const Ctx& c, const float* src, void* dst, size_t n) {
  note_launch(1);
  if (n == 0) return;
  int blocks = ceil_div((long)n, 256);
  if (c.dtype == 0) launch_k(from_float_kernel<float>, blocks, 256, 0, c.stream, src, (float*)dst, n);
  else launch_k(from_float_kernel<bf16>, blocks, 256, 0, c.stream, src, (bf16*)dst, n);
}
void convert_to_float(const Ctx& c, const void* src, float* dst, size_t n) {
  note_launch(1);
  if (n == 0) return;
  int blocks = ceil_div((long)n, 256);
  if (c.dtype == 0) launch_k(to_float_kernel<float>, blocks, 256, 0, c.stream, (const float*)src, dst, n);
  else launch_k(to_float_kernel<bf16>, blocks, 256, 0, c.stream, (const bf16*)src, dst, n);
}
__global__ void int_to_float_kernel(const int* s, float* d, size_t n) {
  dependent_sync();
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) d[i] = (float)s[i];
}
void convert_int_to_float(cudaStream_t st, const int* src, float* dst, size_t n) {
  if (n == 0) return;
  note_launch(1);
  launch_k(int_to_float_kernel, ceil_div((long)n, 256), 256, 0, st, src, dst, n);
}
void fill_float(cudaStream_t s, float* dst, float v, size_t n) {
  note_launch(1);
  if (n == 0) return;
  launch_k(fill_kernel, ceil_div((long)n, 256), 256, 0, s, dst, v, n);
}

}  // namespace bsr
