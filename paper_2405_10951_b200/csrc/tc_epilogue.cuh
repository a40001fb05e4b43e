// Epilogue of the tcgen05 GEMM kernels: a warp turns 32 rows x 32 columns of fp32 accumulators (lane = row) into
// outputs with bias, GELU, GELU-derivative and residual options, moving data to and from global memory through a
// swizzled staging buffer so that every global access is row-contiguous.
#pragma once

#include "common.cuh"
#include "tc_ptx.cuh"

namespace bsr {
namespace tc {

struct Epi {
  const float* bias = nullptr;
  const void* residual = nullptr;
  int res_ld = 0;                   // elements between its rows
  void* aux_out = nullptr;
  const void* aux_in = nullptr;
  int act = 0;
  bool release = false;             // the next kernel may be scheduled while this one runs (set up: GemmEpilogue's product_next)
  // operands quantised with one scale per row of A and per row of B (8-bit floating point): the accumulator of
  // (row, col) is multiplied by row_scale[row] * col_scale[col] before the bias
  const float* row_scale = nullptr;
  const float* col_scale = nullptr;
};

// Two fp32 lanes per instruction (fma.rn.f32x2 and friends): halves the issue slots of the polynomial below.
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t r, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r)); }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t dup2(float a) { return pack2(a, a); }

// Phi(z) - 1/2 = z * q(z^2) with q a polynomial of degree 8 fitted to erf in double precision on |z| <= 4:
// |error of Phi| < 3e-5 everywhere (4e-6 inside the interval), no special-function unit involved.  Returns
// q(min(z^2, 16)) for two values: beyond |z| = 4 the product z * q(16) leaves [-1/2, 1/2], so that adding 1/2 with
// saturation pins Phi to 0 or 1.  Used where the result is rounded to bf16 (resolution 4e-3 relative).
__device__ __forceinline__ void phi_slope2(float u0, float u1, float& q0, float& q1) {
  uint64_t u = pack2(fminf(u0, 16.0f), fminf(u1, 16.0f));
  uint64_t q = dup2(8.065214468500059e-11f);
  q = fma2(q, u, dup2(-7.004623547857136e-09f));
  q = fma2(q, u, dup2(2.716460869578441e-07f));
  q = fma2(q, u, dup2(-6.295422281255014e-06f));
  q = fma2(q, u, dup2(9.891138324746862e-05f));
  q = fma2(q, u, dup2(-0.001133936457335949f));
  q = fma2(q, u, dup2(0.009877507574856281f));
  q = fma2(q, u, dup2(-0.0664106160402298f));
  q = fma2(q, u, dup2(0.3989226818084717f));
  unpack2(q, q0, q1);
}
// z <- GELU(z) = z * Phi(z), two values.
__device__ __forceinline__ void gelu_fast2(float& z0, float& z1) {
  float u0, u1, q0, q1;
  uint64_t z = pack2(z0, z1);
  unpack2(mul2(z, z), u0, u1);
  phi_slope2(u0, u1, q0, q1);
  z0 *= __saturatef(fmaf(z0, q0, 0.5f));
  z1 *= __saturatef(fmaf(z1, q1, 0.5f));
}
// g <- g * GELU'(z), two values: GELU'(z) = Phi(z) + z * phi(z), with the density phi(z) = exp(-z^2 / 2) / sqrt(2 pi)
// from one exponential of the unclamped square.
__device__ __forceinline__ void gelu_grad_mul2(float& g0, float& g1, float z0, float z1) {
  float u0, u1, q0, q1, d0, d1, e0, e1;
  uint64_t z = pack2(z0, z1);
  unpack2(mul2(z, z), u0, u1);
  phi_slope2(u0, u1, q0, q1);
  const float kh = -0.5f * 1.4426950408889634f;          // exp(-u / 2) = 2^(kh u)
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e0) : "f"(u0 * kh));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e1) : "f"(u1 * kh));
  unpack2(mul2(z, dup2(0.39894228040143268f)), d0, d1);
  g0 *= fmaf(d0, e0, __saturatef(fmaf(z0, q0, 0.5f)));
  g1 *= fmaf(d1, e1, __saturatef(fmaf(z1, q1, 0.5f)));
}

// The same, also returning h = GELU(z) = z * Phi(z) (the second FFN layer's input, recomputed in the backward pass
// instead of being kept since the forward pass).
__device__ __forceinline__ void gelu_grad_mul2h(float& g0, float& g1, float z0, float z1, float& h0, float& h1) {
  float u0, u1, q0, q1, d0, d1, e0, e1;
  uint64_t z = pack2(z0, z1);
  unpack2(mul2(z, z), u0, u1);
  phi_slope2(u0, u1, q0, q1);
  const float kh = -0.5f * 1.4426950408889634f;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e0) : "f"(u0 * kh));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e1) : "f"(u1 * kh));
  unpack2(mul2(z, dup2(0.39894228040143268f)), d0, d1);
  float p0 = __saturatef(fmaf(z0, q0, 0.5f)), p1 = __saturatef(fmaf(z1, q1, 0.5f));
  h0 = z0 * p0; h1 = z1 * p1;
  g0 *= fmaf(d0, e0, p0);
  g1 *= fmaf(d1, e1, p1);
}

// The polynomial above is off by up to 4e-6 of Phi, which near z = -4 is a tenth of GELU itself and twenty times its rounding to
// bf16.  The classification rows of the last block and other products of few rows and a long reduction take GELU and its
// derivative to 7e-6 of their values: Phi(-t) = exp(-t^2 / 2) R(t), R a polynomial of degree 11 in 2 t / 5.75 - 1 fitted to
// erfc(t / sqrt 2) exp(t^2 / 2) / 2 in double precision on 0 <= t <= 5.75 (relative error 6e-6; beyond, Phi(-t) < 5e-9 and too large
// by less than t / 5.75).  At many rows its exponential would be felt (25216 x 3072 x 768: GELU already adds 11 us to 75); with
// few a launch waits for its operands (128 x 3072 x 768: 6.5 -> 6.9 us; erff and expf 7.4).
inline bool exact_gelu(int m, int k) { return m <= 256 && k > 448; }
// z <- Phi(z) of two values; e = exp(-z^2 / 2).
__device__ __forceinline__ void phi_exact2(float& z0, float& z1, float& e0, float& e1) {
  float u0, u1, p0, p1;
  uint64_t z = pack2(z0, z1);
  unpack2(mul2(z, z), u0, u1);
  const float kh = -0.5f * 1.4426950408889634f;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e0) : "f"(u0 * kh));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e1) : "f"(u1 * kh));
  const uint64_t x = fma2(pack2(fminf(fabsf(z0), 5.75f), fminf(fabsf(z1), 5.75f)), dup2(2.0f / 5.75f), dup2(-1.0f));
  uint64_t r = dup2(-0.003139214925281772f);
  r = fma2(r, x, dup2(0.006516454073486045f));
  r = fma2(r, x, dup2(-0.0026901766723877356f));
  r = fma2(r, x, dup2(0.0023635298203356254f));
  r = fma2(r, x, dup2(-0.01276389393510076f));
  r = fma2(r, x, dup2(0.022197755375759323f));
  r = fma2(r, x, dup2(-0.02989035800599237f));
  r = fma2(r, x, dup2(0.04333526234265012f));
  r = fma2(r, x, dup2(-0.06198110430277863f));
  r = fma2(r, x, dup2(0.08334893928193564f));
  r = fma2(r, x, dup2(-0.10580940246565074f));
  r = fma2(r, x, dup2(0.12596105591795748f));
  unpack2(mul2(r, pack2(e0, e1)), p0, p1);
  z0 = z0 < 0.0f ? p0 : 1.0f - p0;
  z1 = z1 < 0.0f ? p1 : 1.0f - p1;
}
__device__ __forceinline__ void gelu_exact2(float& z0, float& z1) {
  float p0 = z0, p1 = z1, e0, e1;
  phi_exact2(p0, p1, e0, e1);
  z0 *= p0;
  z1 *= p1;
}
// g <- g * GELU'(z), z <- GELU(z), two values.
__device__ __forceinline__ void gelu_grad_exact2(float& g0, float& g1, float& z0, float& z1) {
  float p0 = z0, p1 = z1, e0, e1;
  phi_exact2(p0, p1, e0, e1);
  g0 *= fmaf(z0 * 0.39894228040143268f, e0, p0);
  g1 *= fmaf(z1 * 0.39894228040143268f, e1, p1);
  z0 *= p0;
  z1 *= p1;
}

// 16-byte global load of data that is read once (residual stream, stored pre-activations).
template <typename T>
__device__ __forceinline__ uint4 ld_stream(const T* p) {
  uint4 x;
  asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(x.x), "=r"(x.y), "=r"(x.z), "=r"(x.w) : "l"(p));
  return x;
}

// A warp moves a 32-row x 32-column chunk between registers (lane = row, v[32] = the row's columns) and global
// memory through its staging buffer, so that the global accesses are row-contiguous: each instruction touches a
// few full rows instead of one 16-byte piece of 32 different rows.
template <typename T>
struct ChunkIO {
  static constexpr int E = 16 / sizeof(T);          // elements per 16-byte unit
  static constexpr int UNITS = 32 / E;               // units per chunk row: 4 (bf16) or 8 (float)
  static constexpr int ROWS_PER_PASS = 32 / UNITS;
  // rows of 128 bytes (float) or 64 bytes (bf16); the order of a row's units depends on the row so that neither direction
  // has bank conflicts
  __device__ static uint32_t slot(int r, int u) {
    return sizeof(T) == 4 ? (uint32_t)(r * 128 + ((u ^ (r & 7)) << 4)) : (uint32_t)(r * 64 + ((u ^ ((r >> 1) & 3)) << 4));
  }

  // All global loads are issued before the first shared-memory store: the staging pointer may alias anything as
  // far as the compiler knows, so a load placed after a store could not be moved ahead of it.
  __device__ static void load(const T* g, int ld, int row0, int col0, int M, int N, unsigned char* st, int lane, float* v) {
    uint4 x[UNITS];
#pragma unroll
    for (int i = 0; i < UNITS; ++i) {
      int r = i * ROWS_PER_PASS + lane / UNITS, u = lane % UNITS;
      int col = col0 + u * E;
      x[i] = make_uint4(0, 0, 0, 0);
      if (row0 + r < M && col < N) x[i] = ld_stream(g + (size_t)(row0 + r) * ld + col);
    }
#pragma unroll
    for (int i = 0; i < UNITS; ++i) {
      int r = i * ROWS_PER_PASS + lane / UNITS, u = lane % UNITS;
      *reinterpret_cast<uint4*>(st + slot(r, u)) = x[i];
    }
    __syncwarp();
#pragma unroll
    for (int u = 0; u < UNITS; ++u) {
      uint4 y = *reinterpret_cast<const uint4*>(st + slot(lane, u));
      unpack(y, v + u * E);
    }
    __syncwarp();
  }
  __device__ static void store(T* g, int ld, int row0, int col0, int M, int N, unsigned char* st, int lane, const float* v) {
#pragma unroll
    for (int u = 0; u < UNITS; ++u) *reinterpret_cast<uint4*>(st + slot(lane, u)) = pack(v + u * E);
    __syncwarp();
    uint4 x[UNITS];
#pragma unroll
    for (int i = 0; i < UNITS; ++i) {
      int r = i * ROWS_PER_PASS + lane / UNITS, u = lane % UNITS;
      x[i] = *reinterpret_cast<const uint4*>(st + slot(r, u));
    }
#pragma unroll
    for (int i = 0; i < UNITS; ++i) {
      int r = i * ROWS_PER_PASS + lane / UNITS, u = lane % UNITS;
      int col = col0 + u * E;
      if (row0 + r < M && col < N) *reinterpret_cast<uint4*>(g + (size_t)(row0 + r) * ld + col) = x[i];
    }
    __syncwarp();
  }
  __device__ static void unpack(const uint4& x, float* f);
  __device__ static uint4 pack(const float* f);
};
template <> __device__ __forceinline__ void ChunkIO<float>::unpack(const uint4& x, float* f) {
  f[0] = __uint_as_float(x.x); f[1] = __uint_as_float(x.y); f[2] = __uint_as_float(x.z); f[3] = __uint_as_float(x.w);
}
template <> __device__ __forceinline__ uint4 ChunkIO<float>::pack(const float* f) {
  return make_uint4(__float_as_uint(f[0]), __float_as_uint(f[1]), __float_as_uint(f[2]), __float_as_uint(f[3]));
}
template <> __device__ __forceinline__ void ChunkIO<bf16>::unpack(const uint4& x, float* f) {
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&x);
#pragma unroll
  for (int i = 0; i < 4; ++i) { float2 t = __bfloat1622float2(h[i]); f[2 * i] = t.x; f[2 * i + 1] = t.y; }
}
template <> __device__ __forceinline__ uint4 ChunkIO<bf16>::pack(const float* f) {
  uint4 x;
  __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&x);
#pragma unroll
  for (int i = 0; i < 4; ++i) h[i] = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
  return x;
}

// v[j]: accumulator of (row0 + lane, col0 + j).  All lanes of the warp take part (row0, col0 are warp-uniform).
// z: the chunk of the stored pre-activation for act == 2, already in this lane's row order (overwritten).
// sbias, scol: the chunk's 32 bias values and column scales in shared memory (null: none), rs: this lane's row scale.
// EXACT: activations as exact_gelu has them.
template <typename TOut, bool EXACT>
__device__ __forceinline__ void epilogue_chunk(const uint32_t* r, const Epi& ep, const float* sbias, const float* scol, float rs, TOut* Cs, int M,
                                               int N, int row0, int col0, unsigned char* st, int lane, float* z) {
  if (row0 < M && col0 < N) {
    float v[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
    if (scol != nullptr) {
#pragma unroll
      for (int g = 0; g < 8; ++g) {
        float4 cs = *reinterpret_cast<const float4*>(scol + g * 4);
        v[g * 4 + 0] *= rs * cs.x; v[g * 4 + 1] *= rs * cs.y; v[g * 4 + 2] *= rs * cs.z; v[g * 4 + 3] *= rs * cs.w;
      }
    }
    if (sbias != nullptr) {
#pragma unroll
      for (int g = 0; g < 8; ++g) {
        float4 bb = *reinterpret_cast<const float4*>(sbias + g * 4);
        v[g * 4 + 0] += bb.x; v[g * 4 + 1] += bb.y; v[g * 4 + 2] += bb.z; v[g * 4 + 3] += bb.w;
      }
    }
    if (ep.act == 1) {
      if (ep.aux_out != nullptr) ChunkIO<TOut>::store((TOut*)ep.aux_out, N, row0, col0, M, N, st, lane, v);
      if (EXACT) {
#pragma unroll
        for (int j = 0; j < 32; j += 2) gelu_exact2(v[j], v[j + 1]);
      } else {
#pragma unroll
        for (int j = 0; j < 32; j += 2) gelu_fast2(v[j], v[j + 1]);
      }
    } else if (ep.act == 2) {
      if (EXACT) {
#pragma unroll
        for (int j = 0; j < 32; j += 2) gelu_grad_exact2(v[j], v[j + 1], z[j], z[j + 1]);
        if (ep.aux_out != nullptr) ChunkIO<bf16>::store((bf16*)ep.aux_out, N, row0, col0, M, N, st, lane, z);
      } else if (ep.aux_out != nullptr) {   // GELU(z) recomputed for the weight gradient of the second FFN layer
#pragma unroll
        for (int j = 0; j < 32; j += 2) gelu_grad_mul2h(v[j], v[j + 1], z[j], z[j + 1], z[j], z[j + 1]);
        ChunkIO<bf16>::store((bf16*)ep.aux_out, N, row0, col0, M, N, st, lane, z);
      } else {
#pragma unroll
        for (int j = 0; j < 32; j += 2) gelu_grad_mul2(v[j], v[j + 1], z[j], z[j + 1]);
      }
    }
    if (ep.residual != nullptr) {
      float rr[32];
      ChunkIO<TOut>::load((const TOut*)ep.residual, ep.res_ld, row0, col0, M, N, st, lane, rr);
#pragma unroll
      for (int j = 0; j < 32; ++j) v[j] += rr[j];
    }
    ChunkIO<TOut>::store(Cs, N, row0, col0, M, N, st, lane, v);
  }
}


// ---- float outputs without activation (projection, second FFN layer, weight gradients) ----------------------------
// The accumulators are transposed once, through the staging buffer, into the row-contiguous order in which global
// memory is read and written; bias and residual are added in that order, so the residual needs no staging at all and
// its loads (issued by chunk_issue a chunk ahead, the first of a tile before the tile's accumulator is complete) stay
// in flight while the tensor-memory read and the transposition proceed.
__device__ __forceinline__ void chunk_issue(const float* g, int ld, int row0, int col0, int M, int N, int lane, uint4* x) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    int r = i * 4 + lane / 8, col = col0 + (lane % 8) * 4;
    x[i] = make_uint4(0, 0, 0, 0);
    if (row0 + r < M && col < N) x[i] = ld_stream(g + (size_t)(row0 + r) * ld + col);
  }
}
// bb: bias of columns col0 + 4 (lane % 8) .. + 3.
__device__ __forceinline__ void epilogue_chunk_f32(const uint32_t* r, float4 bb, float* Cs, int M, int N, int row0, int col0,
                                                   unsigned char* st, int lane, const uint4* xres, bool has_res) {
  if (row0 < M && col0 < N) {
    using IO = ChunkIO<float>;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      *reinterpret_cast<uint4*>(st + IO::slot(lane, u)) = make_uint4(r[4 * u], r[4 * u + 1], r[4 * u + 2], r[4 * u + 3]);
    __syncwarp();
    int u = lane % 8, col = col0 + u * 4;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      int rr = i * 4 + lane / 8;
      uint4 a = *reinterpret_cast<const uint4*>(st + IO::slot(rr, u));
      float4 v = make_float4(__uint_as_float(a.x) + bb.x, __uint_as_float(a.y) + bb.y, __uint_as_float(a.z) + bb.z, __uint_as_float(a.w) + bb.w);
      if (has_res) {
        v.x += __uint_as_float(xres[i].x); v.y += __uint_as_float(xres[i].y); v.z += __uint_as_float(xres[i].z); v.w += __uint_as_float(xres[i].w);
      }
      if (row0 + rr < M && col < N) *reinterpret_cast<float4*>(Cs + (size_t)(row0 + rr) * N + col) = v;
    }
    __syncwarp();
  }
}

// Stored pre-activation chunk (bf16) fetched ahead of use: four 16-byte units per lane in row-contiguous order, later
// turned into this lane's row through the staging buffer.
__device__ __forceinline__ void chunk_issue(const bf16* g, int ld, int row0, int col0, int M, int N, int lane, uint4* x) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    int r = i * 8 + lane / 4, col = col0 + (lane % 4) * 8;
    x[i] = make_uint4(0, 0, 0, 0);
    if (row0 + r < M && col < N) x[i] = ld_stream(g + (size_t)(row0 + r) * ld + col);
  }
}
__device__ __forceinline__ void chunk_land_bf16(const uint4* x, unsigned char* st, int lane, float* v) {
  using IO = ChunkIO<bf16>;
#pragma unroll
  for (int i = 0; i < 4; ++i) *reinterpret_cast<uint4*>(st + IO::slot(i * 8 + lane / 4, lane % 4)) = x[i];
  __syncwarp();
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    uint4 y = *reinterpret_cast<const uint4*>(st + IO::slot(lane, u));
    IO::unpack(y, v + u * 8);
  }
  __syncwarp();
}

// A warp's share of a tile: `nc` (at most four) chunks of 32 columns from column cb of 32 rows, accumulators at taddr.  ready()
// waits for the accumulators; what does not depend on them is fetched before: bias and column scales (read where they
// are added, they came from L2 -- the operand ring leaves hardly any L1 -- and took 900 of the 1700 clocks of a chunk) and
// the first chunk of the residual or of the stored pre-activation, whose next chunk is always on its way.
// st: this warp's staging buffer, 4 KB.
template <typename TOut, bool FP8, bool EXACT, typename Ready>
__device__ __forceinline__ bool epilogue_tile(Ready ready, const Epi& ep, int bias_off, TOut* Cs, int M, int N, int row0, int cb, int nc, uint32_t taddr,
                                              unsigned char* st, int lane) {
  const float* bias = ep.bias == nullptr ? nullptr : ep.bias + bias_off;
  uint4 xn[8];
  if constexpr (sizeof(TOut) == 4) {           // float outputs (never with an activation) are transposed once
    const bool has_res = ep.residual != nullptr;
    auto bias4 = [&](int cc) {
      const int col = cb + cc * 32 + (lane % 8) * 4;
      return bias != nullptr && col < N ? __ldg(reinterpret_cast<const float4*>(bias + col)) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    float4 bn = bias4(0);
    if (has_res) chunk_issue((const float*)ep.residual, ep.res_ld, row0, cb, M, N, lane, xn);
    if (!ready()) return false;
#pragma unroll 1
    for (int cc = 0; cc < nc; ++cc) {
      uint4 xc[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) xc[i] = xn[i];
      const float4 bb = bn;
      if (cc + 1 < nc) {
        bn = bias4(cc + 1);
        if (has_res) chunk_issue((const float*)ep.residual, ep.res_ld, row0, cb + (cc + 1) * 32, M, N, lane, xn);
      }
      uint32_t r[32];
      tmem_ld32(taddr + cc * 32, r);
      tmem_ld_wait();
      epilogue_chunk_f32(r, bb, (float*)Cs, M, N, row0, cb + cc * 32, st, lane, xc, has_res);
    }
  } else {
    float* sbias = reinterpret_cast<float*>(st + 2048);      // behind the 32 rows of 64 bytes a chunk takes: bias, column scales
    if (lane < nc * 8) {
      const int col = cb + lane * 4;
      const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
      if (bias != nullptr) *reinterpret_cast<float4*>(sbias + lane * 4) = col < N ? __ldg(reinterpret_cast<const float4*>(bias + col)) : z4;
      if (FP8) *reinterpret_cast<float4*>(sbias + 128 + lane * 4) = col < N ? __ldg(reinterpret_cast<const float4*>(ep.col_scale + col)) : z4;
    }
    const float rs = FP8 && row0 + lane < M ? __ldg(ep.row_scale + row0 + lane) : 0.f;
    const bool pre_z = ep.act == 2;            // dz of the FFN backward
    if (pre_z) chunk_issue((const bf16*)ep.aux_in, N, row0, cb, M, N, lane, xn);
    if (!ready()) return false;
    __syncwarp();
#pragma unroll 1
    for (int cc = 0; cc < nc; ++cc) {
      float z[32];
      if (pre_z) {
        chunk_land_bf16(xn, st, lane, z);
        if (cc + 1 < nc) chunk_issue((const bf16*)ep.aux_in, N, row0, cb + (cc + 1) * 32, M, N, lane, xn);
      }
      uint32_t r[32];
      tmem_ld32(taddr + cc * 32, r);
      tmem_ld_wait();
      epilogue_chunk<TOut, EXACT>(r, ep, bias != nullptr ? sbias + cc * 32 : nullptr, FP8 ? sbias + 128 + cc * 32 : nullptr, rs, Cs, M, N, row0, cb + cc * 32, st,
                           lane, z);
    }
  }
  return true;
}

}  // namespace tc
}  // namespace bsr
