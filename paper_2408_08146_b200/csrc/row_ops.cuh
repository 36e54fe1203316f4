// Device helpers of the row-wise kernels: block reductions, vector loads, operand stores, and the rows a
// forward starts from (embeddings, or the head's [feature ; embedding]).
#pragma once
#include "common.cuh"

namespace koala {
namespace {

__device__ __forceinline__ float block_sum(float v, float *red) {
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  if (lane == 0) red[w] = v;
  __syncthreads();
  float t = (threadIdx.x < nw) ? red[threadIdx.x] : 0.f;
  if (w == 0) {
    t = warp_sum(t);
    if (lane == 0) red[0] = t;
  }
  __syncthreads();
  t = red[0];
  __syncthreads();
  return t;
}

// Stores v as a matrix-multiply operand.  bf16 operands are kept as a pair hi + lo (lo = the
// rounding residual of hi, itself rounded to bf16), which carries 16 significant bits into the
// tensor cores; fp32 operands are exact and have no lo part.
template <typename T>
__device__ __forceinline__ void store_operand(T *hi, T *lo, size_t i, float v) {
  const T h = from_f<T>(v);
  hi[i] = h;
  if (lo != nullptr) lo[i] = from_f<T>(v - to_f(h));
}

template <typename T> __device__ __forceinline__ float4 load4(const T *p);
template <> __device__ __forceinline__ float4 load4<float>(const float *p) { return *reinterpret_cast<const float4 *>(p); }
template <> __device__ __forceinline__ float4 load4<bf16>(const bf16 *p) {
  const uint2 u = *reinterpret_cast<const uint2 *>(p);
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.x));
  const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.y));
  return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void store_operand4(float *hi, float *lo, size_t i, float4 v) {
  (void)lo;
  *reinterpret_cast<float4 *>(hi + i) = v;
}
__device__ __forceinline__ void store_operand4(bf16 *hi, bf16 *lo, size_t i, float4 v) {
  const __nv_bfloat162 h0 = __floats2bfloat162_rn(v.x, v.y), h1 = __floats2bfloat162_rn(v.z, v.w);
  uint2 u;
  u.x = *reinterpret_cast<const uint32_t *>(&h0);
  u.y = *reinterpret_cast<const uint32_t *>(&h1);
  *reinterpret_cast<uint2 *>(hi + i) = u;
  if (lo != nullptr) {
    const float2 f0 = __bfloat1622float2(h0), f1 = __bfloat1622float2(h1);
    const __nv_bfloat162 l0 = __floats2bfloat162_rn(v.x - f0.x, v.y - f0.y);
    const __nv_bfloat162 l1 = __floats2bfloat162_rn(v.z - f1.x, v.w - f1.y);
    u.x = *reinterpret_cast<const uint32_t *>(&l0);
    u.y = *reinterpret_cast<const uint32_t *>(&l1);
    *reinterpret_cast<uint2 *>(lo + i) = u;
  }
}

// The row a forward starts from, filled by the block that plans it (all threads of a block of ROW_THREADS).
constexpr int ROW_THREADS = 256;

// x <- E[tok]; xn <- T(x * gain) (not normalised); sumsq[row][chunk] <- sums of x^2 over chunks of 1024 columns.
template <typename T>
__device__ __forceinline__ void fill_embedding(const RowFill &f, size_t r, int tok) {
  __shared__ float part[ROW_SUMS][ROW_THREADS / 32];
  tok = tok < 0 ? 0 : (tok >= f.V ? f.V - 1 : tok);
  const T *e = reinterpret_cast<const T *>(f.E) + (size_t)tok * f.H, *g = reinterpret_cast<const T *>(f.gain);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, chunks = (f.H + 1023) >> 10;
#pragma unroll 1
  for (int k = 0; k < chunks; ++k) {
    const int c = k * 1024 + threadIdx.x * 4;
    float ss = 0.f;
    if (c < f.H) {
      const float4 o = load4<T>(e + c), gg = load4<T>(g + c);
      *reinterpret_cast<float4 *>(f.x + r * f.H + c) = o;
      ss = o.x * o.x + o.y * o.y + o.z * o.z + o.w * o.w;
      store_operand4(reinterpret_cast<T *>(f.out.hi), reinterpret_cast<T *>(f.out.lo), r * f.H + c,
                     make_float4(o.x * gg.x, o.y * gg.y, o.z * gg.z, o.w * gg.w));
    }
    ss = warp_sum(ss);
    if (lane == 0) part[k][w] = ss;
  }
  __syncthreads();
  if ((int)threadIdx.x < chunks) {
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < ROW_THREADS / 32; ++i) s += part[threadIdx.x][i];
    f.sumsq[r * ROW_SUMS + threadIdx.x] = s;
  }
}

// out <- [feature row src ; E[tok]]
template <typename T>
__device__ __forceinline__ void fill_concat(const RowFill &f, size_t r, int src, int tok) {
  tok = tok < 0 ? 0 : (tok >= f.V ? f.V - 1 : tok);
  const T *e = reinterpret_cast<const T *>(f.E) + (size_t)tok * f.H;
  const float *x = f.feat + (size_t)src * f.H;
  T *hi = reinterpret_cast<T *>(f.out.hi), *lo = reinterpret_cast<T *>(f.out.lo);
  const size_t base = r * 2 * f.H;
#pragma unroll 2
  for (int c = threadIdx.x * 4; c < f.H; c += ROW_THREADS * 4) {
    const float4 a = *reinterpret_cast<const float4 *>(x + c), b = load4<T>(e + c);
    store_operand4(hi, lo, base + c, a);
    store_operand4(hi, lo, base + f.H + c, b);      // the embedding is exact in T: its residual is zero
  }
}

}  // namespace
}  // namespace koala
