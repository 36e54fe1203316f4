// CUDA-core matrix multiply: Y[R][N] = X[R][K] * W[N][K]^T with fp32 accumulation, for any
// shape and for fp32 or bf16 operands.  Used for the fp32 configuration (strict fp32, no TF32),
// for shapes the tensor-core path does not take, and as the A/B reference of that path.
#include <type_traits>

#include "common.cuh"

namespace koala {
namespace {

constexpr int FPW = 4;       // output features per warp
constexpr int ROWS = 16;     // X rows per block
constexpr int KC = 512;      // K elements staged per step
constexpr int WARPS = 8;
// Multiply-adds up to which the small kernel is taken (see gemm_simt).
constexpr int FEW_ROWS = 16;
constexpr double SMALL_MACS_FEW_ROWS = 4e8, SMALL_MACS = 1e8;

template <typename T>
__global__ void __launch_bounds__(WARPS * 32)
gemm_simt_kernel(const T *X, const T *Xlo, int R, int K_in, const T *__restrict__ W0,
                 const T *__restrict__ W1, const T *__restrict__ W2, int n0, int n1, int n2,
                 float *__restrict__ Y, int ldy) {
  __shared__ float xs[ROWS][KC + 1];
  pdl_launch_dependents();
  pdl_wait();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int r0 = blockIdx.y * ROWS;
  const int ntot = n0 + n1 + n2;
  const T *wrow[FPW];
  int col[FPW];
#pragma unroll
  for (int f = 0; f < FPW; ++f) {
    int g = (blockIdx.x * WARPS + w) * FPW + f;
    col[f] = g;
    if (g >= ntot) g = ntot - 1;
    const T *base = W0;
    if (g >= n0 + n1) { base = W2; g -= n0 + n1; }
    else if (g >= n0) { base = W1; g -= n0; }
    wrow[f] = base + (size_t)g * K_in;
  }
  float acc[FPW][ROWS];
#pragma unroll
  for (int f = 0; f < FPW; ++f)
#pragma unroll
    for (int r = 0; r < ROWS; ++r) acc[f][r] = 0.f;

  for (int k0 = 0; k0 < K_in; k0 += KC) {
    __syncthreads();
    for (int e = threadIdx.x; e < ROWS * KC; e += WARPS * 32) {
      const int r = e / KC, k = e % KC;
      float v = 0.f;
      if (r0 + r < R && k0 + k < K_in) {
        const size_t idx = (size_t)(r0 + r) * K_in + k0 + k;
        v = to_f(X[idx]);
        if (Xlo != nullptr) v += to_f(Xlo[idx]);
      }
      xs[r][k] = v;
    }
    __syncthreads();
    const int kend = min(KC, K_in - k0);
    for (int k = lane; k < kend; k += 32) {
      float wv[FPW];
#pragma unroll
      for (int f = 0; f < FPW; ++f) wv[f] = to_f(wrow[f][k0 + k]);
#pragma unroll
      for (int r = 0; r < ROWS; ++r) {
        const float xv = xs[r][k];
#pragma unroll
        for (int f = 0; f < FPW; ++f) acc[f][r] = fmaf(wv[f], xv, acc[f][r]);
      }
    }
  }
#pragma unroll
  for (int f = 0; f < FPW; ++f)
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      const float v = warp_sum(acc[f][r]);
      if (lane == 0 && col[f] < ntot && r0 + r < R) Y[(size_t)(r0 + r) * ldy + col[f]] = v;
    }
}

// Small problems (few rows, K a multiple of four): latency is all there is, so nothing is staged and
// nothing waits that need not.  A warp owns one output feature and RT rows; a lane owns every 32nd
// group of four K elements.  The weights of the first WPRE groups are read before the dependency wait
// (they do not depend on the kernel before this one), then all loads of X are independent of each
// other and shared by the block's eight warps through L1.  The RT partial sums are reduced together:
// every exchange halves the number of values a lane still carries, RT + log2(32 / RT) shuffles
// instead of 5 RT.  fp32, 15 rows, 256 x 768 and 688 x 256 matrices: 13.3 -> 3.4 us per launch
// against the staged kernel above (32 features per block leave it on eight SMs there).
constexpr int WPRE = 6;

template <typename T> struct Vec4;
template <> struct Vec4<float> {
  static __device__ __forceinline__ float4 load(const float *p) { return *reinterpret_cast<const float4 *>(p); }
};
template <> struct Vec4<bf16> {
  static __device__ __forceinline__ float4 load(const bf16 *p) {
    const uint2 u = *reinterpret_cast<const uint2 *>(p);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.y));
    return make_float4(a.x, a.y, b.x, b.y);
  }
};

template <typename T, int RT>
__global__ void __launch_bounds__(WARPS * 32)
gemm_simt_small_kernel(const T *X, const T *Xlo, int R, int K_in, const T *__restrict__ W0, const T *__restrict__ W1,
                       const T *__restrict__ W2, int n0, int n1, int n2, float *__restrict__ Y, int ldy) {
  pdl_launch_dependents();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int ntot = n0 + n1 + n2;
  const int col = blockIdx.x * WARPS + w;
  if (col >= ntot) return;
  const T *wr = col >= n0 + n1 ? W2 + (size_t)(col - n0 - n1) * K_in
                               : (col >= n0 ? W1 + (size_t)(col - n0) * K_in : W0 + (size_t)col * K_in);
  const int r0 = blockIdx.y * RT;
  float4 pre[WPRE];
#pragma unroll
  for (int i = 0; i < WPRE; ++i) {
    const int k = (lane + 32 * i) * 4;
    pre[i] = k < K_in ? Vec4<T>::load(wr + k) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  pdl_wait();
  float acc[RT];
#pragma unroll
  for (int r = 0; r < RT; ++r) acc[r] = 0.f;
  const int rows = R - r0 < RT ? R - r0 : RT;
  auto step = [&](const float4 wv, int k) {
#pragma unroll
    for (int r = 0; r < RT; ++r) {
      const size_t at = (size_t)(r0 + (r < rows ? r : 0)) * K_in + k;     // rows beyond R repeat row r0, dropped below
      float4 x = Vec4<T>::load(X + at);
      if (Xlo != nullptr) {
        const float4 l = Vec4<T>::load(Xlo + at);
        x.x += l.x; x.y += l.y; x.z += l.z; x.w += l.w;
      }
      acc[r] = fmaf(wv.x, x.x, acc[r]);
      acc[r] = fmaf(wv.y, x.y, acc[r]);
      acc[r] = fmaf(wv.z, x.z, acc[r]);
      acc[r] = fmaf(wv.w, x.w, acc[r]);
    }
  };
#pragma unroll
  for (int i = 0; i < WPRE; ++i) {
    const int k = (lane + 32 * i) * 4;
    if (k < K_in) step(pre[i], k);
  }
  for (int k = (lane + 32 * WPRE) * 4; k < K_in; k += 128) step(Vec4<T>::load(wr + k), k);
  // lane l ends with row (l / (32 / RT)): bit by bit, a lane keeps the half of its rows that its lane index names
#pragma unroll
  for (int n = RT / 2, o = 16; n >= 1; n >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int r = 0; r < n; ++r) {
      const float mine = up ? acc[n + r] : acc[r], give = up ? acc[r] : acc[n + r];
      acc[r] = mine + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  float v = acc[0];
#pragma unroll
  for (int o = 32 / RT / 2; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  constexpr int LPR = 32 / RT;                        // lanes that hold the same row
  const int row = r0 + lane / LPR;
  if (lane % LPR == 0 && row < R) Y[(size_t)row * ldy + col] = v;
}

}  // namespace

cudaError_t gemm_simt(Launch L, int dtype, Operand X, GemmMats m, int K_in, int R, float *Y,
                      int ldy) {
  const int n0 = m.n_out[0], n1 = m.n > 1 ? m.n_out[1] : 0, n2 = m.n > 2 ? m.n_out[2] : 0;
  const int ntot = n0 + n1 + n2;
  // The small kernel reads a weight row once per RT rows of X and X once per block of eight features, all from
  // L1 / L2; up to 16 rows it is taken while that is a few hundred KB per SM, with more rows, where the staged
  // kernel's tile of 16 rows is full and its reuse counts, only for the smallest matrices.  (bf16 forwards whose
  // F is no multiple of 64, small against staged: hidden 1024, 128 rows 700 / 391 us; 1536, 40 rows 557 / 388;
  // 2048, 24 rows 611 / 502; 4096, 8 rows 841 / 970.)
  const size_t esz = dtype == 0 ? 4 : 2;
  const bool aligned = (K_in & 3) == 0 && ((uintptr_t)X.hi % (4 * esz)) == 0 && ((uintptr_t)X.lo % (4 * esz)) == 0 &&
                       ((uintptr_t)m.W[0] % (4 * esz)) == 0 && (m.n < 2 || ((uintptr_t)m.W[1] % (4 * esz)) == 0) &&
                       (m.n < 3 || ((uintptr_t)m.W[2] % (4 * esz)) == 0);
  if (aligned && (double)R * K_in * ntot <= (R <= FEW_ROWS ? SMALL_MACS_FEW_ROWS : SMALL_MACS)) {
    auto go = [&](auto tag, auto rt) {
      typedef decltype(tag) T;
      constexpr int RT = decltype(rt)::value;
      dim3 g((ntot + WARPS - 1) / WARPS, (R + RT - 1) / RT);
      return launch_k(gemm_simt_small_kernel<T, RT>, g, dim3(WARPS * 32), 0, L.st, L.pdl, (const T *)X.hi,
                      (const T *)X.lo, R, K_in, (const T *)m.W[0], (const T *)(m.n > 1 ? m.W[1] : m.W[0]),
                      (const T *)(m.n > 2 ? m.W[2] : m.W[0]), n0, n1, n2, Y, ldy);
    };
    // rows per warp: as few as keep the grid near two blocks per SM (more blocks, shorter chains)
    const bool wide = (long long)((ntot + WARPS - 1) / WARPS) * ((R + 7) / 8) > 2 * 148;
    if (dtype == 0) return R <= 2 ? go(float{}, std::integral_constant<int, 2>{})
                                  : (R <= 4 ? go(float{}, std::integral_constant<int, 4>{})
                                            : (wide && R > 8 ? go(float{}, std::integral_constant<int, 16>{})
                                                             : go(float{}, std::integral_constant<int, 8>{})));
    return R <= 2 ? go(bf16{}, std::integral_constant<int, 2>{})
                  : (R <= 4 ? go(bf16{}, std::integral_constant<int, 4>{})
                            : (wide && R > 8 ? go(bf16{}, std::integral_constant<int, 16>{})
                                             : go(bf16{}, std::integral_constant<int, 8>{})));
  }
  dim3 grid((ntot + WARPS * FPW - 1) / (WARPS * FPW), (R + ROWS - 1) / ROWS);
  if (dtype == 0)
    return launch_k(gemm_simt_kernel<float>, grid, dim3(WARPS * 32), 0, L.st, L.pdl, (const float *)X.hi,
                    (const float *)X.lo, R, K_in, (const float *)m.W[0], (const float *)(m.n > 1 ? m.W[1] : m.W[0]),
                    (const float *)(m.n > 2 ? m.W[2] : m.W[0]), n0, n1, n2, Y, ldy);
  return launch_k(gemm_simt_kernel<bf16>, grid, dim3(WARPS * 32), 0, L.st, L.pdl, (const bf16 *)X.hi,
                  (const bf16 *)X.lo, R, K_in, (const bf16 *)m.W[0], (const bf16 *)(m.n > 1 ? m.W[1] : m.W[0]),
                  (const bf16 *)(m.n > 2 ? m.W[2] : m.W[0]), n0, n1, n2, Y, ldy);
}

}  // namespace koala
