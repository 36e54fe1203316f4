// fp32 matrix multiplies of the sizes where latency is all there is, with the row-wise steps around them
// in the same launch.
//
// In a small model every kernel is a few microseconds of dependency latency whatever it does, so what
// counts is their number.  Every output is finished by one warp, so the step that follows a multiply
// happens where the result is:
//   FEW_ROPE      Q, K, V: rotary embedding, queries and cache rows written
//   FEW_SWIGLU    gate and up: SiLU(gate) * up
//   FEW_RESIDUAL  x += result, or x = result + bias
// and the RMSNorm in front of the first two is part of them (its gain folded into the weights before the
// dependency wait, the sum of squares of the row accumulated beside the products).  A layer is five
// launches (with attention) instead of nine: tiny iteration of 15 nodes and 4 draft passes 363 -> 310 us.
//
// The unit of work is a pair of weight rows whose results are needed together: (i, i + half) of a head for
// FEW_ROPE, (gate f, up f) for FEW_SWIGLU, two neighbours otherwise; a warp per unit and group of rows.
// (The same in bf16 with the weights as mma.sync operands streamed by bulk copies lost to the tcgen05
// multiply and its row-wise kernels: 3.43 against 3.03 ms per 7B one-token step.)
#include <type_traits>

#include "common.cuh"

namespace koala {
namespace {

constexpr int WPRE = 6;              // 128-element groups of both weight rows read before the dependency wait
constexpr int F32_WARPS = 4;

struct FewParams {
  const float *x, *w0, *w1, *w2;
  int R, K, units, n_out;            // n_out: rows of one matrix
  float inv_h, eps;                  // of the norm in front
  const float *gain, *bias;
  float *xres, *out, *out2;
  RowPlan plan;                      // ROPE
  float *q_out, *kc, *vc;
  int rows_per_seq, n_heads, head_dim, S_max;
};

// the two weight rows of a unit
template <int MODE>
__device__ __forceinline__ void unit_rows(const FewParams &P, int u, const float *&a, const float *&b) {
  if constexpr (MODE == FEW_SWIGLU) {
    a = P.w0 + (size_t)u * P.K;
    b = P.w1 + (size_t)u * P.K;
  } else if constexpr (MODE == FEW_ROPE) {
    const int per = P.n_out >> 1, half = P.head_dim >> 1;
    const int m = u / per, v = u - m * per, h = v / half, i = v - h * half;
    const float *w = m == 0 ? P.w0 : (m == 1 ? P.w1 : P.w2);
    a = w + (size_t)(h * P.head_dim + i) * P.K;
    b = a + (size_t)half * P.K;
  } else {
    a = P.w0 + (size_t)(2 * u) * P.K;
    b = 2 * u + 1 < P.n_out ? a + P.K : a;
  }
}

// What becomes of the two results of unit u for row r (s: the row's RMSNorm scale).
template <int MODE>
__device__ __forceinline__ void finish_unit(const FewParams &P, int u, int r, float a, float b, float s) {
  if constexpr (MODE == FEW_SWIGLU) {
    const float g = s * a;
    P.out[(size_t)r * P.n_out + u] = g / (1.f + expf(-g)) * (s * b);
  } else if constexpr (MODE == FEW_ROPE) {
    const int per = P.n_out >> 1, half = P.head_dim >> 1;
    const int m = u / per, v = u - m * per, h = v / half, i = v - h * half;
    a *= s;
    b *= s;
    if (m < 2) {
      const float2 cs = P.plan.rope[(size_t)r * half + i];
      const float ra = a * cs.x - b * cs.y, rb = b * cs.x + a * cs.y;
      a = ra;
      b = rb;
    }
    float *to;
    if (m == 0) {
      to = P.q_out + (size_t)r * P.n_out + h * P.head_dim + i;
    } else {
      const int slot = P.plan.slot[r];
      if (slot < 0 || slot >= P.S_max) return;
      const int seq = P.plan.cache_of(r / P.rows_per_seq);
      to = (m == 1 ? P.kc : P.vc) + (((size_t)seq * P.n_heads + h) * P.S_max + slot) * P.head_dim + i;
    }
    to[0] = a;
    to[half] = b;
  } else {
    const int c = 2 * u;
    const bool two = c + 1 < P.n_out;
    const size_t at = (size_t)r * P.n_out + c;
    const float *add = P.bias != nullptr ? P.bias + c : P.xres + at;
    const float v0 = a + add[0], v1 = two ? b + add[1] : 0.f;
    P.xres[at] = v0;
    if (two) P.xres[at + 1] = v1;
    if (P.out != nullptr) {
      P.out[at] = v0;
      if (two) P.out[at + 1] = v1;
    }
    if (P.out2 != nullptr) {
      P.out2[at] = v0;
      if (two) P.out2[at + 1] = v1;
    }
  }
}

// Reduces RT values over the warp; lane l ends with the sum of value l / (32 / RT).  Bit by bit a lane keeps
// the half of its values that its lane index names: RT - 1 + log2(32 / RT) shuffles.
template <int RT>
__device__ __forceinline__ float reduce_rows(float (&v)[RT], int lane) {
#pragma unroll
  for (int n = RT / 2, o = 16; n >= 1; n >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int r = 0; r < n; ++r) {
      const float mine = up ? v[n + r] : v[r], give = up ? v[r] : v[n + r];
      v[r] = mine + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  float s = v[0];
#pragma unroll
  for (int o = 32 / RT / 2; o >= 1; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

template <int MODE, int RT>
__global__ void __launch_bounds__(F32_WARPS * 32)
gemm_few_f32_kernel(const FewParams P) {
  constexpr bool NORM = MODE == FEW_ROPE || MODE == FEW_SWIGLU;
  pdl_launch_dependents();
  const int lane = threadIdx.x & 31, u = blockIdx.x * F32_WARPS + (threadIdx.x >> 5);
  if (u >= P.units) return;
  const float *ra, *rb;
  unit_rows<MODE>(P, u, ra, rb);
  auto ld4 = [](const float *p) { return *reinterpret_cast<const float4 *>(p); };
  auto mul4 = [](float4 a, float4 b) { return make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w); };
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  float4 wa[WPRE], wb[WPRE];
#pragma unroll
  for (int i = 0; i < WPRE; ++i) {
    const int k = (lane + 32 * i) * 4;
    const bool in = k < P.K;
    wa[i] = in ? ld4(ra + k) : zero;
    wb[i] = in ? ld4(rb + k) : zero;
    if (NORM && in) {
      const float4 gg = ld4(P.gain + k);
      wa[i] = mul4(wa[i], gg);
      wb[i] = mul4(wb[i], gg);
    }
  }
  pdl_wait();
  const int r0 = blockIdx.y * RT, rows = P.R - r0 < RT ? P.R - r0 : RT;
  const float *x = P.x + (size_t)r0 * P.K;
  float a[RT], b[RT], q[RT];
#pragma unroll
  for (int r = 0; r < RT; ++r) a[r] = b[r] = q[r] = 0.f;
  auto step = [&](const float4 &va, const float4 &vb, int k) {
#pragma unroll
    for (int r = 0; r < RT; ++r) {
      const float4 xx = ld4(x + (size_t)(r < rows ? r : 0) * P.K + k);     // rows beyond R repeat the first, dropped below
      a[r] = fmaf(va.x, xx.x, a[r]); a[r] = fmaf(va.y, xx.y, a[r]); a[r] = fmaf(va.z, xx.z, a[r]); a[r] = fmaf(va.w, xx.w, a[r]);
      b[r] = fmaf(vb.x, xx.x, b[r]); b[r] = fmaf(vb.y, xx.y, b[r]); b[r] = fmaf(vb.z, xx.z, b[r]); b[r] = fmaf(vb.w, xx.w, b[r]);
      if (NORM) { q[r] = fmaf(xx.x, xx.x, q[r]); q[r] = fmaf(xx.y, xx.y, q[r]); q[r] = fmaf(xx.z, xx.z, q[r]); q[r] = fmaf(xx.w, xx.w, q[r]); }
    }
  };
#pragma unroll
  for (int i = 0; i < WPRE; ++i) {
    const int k = (lane + 32 * i) * 4;
    if (k < P.K) step(wa[i], wb[i], k);
  }
#pragma unroll 1
  for (int k = (lane + 32 * WPRE) * 4; k < P.K; k += 128) {
    float4 va = ld4(ra + k), vb = ld4(rb + k);
    if (NORM) {
      const float4 gg = ld4(P.gain + k);
      va = mul4(va, gg);
      vb = mul4(vb, gg);
    }
    step(va, vb, k);
  }
  const float sa = reduce_rows<RT>(a, lane), sb = reduce_rows<RT>(b, lane);
  float s = 1.f;
  if (NORM) s = rsqrtf(reduce_rows<RT>(q, lane) * P.inv_h + P.eps);
  constexpr int LPR = 32 / RT;                        // lanes that hold the same row
  const int r = r0 + lane / LPR;
  if (lane % LPR == 0 && r < P.R) finish_unit<MODE>(P, u, r, sa, sb, s);
}

}  // namespace

// The sizes at which every kernel is latency; 16-byte rows.  Every multiply of the layers has to be one of them.
// (fp32 forwards, fused / one kernel per step, us: hidden 512 in four layers, 30 rows 213 / 285, 60 rows 318 / 560; hidden
// 1024, 15 rows 327 / 785.  The line is low: hidden 1024 and 60 rows, past it, would take 842 fused against 1306.)
bool few_supported(const void *X, int R, int K, int units, const void *const *W, int n_w) {
  if (R < 1 || units < 1 || ((uintptr_t)X & 15)) return false;
  for (int i = 0; i < n_w; ++i)
    if ((uintptr_t)W[i] & 15) return false;
  return K % 4 == 0 && (double)R * K * units <= 1e8;
}

cudaError_t gemm_few(Launch L, const FewJob &j, int num_sms) {
  FewParams P;
  memset(&P, 0, sizeof(P));
  P.x = (const float *)j.X;
  P.w0 = (const float *)j.W[0]; P.w1 = (const float *)j.W[1]; P.w2 = (const float *)j.W[2];
  P.R = j.R; P.K = j.K; P.n_out = j.n_out;
  P.units = j.mode == FEW_ROPE ? 3 * j.n_out / 2 : (j.mode == FEW_SWIGLU ? j.n_out : (j.n_out + 1) / 2);
  P.inv_h = 1.f / (float)j.K; P.eps = j.eps; P.gain = (const float *)j.gain;
  P.bias = (const float *)j.bias; P.xres = j.x; P.out = (float *)j.out; P.out2 = j.out2;
  P.plan = j.plan; P.q_out = j.q_out; P.kc = (float *)j.k_cache; P.vc = (float *)j.v_cache;
  P.rows_per_seq = j.rows_per_seq; P.n_heads = j.n_heads; P.head_dim = j.head_dim; P.S_max = j.S_max;
  auto run = [&](auto mode) -> cudaError_t {
    constexpr int M = decltype(mode)::value;
    const unsigned gx = (unsigned)((P.units + F32_WARPS - 1) / F32_WARPS);
    auto go = [&](auto *kern, int rt) {
      return launch_k(kern, dim3(gx, (unsigned)((P.R + rt - 1) / rt)), dim3(F32_WARPS * 32), 0, L.st, L.pdl, P);
    };
    // rows per warp: few rows keep the chains short, eight share the weights where blocks abound
    if (P.R <= 2) return go(gemm_few_f32_kernel<M, 2>, 2);
    if (P.R <= 4 || (size_t)gx * ((P.R + 3) / 4) <= 4 * (size_t)num_sms) return go(gemm_few_f32_kernel<M, 4>, 4);
    return go(gemm_few_f32_kernel<M, 8>, 8);
  };
  if (j.mode == FEW_ROPE) return run(std::integral_constant<int, FEW_ROPE>{});
  if (j.mode == FEW_SWIGLU) return run(std::integral_constant<int, FEW_SWIGLU>{});
  return run(std::integral_constant<int, FEW_RESIDUAL>{});
}

}  // namespace koala
