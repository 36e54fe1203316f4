// Row-wise kernels of the decoder layers and heads: embedding gather, RMSNorm / residual
// epilogues, RoPE + KV-cache write, SwiGLU, arg-max and top-k with log-probabilities.  All statistics are fp32.
#include "common.cuh"
#include "row_ops.cuh"

namespace koala {

namespace {

__device__ __forceinline__ float silu(float v) { return v / (1.f + expf(-v)); }
// (not inlined: an exponential and a division, used a dozen times by kernels that run their instructions once)
__device__ __noinline__ float silu_f(float v) { return silu(v); }

// ------------------------------------------------------------------------------- embedding + norm
template <typename T>
__global__ void embed_norm_kernel(const int32_t *tok, const T *__restrict__ E,
                                  const T *__restrict__ g, float *__restrict__ x,
                                  T *__restrict__ xn, T *__restrict__ xn_lo, int H, int V, float eps) {
  __shared__ float red[32];
  pdl_launch_dependents();
  pdl_wait();
  const int r = blockIdx.x;
  int t = tok[r];
  t = t < 0 ? 0 : (t >= V ? V - 1 : t);
  const T *e = E + (size_t)t * H;
  float ss = 0.f;
  for (int i = threadIdx.x; i < H; i += blockDim.x) {
    const float v = to_f(e[i]);
    x[(size_t)r * H + i] = v;
    ss += v * v;
  }
  const float inv = rsqrtf(block_sum(ss, red) / (float)H + eps);
  for (int i = threadIdx.x; i < H; i += blockDim.x)
    store_operand(xn, xn_lo, (size_t)r * H + i, x[(size_t)r * H + i] * inv * to_f(g[i]));
}

// ------------------------------------------------------------------------------- row epilogue
template <typename T>
__global__ void row_epilogue_kernel(int mode, float *__restrict__ x, SplitIn P,
                                    const T *__restrict__ bias, const T *__restrict__ g,
                                    T *__restrict__ xn, T *__restrict__ xn_lo,
                                    float *__restrict__ out_f32, RowMap out_map, int H, float eps) {
  __shared__ float red[32];
  pdl_launch_dependents();
  pdl_wait();
  const int r = blockIdx.x;
  float *xr = x + (size_t)r * H;
  float ss = 0.f;
  for (int i = threadIdx.x; i < H; i += blockDim.x) {
    float p = P.at(r, i);
    float v;
    if (mode == 0) v = xr[i] + p;
    else if (mode == 1) v = p + to_f(bias[i]);
    else v = xr[i] + silu_f(p + to_f(bias[i]));
    xr[i] = v;
    ss += v * v;
  }
  float inv = 1.f;
  if (g != nullptr) inv = rsqrtf(block_sum(ss, red) / (float)H + eps);
  for (int i = threadIdx.x; i < H; i += blockDim.x) {
    float n = xr[i];
    if (g != nullptr) n = n * inv * to_f(g[i]);
    if (xn != nullptr) store_operand(xn, xn_lo, (size_t)r * H + i, n);
    if (out_f32 != nullptr) out_f32[(size_t)out_map(r) * H + i] = n;
  }
}

// Vectorised variant for H % 4 == 0: one CTA per row, every thread owns up to VPT groups of four
// consecutive columns, keeps them in registers between the two passes and issues all split-K
// partial loads of a group back to back.
// NS bounds the partial sums of a column: all of them are requested before the first is added - one
// trip to L2 instead of one per partial; the additions keep the slot order.  SK: the number varies
// with the tile (stream-K).  NS is a template argument so that the code is as short as the launch
// allows: with one body for every factor the rotary kernel was 42 KB of instructions run once each,
// and fetching them was most of its time (see the dispatch, FOR_SPLIT).
template <int NS, bool SK>
__device__ __forceinline__ int slots_at(const SplitIn &P, int r, int c) {
  if (!SK) return P.n;
  return sk_count(P.tile_of(r, c), P.sk_ctas, P.sk_uinv, P.sk_kb);
}
template <int NS>
__device__ __forceinline__ float4 split_sum4(const SplitIn &P, int r, int c, int k) {
  const float *q = P.p + (size_t)r * P.ld + c;
  float4 u[NS];
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    u[s] = (s == 0 || s < k) ? *reinterpret_cast<const float4 *>(q) : make_float4(0.f, 0.f, 0.f, 0.f);
    q += P.stride;
  }
  float4 v = u[0];
#pragma unroll
  for (int s = 1; s < NS; ++s) { v.x += u[s].x; v.y += u[s].y; v.z += u[s].z; v.w += u[s].w; }
  return v;
}
template <typename T, int VPT, int NS, bool SK>
__global__ void __launch_bounds__(1024)
row_epilogue_vec_kernel(int mode, float *__restrict__ x, SplitIn P, const T *__restrict__ bias,
                        const T *__restrict__ g, T *__restrict__ xn, T *__restrict__ xn_lo,
                        float *__restrict__ out_f32, RowMap out_map, int H, float eps) {
  __shared__ float red[32];
  pdl_launch_dependents();
  pdl_wait();
  const int r = blockIdx.x;
  float *xr = x + (size_t)r * H;
  float4 v[VPT];
  float ss = 0.f;
#pragma unroll
  for (int k = 0; k < VPT; ++k) {
    const int c = (threadIdx.x + k * blockDim.x) * 4;
    if (c < H) {
      const float4 p = split_sum4<NS>(P, r, c, slots_at<NS, SK>(P, r, c));
      float4 o;
      if (mode == 0) {
        const float4 xv = *reinterpret_cast<const float4 *>(xr + c);
        o = make_float4(xv.x + p.x, xv.y + p.y, xv.z + p.z, xv.w + p.w);
      } else {
        const float4 b = load4<T>(bias + c);
        if (mode == 1) {
          o = make_float4(p.x + b.x, p.y + b.y, p.z + b.z, p.w + b.w);
        } else {
          const float4 xv = *reinterpret_cast<const float4 *>(xr + c);
          o = make_float4(xv.x + silu_f(p.x + b.x), xv.y + silu_f(p.y + b.y), xv.z + silu_f(p.z + b.z),
                          xv.w + silu_f(p.w + b.w));
        }
      }
      *reinterpret_cast<float4 *>(xr + c) = o;
      v[k] = o;
      ss += o.x * o.x + o.y * o.y + o.z * o.z + o.w * o.w;
    }
  }
  // the gains are fetched before the block-wide reduction so that their latency hides behind it
  float4 gg[VPT];
#pragma unroll
  for (int k = 0; k < VPT; ++k) {
    const int c = (threadIdx.x + k * blockDim.x) * 4;
    gg[k] = (g != nullptr && c < H) ? load4<T>(g + c) : make_float4(1.f, 1.f, 1.f, 1.f);
  }
  float inv = 1.f;
  if (g != nullptr) inv = rsqrtf(block_sum(ss, red) / (float)H + eps);
#pragma unroll
  for (int k = 0; k < VPT; ++k) {
    const int c = (threadIdx.x + k * blockDim.x) * 4;
    if (c < H) {
      float4 n = v[k];
      if (g != nullptr) {
        n = make_float4(n.x * inv * gg[k].x, n.y * inv * gg[k].y, n.z * inv * gg[k].z, n.w * inv * gg[k].w);
      }
      if (xn != nullptr) store_operand4(xn, xn_lo, (size_t)r * H + c, n);
      if (out_f32 != nullptr) *reinterpret_cast<float4 *>(out_f32 + (size_t)out_map(r) * H + c) = n;
    }
  }
}

// Residual update with the RMSNorm deferred: grid (chunks of 1024 columns, rows).  Many CTAs per
// row pull the split-K partial sums; the row statistic is left as per-chunk partial sums of
// squares for the consumer of the next GEMM's output (RowScale).
template <typename T, int NS, bool SK>
__global__ void __launch_bounds__(256)
row_update_kernel(float *__restrict__ x, SplitIn P, const T *__restrict__ g, T *__restrict__ xg,
                  T *__restrict__ xg_lo, float *__restrict__ sumsq, int H) {
  __shared__ float red[32];
  pdl_launch_dependents();
  pdl_wait();
  const int r = blockIdx.y;
  const int c = (blockIdx.x * 256 + threadIdx.x) * 4;
  float ss = 0.f;
  if (c < H) {
    const float4 gg = load4<T>(g + c);
    const float4 p = split_sum4<NS>(P, r, c, slots_at<NS, SK>(P, r, c));
    float *xr = x + (size_t)r * H + c;
    const float4 xv = *reinterpret_cast<const float4 *>(xr);
    const float4 o = make_float4(xv.x + p.x, xv.y + p.y, xv.z + p.z, xv.w + p.w);
    *reinterpret_cast<float4 *>(xr) = o;
    ss = o.x * o.x + o.y * o.y + o.z * o.z + o.w * o.w;
    store_operand4(xg, xg_lo, (size_t)r * H + c, make_float4(o.x * gg.x, o.y * gg.y, o.z * gg.z, o.w * gg.w));
  }
  const float tot = block_sum(ss, red);
  if (threadIdx.x == 0) sumsq[(size_t)r * ROW_SUMS + blockIdx.x] = tot;
}

template <typename T, int NS>
__global__ void __launch_bounds__(256)
resblock_update_kernel(float *__restrict__ x, SplitIn P, HeadTab tab, T *__restrict__ xn, T *__restrict__ xn_lo, int H) {
  pdl_launch_dependents();
  pdl_wait();
  const int r = blockIdx.y;
  const int c = (blockIdx.x * 256 + threadIdx.x) * 4;
  if (c >= H) return;
  const int head = r / tab.rows_per_head;
  P.p = tab.p[head];
  const float4 p = split_sum4<NS>(P, r - head * tab.rows_per_head, c, P.n);
  const float4 b = load4<T>(reinterpret_cast<const T *>(tab.bias[head]) + c);
  float *xr = x + (size_t)r * H + c;
  const float4 xv = *reinterpret_cast<const float4 *>(xr);
  const float4 o = make_float4(xv.x + silu_f(p.x + b.x), xv.y + silu_f(p.y + b.y), xv.z + silu_f(p.z + b.z),
                               xv.w + silu_f(p.w + b.w));
  *reinterpret_cast<float4 *>(xr) = o;
  store_operand4(xn, xn_lo, (size_t)r * H + c, o);
}

// ------------------------------------------------------------------------------- EAGLE fc input
template <typename T>
__global__ void eagle_concat_kernel(const float *feat_src,
                                    const int32_t *row_src,
                                    const int32_t *row_tok, const T *__restrict__ E,
                                    T *__restrict__ cat, T *__restrict__ cat_lo, int H, int V) {
  pdl_launch_dependents();
  pdl_wait();
  const int r = blockIdx.x;
  const int src = row_src[r];
  int t = row_tok[r];
  t = t < 0 ? 0 : (t >= V ? V - 1 : t);
  const float *f = feat_src + (size_t)src * H;
  const T *e = E + (size_t)t * H;
  const size_t base = (size_t)r * 2 * H;
  for (int i = threadIdx.x; i < H; i += blockDim.x) {
    store_operand(cat, cat_lo, base + i, f[i]);
    cat[base + H + i] = e[i];
    if (cat_lo != nullptr) cat_lo[base + H + i] = from_f<T>(0.f);
  }
}

template <typename T>
__global__ void cast_rows_kernel(const float *src, const int32_t *row_src,
                                 T *__restrict__ dst, T *__restrict__ dst_lo,
                                 float *__restrict__ dst32, int dst32_stride, int H) {
  pdl_launch_dependents();
  pdl_wait();
  const int r = blockIdx.x;
  const int s = row_src ? row_src[r] : r;
  for (int i = threadIdx.x; i < H; i += blockDim.x) {
    const float v = src[(size_t)s * H + i];
    store_operand(dst, dst_lo, (size_t)r * H + i, v);
    if (dst32) dst32[(size_t)r * dst32_stride * H + i] = v;
  }
}

// Rows of a prompt forward that belong to their sequence's last part, to where a verification leaves them.
template <typename T>
__global__ void ingest_last_kernel(const __grid_constant__ IngestBlocks k, const float *hid, float *__restrict__ verify_hid,
                                   T *__restrict__ xn, T *__restrict__ xn_lo, int N, int n_max, int H) {
  pdl_launch_dependents();
  pdl_wait();
  const int v = blockIdx.x, i = blockIdx.y, u = i - k.last[v];
  if (i >= k.count[v] || u < 0 || u >= n_max) return;
  const float *src = hid + (size_t)(v * k.q + i) * H;
  float *to = verify_hid + (size_t)(k.seq[v] * N + u) * H;
  const size_t at = (size_t)(k.seq[v] * n_max + u) * H;
  for (int d = threadIdx.x; d < H; d += blockDim.x) {
    const float x = src[d];
    to[d] = x;
    store_operand(xn, xn_lo, at + d, x);
  }
}

__global__ void reduce_splits_kernel(SplitIn P, float *__restrict__ Y, int ldy, int ncols) {
  pdl_launch_dependents();
  pdl_wait();
  const int r = blockIdx.y;
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c < ncols) Y[(size_t)r * ldy + c] = P.at(r, c);
}

// ------------------------------------------------------------------------------- RoPE + KV write
// grid (R, n_heads), block head_dim/2: thread i rotates the pair (i, i + head_dim/2).
template <typename T>
__global__ void rope_kv_kernel(SplitIn qkv, RowScale sc, RowPlan plan, float *__restrict__ q_out,
                               bf16 *__restrict__ qp_hi, bf16 *__restrict__ qp_lo,
                               T *__restrict__ k_cache, T *__restrict__ v_cache, int rows_per_seq,
                               int n_heads, int head_dim, int S_max) {
  pdl_wait();
  pdl_launch_dependents();                // in this order: see rope_kv_write
  const int r = blockIdx.x, h = blockIdx.y, i = threadIdx.x;
  const int half = head_dim >> 1, H = n_heads * head_dim;
  const int b = plan.cache_of(r / rows_per_seq);
  const int slot = plan.slot[r];
  const float2 cs = plan.rope[(size_t)r * half + i];
  const int c0 = h * head_dim + i, c1 = c0 + half;
  const float rs = sc.of(r);
  const float q0 = rs * qkv.at(r, c0), q1 = rs * qkv.at(r, c1);
  const float qr0 = q0 * cs.x - q1 * cs.y, qr1 = q1 * cs.x + q0 * cs.y;
  q_out[(size_t)r * H + c0] = qr0;
  q_out[(size_t)r * H + c1] = qr1;
  if (qp_hi != nullptr) {
    store_operand(qp_hi, qp_lo, (size_t)r * H + c0, qr0);
    store_operand(qp_hi, qp_lo, (size_t)r * H + c1, qr1);
  }
  if (slot < 0 || slot >= S_max) return;
  const float k0 = rs * qkv.at(r, H + c0), k1 = rs * qkv.at(r, H + c1);
  const float v0 = rs * qkv.at(r, 2 * H + c0), v1 = rs * qkv.at(r, 2 * H + c1);
  const size_t base = (((size_t)b * n_heads + h) * S_max + slot) * head_dim;
  k_cache[base + i] = from_f<T>(k0 * cs.x - k1 * cs.y);
  k_cache[base + i + half] = from_f<T>(k1 * cs.x + k0 * cs.y);
  v_cache[base + i] = from_f<T>(v0);
  v_cache[base + i + half] = from_f<T>(v1);
}

// One CTA per row (or ROWS of them); a thread rotates two adjacent pairs (i, i+1) and (i + half, i + half + 1) of
// one head with 8-byte loads.
template <int NS>
__device__ __forceinline__ float2 split_sum2(const SplitIn &P, int r, int c, int k) {
  const float *q = P.p + (size_t)r * P.ld + c;
  float2 u[NS];
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    u[s] = (s == 0 || s < k) ? *reinterpret_cast<const float2 *>(q) : make_float2(0.f, 0.f);
    q += P.stride;
  }
  float2 v = u[0];
#pragma unroll
  for (int s = 1; s < NS; ++s) { v.x += u[s].x; v.y += u[s].y; }
  return v;
}
__device__ __forceinline__ void store2(float *p, float a, float b) { *reinterpret_cast<float2 *>(p) = make_float2(a, b); }
__device__ __forceinline__ void store2(bf16 *p, float a, float b) {
  *reinterpret_cast<__nv_bfloat162 *>(p) = __floats2bfloat162_rn(a, b);
}
// ROWS: consecutive rows of a thread, see rope_rows_per_thread.
template <typename T, int NS, bool SK, int ROWS>
__global__ void __launch_bounds__(128)
rope_kv_vec_kernel(SplitIn qkv, RowScale sc, RowPlan plan, float *__restrict__ q_out, bf16 *__restrict__ qp_hi,
                   bf16 *__restrict__ qp_lo, T *__restrict__ k_cache, T *__restrict__ v_cache, int rows_per_seq,
                   int n_heads, int head_dim, int S_max, int R) {
  pdl_wait();
  pdl_launch_dependents();                // in this order: see rope_kv_write
  const int r0 = blockIdx.x * ROWS;
  const int half = head_dim >> 1, H = n_heads * head_dim, hq = half >> 1;
  // grid.y slices the row's work so that many SMs pull the partial sums
  const int p = blockIdx.y * blockDim.x + threadIdx.x;
  if (p < n_heads * hq) {
    const int h = p / hq, i = (p - h * hq) * 2;
    const int c0 = h * head_dim + i, c1 = c0 + half;
    // all partial sums of this thread are requested before the first store (a head lies in one weight
    // tile where tiles are dealt unevenly: there head_dim is 128 and a tile is a multiple of it)
    const int kq = slots_at<NS, SK>(qkv, r0, c0), kk = slots_at<NS, SK>(qkv, r0, H + c0), kv = slots_at<NS, SK>(qkv, r0, 2 * H + c0);
#pragma unroll
    for (int ri = 0; ri < ROWS; ++ri) {
      const int r = r0 + ri;
      if (ROWS > 1 && r >= R) break;
      const int b = plan.cache_of(r / rows_per_seq);
      const int slot = plan.slot[r];
      const bool wr = slot >= 0 && slot < S_max;
      const float rs = sc.of(r);
      const float4 cs = *reinterpret_cast<const float4 *>(&plan.rope[(size_t)r * half + i]);   // c0 s0 c1 s1
      float2 qa = split_sum2<NS>(qkv, r, c0, kq), qb = split_sum2<NS>(qkv, r, c1, kq);
      float2 ka = split_sum2<NS>(qkv, r, H + c0, kk), kb = split_sum2<NS>(qkv, r, H + c1, kk);
      float2 va = split_sum2<NS>(qkv, r, 2 * H + c0, kv), vb = split_sum2<NS>(qkv, r, 2 * H + c1, kv);
      qa.x *= rs; qa.y *= rs; qb.x *= rs; qb.y *= rs;
      const float2 ra = make_float2(qa.x * cs.x - qb.x * cs.y, qa.y * cs.z - qb.y * cs.w);
      const float2 rb = make_float2(qb.x * cs.x + qa.x * cs.y, qb.y * cs.z + qa.y * cs.w);
      store2(q_out + (size_t)r * H + c0, ra.x, ra.y);
      store2(q_out + (size_t)r * H + c1, rb.x, rb.y);
      if (qp_hi != nullptr) {      // the same values as a bf16 pair (value + rounding residual)
        const __nv_bfloat162 ha = __floats2bfloat162_rn(ra.x, ra.y), hb = __floats2bfloat162_rn(rb.x, rb.y);
        const float2 fa = __bfloat1622float2(ha), fb = __bfloat1622float2(hb);
        *reinterpret_cast<__nv_bfloat162 *>(qp_hi + (size_t)r * H + c0) = ha;
        *reinterpret_cast<__nv_bfloat162 *>(qp_hi + (size_t)r * H + c1) = hb;
        *reinterpret_cast<__nv_bfloat162 *>(qp_lo + (size_t)r * H + c0) = __floats2bfloat162_rn(ra.x - fa.x, ra.y - fa.y);
        *reinterpret_cast<__nv_bfloat162 *>(qp_lo + (size_t)r * H + c1) = __floats2bfloat162_rn(rb.x - fb.x, rb.y - fb.y);
      }
      if (!wr) continue;
      ka.x *= rs; ka.y *= rs; kb.x *= rs; kb.y *= rs;
      va.x *= rs; va.y *= rs; vb.x *= rs; vb.y *= rs;
      const size_t base = (((size_t)b * n_heads + h) * S_max + slot) * head_dim + i;
      store2(k_cache + base, ka.x * cs.x - kb.x * cs.y, ka.y * cs.z - kb.y * cs.w);
      store2(k_cache + base + half, kb.x * cs.x + ka.x * cs.y, kb.y * cs.z + ka.y * cs.w);
      store2(v_cache + base, va.x, va.y);
      store2(v_cache + base + half, vb.x, vb.y);
    }
  }
}

// ------------------------------------------------------------------------------- SwiGLU
template <typename T>
__global__ void swiglu_kernel(SplitIn gu, RowScale sc, T *__restrict__ act, T *__restrict__ act_lo, int F) {
  pdl_launch_dependents();
  pdl_wait();
  const int r = blockIdx.y;
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= F) return;
  const float rs = sc.of(r);
  store_operand(act, act_lo, (size_t)r * F + f, silu_f(rs * gu.at(r, f)) * (rs * gu.at(r, F + f)));
}

// SiLU is inlined: behind the calls of silu_f the second operand's partial sums were not requested before the first's were
// used (us per launch, calls / inlined: one row of the 7B shape 3.18 / 2.95, 64 rows 5.8 / 5.5, 512 rows 24.4 / 22.7, prompts
// of 509 tokens 22.5 / 20.9, 860 tokens 35.4 / 33.8, 13B 46.7 / 43.8).  One row per thread; one / two / four, inlined, at the
// power cap: prompts 7B 360 tokens 14.4 / 15.4 / 17.6, 509 20.9 / 21.5 / 22.0, 860 34.2 / 34.5 / 33.6, 1020 40.6 / 40.9 / 41.7, 13B
// 509 26.1 / 26.9 / 25.9, 860 44.1 / 42.6 / 42.2, 1020 52.2 / 51.2 / 49.4, verifications of 512 rows 19.7 / 21.7 / 22.0 and 25.3 / 26.7
// / 28.3: four gain in the longest 13B prompts only, 0.3 % of a pass at most.
template <typename T, int NS, bool SK>
__global__ void __launch_bounds__(256) swiglu_vec_kernel(SplitIn gu, RowScale sc, T *__restrict__ act, T *__restrict__ act_lo, int F) {
  pdl_launch_dependents();
  pdl_wait();
  const int r = blockIdx.y;
  const int f = (blockIdx.x * blockDim.x + threadIdx.x) * 4;
  if (f >= F) return;
  const float rs = sc.of(r);
  const float4 a = split_sum4<NS>(gu, r, f, slots_at<NS, SK>(gu, r, f)), b = split_sum4<NS>(gu, r, F + f, slots_at<NS, SK>(gu, r, F + f));
  store_operand4(act, act_lo, (size_t)r * F + f,
                 make_float4(silu(rs * a.x) * (rs * b.x), silu(rs * a.y) * (rs * b.y),
                             silu(rs * a.z) * (rs * b.z), silu(rs * a.w) * (rs * b.w)));
}

// ------------------------------------------------------------------------------- arg-max / top-k
struct ValIdx {
  float v;
  int i;
};
__device__ __forceinline__ ValIdx better(ValIdx a, ValIdx b) {
  return (b.v > a.v || (b.v == a.v && b.i < a.i)) ? b : a;
}
__device__ __forceinline__ ValIdx block_argmax(ValIdx x, ValIdx *red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    ValIdx y;
    y.v = __shfl_xor_sync(0xffffffffu, x.v, o);
    y.i = __shfl_xor_sync(0xffffffffu, x.i, o);
    x = better(x, y);
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  if (lane == 0) red[w] = x;
  __syncthreads();
  if (w == 0) {
    ValIdx y = lane < nw ? red[lane] : ValIdx{-INFINITY, 0x7fffffff};
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      ValIdx z;
      z.v = __shfl_xor_sync(0xffffffffu, y.v, o);
      z.i = __shfl_xor_sync(0xffffffffu, y.i, o);
      y = better(y, z);
    }
    if (lane == 0) red[0] = y;
  }
  __syncthreads();
  x = red[0];
  __syncthreads();
  return x;
}

// Arg-max of rows wider than the kernel below takes.
__global__ void argmax_rows_kernel(const float *logits, int32_t *__restrict__ out, float *spread, RowMap map, int V) {
  __shared__ ValIdx red[32];
  pdl_launch_dependents();
  pdl_wait();
  const float *row = logits + (size_t)blockIdx.x * V;
  const int to = map(blockIdx.x);
  ValIdx best{-INFINITY, 0x7fffffff};
  for (int i = threadIdx.x; i < V; i += blockDim.x) {
    const float v = row[i];
    best = better(best, ValIdx{v, i});
    if (spread != nullptr) spread[(size_t)to * V + i] = v;
  }
  best = block_argmax(best, red);
  if (threadIdx.x == 0) out[to] = best.i;
}

// Per row: the k largest logits (ties: smaller id) and their natural-log softmax probabilities.
// The row is staged in shared memory; each round removes the current maximum.
__global__ void topk_logp_kernel(const float *logits, int32_t *__restrict__ tok,
                                 float *__restrict__ logp, int V, int k) {
  extern __shared__ float srow[];
  __shared__ ValIdx red[32];
  __shared__ float redf[32];
  pdl_launch_dependents();
  pdl_wait();
  const float *row = logits + (size_t)blockIdx.x * V;
  ValIdx best{-INFINITY, 0x7fffffff};
  for (int i = threadIdx.x; i < V; i += blockDim.x) {
    const float v = row[i];
    srow[i] = v;
    best = better(best, ValIdx{v, i});
  }
  best = block_argmax(best, red);
  const float mx = best.v;
  float se = 0.f;
  for (int i = threadIdx.x; i < V; i += blockDim.x) se += expf(srow[i] - mx);
  const float lse = mx + logf(block_sum(se, redf));
  for (int j = 0; j < k; ++j) {
    if (j > 0) {
      best = ValIdx{-INFINITY, 0x7fffffff};
      for (int i = threadIdx.x; i < V; i += blockDim.x) best = better(best, ValIdx{srow[i], i});
      best = block_argmax(best, red);
    }
    if (threadIdx.x == 0) {
      tok[(size_t)blockIdx.x * k + j] = best.i;
      logp[(size_t)blockIdx.x * k + j] = best.v - lse;
      srow[best.i] = -INFINITY;
    }
    __syncthreads();
  }
}

// The same result for V <= 32768 and k <= 32, the row read once: one CTA per row up to 4096 columns, beyond
// that eight as a thread-block cluster.  A CTA holds its part of the row, 16 strided elements per thread in
// registers; every warp extracts the k best of its 512 elements, warp 0 merges the eight sorted lists, and
// CTA 0 merges the parts' lists and (max, sum of exponentials) pairs through distributed shared memory.
// Values are compared as order-preserving integers, so that a round is two warp-wide integer reductions
// (largest key, then smallest id among equals) and only the winning lane looks at its elements again.
// logp == nullptr: only the ids are wanted (the arg-max of a row is its top-1), no exponentials.
// spread: the row is also copied to row map(r) of it.
// (Rounds of five shuffle steps over (value, id) pairs with 16 comparisons in every lane took 20 us per call
// at V = 32000, k = 10 in a running step, and a 32-element body for narrow rows 12 us at V = 1024.)
constexpr int TKP = 8;            // CTAs per row of more than 256 * TKE columns
constexpr int TKE = 16;           // elements per thread
constexpr uint32_t NO_KEY = 0u;   // below every number's key
constexpr uint32_t NO_ID = 0x7fffffffu;
__device__ __forceinline__ uint32_t order_key(float v) {
  const uint32_t b = __float_as_uint(v + 0.f);           // -0 counts as +0
  return v == v ? b ^ ((uint32_t)((int32_t)b >> 31) | 0x80000000u) : NO_KEY;
}
__device__ __forceinline__ float key_value(uint32_t k) {
  return __uint_as_float(k ^ ((k >> 31) ? 0x80000000u : 0xffffffffu));
}

// Merges `lists` lists of k (key, id) pairs, each sorted from best to worst, into dst[0..k): lane l of the
// calling warp walks list l.
__device__ __noinline__ void merge_lists(const uint2 *src, int lists, int k, uint2 *dst) {
  const int lane = threadIdx.x & 31;
  int at = 0;
  uint2 head = lane < lists ? src[lane * k] : make_uint2(NO_KEY, NO_ID);
#pragma unroll 1
  for (int rnd = 0; rnd < k; ++rnd) {
    const uint32_t m = __reduce_max_sync(0xffffffffu, head.x);
    const uint32_t id = __reduce_min_sync(0xffffffffu, head.x == m ? head.y : 0xffffffffu);
    if (head.x == m && head.y == id) {
      dst[rnd] = head;
      ++at;
      head = lane < lists && at < k ? src[lane * k + at] : make_uint2(NO_KEY, NO_ID);
    }
  }
  __syncwarp();
}

__global__ void __launch_bounds__(256)
topk_logp_cluster_kernel(const float *logits, int32_t *__restrict__ tok, float *__restrict__ logp, float *spread,
                         RowMap map, int V, int k) {
  __shared__ __align__(8) uint2 cand[8 * 32];   // the warps' lists, then the parts'
  __shared__ __align__(8) uint2 mine[32];       // this CTA's k best, read by CTA 0
  __shared__ __align__(8) uint2 result[32];
  __shared__ __align__(8) float s_ms[2];        // this CTA's (max, sum of exp(v - max))
  __shared__ float redf[32];
  pdl_launch_dependents();
  pdl_wait();
  const int part = blockIdx.x, parts = gridDim.x, r = map(blockIdx.y);   // the row is read at blockIdx.y, its results go to r
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int chunk = (((V + parts - 1) / parts) + 255) & ~255;      // ids per CTA, a multiple of 256
  const int base = part * chunk;
  const int end = min(chunk, V - base);                            // this CTA's elements (may be <= 0)
  const float *row = logits + (size_t)blockIdx.y * V + base;
  float vals[TKE];
  float mx = -INFINITY;
#pragma unroll
  for (int j = 0; j < TKE; ++j) {
    const int o = tid + 256 * j;
    vals[j] = o < end ? row[o] : -INFINITY;
    mx = fmaxf(mx, vals[j]);
  }
  if (spread != nullptr) {
    float *to = spread + (size_t)r * V + base;
#pragma unroll
    for (int j = 0; j < TKE; ++j)
      if (tid + 256 * j < end) to[tid + 256 * j] = vals[j];
  }
  if (logp != nullptr) {
    mx = warp_max(mx);
    if (lane == 0) redf[w] = mx;
    __syncthreads();
    mx = warp_max(lane < 8 ? redf[lane] : -INFINITY);
    __syncthreads();
    float se = 0.f;
    if (mx != -INFINITY) {
#pragma unroll 4
      for (int j = 0; j < TKE; ++j) se += expf(vals[j] - mx);
    }
    se = warp_sum(se);
    if (lane == 0) redf[w] = se;
    __syncthreads();
    se = warp_sum(lane < 8 ? redf[lane] : 0.f);
    if (tid == 0) { s_ms[0] = mx; s_ms[1] = se; }
  }
  // this warp's k best
  uint32_t keys[TKE];
#pragma unroll
  for (int j = 0; j < TKE; ++j) keys[j] = tid + 256 * j < end ? order_key(vals[j]) : NO_KEY;
  uint32_t best = NO_KEY;
  int at = TKE;                     // rescan first
#pragma unroll 1
  for (int rnd = 0, scan = 1; rnd < k; ++rnd) {
    if (scan) {
      best = NO_KEY;
      int next = 0;
#pragma unroll
      for (int j = 0; j < TKE; ++j) {
        if (j == at) keys[j] = NO_KEY;                   // taken in the round before
        if (keys[j] > best) { best = keys[j]; next = j; }   // the first of equals: the smaller id
      }
      at = next;
    }
    const uint32_t id = best == NO_KEY ? NO_ID : (uint32_t)(base + tid + 256 * at);
    const uint32_t m = __reduce_max_sync(0xffffffffu, best);
    const uint32_t win = __reduce_min_sync(0xffffffffu, best == m ? id : 0xffffffffu);
    if (lane == 0) cand[w * k + rnd] = make_uint2(m, win);
    scan = m != NO_KEY && best == m && id == win;
  }
  __syncthreads();
  if (w == 0) merge_lists(cand, 8, k, parts > 1 ? mine : result);
  if (parts > 1) {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  }
  if (part == 0 && w == 0) {
    float M = 0.f, S = 1.f;
    if (logp != nullptr && parts == 1) { M = s_ms[0]; S = s_ms[1]; }
    if (parts > 1) {
      // every part's list and (max, sum) into this CTA, then the same merge
      const uint32_t a_mine = (uint32_t)__cvta_generic_to_shared(&mine[lane < k ? lane : 0]);
      const uint32_t a_ms = (uint32_t)__cvta_generic_to_shared(&s_ms[0]);
      uint2 c8[TKP];
#pragma unroll
      for (int j = 0; j < TKP; ++j) {
        uint32_t ra;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a_mine), "r"(j));
        asm volatile("ld.shared::cluster.v2.u32 {%0, %1}, [%2];" : "=r"(c8[j].x), "=r"(c8[j].y) : "r"(ra) : "memory");
      }
      if (logp != nullptr) {
        uint32_t rb;
        float mj, sj;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rb) : "r"(a_ms), "r"(lane & 7));
        asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(mj), "=f"(sj) : "r"(rb) : "memory");
        M = warp_max(mj);
        S = warp_sum((lane < 8 && mj != -INFINITY) ? sj * expf(mj - M) : 0.f);
      }
      if (lane < k) {
#pragma unroll
        for (int j = 0; j < TKP; ++j) cand[j * k + lane] = c8[j];
      }
      __syncwarp();
      merge_lists(cand, TKP, k, result);
    }
    if (lane < k) {
      tok[(size_t)r * k + lane] = (int)result[lane].y;
      if (logp != nullptr) logp[(size_t)r * k + lane] = key_value(result[lane].x) - (M + logf(S));
    }
  }
  if (parts > 1) {
    // no CTA leaves while CTA 0 may still read its shared memory
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  }
}

}  // namespace

#define DISPATCH_T(dtype, ...)                \
  if ((dtype) == 0) {                         \
    typedef float T;                          \
    __VA_ARGS__                               \
  } else {                                    \
    typedef bf16 T;                           \
    __VA_ARGS__                               \
  }

// Runs BODY with NS (a bound of the partial sums per column) and SK (whether their number varies) as
// constants.  fp32 operands come from the CUDA-core multiply, which leaves one whole result.
#define SPLIT_CASE(n_, sk_, ...)              \
  {                                           \
    constexpr int NS = n_;                    \
    constexpr bool SK = sk_;                  \
    __VA_ARGS__                               \
  }
#define FOR_SPLIT(dtype, P, ...)                                                  \
  if ((dtype) == 0) {                                                             \
    typedef float T;                                                              \
    if ((P).n != 1 || (P).sk_ctas != 0) return cudaErrorInvalidValue;             \
    SPLIT_CASE(1, false, __VA_ARGS__)                                             \
  } else {                                                                        \
    typedef bf16 T;                                                               \
    if ((P).n > 12) return cudaErrorInvalidValue;                                 \
    if ((P).sk_ctas == 0) {                                                       \
      if ((P).n <= 1) SPLIT_CASE(1, false, __VA_ARGS__)                           \
      if ((P).n == 2) SPLIT_CASE(2, false, __VA_ARGS__)                           \
      if ((P).n == 3) SPLIT_CASE(3, false, __VA_ARGS__)                           \
      if ((P).n <= 5) SPLIT_CASE(5, false, __VA_ARGS__)                           \
      if ((P).n <= 8) SPLIT_CASE(8, false, __VA_ARGS__)                           \
      SPLIT_CASE(12, false, __VA_ARGS__)                                          \
    }                                                                             \
    if ((P).n <= 3) SPLIT_CASE(3, true, __VA_ARGS__)                              \
    if ((P).n <= 5) SPLIT_CASE(5, true, __VA_ARGS__)                              \
    if ((P).n <= 8) SPLIT_CASE(8, true, __VA_ARGS__)                              \
    SPLIT_CASE(12, true, __VA_ARGS__)                                             \
  }

// The rotary kernel takes two consecutive rows per thread where most columns have one or two partial sums (at least five
// weight tiles per four clusters: prompt forwards; token tiles are multiples of 32 rows, so both rows have the same number)
// and half as many CTAs still give an SM 1280 threads; a row's loads follow the other's stores, so with more sums or fewer
// threads the second trip is exposed.  us per launch, one / two rows: prompts 7B 257 tokens 8.7 / 9.2, 300 9.7 / 9.8, 430 14.1 /
// 13.8, 509 16.2 / 16.0, 640 21.0 / 18.3, 860 25.6 / 22.5, 13B 300 12.4 / 12.2, 509 20.3 / 18.2, 860 32.0 / 28.6; verifications 7B
// 260 rows 10.1 / 11.4, 360 12.4 / 12.9, 512 18.6 / 19.4, 13B 300 12.3 / 12.9.
int rope_rows_per_thread(const SplitIn &P, int R, int threads_per_row) {
  const bool short_columns = P.sk_ctas != 0 && P.n <= 3 && 4ull * P.sk_units >= 5ull * P.sk_ctas * P.sk_kb;
  return short_columns && (R + 1LL) / 2 * threads_per_row >= 1280LL * 148 ? 2 : 1;
}

cudaError_t embed_norm(Launch L, int dtype, const int32_t *tok, const void *E, const void *g,
                       float *x, Operand xn, int R, int H, int V, float eps) {
  DISPATCH_T(dtype, return launch_k(embed_norm_kernel<T>, dim3(R), dim3(256), 0, L.st, L.pdl, tok,
                                    (const T *)E, (const T *)g, x, (T *)xn.hi, (T *)xn.lo, H, V, eps);)
}

cudaError_t row_epilogue(Launch L, int dtype, int mode, float *x, SplitIn P, const void *bias,
                         const void *g, Operand xn, float *out_f32, RowMap out_map, int R, int H, float eps) {
  if (H % 4 == 0 && P.ld % 4 == 0 && P.stride % 4 == 0 && H <= 8192) {
    const int groups = H / 4;
    int threads = groups <= 1024 ? ((groups + 31) / 32) * 32 : (((groups + 1) / 2 + 31) / 32) * 32;
    if (groups <= 1024) {
      FOR_SPLIT(dtype, P, return launch_k(row_epilogue_vec_kernel<T, 1, NS, SK>, dim3(R), dim3(threads), 0, L.st, L.pdl,
                                          mode, x, P, (const T *)bias, (const T *)g, (T *)xn.hi, (T *)xn.lo,
                                          out_f32, out_map, H, eps);)
    }
    FOR_SPLIT(dtype, P, return launch_k(row_epilogue_vec_kernel<T, 2, NS, SK>, dim3(R), dim3(threads), 0, L.st, L.pdl,
                                        mode, x, P, (const T *)bias, (const T *)g, (T *)xn.hi, (T *)xn.lo,
                                        out_f32, out_map, H, eps);)
  }
  DISPATCH_T(dtype, return launch_k(row_epilogue_kernel<T>, dim3(R), dim3(256), 0, L.st, L.pdl, mode,
                                    x, P, (const T *)bias, (const T *)g, (T *)xn.hi, (T *)xn.lo, out_f32,
                                    out_map, H, eps);)
}

cudaError_t eagle_concat(Launch L, int dtype, const float *feat_src, const int32_t *row_src,
                         const int32_t *row_tok, const void *E, Operand cat, int R, int H, int V) {
  DISPATCH_T(dtype, return launch_k(eagle_concat_kernel<T>, dim3(R), dim3(256), 0, L.st, L.pdl,
                                    feat_src, row_src, row_tok, (const T *)E, (T *)cat.hi, (T *)cat.lo, H,
                                    V);)
}

cudaError_t cast_rows(Launch L, int dtype, const float *src, const int32_t *row_src, Operand dst,
                      float *dst32, int dst32_stride, int R, int H) {
  DISPATCH_T(dtype, return launch_k(cast_rows_kernel<T>, dim3(R), dim3(256), 0, L.st, L.pdl, src,
                                    row_src, (T *)dst.hi, (T *)dst.lo, dst32, dst32_stride, H);)
}

cudaError_t ingest_last(Launch L, int dtype, IngestBlocks k, const float *hid, float *verify_hid, Operand xn, int N, int n_max,
                        int H) {
  DISPATCH_T(dtype, return launch_k(ingest_last_kernel<T>, dim3(k.n, k.q), dim3(256), 0, L.st, L.pdl, k, hid, verify_hid,
                                    (T *)xn.hi, (T *)xn.lo, N, n_max, H);)
}

cudaError_t reduce_splits(Launch L, SplitIn P, float *Y, int ldy, int R, int ncols) {
  return launch_k(reduce_splits_kernel, dim3((ncols + 255) / 256, R), dim3(256), 0, L.st, L.pdl, P, Y,
                  ldy, ncols);
}

cudaError_t resblock_update(Launch L, int dtype, float *x, SplitIn P, HeadTab tab, Operand xn, int R, int H) {
  if (H % 4 != 0 || P.ld % 4 != 0 || P.stride % 4 != 0 || tab.rows_per_head < 1) return cudaErrorInvalidValue;
  if (P.sk_ctas != 0) return cudaErrorInvalidValue;
  FOR_SPLIT(dtype, P, return launch_k(resblock_update_kernel<T, NS>, dim3((H + 1023) / 1024, R), dim3(256), 0, L.st,
                                      L.pdl, x, P, tab, (T *)xn.hi, (T *)xn.lo, H);)
}

cudaError_t row_update(Launch L, int dtype, float *x, SplitIn P, const void *g, Operand xg, float *sumsq,
                       int R, int H) {
  if (H % 4 != 0 || P.ld % 4 != 0 || P.stride % 4 != 0) return cudaErrorInvalidValue;
  FOR_SPLIT(dtype, P, return launch_k(row_update_kernel<T, NS, SK>, dim3((H + 1023) / 1024, R), dim3(256), 0, L.st,
                                      L.pdl, x, P, (const T *)g, (T *)xg.hi, (T *)xg.lo, sumsq, H);)
}

// The rotary kernels let their successor, the attention, start only once their own predecessor is done: every
// earlier kernel is complete then, and the attention may read the plan and the cached context before
// its dependency wait (`early`).  (7B one-token step 2.91 -> 2.88 ms from the order alone, with the early reads
// Medusa iteration 3.85 -> 3.82, EAGLE 5.07 -> 5.04.)
cudaError_t rope_kv_write(Launch L, int dtype, SplitIn qkv, RowScale sc, RowPlan plan, float *q_out,
                          Operand q_pair, void *k_cache, void *v_cache, int R, int rows_per_seq, int n_heads,
                          int head_dim, int S_max) {
  bf16 *qh = (bf16 *)q_pair.hi, *ql = (bf16 *)q_pair.lo;
  if (dtype == 0 || ql == nullptr) qh = ql = nullptr;      // the pair exists for bf16 storage only
  const bool one_tile = qkv.sk_ctas == 0 || head_dim == 128;      // a head's columns have one number of partial sums
  if (head_dim % 4 == 0 && qkv.ld % 2 == 0 && qkv.stride % 2 == 0 && one_tile) {
    const int work = n_heads * head_dim / 4;
    const int threads = work < 128 ? ((work + 31) / 32) * 32 : 128;
    const int slices = (work + threads - 1) / threads;
    if (dtype != 0 && rope_rows_per_thread(qkv, R, work) == 2)
      return launch_k(rope_kv_vec_kernel<bf16, 3, true, 2>, dim3((R + 1) / 2, slices), dim3(threads), 0, L.st, L.pdl, qkv, sc, plan,
                      q_out, qh, ql, (bf16 *)k_cache, (bf16 *)v_cache, rows_per_seq, n_heads, head_dim, S_max, R);
    FOR_SPLIT(dtype, qkv, return launch_k(rope_kv_vec_kernel<T, NS, SK, 1>, dim3(R, slices), dim3(threads), 0, L.st, L.pdl,
                                          qkv, sc, plan, q_out, qh, ql, (T *)k_cache, (T *)v_cache, rows_per_seq,
                                          n_heads, head_dim, S_max, R);)
  }
  DISPATCH_T(dtype, return launch_k(rope_kv_kernel<T>, dim3(R, n_heads), dim3(head_dim / 2), 0, L.st,
                                    L.pdl, qkv, sc, plan, q_out, qh, ql, (T *)k_cache, (T *)v_cache,
                                    rows_per_seq, n_heads, head_dim, S_max);)
}

cudaError_t swiglu(Launch L, int dtype, SplitIn gu, RowScale sc, Operand act, int R, int F) {
  if (F % 4 == 0 && gu.ld % 4 == 0 && gu.stride % 4 == 0) {
    FOR_SPLIT(dtype, gu, return launch_k(swiglu_vec_kernel<T, NS, SK>, dim3((F / 4 + 255) / 256, R), dim3(256), 0, L.st,
                                         L.pdl, gu, sc, (T *)act.hi, (T *)act.lo, F);)
  }
  DISPATCH_T(dtype, return launch_k(swiglu_kernel<T>, dim3((F + 255) / 256, R), dim3(256), 0, L.st,
                                    L.pdl, gu, sc, (T *)act.hi, (T *)act.lo, F);)
}

static cudaError_t topk_cluster_launch(Launch L, const float *logits, int32_t *tok, float *logp, float *spread, RowMap map,
                                       int R, int V, int k) {
  cudaLaunchConfig_t cfg = {};
  const int parts = V <= 256 * TKE ? 1 : TKP;      // a row that fits in one CTA's registers needs no cluster
  cfg.gridDim = dim3(parts, R);
  cfg.blockDim = dim3(256);
  cfg.stream = L.st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = L.pdl ? 1 : 0;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = TKP;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = parts > 1 ? 2 : 1;
  ++g_launches;
  return cudaLaunchKernelEx(&cfg, topk_logp_cluster_kernel, logits, tok, logp, spread, map, V, k);
}

cudaError_t argmax_rows(Launch L, const float *logits, int32_t *out, float *spread, RowMap map, int R, int V) {
  // the arg-max (ties: smaller id) is the top-1
  if (V <= 256 * TKE * TKP) return topk_cluster_launch(L, logits, out, nullptr, spread, map, R, V, 1);
  return launch_k(argmax_rows_kernel, dim3(R), dim3(1024), 0, L.st, L.pdl, logits, out, spread, map, V);
}

cudaError_t topk_logp(Launch L, const float *logits, int32_t *tok, float *logp, int R, int V, int k) {
  if (V <= 256 * TKE * TKP && k <= 32) return topk_cluster_launch(L, logits, tok, logp, nullptr, RowMap{0, 0}, R, V, k);
  const size_t smem = (size_t)V * sizeof(float);
  static SmemOptIn optin;
  {
    cudaError_t e = optin.ensure((const void *)topk_logp_kernel, smem);
    if (e != cudaSuccess) return e;
  }
  return launch_k(topk_logp_kernel, dim3(R), dim3(1024), smem, L.st, L.pdl, logits, tok, logp, V, k);
}

}  // namespace koala
