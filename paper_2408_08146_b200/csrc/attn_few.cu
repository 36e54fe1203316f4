// Tree-masked attention on CUDA cores: one or two query rows per sequence (one-token steps) of bf16 caches
// with head_dim 128, and every size of the fp32 and head_dim 64 configurations, whose rows are taken in
// groups (grid z).
//
// With so few rows the cached keys and values are all there is to move: 512 bytes per key and head
// against a few hundred multiply-adds, so the products run in fp32 on the CUDA cores (the tensor-core
// kernels would multiply a 16- or 128-row operand that is mostly padding: 0.7 us of mma.sync per
// 64-key tile).  One CTA = one (key chunk, head, sequence); a warp takes eight keys of every 64-key
// tile, half a warp one key per step: 16 lanes x 16 bytes of K and of V, the next tile's loads in
// flight in registers while this one's are used.  Softmax is online, per half-warp; the sixteen
// partial results of a CTA are merged through shared memory, the chunks (a thread-block cluster)
// through distributed shared memory, each CTA finishing its share of the output, in chunk order.
// Tried and dropped: tiles dealt evenly over all CTAs with partials in global memory and the last
// arriver adding them (fence, counter and the re-read: 4 us at the end of every launch; 14 us per
// launch, ragged batch 22 us).
#include <type_traits>

#include "common.cuh"

namespace koala {
namespace {

constexpr int TILE = 64;
constexpr int WARPS = 8;
constexpr int MAX_CHUNKS = 8;

// E consecutive cache elements of a lane, as loaded and as floats.
template <typename T, int E> struct Frag;
template <int E> struct Frag<bf16, E> {
  uint32_t w[E / 2];
  __device__ __forceinline__ void load(const bf16 *p, bool in) {
    if constexpr (E == 8) {
      const uint4 u = in ? *reinterpret_cast<const uint4 *>(p) : make_uint4(0u, 0u, 0u, 0u);
      w[0] = u.x; w[1] = u.y; w[2] = u.z; w[3] = u.w;
    } else {
      const uint2 u = in ? *reinterpret_cast<const uint2 *>(p) : make_uint2(0u, 0u);
      w[0] = u.x; w[1] = u.y;
    }
  }
  __device__ __forceinline__ void unpack(float *f) const {
#pragma unroll
    for (int i = 0; i < E / 2; ++i) {
      f[2 * i] = __uint_as_float(w[i] << 16);
      f[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
  }
};
template <int E> struct Frag<float, E> {
  float4 w[E / 4];
  __device__ __forceinline__ void load(const float *p, bool in) {
#pragma unroll
    for (int i = 0; i < E / 4; ++i) w[i] = in ? reinterpret_cast<const float4 *>(p)[i] : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __device__ __forceinline__ void unpack(float *f) const {
#pragma unroll
    for (int i = 0; i < E / 4; ++i) { f[4 * i] = w[i].x; f[4 * i + 1] = w[i].y; f[4 * i + 2] = w[i].z; f[4 * i + 3] = w[i].w; }
  }
};

__device__ __forceinline__ float ld_cluster(uint32_t local_addr, uint32_t rank) {
  uint32_t ra;
  float v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(local_addr), "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(ra) : "memory");
  return v;
}

// ROPE: the queries come as the partial sums of the Q/K/V multiply, as do the new keys and values: the CTA whose tiles
// hold a new row's slot writes it to the cache and reads it back with the tile.  A launch less per layer, whose 5 us
// were one trip to the partial sums and back (rule and figures at attn_few_takes_sums).
constexpr int ROPE_PARTS = 4;                              // partial sums that are requested side by side
template <typename T, int DH, int RT, bool ROPE>
__global__ void __launch_bounds__(WARPS * 32, RT <= 2 ? 2 : 1)
tree_attn_few_kernel(const float *q, T *kc, T *vc, RowPlan plan, T *__restrict__ out, T *__restrict__ out_lo,
                     int rows_per_seq, int n_heads, int S_max, int early, SplitIn qkv, RowScale scale) {
  constexpr int E = DH / 16;                               // dims of a lane
  constexpr int PSTRIDE = DH + 4;                          // floats of a partial: O[DH], m, l, pad (16-byte rows)
  __shared__ __align__(16) float s_q[RT][DH];
  __shared__ __align__(16) float s_o[2 * WARPS][RT][PSTRIDE];
  __shared__ __align__(16) float s_c[RT][PSTRIDE];         // this chunk's result, read by the cluster
  pdl_launch_dependents();
  if (!early) pdl_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, hf = lane >> 4, d0 = (lane & 15) * E;
  const int H = n_heads * DH;
  const int c = (int)blockIdx.x, chunks = (int)gridDim.x;
  const int b = (int)blockIdx.y / n_heads, h = (int)blockIdx.y % n_heads;
  const float sc = (DH == 128 ? 0.08838834764831845f : 0.125f) * 1.4426950408889634f;    // 1/sqrt(DH) * log2(e)
  const int i0 = (int)blockIdx.z * RT;                     // this CTA's rows of the sequence: i0 ..
  const int ctx = plan.ctx_len[b];
  const int kv_len = min(plan.kv_len[b], S_max);
  const int tiles = (kv_len + TILE - 1) / TILE;
  const int t_lo = tiles * c / chunks, t_hi = tiles * (c + 1) / chunks;
  const size_t base = ((size_t)plan.cache_of(b) * n_heads + h) * S_max;
  const T *kb = kc + base * DH + d0, *vb = vc + base * DH + d0;
  const int k_off = warp * 8 + hf;                       // this half-warp's keys of a tile: k_off + 2 j
  Frag<T, E> kn[4], vn[4];
  auto load = [&](int t) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int key = t * TILE + k_off + 2 * j;
      const bool in = key < kv_len;                      // slots past the end were never written
      kn[j].load(kb + (size_t)key * DH, in);
      vn[j].load(vb + (size_t)key * DH, in);
    }
  };
  if (early) {
    // a tile of nothing but context does not depend on the kernel before
    const bool context = (t_lo + 1) * TILE <= ctx;
    if (context) load(t_lo);
    pdl_wait();
    if (!ROPE && !context) load(t_lo);
  } else {
    load(t_lo);                                          // first of all: the longest way
  }
  uint64_t mk0[RT], mk1[RT];
  unsigned row_ok = 0;
#pragma unroll
  for (int r = 0; r < RT; ++r) {
    const int rg = b * rows_per_seq + (i0 + r < rows_per_seq ? i0 + r : 0);
    const int slot = plan.slot[rg];
    mk0[r] = plan.mask[(size_t)rg * 2];
    mk1[r] = plan.mask[(size_t)rg * 2 + 1];
    if (i0 + r < rows_per_seq && slot >= 0) row_ok |= 1u << r;
  }
  if constexpr (ROPE) {
    constexpr int HALF = DH / 2;
#pragma unroll
    for (int e = threadIdx.x; e < RT * 3 * HALF; e += WARPS * 32) {      // (row, Q / K / V, pair of dims)
      const int r = e / (3 * HALF), mat = e / HALF % 3, i = e % HALF;
      const int rg = b * rows_per_seq + (i0 + r < rows_per_seq ? i0 + r : 0), slot = plan.slot[rg];
      if (mat > 0) {
        const int tile = min(slot / TILE, tiles - 1);      // the chunk that holds the row's slot writes it
        if (i0 + r >= rows_per_seq || slot < 0 || slot >= S_max || tile < t_lo || tile >= t_hi) continue;
      }
      const float *p = qkv.p + (size_t)rg * qkv.ld + mat * H + h * DH + i;
      float ua[ROPE_PARTS], ub[ROPE_PARTS];
#pragma unroll
      for (int s = 0; s < ROPE_PARTS; ++s) {
        ua[s] = s < qkv.n ? p[(size_t)s * qkv.stride] : 0.f;
        ub[s] = s < qkv.n ? p[(size_t)s * qkv.stride + HALF] : 0.f;
      }
      const float rs = scale.of(rg);
      const float2 cs = plan.rope[(size_t)rg * HALF + i];
      float a = ua[0], c2 = ub[0];
#pragma unroll
      for (int s = 1; s < ROPE_PARTS; ++s) { a += ua[s]; c2 += ub[s]; }
      a *= rs;
      c2 *= rs;
      const float ra = a * cs.x - c2 * cs.y, rb = c2 * cs.x + a * cs.y;
      if (mat == 0) {
        s_q[r][i] = ra * sc;
        s_q[r][i + HALF] = rb * sc;
      } else {
        T *to = (mat == 1 ? kc : vc) + (base + slot) * DH + i;
        to[0] = from_f<T>(mat == 1 ? ra : a);
        to[HALF] = from_f<T>(mat == 1 ? rb : c2);
      }
    }
  } else {
    for (int e = threadIdx.x; e < RT * DH; e += WARPS * 32) {
      const int r = e / DH, d = e % DH;
      s_q[r][d] = q[(size_t)(b * rows_per_seq + (i0 + r < rows_per_seq ? i0 + r : 0)) * H + h * DH + d] * sc;
    }
  }
  __syncthreads();
  if (ROPE && (t_lo + 1) * TILE > ctx) load(t_lo);         // its new rows stand now
  float m[RT], l[RT], o[RT][E];
#pragma unroll
  for (int r = 0; r < RT; ++r) {
    m[r] = -INFINITY;
    l[r] = 0.f;
#pragma unroll
    for (int d = 0; d < E; ++d) o[r][d] = 0.f;
  }
  for (int t = t_lo; t < t_hi; ++t) {
    Frag<T, E> kx[4], vx[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) { kx[j] = kn[j]; vx[j] = vn[j]; }
    if (t + 1 < t_hi) load(t + 1);
    float s[RT][4];
    {
      float kf[4][E];
#pragma unroll
      for (int j = 0; j < 4; ++j) kx[j].unpack(kf[j]);
#pragma unroll
      for (int r = 0; r < RT; ++r) {
        float qr[E];
#pragma unroll
        for (int d = 0; d < E; d += 4) {
          const float4 qa = *reinterpret_cast<const float4 *>(&s_q[r][d0 + d]);
          qr[d] = qa.x; qr[d + 1] = qa.y; qr[d + 2] = qa.z; qr[d + 3] = qa.w;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float a = 0.f;
#pragma unroll
          for (int d = 0; d < E; ++d) a = fmaf(qr[d], kf[j][d], a);
          s[r][j] = a;
        }
      }
    }
#pragma unroll
    for (int o2 = 8; o2 >= 1; o2 >>= 1)
#pragma unroll
      for (int r = 0; r < RT; ++r)
#pragma unroll
        for (int j = 0; j < 4; ++j) s[r][j] += __shfl_xor_sync(0xffffffffu, s[r][j], o2);
    const int key0 = t * TILE + k_off;
#pragma unroll
    for (int r = 0; r < RT; ++r) {
      float mx = m[r];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int rel = key0 + 2 * j - ctx;
        bool vis = ((row_ok >> r) & 1u) != 0 && key0 + 2 * j < kv_len;
        if (rel >= 0) vis = vis && (rel < 64 ? ((mk0[r] >> rel) & 1ull) : (rel < 128 ? ((mk1[r] >> (rel - 64)) & 1ull) : 0ull)) != 0ull;
        s[r][j] = vis ? s[r][j] : -INFINITY;
        mx = fmaxf(mx, s[r][j]);
      }
      const float mu = mx == -INFINITY ? 0.f : mx;
      const float corr = exp2f(m[r] - mu);               // exp2(-inf) = 0
      m[r] = mx;
      l[r] *= corr;
#pragma unroll
      for (int d = 0; d < E; ++d) o[r][d] *= corr;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        s[r][j] = exp2f(s[r][j] - mu);
        l[r] += s[r][j];
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float vf[E];
      vx[j].unpack(vf);
#pragma unroll
      for (int r = 0; r < RT; ++r)
#pragma unroll
        for (int d = 0; d < E; ++d) o[r][d] = fmaf(s[r][j], vf[d], o[r][d]);
    }
  }
// ---- the CTA's sixteen half-warps
  const int src = warp * 2 + hf;
#pragma unroll
  for (int r = 0; r < RT; ++r) {
#pragma unroll
    for (int d = 0; d < E; d += 4)
      *reinterpret_cast<float4 *>(&s_o[src][r][d0 + d]) = make_float4(o[r][d], o[r][d + 1], o[r][d + 2], o[r][d + 3]);
    if ((lane & 15) == 0) { s_o[src][r][DH] = m[r]; s_o[src][r][DH + 1] = l[r]; }
  }
  __syncthreads();
  auto emit = [&](int r, int d, float v) {
    const size_t at = (size_t)(b * rows_per_seq + i0 + r) * H + h * DH + d;
    const T hi = from_f<T>(v);
    out[at] = hi;
    if (out_lo != nullptr) out_lo[at] = from_f<T>(v - to_f(hi));
  };
  for (int e = threadIdx.x; e < RT * DH; e += WARPS * 32) {
    const int r = e / DH, d = e % DH;
    float mm = -INFINITY;
#pragma unroll
    for (int w = 0; w < 2 * WARPS; ++w) mm = fmaxf(mm, s_o[w][r][DH]);
    float acc = 0.f, ll = 0.f;
    if (mm != -INFINITY) {
#pragma unroll
      for (int w = 0; w < 2 * WARPS; ++w) {
        const float wt = exp2f(s_o[w][r][DH] - mm);
        acc += wt * s_o[w][r][d];
        ll += wt * s_o[w][r][DH + 1];
      }
    }
    if (chunks == 1) {
      if (i0 + r < rows_per_seq) emit(r, d, ll > 0.f ? acc / ll : 0.f);
    } else {
      s_c[r][d] = acc;
      if (d == 0) { s_c[r][DH] = mm; s_c[r][DH + 1] = ll; }
    }
  }
  if (chunks == 1) return;
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  const int share = RT * DH / chunks;                      // outputs this CTA finishes
  for (int e = c * share + (int)threadIdx.x; e < (c + 1) * share; e += WARPS * 32) {
    const int r = e / DH, d = e % DH;
    const uint32_t at = (uint32_t)__cvta_generic_to_shared(&s_c[r][0]);
    float pm[MAX_CHUNKS], pl[MAX_CHUNKS], po[MAX_CHUNKS];  // all requested before the first is used
#pragma unroll
    for (int k = 0; k < MAX_CHUNKS; ++k) {
      const bool in = k < chunks;
      const uint32_t rk = in ? k : 0;
      const float a0 = ld_cluster(at + DH * 4, rk), a1 = ld_cluster(at + DH * 4 + 4, rk), a2 = ld_cluster(at + d * 4, rk);
      pm[k] = in ? a0 : -INFINITY;
      pl[k] = a1;
      po[k] = a2;
    }
    float mm = pm[0];
#pragma unroll
    for (int k = 1; k < MAX_CHUNKS; ++k) mm = fmaxf(mm, pm[k]);
    float acc = 0.f, ll = 0.f;
    if (mm != -INFINITY) {
#pragma unroll
      for (int k = 0; k < MAX_CHUNKS; ++k) {               // in chunk order
        const float wt = exp2f(pm[k] - mm);
        acc += wt * po[k];
        ll += wt * pl[k];
      }
    }
    if (i0 + r < rows_per_seq) emit(r, d, ll > 0.f ? acc / ll : 0.f);
  }
  // no CTA leaves while another may still read its result
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

}  // namespace

// Rows per CTA: in bf16 at head_dim 128 one, two or (tensor cores switched off) groups of four; elsewhere one
// while that makes few CTAs (latency), four (two with fp32 rows of 128) where the cache would be re-read too often.
// Key chunks (= cluster size) per (sequence, head): the largest of 1, 2, 4, 8 that keeps the launch
// within what is resident at once (two CTAs per SM up to two rows, else one; clusters of eight do not
// fill every GPC, hence seven eighths), and at least `min_keys` of capacity per chunk: two tiles, eight
// in the small configurations, where the cluster's two barriers cost more than a few tiles.  Single rows of bf16
// caches take two chunks of at least 1024 keys also where not all are resident at once: one chunk leaves most
// SMs a single CTA, which cannot draw the SM's share of the bandwidth (160 pairs, four layers: context 2000
// 602 -> 544 us with equal, 515 -> 475 with ragged lengths, context 4000 776 -> 656 and 627 -> 552; 256 pairs
// 609 -> 584, 563 -> 526), up to as many pairs as two CTAs per SM take (320 pairs 477 -> 456 and 322 -> 333).  Two
// rows do up to a tenth more pairs than SMs (160 pairs, context 4000 697 -> 665 and 632 -> 549; 192 pairs 702 ->
// 727 and 662 -> 594: left at one).
static int few_chunks(bool bf128, int rt, int B, int n_heads, int groups, int S_max, int num_sms) {
  const int room = (rt <= 2 ? 2 : 1) * num_sms * 7 / 8, min_keys = (bf128 ? 2 : 8) * TILE;
  int chunks = 1;
  while (chunks < MAX_CHUNKS && 2 * chunks * B * n_heads * groups <= room && 2 * chunks * min_keys <= S_max) chunks *= 2;
  const bool halve = rt <= 2 && 10 * B * n_heads <= (rt == 1 ? 20 : 11) * num_sms;
  return bf128 && halve && chunks == 1 && S_max >= 2048 ? 2 : chunks;
}

static cudaError_t attention_few(Launch L, int dtype, const float *q, const SplitIn *qkv, RowScale sc, void *k_cache, void *v_cache,
                                 RowPlan plan, Operand out, int rows_per_seq, int B, int n_heads, int head_dim, int S_max, int num_sms, bool early) {
  if (rows_per_seq < 1 || (head_dim != 64 && head_dim != 128)) return cudaErrorInvalidValue;
  const bool bf = dtype != 0;
  auto go = [&](auto tag, auto dh, auto rt, auto rope) -> cudaError_t {
    typedef decltype(tag) T;
    constexpr int DH = decltype(dh)::value, RT = decltype(rt)::value;
    const int groups = (rows_per_seq + RT - 1) / RT;
    const int chunks = few_chunks(bf && DH == 128, RT, B, n_heads, groups, S_max, num_sms);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(chunks, n_heads * B, groups);
    cfg.blockDim = dim3(WARPS * 32);
    cfg.stream = L.st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = L.pdl ? 1 : 0;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = chunks;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = chunks > 1 ? 2 : 1;
    ++g_launches;
    return cudaLaunchKernelEx(&cfg, tree_attn_few_kernel<T, DH, RT, decltype(rope)::value>, q, (T *)k_cache, (T *)v_cache, plan,
                              (T *)out.hi, (T *)out.lo, rows_per_seq, n_heads, S_max, early ? 1 : 0, qkv != nullptr ? *qkv : SplitIn{}, sc);
  };
  std::integral_constant<int, 64> d64;
  std::integral_constant<int, 128> d128;
  std::integral_constant<int, 1> r1;
  std::integral_constant<int, 2> r2;
  std::integral_constant<int, 4> r4;
  const bool one = rows_per_seq == 1 || (!(bf && head_dim == 128) && (long long)rows_per_seq * B * n_heads <= 4LL * num_sms);
  std::false_type plain;
  if (qkv != nullptr) return one ? go(bf16{}, d128, r1, std::true_type{}) : go(bf16{}, d128, r2, std::true_type{});
  if (bf && head_dim == 128) return one ? go(bf16{}, d128, r1, plain) : (rows_per_seq == 2 ? go(bf16{}, d128, r2, plain) : go(bf16{}, d128, r4, plain));
  if (bf) return one ? go(bf16{}, d64, r1, plain) : go(bf16{}, d64, r4, plain);
  if (head_dim == 64) return one ? go(float{}, d64, r1, plain) : go(float{}, d64, r4, plain);
  return one ? go(float{}, d128, r1, plain) : go(float{}, d128, r2, plain);
}

cudaError_t tree_attention_few(Launch L, int dtype, const float *q, const void *k_cache, const void *v_cache, RowPlan plan,
                               Operand out, int rows_per_seq, int B, int n_heads, int head_dim, int S_max, int num_sms, bool early) {
  return attention_few(L, dtype, q, nullptr, RowScale{}, const_cast<void *>(k_cache), const_cast<void *>(v_cache), plan, out, rows_per_seq, B,
                       n_heads, head_dim, S_max, num_sms, early);
}

// Whether a forward of so many rows takes the partial sums itself.  The rotary launch it saves is a time in which the O
// projection's first weights arrive, and the CTAs come to lie where the multiply's end, not evenly; where they have many keys
// to walk that costs more.  Six layers, us per one-token pass, rotary launch / sums by keys of capacity per chunk: 7B one
// sequence (eight chunks) 160 598 / 583, 528 676 / 653; two 416 630 / 631, 560 ragged 605 / 604, 1056 equal 730 / 696 but
// ragged 648 / 686; four 256 609 / 591, 320 ragged 575 / 563, 448 650 / 629, 576 ragged 595 / 598, 832 equal 687 / 658 but ragged
// 626 / 649; eight 621 / 604; 13B one 304 784 / 777, 560 811 / 816, 1056 869 / 898; two 608 ragged 794 / 809; three 320 ragged
// 785 / 775.  The host does not know the lengths, so the capacity stands for them: an engine of more capacity takes the
// rotary launch for the same contexts.  (Against the rotary launch and unpaced weights, one and two rows of one to 64
// sequences at contexts of 150 to 3000, 63 cases of 7B and 13B shapes: 1.00 to 1.08 times as fast.)
bool attn_few_takes_sums(int rows_per_seq, int B, int n_heads, int S_max, int num_sms) {
  if (rows_per_seq < 1 || rows_per_seq > ATTN_FEW_ROWS) return false;
  const int chunks = few_chunks(true, rows_per_seq, B, n_heads, 1, S_max, num_sms);
  return S_max <= (chunks == MAX_CHUNKS ? 640 : 448) * chunks;
}
bool attn_few_rope_supported(const SplitIn &qkv) { return qkv.sk_ctas == 0 && qkv.n <= ROPE_PARTS; }

cudaError_t tree_attention_few_rope(Launch L, SplitIn qkv, RowScale sc, void *k_cache, void *v_cache, RowPlan plan, Operand out,
                                    int rows_per_seq, int B, int n_heads, int S_max, int num_sms) {
  if (rows_per_seq > ATTN_FEW_ROWS || !attn_few_rope_supported(qkv)) return cudaErrorInvalidValue;
  return attention_few(L, 1, nullptr, &qkv, sc, k_cache, v_cache, plan, out, rows_per_seq, B, n_heads, 128, S_max, num_sms, true);
}

}  // namespace koala
