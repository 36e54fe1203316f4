// Tree-masked attention for bf16 caches with head_dim 128 on the 5th-generation tensor cores.
//
// One CTA = one (key chunk, head, sequence) and ALL query rows of that sequence (at most 128 =
// the MMA's M).  The chunk's keys are walked in tiles of 64.  Per tile:
//   S[128 x 64]  = Q K^T          tcgen05.mma, A = Q (K-major), B = K tile (K-major), fp32 in TMEM
//   P            = exp2(S*c - m)  by the thread that owns the query row's TMEM lane: tcgen05.ld,
//                                 mask, row max / sum without shuffles, P written to shared memory
//   O[128x128]  += P V            tcgen05.mma, A = P (K-major), B = V tile as stored, [key][dim],
//                                 which is the MN-major operand form; O stays in tensor memory
// O accumulates over all tiles of the chunk.  A row's exponentials are relative to a reference
// maximum that is raised only when a tile's maximum exceeds it by more than 2^8; only then is the
// row's O rescaled in tensor memory (tcgen05.ld / st), so in the common case the rows never wait
// for P V: the tensor pipe computes S of tile t+1 and P V of tile t-1 while the rows turn S of tile
// t into P (two S buffers in tensor memory, two P buffers in shared memory).  Q and P enter the
// MMAs as bf16 pairs (value + rounding residual: two accumulating MMAs), so only the cached K and V
// carry bf16 rounding.  Q (written as a pair by the rotary-embedding kernel) and the K/V tiles
// arrive by TMA with the 128-byte swizzle, K/V in a ring of two (up to 64 rows) or three stages.
// Warps 0..3 own the rows, warp 4 lane 0 issues the copies, warp 5 lane 0 the MMAs (with more than 64 rows warp 6 lane 0
// those of S).
// With several chunks the CTAs of one (head, sequence) form a thread-block cluster: every CTA leaves
// its unnormalised (O, m, l) in its own shared memory (the K/V ring is free by then); after a cluster
// barrier every CTA reads its slice of the head dimension from all of them, merges it in chunk order
// and writes it as a matrix-multiply operand pair; a second barrier keeps the CTAs alive until all
// have read.
// The mask is: slots below ctx_len visible to every row; slot ctx_len + j visible to a row iff
// bit j of its 128-bit mask; slots from kv_len on invisible.
// Every wait is bounded: on expiry the kernel records a timeout in *status and returns.
#include "common.cuh"
#include "tc_ptx.cuh"

namespace koala {

bool tc_get_map(const void *ptr, int rows, int K_in, int box_rows, CUtensorMap *out);
int tc_num_sms();

namespace {

constexpr int DH = 128;
constexpr int TK = 64;                       // keys per tile
constexpr int NKV_MAX = 3;
constexpr int SUB = 64 * 64 * 2;             // one [64 keys][64 dims] block: 8 KB
constexpr int QSUB = 128 * 64 * 2;           // one [128 rows][64 columns] block: 16 KB
// Shared memory by form.  Up to 64 rows: Q 32 KB, two K and two V buffers of 16 KB, one P buffer of 16 KB =
// 112 KB, so that two CTAs share an SM (their row warps' dependent chains overlap), or one CTA leaves
// half an SM to the next kernel, whose weight loads then start while attention still runs.  More rows:
// Q 64 KB, three K/V buffers, two P buffers = 224 KB.
template <bool DUP> struct Lay {
  static constexpr int NST = DUP ? 2 : 3;              // K and V buffers
  static constexpr int NP = DUP ? 1 : 2;               // P buffers
  static constexpr int PB = DUP ? QSUB : 2 * QSUB;     // bytes of one: value and residual rows in one operand, or two
  static constexpr int Q = 0;
  static constexpr int K = DUP ? 2 * QSUB : 4 * QSUB;
  static constexpr int V = K + NST * 2 * SUB;
  static constexpr int P = V + NST * 2 * SUB;
  static constexpr int BYTES = P + NP * PB;
};
// The kernel's only static shared variables.  They come first, then the gap up to the 1 KB boundary that the
// buffers start at: the two share 1 KB, so that two CTAs of the 112 KB form fit on an SM to the byte.
struct alignas(16) SyncVars {
  uint64_t q_full, k_full[NKV_MAX], k_empty[NKV_MAX], v_full[NKV_MAX], v_empty[NKV_MAX], s_full[2], p_full[2], pv_done[2], drain_bar;
  uint32_t tmem_base_slot;
  int s_error;
};
static_assert(sizeof(SyncVars) <= 1024, "the static variables and the alignment gap share 1 KB");
template <bool DUP> constexpr unsigned SMEM_BYTES = Lay<DUP>::BYTES + 1024 - (unsigned)sizeof(SyncVars);
template <bool DUP> constexpr int THREADS = DUP ? 192 : 224;
constexpr int E_INVALID = 1, E_TIMEOUT = 6;
constexpr int TMEM_COLS = 256;               // S: 2 x 64 columns, O: 128 columns
constexpr int COL_S = 0, COL_O = 128;
constexpr float RESCALE_STEP = 8.f;          // O is rescaled only when a row's maximum grows by more than 2^8
constexpr int OSTRIDE = DH + 4;              // floats of a row of the chunk's result: O[128], m, l, pad
// the chunk's result goes where the K/V buffers were
static_assert(64 * OSTRIDE * 4 <= 2 * 4 * SUB && 128 * OSTRIDE * 4 <= 3 * 4 * SUB, "the chunk's result fits");

// Two floats as bf16 value + rounding residual.  (Probabilities too: cutting their value part off instead of rounding it is no
// faster and leaves a residual twice as large; whole layer of the 7B shape against float64 1.02e-5 instead of 8.4e-6.)
__device__ __forceinline__ void split_pack(float x, float y, uint32_t &hi, uint32_t &lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  const float2 hf = __bfloat1622float2(h);
  const __nv_bfloat162 l = __floats2bfloat162_rn(x - hf.x, y - hf.y);
  hi = *reinterpret_cast<const uint32_t *>(&h);
  lo = *reinterpret_cast<const uint32_t *>(&l);
}
// 2^x for x <= 0 (or -inf): one MUFU instruction; results below 2^-126 flush to zero
__device__ __forceinline__ float ex2_fast(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ uint32_t peer_addr(uint32_t local_addr, uint32_t rank) {
  uint32_t ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(local_addr), "r"(rank));
  return ra;
}
__device__ __forceinline__ float4 ld_cluster_v4(uint32_t ra) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(ra) : "memory");
  return v;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 64-bit visibility of the keys key0 .. key0+63 for a row with tree mask (m1:m0)
__device__ __forceinline__ uint64_t tile_visibility(uint64_t m0, uint64_t m1, int key0, int ctx, int kv_len) {
  uint64_t w;
  const int shift = key0 - ctx;
  if (shift <= -64) w = ~0ull;
  else if (shift < 0) w = (m0 << (-shift)) | ((1ull << (-shift)) - 1ull);
  else if (shift == 0) w = m0;
  else if (shift < 64) w = (m0 >> shift) | (m1 << (64 - shift));
  else if (shift < 128) w = m1 >> (shift - 64);
  else w = 0ull;
  const int n_valid = kv_len - key0;
  if (n_valid <= 0) w = 0ull;
  else if (n_valid < 64) w &= (1ull << n_valid) - 1ull;
  return w;
}

struct AttnParams {
  RowPlan plan;
  bf16 *out, *out_lo;      // [R][n_heads * 128]
  int rows_per_seq, n_heads, S_max, chunks, chunk_bits;
  int longest_first;       // 1: grid slot y / n_heads takes the sequence with that rank in descending cache length
  int early;               // 1: the plan and the cached context may be read before the dependency wait
  int dry_pass;            // 1: the row warps make a dry pass over the tile loop body before the dependency wait
  int *status;
};

// DUP (at most 64 query rows): the MMA's 128 rows hold both parts of the operand pair (of Q for S,
// of P for P V), so that one pass of MMAs gives both partial products, to be added: warp w owns
// queries 16w .. 16w+15, whose value parts are MMA rows (= tensor-memory lanes) 32w .. 32w+15 and
// whose residual parts are rows 32w+16 .. 32w+31.  Lanes l and l+16 of a warp therefore hold the
// two partial scores S_v, S_r of one query: they swap halves by shuffles (no shared memory, no
// barrier), after which lane l has S = S_v + S_r for keys 0..31 of the tile and lane l+16 for keys
// 32..63; the row maximum is one more shuffle; at the end they swap halves of O_v, O_r the same
// way and write dims 0..63 and 64..127.  Otherwise warp w owns rows 32w .. 32w+31 entirely and
// the pair is two accumulating MMAs.
// ONE: a single chunk (its end phase instead of the merge).  Both are template arguments because a launch
// fetches its instructions anew and runs most of them once: 60 KB of code in one body were a third of
// the fixed cost of a launch.
template <bool DUP, bool ONE>
__global__ void __launch_bounds__(THREADS<DUP>, DUP ? 2 : 1)
tree_attn_tc_kernel(const __grid_constant__ CUtensorMap tmQh, const __grid_constant__ CUtensorMap tmQl,
                    const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                    const AttnParams P) {
  constexpr int NC = DUP ? 32 : 64;      // keys of a tile per thread
  typedef Lay<DUP> LY;
  constexpr int NST = LY::NST, NP = LY::NP;
  extern __shared__ unsigned char smem_raw[];
  __shared__ SyncVars sync;
  auto &q_full = sync.q_full, &drain_bar = sync.drain_bar;
  auto &k_full = sync.k_full, &k_empty = sync.k_empty, &v_full = sync.v_full, &v_empty = sync.v_empty;
  auto &s_full = sync.s_full, &p_full = sync.p_full, &pv_done = sync.pv_done;
  auto &tmem_base_slot = sync.tmem_base_slot;
  auto &s_error = sync.s_error;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t raw = smem_u32(smem_raw);
  unsigned char *sm = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
  const uint32_t sb = smem_u32(sm);
  if (sb + LY::BYTES > raw + SMEM_BYTES<DUP>) {       // the static variables are not where SyncVars counts on them
    if (threadIdx.x == 0 && P.status) atomicMax(P.status, E_INVALID);
    return;
  }
  const int c = blockIdx.x;
  int b = blockIdx.y / P.n_heads;
  const int h = blockIdx.y % P.n_heads;
  const int H = P.n_heads * DH;
  const int n_q = DUP ? (P.rows_per_seq + 15) >> 4 : (P.rows_per_seq + 31) >> 5;   // row warps in use (16 or 32 queries each)
  const int n_arrive = n_q;

  pdl_launch_dependents();
  if (threadIdx.x == 0) {
    mbar_init(&q_full, 1);
    for (int s = 0; s < NST; ++s) { mbar_init(&k_full[s], 1); mbar_init(&k_empty[s], 1); mbar_init(&v_full[s], 1); mbar_init(&v_empty[s], 1); }
    mbar_init(&drain_bar, DUP ? 1 : 2);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&s_full[i], 1);
      mbar_init(&p_full[i], (uint32_t)n_arrive);
      mbar_init(&pv_done[i], 1);
    }
    s_error = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmQh) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmQl) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmK) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmV) : "memory");
  }
  if (warp == 5) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(&tmem_base_slot)), "r"((uint32_t)TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_slot;

  // Q and the K/V rows of this forward come from the kernel before: what reads them comes after the dependency
  // wait.  With `early` the plan and the cached context are older and are read before it, except by the row warps,
  // which call read_plan inside their tile loop, after a dry pass over the loop body (see there).
  int ctx = 0, kv_len = 0, tile_lo = 0, T = 0;
  auto read_plan = [&](bool wait) {
    if (wait) pdl_wait();
    if (P.longest_first) {
      // More CTAs than SMs: the CTAs beyond the first round start when the first ones finish, so the
      // sequences are taken longest first and the late CTAs belong to the shortest one.  Lane l holds
      // sequence l's length; its rank is the number of sequences that are longer (ties: lower index).
      const int nb = (int)gridDim.y / P.n_heads;              // <= 32 here
      const int len_l = lane < nb ? P.plan.kv_len[lane] : -1;
      int rank = 0;
#pragma unroll 1
      for (int j = 0; j < nb; ++j) {
        const int len_j = __shfl_sync(0xffffffffu, len_l, j);
        rank += (len_j > len_l || (len_j == len_l && j < lane)) ? 1 : 0;
      }
      const unsigned hit = __ballot_sync(0xffffffffu, lane < nb && rank == b);
      b = hit ? __ffs(hit) - 1 : b;
    }
    ctx = P.plan.ctx_len[b];
    kv_len = P.plan.kv_len[b];
    kv_len = kv_len > P.S_max ? P.S_max : kv_len;
    const int n_tiles = (kv_len + TK - 1) / TK;
    tile_lo = (n_tiles * c) >> P.chunk_bits;          // a power of two of chunks
    T = ((n_tiles * (c + 1)) >> P.chunk_bits) - tile_lo;
  };
  // row ownership of warps 0..3
  const int half = DUP ? (lane >> 4) : 0;                   // DUP: residual lane; takes the second half of the keys / dims
  const int row = DUP ? warp * 16 + (lane & 15) : warp * 32 + lane;
  const bool row_warp = warp < 4 && warp < n_q;
  const bool row_in = row_warp && row < P.rows_per_seq;
  if (!row_warp) read_plan(!P.early);
  auto load_q = [&]() {            // warp 4 lane 0, after the dependency wait
    if (DUP) {
      // of every 32 MMA rows the first 16 are the values of 16 queries, the other 16 their residuals
      mbar_expect_tx(&q_full, (uint32_t)(2 * QSUB));
#pragma unroll 1
      for (int i = 0; i < 16; ++i) {
        const int part = i & 1, hb = (i >> 1) & 1, g = i >> 2;
        tma_load_2d(part ? &tmQl : &tmQh, &q_full, sm + LY::Q + hb * QSUB + (32 * g + 16 * part) * 128,
                    h * DH + 64 * hb, b * P.rows_per_seq + 16 * g);
      }
    } else {
      mbar_expect_tx(&q_full, (uint32_t)(4 * QSUB));
#pragma unroll 1
      for (int i = 0; i < 8; ++i) {
        const int rh = i & 1, hb = (i >> 1) & 1, part = i >> 2;
        tma_load_2d(part ? &tmQl : &tmQh, &q_full, sm + LY::Q + (part * 2 + hb) * QSUB + rh * (QSUB / 2),
                    h * DH + 64 * hb, b * P.rows_per_seq + 64 * rh);
      }
    }
  };
  int r_glob = 0;
  float m_run = -INFINITY, l_run = 0.f;
  bool have_o = false;             // this warp's O in tensor memory is complete (warp-uniform)

  if (warp == 4) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      const int y0 = (P.plan.cache_of(b) * P.n_heads + h) * P.S_max;
      const uint64_t policy = stream_policy(P.plan.seq == nullptr);     // prompt blocks share their sequence's keys
      bool ok = true;
      int issued = 0;
      // K's buffer is free once S has been computed, V's only after P V: K runs ahead
      auto load_kv = [&](int i) {
        const int t = i >> 1, v = i & 1, s = t % NST;
        uint64_t *full = v ? &v_full[s] : &k_full[s];
        mbar_expect_tx(full, (uint32_t)(2 * SUB));
        unsigned char *dst = sm + (v ? LY::V : LY::K) + s * 2 * SUB;
        const int y = y0 + (tile_lo + t) * TK;
        const CUtensorMap *map = v ? &tmV : &tmK;
        tma_load_2d_hint(map, full, dst, 0, y, policy);
        tma_load_2d_hint(map, full, dst + SUB, 64, y, policy);
        issued = i + 1;
      };
      // before the wait: the first tiles, as far as they hold nothing but context
      const int n_pre = P.early ? 2 * min(min(NST, T), max(0, ctx / TK - tile_lo)) : 0;
      bool waited = !P.early;
      if (waited) load_q();
#pragma unroll 1
      for (int i = 0; i < 2 * T; ++i) {
        if (!waited && i == n_pre) { waited = true; pdl_wait(); load_q(); }
        const int t = i >> 1;
        if (t >= NST) {
          ok = mbar_wait((i & 1) ? &v_empty[t % NST] : &k_empty[t % NST], (uint32_t)((t / NST) - 1) & 1u);
          if (!ok) break;
        }
        load_kv(i);
      }
      if (!waited) { pdl_wait(); load_q(); }
      if (!ok) {
        atomicExch(&s_error, 1);
        // let the copies already requested land before the block's memory goes away
        for (int i = issued > 2 * NST ? issued - 2 * NST : 0; i < issued; ++i)
          (void)mbar_wait((i & 1) ? &v_full[(i >> 1) % NST] : &k_full[(i >> 1) % NST], (uint32_t)((i >> 1) / NST) & 1u);
      }
      if (T == 0 || !ok) (void)mbar_wait(&q_full, 0);      // nobody else waits for Q then
    }
  } else if (warp >= 5) {
    // ------------------------------------------------------------------ MMA issuers
    // A thread hands over an MMA of these sizes every 50 to 100 cycles, about as fast as they execute, and prepares nothing
    // meanwhile.  With more than 64 rows (16 MMAs of S and 8 of P V per tile) one thread for both was what a tile took,
    // 2700 cycles of which the rows worked 1700: S and P V have a thread each there (128 rows, context 3989, 32 heads:
    // 38.2 -> 32.9 us per launch).  Up to 64 rows it is half as many MMAs, and a second thread gained nothing.
    // D fp32, A and B bf16; S: N = 64, both K-major; O: N = 128, B MN-major
    const uint32_t idesc_s = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TK >> 3) << 17) | ((128u >> 4) << 24);
    const uint32_t idesc_o = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(DH >> 3) << 17) | ((128u >> 4) << 24);
    auto issue_s = [&](int t) -> bool {
      const int s = t % NST;
      // the rows have read S of tile t - 2 out of this buffer (one thread for both has waited for that before its P V)
      if (!DUP && t >= 2 && !mbar_wait(&p_full[t & 1], (uint32_t)((t - 2) >> 1) & 1u)) return false;
      if (!mbar_wait(&k_full[s], (uint32_t)(t / NST) & 1u)) return false;
      tc_fence_after();
      const uint32_t kb = sb + LY::K + s * 2 * SUB;
      const uint32_t d = tmem + (uint32_t)(COL_S + (t & 1) * TK);
#pragma unroll
      for (int part = 0; part < (DUP ? 1 : 2); ++part) {   // Q value, then Q residual (DUP: both in one operand)
#pragma unroll
        for (int hb = 0; hb < 2; ++hb) {                   // 64-dim block
          const uint64_t da = smem_desc_sw128(sb + LY::Q + (DUP ? hb : part * 2 + hb) * QSUB);
          const uint64_t db = smem_desc_sw128(kb + hb * SUB);
#pragma unroll
          for (int k = 0; k < 4; ++k)
            umma_bf16(d, da + (uint64_t)(2 * k), db + (uint64_t)(2 * k), idesc_s, (part | hb | k) ? 1u : 0u);
        }
      }
      umma_commit(&s_full[t & 1]);
      umma_commit(&k_empty[s]);
      return true;
    };
    auto issue_pv = [&](int t) -> bool {
      if (!mbar_wait(&p_full[t & 1], (uint32_t)(t >> 1) & 1u)) return false;
      if (!mbar_wait(&v_full[t % NST], (uint32_t)(t / NST) & 1u)) return false;
      tc_fence_after();
      const uint32_t vb = sb + LY::V + (t % NST) * 2 * SUB;
      const uint32_t pb = sb + LY::P + (t % NP) * LY::PB;
      const uint32_t d = tmem + (uint32_t)COL_O;
#pragma unroll
      for (int part = 0; part < (DUP ? 1 : 2); ++part) {   // P value, then P residual (DUP: both in one operand)
        const uint64_t da = smem_desc_sw128(pb + part * QSUB);
#pragma unroll
        for (int k = 0; k < 4; ++k) {                      // 16 keys per MMA
          const uint64_t db = smem_desc_mn_sw128(vb + k * 2048, SUB, 1024);
          umma_bf16(d, da + (uint64_t)(2 * k), db, idesc_o, (t | part | k) ? 1u : 0u);   // O accumulates over the tiles
        }
      }
      umma_commit(&v_empty[t % NST]);
      umma_commit(&pv_done[t & 1]);
      return true;
    };
    if (lane == 0) {
      const bool do_s = DUP || warp == 6, do_pv = DUP || warp == 5;
      bool ok = T > 0 && do_s ? mbar_wait(&q_full, 0) : true;
#pragma unroll 1
      for (int t = T > 0 ? -1 : 0; t < T && ok; ++t) {     // one place that issues S: the first one at t = -1
        if (do_s && t + 1 < T) ok = issue_s(t + 1);
        if (do_pv && t >= 0 && ok) ok = issue_pv(t);
      }
      if (!ok) atomicExch(&s_error, 1);
    }
  } else if (row_warp) {
    // ------------------------------------------------------------------ softmax rows
    // O accumulates in tensor memory over all tiles of the chunk.  A row's exponentials are taken
    // relative to a reference maximum m_run that is raised only when a tile's maximum exceeds it
    // by more than RESCALE_STEP (then the row's O and l are multiplied by 2^(old - new) in place);
    // in between the probabilities may exceed 1 (by at most 2^RESCALE_STEP), which costs nothing in
    // fp32 / bf16-pair arithmetic, and the rows never wait for P V except to reuse a P buffer.
    bool ok_row = false;
    uint64_t mk0 = 0ull, mk1 = 0ull;
    const float sc = 0.08838834764831845f * 1.4426950408889634f;    // 1/sqrt(128) * log2(e)
    const uint32_t lane_sel = (uint32_t)(warp * 32) << 16;          // this warp's 32 TMEM lanes
    const uint32_t prow = (uint32_t)((DUP ? warp * 32 + (lane & 15) : row) * 128);   // this query's (value) row of the P operand
    const uint32_t psw = (uint32_t)(row & 7);
    const uint32_t o_base = tmem + lane_sel + (uint32_t)COL_O;     // all 128 dims of this thread's lane
    bool ok = true;

    // Pass t = -1 is a dry pass over the loop body, made before the dependency wait while the kernel
    // before this one still runs: no waits, no row visible (every probability is 0), nothing handed
    // to the MMA warp.  The body is some 20 KB of instructions that run a few times per launch; the
    // dry pass takes their first, slow fetch off the path between the arrival of S and the first P.
    int T_run = 1;
    for (int t = P.dry_pass ? -1 : 0; t < T_run; ++t) {
      if (t == 0) {
        read_plan(true);
        T_run = T;
        r_glob = b * P.rows_per_seq + (row_in ? row : 0);    // also needed by a chunk without tiles: it still merges and stores its dims
        if (T == 0) break;
        ok_row = row_in && P.plan.slot[r_glob] >= 0;
        mk0 = ok_row ? P.plan.mask[(size_t)r_glob * 2] : 0ull;
        mk1 = ok_row ? P.plan.mask[(size_t)r_glob * 2 + 1] : 0ull;
      }
      const bool live = t >= 0;
      if (live && (DUP || t == 0)) {
        ok = __all_sync(0xffffffffu, mbar_wait(&s_full[t & 1], (uint32_t)(t >> 1) & 1u));   // warp-uniform
        if (!ok) break;
      }
      tc_fence_after();
      uint32_t v[NC];
      const uint32_t base = tmem + lane_sel + (uint32_t)(COL_S + (t & 1) * TK);
      if constexpr (DUP) {
        // this lane holds one part (value or residual) of the query's 64 raw scores: keep the part of
        // this lane's 32 keys, hand the other 32 to the query's second lane, add what it hands back
        uint32_t raw[TK];
#pragma unroll
        for (int c0 = 0; c0 < TK; c0 += 16) tmem_ld16(base + (uint32_t)c0, raw + c0);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const float got = __shfl_xor_sync(0xffffffffu, __uint_as_float(half ? raw[j] : raw[32 + j]), 16);
          v[j] = __float_as_uint(__uint_as_float(half ? raw[32 + j] : raw[j]) + got);
        }
      } else {
#pragma unroll
        for (int c0 = 0; c0 < NC; c0 += 16) tmem_ld16(base + (uint32_t)c0, v + c0);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      }
      const int key0 = (tile_lo + t) * TK;
      if (kv_len - key0 < TK) {
        // The last tile reaches past kv_len: those cache slots were never written and may hold
        // anything, NaN bit patterns included, and 0 x NaN in P V would poison every row.  Zero
        // the value rows from kv_len on (a row is 128 bytes of each 64-dim block; the swizzle
        // only permutes inside the row), once the tile has landed.  Every row warp in use writes the
        // same zeros.
        if (live) {
          ok = __all_sync(0xffffffffu, mbar_wait(&v_full[t % NST], (uint32_t)(t / NST) & 1u));
          if (!ok) break;
        }
        const uint32_t vb = sb + LY::V + (live ? t % NST : 0) * 2 * SUB;
        for (int kr = (live ? kv_len - key0 : TK) + lane; kr < TK; kr += 32) {
#pragma unroll
          for (int blk = 0; blk < 2; ++blk)
#pragma unroll
            for (int q = 0; q < 8; ++q) st_shared_v4(vb + blk * SUB + kr * 128 + q * 16, 0u, 0u, 0u, 0u);
        }
      }
      // (more than 64 rows, where a thread has 64 keys: a tile that every row in use sees whole is not masked key by key)
      const bool open = !DUP && key0 + TK <= ctx && __all_sync(0xffffffffu, ok_row || !row_in);
      if (!open) {
        uint64_t vis = ok_row ? tile_visibility(mk0, mk1, key0, ctx, kv_len) : 0ull;
        if (DUP) vis >>= 32 * half;
#pragma unroll
        for (int j = 0; j < NC; ++j) v[j] = ((vis >> j) & 1ull) ? v[j] : 0xff800000u;      // -inf
      }
      float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
      for (int j = 0; j < NC; ++j) m4[j & 3] = fmaxf(m4[j & 3], __uint_as_float(v[j]));
      float m_t = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])) * sc;
      if (DUP) m_t = fmaxf(m_t, __shfl_xor_sync(0xffffffffu, m_t, 16));   // over all 64 keys: both lanes keep the same reference
      // raise the reference maximum?  (the first visible key sets it; O holds nothing of this row yet then)
      float factor = 1.f;
      if (m_t > m_run + RESCALE_STEP || (m_run == -INFINITY && m_t > -INFINITY)) {
        factor = m_run == -INFINITY ? 0.f : exp2f(m_run - m_t);
        m_run = m_t;
      }
      const bool rescale = t > 0 && __any_sync(0xffffffffu, factor != 1.f);
      if (rescale) {
        // every P V issued so far must have landed before O is touched; none can be issued before
        // this warp has handed in its P of tile t
        ok = __all_sync(0xffffffffu, mbar_wait(&pv_done[(t - 1) & 1], (uint32_t)((t - 1) >> 1) & 1u));
        if (!ok) break;
        tc_fence_after();
#pragma unroll 1
        for (int c0 = 0; c0 < DH; c0 += 16) {          // rare: kept short
          uint32_t o[16];
          tmem_ld16(o_base + (uint32_t)c0, o);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int j = 0; j < 16; ++j) o[j] = __float_as_uint(__uint_as_float(o[j]) * factor);
          tmem_st16(o_base + (uint32_t)c0, o);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        l_run *= factor;
      } else if (t == 0) {
        l_run = 0.f;
      }
      // the P buffer of tile t was last read by the P V of tile t - NP
      if (t >= NP) {
        ok = __all_sync(0xffffffffu, mbar_wait(&pv_done[(t - NP) & 1], (uint32_t)((t - NP) >> 1) & 1u));
        if (!ok) break;
      }
      const float mu = m_run == -INFINITY ? 0.f : m_run;
      float l_t = 0.f;
      const uint32_t pb = sb + LY::P + (uint32_t)((t & (NP - 1)) * LY::PB) + prow;
#pragma unroll
      for (int ch = 0; ch < NC / 8; ++ch) {
        uint32_t hi[4], lo[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float p0 = ex2_fast(fmaf(__uint_as_float(v[ch * 8 + 2 * e]), sc, -mu));
          const float p1 = ex2_fast(fmaf(__uint_as_float(v[ch * 8 + 2 * e + 1]), sc, -mu));
          l_t += p0 + p1;
          split_pack(p0, p1, hi[e], lo[e]);
        }
        const uint32_t off = (((uint32_t)(ch + (NC / 8) * half)) ^ psw) << 4;
        st_shared_v4(pb + off, hi[0], hi[1], hi[2], hi[3]);
        // the residuals: 16 rows further down in the same operand (DUP) or the second operand
        st_shared_v4(pb + (DUP ? 16 * 128 : QSUB) + off, lo[0], lo[1], lo[2], lo[3]);
      }
      l_run += l_t;
      // S of the next tile was asked for a tile ago.  With a thread of its own for S its barrier is looked at here, before P
      // is handed over: P V's operands then take all of the shared memory's bandwidth, and a try of a barrier 600 cycles.
      if (!DUP && live && t + 1 < T_run) {
        ok = __all_sync(0xffffffffu, mbar_wait(&s_full[(t + 1) & 1], (uint32_t)((t + 1) >> 1) & 1u));
        if (!ok) break;
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      tc_fence_before();
      __syncwarp();
      if (live && lane == 0) mbar_arrive(&p_full[t & 1]);
    }
    // every P V of the chunk has landed in tensor memory before O is read below
    if (ok && T > 0) ok = __all_sync(0xffffffffu, mbar_wait(&pv_done[(T - 1) & 1], (uint32_t)((T - 1) >> 1) & 1u));
    have_o = ok && T > 0;
    if (!ok) atomicExch(&s_error, 1);
  }

  tc_fence_before();
  __syncthreads();                       // all tiles consumed
  const bool failed = s_error != 0;
  // ---- the end phase runs once per CTA, so it is written as short loops rather than unrolled over the dims
  if (ONE && row_warp) {
    // one chunk: nothing to merge - O out of tensor memory 16 dims at a time, normalised and stored
    tc_fence_after();
    const uint32_t o_lane = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)COL_O;   // this thread's lane, dim 0
    float l = l_run;
    if (DUP) l += __shfl_xor_sync(0xffffffffu, l_run, 16);      // the query's other 32 keys of every tile
    const float inv = (m_run != -INFINITY && l > 0.f) ? 1.f / l : 0.f;
    const size_t ob = (size_t)r_glob * H + h * DH;
#pragma unroll 1
    for (int c0 = 0; c0 < DH; c0 += 16) {
      uint32_t o[16];
      if (have_o) {
        tmem_ld16(o_lane + (uint32_t)c0, o);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) o[j] = 0u;
      }
      if constexpr (DUP) {
        // the query's two lanes hold the two parts of the pair's product: add them; each lane stores eight dims
        float x[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const float lo8 = __uint_as_float(o[k]) + __shfl_xor_sync(0xffffffffu, __uint_as_float(o[k]), 16);
          const float hi8 = __uint_as_float(o[8 + k]) + __shfl_xor_sync(0xffffffffu, __uint_as_float(o[8 + k]), 16);
          x[k] = (half ? hi8 : lo8) * inv;
        }
        if (row_in && !failed) {
          uint32_t hi[4], lo[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) split_pack(x[2 * e], x[2 * e + 1], hi[e], lo[e]);
          const size_t at = ob + c0 + 8 * half;
          *reinterpret_cast<uint4 *>(P.out + at) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
          if (P.out_lo != nullptr) *reinterpret_cast<uint4 *>(P.out_lo + at) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
      } else if (row_in && !failed) {
#pragma unroll
        for (int g8 = 0; g8 < 2; ++g8) {
          uint32_t hi[4], lo[4];
#pragma unroll
          for (int e = 0; e < 4; ++e)
            split_pack(__uint_as_float(o[8 * g8 + 2 * e]) * inv, __uint_as_float(o[8 * g8 + 2 * e + 1]) * inv, hi[e], lo[e]);
          const size_t at = ob + c0 + 8 * g8;
          *reinterpret_cast<uint4 *>(P.out + at) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
          if (P.out_lo != nullptr) *reinterpret_cast<uint4 *>(P.out_lo + at) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
      }
    }
  }
  if constexpr (!ONE) {
    // Merge over the chunks: every CTA leaves its unnormalised O (relative to m), m and l per row in its own
    // shared memory; after one cluster barrier CTA c finishes the dims [c * wc, (c + 1) * wc) of all rows,
    // reading them from every CTA of the cluster, in chunk order.  (Pushing each peer's dims into its
    // shared memory needed a barrier before and after and took 5.9 us per launch, 11.5 us with 128 rows.)
    float *stage = reinterpret_cast<float *>(sm + LY::K);
    if (row_warp) {
      tc_fence_after();
      const uint32_t o_lane = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)COL_O;   // this thread's lane, dim 0
      float *mine = stage + (size_t)row * OSTRIDE;
#pragma unroll 1
      for (int c0 = 0; c0 < DH; c0 += 16) {
        uint32_t o[16];
        if (have_o) {
          tmem_ld16(o_lane + (uint32_t)c0, o);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        } else {
#pragma unroll
          for (int j = 0; j < 16; ++j) o[j] = 0u;
        }
        if constexpr (DUP) {
          // the query's two lanes hold the two parts of the pair's product: add them; each lane stores eight dims
          float x[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const float lo8 = __uint_as_float(o[k]) + __shfl_xor_sync(0xffffffffu, __uint_as_float(o[k]), 16);
            const float hi8 = __uint_as_float(o[8 + k]) + __shfl_xor_sync(0xffffffffu, __uint_as_float(o[8 + k]), 16);
            x[k] = half ? hi8 : lo8;
          }
          float4 *to = reinterpret_cast<float4 *>(mine + c0 + 8 * half);
          to[0] = make_float4(x[0], x[1], x[2], x[3]);
          to[1] = make_float4(x[4], x[5], x[6], x[7]);
        } else {
          float4 *to = reinterpret_cast<float4 *>(mine + c0);
#pragma unroll
          for (int k = 0; k < 4; ++k)
            to[k] = make_float4(__uint_as_float(o[4 * k]), __uint_as_float(o[4 * k + 1]), __uint_as_float(o[4 * k + 2]),
                                __uint_as_float(o[4 * k + 3]));
        }
      }
      float l = l_run;
      if (DUP) l += __shfl_xor_sync(0xffffffffu, l_run, 16);      // the query's other 32 keys of every tile
      if (half == 0) *reinterpret_cast<float2 *>(mine + DH) = make_float2(m_run, l);
    }
    cluster_sync_all();
    if (!failed) {
      const int wc = DH >> P.chunk_bits, per_row = wc >> 3;          // eight dims per thread and step
      const uint32_t st0 = smem_u32(stage);
#pragma unroll 1
      for (int e = threadIdx.x; e < P.rows_per_seq * per_row; e += THREADS<DUP>) {
        const int r = e / per_row, d = c * wc + (e - r * per_row) * 8;
        const uint32_t at = st0 + (uint32_t)(r * OSTRIDE) * 4u;
        float mm = -INFINITY, l = 0.f;
        float o[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
        for (int j0 = 0; j0 < P.chunks; j0 += 4) {           // four chunks at a time, all requested before the first is used
          float4 ml[4], x0[4], x1[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            ml[j] = make_float4(-INFINITY, 0.f, 0.f, 0.f);
            x0[j] = x1[j] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (j0 + j >= P.chunks) continue;
            const uint32_t pa = peer_addr(at, (uint32_t)(j0 + j));
            ml[j] = ld_cluster_v4(pa + DH * 4u);
            x0[j] = ld_cluster_v4(pa + (uint32_t)d * 4u);
            x1[j] = ld_cluster_v4(pa + (uint32_t)d * 4u + 16u);
          }
          float mn = mm;
#pragma unroll
          for (int j = 0; j < 4; ++j) mn = fmaxf(mn, ml[j].x);
          const float mu = mn == -INFINITY ? 0.f : mn, back = exp2f(mm - mu);      // exp2(-inf) = 0; such a chunk's O is zero
          mm = mn;
          l *= back;
#pragma unroll
          for (int k = 0; k < 8; ++k) o[k] *= back;
#pragma unroll
          for (int j = 0; j < 4; ++j) {                      // in chunk order
            const float w = exp2f(ml[j].x - mu);
            l += w * ml[j].y;
            o[0] += w * x0[j].x; o[1] += w * x0[j].y; o[2] += w * x0[j].z; o[3] += w * x0[j].w;
            o[4] += w * x1[j].x; o[5] += w * x1[j].y; o[6] += w * x1[j].z; o[7] += w * x1[j].w;
          }
        }
        const float inv = l > 0.f ? 1.f / l : 0.f;
        uint32_t hi[4], lo[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) split_pack(o[2 * k] * inv, o[2 * k + 1] * inv, hi[k], lo[k]);
        const size_t ob = (size_t)(b * P.rows_per_seq + r) * H + h * DH + d;
        *reinterpret_cast<uint4 *>(P.out + ob) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
        if (P.out_lo != nullptr) *reinterpret_cast<uint4 *>(P.out_lo + ob) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
      }
    }
    // no CTA leaves while another may still read its shared memory
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  }
  // MMAs issued before a wait ran out may still be running: no free under them
  if (failed && warp >= 5 && lane == 0) umma_commit(&drain_bar);
  if (warp == 5) {
    if (failed) (void)mbar_wait(&drain_bar, 0);
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)TMEM_COLS) : "memory");
  }
  if (threadIdx.x == 0 && failed && P.status) atomicMax(P.status, E_TIMEOUT);
  if constexpr (!ONE) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

// Fewer query rows per sequence than this: the mma.sync kernel.  (tcgen05 / mma.sync, 32 heads, eight layers, us per
// forward: one sequence at context 2000 12 rows 829 / 808, 16 rows 834 / 817, 20 rows 843 / 879; four sequences at
// 500 8 rows 810 / 835, 15 rows 915 / 966.  Batches of 0.6 to 1 (sequence, head) pairs per SM would gain from three rows on, fifteen
// rows of four sequences 947 / 902 us a pass, but P V is summed over all of a chunk's tiles in one truncating accumulator here:
// whole layer against float64 8.4e-6 where mma.sync leaves 8.0e-6.)
int g_attn_tc_min_rows = 16;
int g_attn_tc_chunks = 0;      // > 0: this many key chunks whatever the shape (A/B runs)
int g_attn_tc_dry_pass = 1;

}  // namespace

void attn_tc_set_min_rows(int rows) { g_attn_tc_min_rows = rows; }
void attn_tc_set_chunks(int chunks) { g_attn_tc_chunks = chunks; }
void attn_tc_set_dry_pass(int on) { g_attn_tc_dry_pass = on ? 1 : 0; }

// Key chunks (= cluster size) per (sequence, head): the largest of 1, 2, 4, 8 that keeps the CTA count
// within the SMs, each chunk with at least 128 keys of capacity.  Up to 64 rows two CTAs share an SM: two chunks
// while they fit so (144 pairs, eight layers, context 1000, one / two chunks: 32 rows 1126 / 1099 us, 16 rows 892 /
// 858), and up to a tenth more pairs than SMs, where a few SMs with two whole sequences are what the launch waits
// for.  There ragged lengths, which the host does not know, gain and equal ones lose.  Equal and ragged lengths, 64
// rows, context 2000: 156 pairs 3695 / 3803 and 3553 / 3522 us, 160 pairs 3258 / 3356 and 3220 / 3116 (40 heads),
// 2904 / 3010 and 2865 / 2782 (32 heads); 176 pairs 2060 / 2160 and 1959 / 1954, 200 pairs 4214 / 4321 and 4097 /
// 4102; 16 rows, four layers, 160 pairs at context 4000 720 / 783 and 706 / 611, at 2000 594 / 640 and 585 / 555;
// 32 rows at context 1000 1824 / 1949 and 1803 / 1901: up to 32 rows only from 2048 keys of capacity.  13B
// shape, four ragged sequences: 17.9 -> 17.5 ms per iteration.  (More chunks where they fit twice over are
// slower, 7B at batch 1 5.09 -> 5.29 ms with eight.)
int attn_tc_chunks(int B, int n_heads, int rows_per_seq, int S_max, int num_sms) {
  int c = 1;
  if (g_attn_tc_chunks > 0) {
    while (2 * c <= g_attn_tc_chunks && 2 * c <= 8 && 2 * c * 128 <= S_max) c *= 2;
    return c;
  }
  while (c < 8 && 2 * c * B * n_heads <= num_sms && 2 * c * 128 <= S_max) c *= 2;
  const int pairs = B * n_heads, longest = rows_per_seq > 32 || pairs <= num_sms ? 256 : 2048;
  if (c == 1 && rows_per_seq <= 64 && 10 * pairs <= 11 * num_sms && S_max >= longest) c = 2;
  return c;
}

bool attn_tc_supported(int rows_per_seq, int head_dim, int S_max) {
  return head_dim == DH && rows_per_seq >= g_attn_tc_min_rows && rows_per_seq <= 128 && S_max >= 1;
}

cudaError_t tree_attention_tc(Launch L, Operand q_pair, int q_rows_alloc, const void *k_cache, const void *v_cache,
                              RowPlan plan, Operand out, int rows_per_seq, int B, int cache_seqs, int n_heads, int S_max, int chunks,
                              bool early, int *status) {
  const bool dup = rows_per_seq <= 64;
  if (chunks != 1 && chunks != 2 && chunks != 4 && chunks != 8) return cudaErrorInvalidValue;
  if (q_pair.hi == nullptr || q_pair.lo == nullptr) return cudaErrorInvalidValue;
  const long long rows = (long long)cache_seqs * n_heads * S_max;
  if (rows > 0x7fffffffLL) return cudaErrorInvalidValue;
  const int H = n_heads * DH;
  CUtensorMap tmQh, tmQl, tmK, tmV;
  const int q_box = rows_per_seq <= 64 ? 16 : 64;      // rows per copy of the query operand
  if (!tc_get_map(q_pair.hi, q_rows_alloc, H, q_box, &tmQh) || !tc_get_map(q_pair.lo, q_rows_alloc, H, q_box, &tmQl) ||
      !tc_get_map(k_cache, (int)rows, DH, TK, &tmK) || !tc_get_map(v_cache, (int)rows, DH, TK, &tmV))
    return cudaErrorInvalidValue;
  const int longest_first = (B > 1 && B <= 32 && (long long)chunks * B * n_heads > (dup ? 2 : 1) * tc_num_sms()) ? 1 : 0;
  AttnParams P{plan, (bf16 *)out.hi, (bf16 *)out.lo, rows_per_seq, n_heads, S_max, chunks,
               31 - __builtin_clz((unsigned)chunks), longest_first, early ? 1 : 0, g_attn_tc_dry_pass, status};
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(chunks, n_heads * B);
  cfg.blockDim = dim3(dup ? THREADS<true> : THREADS<false>);
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
  auto go = [&](auto *kern, unsigned smem) -> cudaError_t {
    cfg.dynamicSmemBytes = smem;
    ++g_launches;
    return cudaLaunchKernelEx(&cfg, kern, tmQh, tmQl, tmK, tmV, P);
  };
  if (dup) return chunks == 1 ? go(tree_attn_tc_kernel<true, true>, SMEM_BYTES<true>) : go(tree_attn_tc_kernel<true, false>, SMEM_BYTES<true>);
  return chunks == 1 ? go(tree_attn_tc_kernel<false, true>, SMEM_BYTES<false>) : go(tree_attn_tc_kernel<false, false>, SMEM_BYTES<false>);
}

// Once per device (tc_init_driver): whether the kernels can run as laid out, and their shared-memory limit.
bool attn_tc_prepare(int smem_optin) {
  if (smem_optin < Lay<false>::BYTES + 1024) return false;
  const void *kern[4] = {(const void *)tree_attn_tc_kernel<true, true>, (const void *)tree_attn_tc_kernel<true, false>,
                         (const void *)tree_attn_tc_kernel<false, true>, (const void *)tree_attn_tc_kernel<false, false>};
  for (int i = 0; i < 4; ++i) {
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, kern[i]) != cudaSuccess || fa.sharedSizeBytes != sizeof(SyncVars)) return false;
    if (cudaFuncSetAttribute(kern[i], cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(i < 2 ? SMEM_BYTES<true> : SMEM_BYTES<false>)) != cudaSuccess)
      return false;
  }
  return true;
}

}  // namespace koala
