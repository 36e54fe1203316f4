// Weight-streaming skinny GEMM on the 5th-generation tensor cores (sm_100a):
//   Y[R][N_out] (fp32) = X[R][K_in] (bf16) * W[N_out][K_in]^T (bf16)
// with R (tokens = tree nodes x batch) small and the weight matrix read exactly once.
//
// Operands are swapped so that the weights fill the MMA's M dimension: one CTA owns 128 weight
// rows and a range of K, and issues tcgen05.mma with M = 128 (weight rows), N = token tile,
// K = 16, both operands K-major in shared memory with the 128-byte swizzle that TMA writes.
// The fp32 accumulator [128 x tokens] lives in tensor memory.  Warp 0 streams weight and
// activation tiles with TMA through a ring of shared-memory stages (mbarrier full/empty pairs),
// warp 1 issues the MMAs, four or sixteen epilogue warps read the accumulator back (tcgen05.ld)
// and store it.
// The weight stream does not depend on the previous kernel, so under programmatic dependent
// launch the first stages are requested before waiting for the producer of X.
// Activations may come as a pair hi + lo of bf16 matrices (lo = rounding residual of hi): the
// token tile then holds the hi rows followed by the lo rows of the same tokens (MMA N doubles),
// and the epilogue adds the two halves of the accumulator, so the product carries 16 significant
// bits of the activations at no extra weight traffic.
// More than 128 tokens as a pair: value rows and residual rows are two accumulating MMAs into the same
// accumulator columns, so a tile holds up to 256 tokens and the weights are passed over once.  With
// 256 tokens a CTA takes 256 weight rows: four MMAs per K step share the activation tile and fill two
// accumulators (all 512 tensor-memory columns); a stage is 32 KB of weights + 64 KB of activations,
// two stages, one CTA per SM.  From 113 rows up (as a pair; prompt forwards from 65) gemm_tc_pair_kernel takes over
// where it applies: two CTAs of a cluster as one MMA unit, see there.
// Split-K: grid.y CTAs share a weight tile and write separate partial outputs that the consumer
// kernel sums in a fixed order (deterministic).
// Every wait is bounded: on expiry the kernel records KOALA_E_TIMEOUT in *status, drains, frees
// its tensor memory and returns.
#include <cuda.h>

#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <tuple>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace koala {
namespace {

constexpr int BM = 128;             // weight rows per CTA (MMA M)
constexpr int BK = 64;              // K elements per stage: 128 bytes of bf16 = one swizzle row
constexpr int UMMA_K = 16;
constexpr int THREADS_WIDE = 576;   // most threads a launch uses: producer warp, MMA warp and sixteen epilogue
                                    // warps (256-row weight tiles); 128-row tiles launch 192 threads
constexpr int W_STAGE_BYTES = BM * BK * 2;
constexpr int E_TIMEOUT = 6;
constexpr int MAX_STAGES = 8;
constexpr int EARLY_STAGES = 2, PACE_CYCLES = 1600, ALONE_STAGES = 5;      // see tc_ring()

struct TcParams {
  float *Y;
  int ldy;
  int R;              // valid tokens
  int bn;             // MMA N = rows of the activation tile in shared memory, multiple of 16, <= 256
  int tt;             // tokens per tile: bn, or bn / 2 (a multiple of 8) when the activations are a hi/lo pair
  int ztiles;         // token tiles (classic mode; fastest-varying part of blockIdx.x)
  int wtiles;         // CTA pairs in chains: weight tiles
  int tmem_cols;      // power of two >= max(32, bn), per accumulator buffer
  int nbuf;           // accumulator buffers in tensor memory (2 when they fit in 256 columns)
  int tiles0, tiles1; // weight tiles of matrix 0 and of matrices 0+1 (cumulative)
  int n0, n1, n2;     // rows of each matrix
  int kblocks;        // K_in / 64
  int split;          // classic mode: CTAs along K (grid.y)
  int sk_ctas;        // stream-K mode (> 0): the grid's CTAs share all (tile, K-block) units evenly
  unsigned sk_units;  // tiles * kblocks
  size_t split_stride;
  int stages;
  int early_w;        // how many of the first stages' weight tiles are requested before the dependency wait
  int pace;           // > 0: the MMA thread requests the stages past early_w, one per so many cycles, until the first stage is complete
  int late_dep;       // 1: the next kernel may start only once everything before this one is complete (one-CTA form)
  int epi_dry;        // 1: the epilogue warps make a dry pass over their loop body (nothing stored) at kernel start
  int *status;
};

// CTA that owns unit u when `units` units are dealt to `ctas` CTAs as [g*units/ctas, (g+1)*units/ctas)
__device__ __forceinline__ unsigned sk_owner(unsigned u, unsigned ctas, unsigned units) {
  return ((u + 1u) * ctas - 1u) / units;
}

// The form of the activations is a template argument: a launch fetches its instructions anew (the
// kernels of a layer together overflow the instruction caches), so a body holds one form's code only.
//   FORM_PLAIN  one matrix
//   FORM_COLS   pair, the residual rows as extra accumulator columns (up to 128 tokens per tile)
//   FORM_ACC    pair, the residual rows as a second MMA into the same columns (up to 256 tokens)
// WIDE: 256 weight rows per CTA (FORM_ACC only).  One form for all and unrolled double-buffered stores
// were 49 KB of instructions, FORM_COLS is 21 KB now: with the same
// treatment of the row-wise kernels (rotary 42 -> 6 KB, SwiGLU 16 -> 7, residual 9 -> 4) a 7B one-token step
// went from 3.33 to 3.02 ms, a 60-node EAGLE iteration from 5.76 to 5.24 ms.
enum { FORM_PLAIN = 0, FORM_COLS = 1, FORM_ACC = 2 };

template <int FORM, bool WIDE>
__global__ void __launch_bounds__(THREADS_WIDE, 1)
gemm_tc_kernel(const __grid_constant__ CUtensorMap tmW0, const __grid_constant__ CUtensorMap tmW1,
               const __grid_constant__ CUtensorMap tmW2, const __grid_constant__ CUtensorMap tmX,
               const __grid_constant__ CUtensorMap tmXlo, const TcParams P) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ uint64_t full_bar[MAX_STAGES];
  __shared__ uint64_t empty_bar[MAX_STAGES];
  __shared__ uint64_t acc_full[2];      // accumulator buffer complete (MMA -> epilogue)
  __shared__ uint64_t acc_empty[2];     // accumulator buffer drained (epilogue -> MMA)
  __shared__ uint64_t drain_bar;        // error path: every MMA issued so far has finished
  __shared__ uint32_t tmem_base_slot;
  __shared__ int s_error;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t raw = smem_u32(smem_raw);
  unsigned char *tiles = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
  const int x_stage_bytes = (FORM == FORM_ACC ? 2 : 1) * P.bn * BK * 2;
  const int w_stage_bytes = WIDE ? 2 * W_STAGE_BYTES : W_STAGE_BYTES;
  const int stage_bytes = w_stage_bytes + x_stage_bytes;   // both multiples of 1024
  const int bm = WIDE ? 2 * BM : BM;                     // weight rows per tile
  const int KB = P.kblocks;

  // this CTA's run of (tile, K-block) units, tile-major; a run may cross tile boundaries (stream-K)
  unsigned u_lo, u_hi;
  int tok0 = 0;
  if (P.sk_ctas > 0) {
    u_lo = blockIdx.x * P.sk_units / (unsigned)P.sk_ctas;           // units x CTAs fits in 32 bits (host)
    u_hi = (blockIdx.x + 1u) * P.sk_units / (unsigned)P.sk_ctas;
  } else {
    const int tile = blockIdx.x / P.ztiles;
    tok0 = (blockIdx.x % P.ztiles) * P.tt;
    u_lo = (unsigned)(tile * KB) + (unsigned)KB * blockIdx.y / (unsigned)P.split;
    u_hi = (unsigned)(tile * KB) + (unsigned)KB * (blockIdx.y + 1u) / (unsigned)P.split;
  }
  const int n_units = (int)(u_hi - u_lo);

  // weight tensor map and first row of a tile
  auto tile_map = [&](int tile, int &row0) -> const CUtensorMap * {
    if (tile >= P.tiles1) { row0 = (tile - P.tiles1) * bm; return &tmW2; }
    if (tile >= P.tiles0) { row0 = (tile - P.tiles0) * bm; return &tmW1; }
    row0 = tile * bm;
    return &tmW0;
  };
  // One weight tile of a stage: 128 rows per copy.  Evict-first in L2 unless several token tiles read it (per step,
  // against the default policy: 7B one-token step 3.03 -> 2.92 ms, 64 rows 4.12 -> 4.00, 128 rows 7.25 -> 7.05;
  // with two token tiles of 256 rows it costs 1.5 %).
  const uint64_t policy = stream_policy(P.ztiles == 1);
  auto load_w = [&](const CUtensorMap *tmW, uint64_t *bar, unsigned char *dst, int kb, int row0) {
    tma_load_2d_hint(tmW, bar, dst, kb * BK, row0, policy);
    if (WIDE) tma_load_2d_hint(tmW, bar, dst + W_STAGE_BYTES, kb * BK, row0 + BM, policy);
  };
  const int pre = n_units < P.stages ? n_units : P.stages;

  if (!P.late_dep) pdl_launch_dependents();
  if (threadIdx.x == 0) {
#pragma unroll 1
    for (int s = 0; s < P.stages; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&acc_full[i], 1);
      mbar_init(&acc_empty[i], (blockDim.x >> 5) - 2);   // one arrival per epilogue warp
    }
    mbar_init(&drain_bar, 1);
    s_error = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    // The weight stream starts right here, before the block-wide set-up barrier and before the
    // dependency wait: weights do not depend on the kernel before this one.
    int tile = (int)(u_lo / KB), kb = (int)(u_lo % KB), row0;
    const CUtensorMap *tmW = tile_map(tile, row0);
    const int early = pre < P.early_w ? pre : P.early_w;
#pragma unroll 1
    for (int it = 0; it < early; ++it) {
      mbar_expect_tx(&full_bar[it], (uint32_t)stage_bytes);
      load_w(tmW, &full_bar[it], tiles + (size_t)it * stage_bytes, kb, row0);
      if (++kb == KB) { kb = 0; ++tile; tmW = tile_map(tile, row0); }
    }
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmX) : "memory");
    if (FORM != FORM_PLAIN) asm volatile("prefetch.tensormap [%0];" ::"l"(&tmXlo) : "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(&tmem_base_slot)), "r"((uint32_t)(P.tmem_cols * P.nbuf * (WIDE ? 2 : 1)))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_acc = tmem_base_slot;

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      int tile, kb, row0;
      const CUtensorMap *tmW;
      pdl_wait();
      if (P.late_dep) pdl_launch_dependents();
      const int lo_off = P.tt * BK * 2;          // the lo rows follow the hi rows of the tile
      tile = (int)(u_lo / KB);
      kb = (int)(u_lo % KB);
      tmW = tile_map(tile, row0);
#pragma unroll 1
      for (int it = 0; it < pre; ++it) {
        unsigned char *xd = tiles + (size_t)it * stage_bytes + w_stage_bytes;
        if (it >= P.early_w && P.pace == 0) {
          mbar_expect_tx(&full_bar[it], (uint32_t)stage_bytes);
          load_w(tmW, &full_bar[it], tiles + (size_t)it * stage_bytes, kb, row0);
        }
        tma_load_2d(&tmX, &full_bar[it], xd, kb * BK, tok0);
        if (FORM != FORM_PLAIN) tma_load_2d(&tmXlo, &full_bar[it], xd + lo_off, kb * BK, tok0);
        if (++kb == KB) { kb = 0; ++tile; tmW = tile_map(tile, row0); }
      }
      bool ok = true;
      int s = pre % P.stages;
      uint32_t ph = (uint32_t)(pre / P.stages) & 1u;
#pragma unroll 1
      for (int it = pre; it < n_units; ++it) {
        ok = mbar_wait(&empty_bar[s], ph ^ 1u);
        if (!ok) break;
        mbar_expect_tx(&full_bar[s], (uint32_t)stage_bytes);
        unsigned char *dst = tiles + (size_t)s * stage_bytes;
        load_w(tmW, &full_bar[s], dst, kb, row0);
        tma_load_2d(&tmX, &full_bar[s], dst + w_stage_bytes, kb * BK, tok0);
        if (FORM != FORM_PLAIN) tma_load_2d(&tmXlo, &full_bar[s], dst + w_stage_bytes + lo_off, kb * BK, tok0);
        if (++kb == KB) { kb = 0; ++tile; tmW = tile_map(tile, row0); }
        if (++s == P.stages) { s = 0; ph ^= 1u; }
      }
      if (!ok) {
        atomicExch(&s_error, 1);
        // let the copies already requested land before the block's memory goes away
        for (int q = 0; q < P.stages; ++q) (void)mbar_wait(&full_bar[q], 0);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      // instruction descriptor: D fp32, A and B bf16, both K-major, N = bn, M = 128
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(P.bn >> 3) << 17) |
                             ((uint32_t)(BM >> 4) << 24);
      if (P.pace > 0) {
        // the weight stages past the early ones, spread over the time of the kernel before, until the first stage is complete
        int tile = (int)(u_lo / KB), kb = (int)(u_lo % KB), row0;
        for (int it = 0; it < P.early_w && it < pre; ++it)
          if (++kb == KB) { kb = 0; ++tile; }
        const CUtensorMap *tmW = tile_map(tile, row0);
        const long long t0 = clock64();
#pragma unroll 1
        for (int it = P.early_w; it < pre; ++it) {
          while (clock64() - t0 < (long long)(it - P.early_w + 1) * P.pace && !mbar_try(smem_u32(&full_bar[0]), 0)) {}
          mbar_expect_tx(&full_bar[it], (uint32_t)stage_bytes);
          load_w(tmW, &full_bar[it], tiles + (size_t)it * stage_bytes, kb, row0);
          if (++kb == KB) { kb = 0; ++tile; tmW = tile_map(tile, row0); }
        }
      }
      bool ok = true;
      int seg = 0;                        // segment = run of units inside one tile
      bool seg_start = true;
      int kb = (int)(u_lo % KB), s = 0, buf = 0;
      uint32_t ph = 0;
      for (int it = 0; it < n_units; ++it) {
        if (seg_start && seg >= P.nbuf) {
          // the accumulator buffer must have been drained by the epilogue of segment seg - nbuf
          ok = mbar_wait(&acc_empty[buf], (uint32_t)((seg / P.nbuf) - 1) & 1u);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        }
        ok = mbar_wait(&full_bar[s], ph);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t wa = smem_u32(tiles + (size_t)s * stage_bytes);
        const uint64_t da = smem_desc_sw128(wa);
        const uint64_t da2 = smem_desc_sw128(wa + W_STAGE_BYTES);      // wide: the second 128 weight rows
        const uint64_t db = smem_desc_sw128(wa + (uint32_t)w_stage_bytes);
        const uint64_t db2 = smem_desc_sw128(wa + (uint32_t)(w_stage_bytes + P.tt * BK * 2));   // accp: the residual rows
        const uint32_t dacc = tmem_acc + (uint32_t)(buf * P.tmem_cols);
#pragma unroll
        for (int k = 0; k < BK / UMMA_K; ++k) {
          // advance 32 bytes (16 bf16) inside the swizzled row: +2 in the 16-byte address field
          const uint32_t acc = (!seg_start || k > 0) ? 1u : 0u;
          umma_bf16(dacc, da + (uint64_t)(2 * k), db + (uint64_t)(2 * k), idesc, acc);
          if (FORM == FORM_ACC) umma_bf16(dacc, da + (uint64_t)(2 * k), db2 + (uint64_t)(2 * k), idesc, 1u);
          if (WIDE) {
            umma_bf16(dacc + (uint32_t)P.tmem_cols, da2 + (uint64_t)(2 * k), db + (uint64_t)(2 * k), idesc, acc);
            if (FORM == FORM_ACC) umma_bf16(dacc + (uint32_t)P.tmem_cols, da2 + (uint64_t)(2 * k), db2 + (uint64_t)(2 * k), idesc, 1u);
          }
        }
        umma_commit(&empty_bar[s]);      // stage reusable once these MMAs have read it
        const bool seg_end = (kb == KB - 1) || it == n_units - 1;
        if (seg_end) {
          umma_commit(&acc_full[buf]);   // this segment's accumulator is complete
          ++seg;
          buf = (P.nbuf == 2) ? (buf ^ 1) : 0;
        }
        seg_start = seg_end;
        if (++kb == KB) kb = 0;
        if (++s == P.stages) { s = 0; ph ^= 1u; }
      }
      if (!ok) atomicExch(&s_error, 1);
    }
  } else {
    // ------------------------------------------------------------------ epilogue (warps 2..5)
    const int quarter = warp & 3;        // the 32 tensor-memory lanes this warp may read
    // with more than four epilogue warps the warps of a lane quarter share the token columns
    const int n_ch = ((int)(blockDim.x >> 5) - 2) >> 2;
    const int c_per = ((((P.tt + 15) >> 4) + n_ch - 1) / n_ch) << 4;
    const int c_lo = min(((warp - 2) >> 2) * c_per, P.tt);
    const int c_hi = min(c_lo + c_per, P.tt);
    // A dry pass first: the loop body once with nothing stored and nothing waited for, while the
    // first tiles stream - the epilogue's instructions are then already fetched when the first
    // accumulator is complete.
    bool dry = P.epi_dry != 0;
    if (!dry) pdl_wait();                // the output buffer may still be read by the previous kernel
    bool ok = true;
    int seg = 0;
    unsigned u = u_lo;
    while (u < u_hi && ok) {
      const int tile = (int)(u / KB);
      unsigned seg_hi = (unsigned)(tile + 1) * KB;
      if (seg_hi > u_hi) seg_hi = u_hi;
      const int buf = seg % P.nbuf;
      int row0, col_off = 0, n_rows = P.n0;                // (where the sums go is found before the wait)
      if (tile >= P.tiles1) { row0 = (tile - P.tiles1) * bm; col_off = P.n0 + P.n1; n_rows = P.n2; }
      else if (tile >= P.tiles0) { row0 = (tile - P.tiles0) * bm; col_off = P.n0; n_rows = P.n1; }
      else row0 = tile * bm;
      if (dry) n_rows = 0;
      // which partial-sum slot: classic = the split index; stream-K = rank among the tile's contributors
      int slot = blockIdx.y;
      if (P.sk_ctas > 0)
        slot = (int)blockIdx.x - (int)sk_owner((unsigned)tile * KB, (unsigned)P.sk_ctas, P.sk_units);
      if (!dry) {
        ok = mbar_wait(&acc_full[buf], (uint32_t)(seg / P.nbuf) & 1u);
        if (!ok) break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
      for (int hw = 0; hw < (WIDE ? 2 : 1); ++hw) {      // wide: one accumulator per 128 weight rows
      const int feat = row0 + hw * BM + quarter * 32 + lane;
      float *Yp = P.Y + (size_t)slot * P.split_stride + col_off + feat;
      const uint32_t lane_base = tmem_acc + (uint32_t)((buf + hw) * P.tmem_cols) + ((uint32_t)(quarter * 32) << 16);
      // 16 token columns per step (the last eight of a tile may bring eight that are not stored), in a rolled loop: the
      // accumulator reads of one warp hide behind the stores of the others, and the loop's instructions are fetched once.
#pragma unroll 1
      for (int c0 = c_lo; c0 < c_hi; c0 += 16) {
        uint32_t va[16];
        tmem_ld16(lane_base + (uint32_t)c0, va);
        if constexpr (FORM == FORM_COLS) {
          // value and residual rows in separate accumulator columns: added here
          uint32_t vb[16];
          tmem_ld16(lane_base + (uint32_t)(P.tt + c0), vb);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int j = 0; j < 16; ++j) va[j] = __float_as_uint(__uint_as_float(va[j]) + __uint_as_float(vb[j]));
        } else {
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        }
        const int left = feat < n_rows ? P.R - (tok0 + c0) : 0;      // tokens of this step that exist
        float *yp = Yp + (size_t)(tok0 + c0) * P.ldy;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          if (j < left) *yp = __uint_as_float(va[j]);
          yp += P.ldy;
        }
      }
      }
      if (dry) {                         // the same segment again, for real
        dry = false;
        pdl_wait();
        continue;
      }
      // hand the accumulator buffer back to the MMA issuer
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&acc_empty[buf])) : "memory");
      ++seg;
      u = seg_hi;
    }
    if (!ok) atomicExch(&s_error, 1);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    if (s_error) {
      // a wait ran out somewhere in the block: MMAs issued before that may still be running, and
      // tensor memory must not be freed under them
      if (lane == 0) {
        umma_commit(&drain_bar);
        (void)mbar_wait(&drain_bar, 0);
      }
      __syncwarp();
    }
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                 ::"r"(tmem_acc), "r"((uint32_t)(P.tmem_cols * P.nbuf * (WIDE ? 2 : 1)))
                 : "memory");
  }
  if (threadIdx.x == 0 && s_error && P.status) atomicMax(P.status, E_TIMEOUT);
}

// ------------------------------------------------------------------------------- CTA pairs
// 113 tokens and more as a pair of activations, two CTAs of a cluster as one MMA unit (cta_group::2), token
// tiles of tt = 128 to 256 rows, a multiple of 32 (several of them in one launch above 256 rows).  With one CTA
// per tile these forms are bound by what L2 delivers into shared memory (128 tokens: 48 KB per 128 weight rows and K block, three times the
// weight bytes; 256 tokens: 96 KB per 256 weight rows).  Here a pair of CTAs owns 512 weight rows:
// every MMA has M = 256 (128 weight rows from each CTA) and N = tt tokens, of which each CTA loads
// only its half (value rows and residual rows).  Per CTA and stage: weight rows
// [a*256 + rank*128, +128) for the accumulators a = 0, 1 (2 x 16 KB) and tokens [rank*tt/2, +tt/2)
// as value and residual rows (2 x tt/2 x 128 B): 48 KB (four stages) at 128 tokens, 64 KB (three) at 256.  With
// 128 tokens the two accumulators take 256 tensor-memory columns and there are two sets, so the
// epilogue of one segment overlaps the MMAs of the next.  Every load of both CTAs is counted on
// the even CTA's full barrier; that CTA's MMA thread issues for the pair and its commits arrive on
// the empty / accumulator barriers of both CTAs; each CTA's epilogue warps read its own 128
// accumulator lanes and arrive on the even CTA's accumulator-empty barrier.  Stream-K over the
// clusters, one cluster per SM pair.
constexpr int PAIR_THREADS = 576;
constexpr int PAIR_PART_BYTES = BM * BK * 2;          // 16 KB: 128 rows of one operand part
constexpr int PAIR_MAX_STAGES = 4;
constexpr int PAIR_ROWS = 4 * BM;                     // weight rows per cluster tile

// CHAIN: the tensor core adds into its fp32 accumulators by truncation, so the error of a sum grows with the
// number of MMAs that went into it (towards zero; K = 4096 as value and residual, 512 MMAs: 9.2e-6 of the
// result, as much as four times what the pairs leave out).  Where a product has several token tiles its
// partial sums are too large to be cut along K into global memory as with few rows (where the longest sum is
// 64 to 256 MMAs; hidden state after 32 layers of the 7B shape, 509 prompt tokens, against float64: 1.7e-3 in
// parts of 64 rows, 2.7e-3 with 512-MMA sums, 1.4e-3 in this form); instead every CHAIN_KB K blocks the MMAs
// change to the other accumulator set, and the epilogue warps add the finished one to sums in registers,
// rounding to nearest, while it fills: 32 MMAs per sum, 5.6e-7.  256 weight rows per cluster, one
// accumulator of up to 256 tokens: two sets in tensor memory, 128 sums per thread of eight warps.  (512 rows x
// 128 tokens, the same loads, read more of shared memory per MMA: 7B prompt of 509 tokens 17.0 ms against
// 14.3; chains of 8 K blocks: the same time, twice the error.)
constexpr int CHAIN_KB = 4;
constexpr int CHAIN_THREADS = 320;
constexpr int CHAIN_ROWS = 2 * BM;                    // weight rows per cluster tile

template <bool CHAIN>
__global__ void __launch_bounds__(CHAIN ? CHAIN_THREADS : PAIR_THREADS, 1)
gemm_tc_pair_kernel(const __grid_constant__ CUtensorMap tmW0, const __grid_constant__ CUtensorMap tmW1,
                    const __grid_constant__ CUtensorMap tmW2, const __grid_constant__ CUtensorMap tmX,
                    const __grid_constant__ CUtensorMap tmXlo, const TcParams P) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ uint64_t full_bar[PAIR_MAX_STAGES];    // used in the even CTA: both CTAs' loads of a stage landed
  __shared__ uint64_t empty_bar[PAIR_MAX_STAGES];   // per CTA: the pair's MMAs have read this stage
  __shared__ uint64_t acc_full[2];              // per CTA: a segment's accumulators are complete
  __shared__ uint64_t acc_empty[2];             // used in the even CTA: both CTAs' epilogues drained them
  __shared__ uint64_t drain_bar;
  __shared__ uint32_t tmem_base_slot;
  __shared__ int s_error;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const unsigned cid = blockIdx.x >> 1;                       // cluster index
  const uint32_t raw = smem_u32(smem_raw);
  unsigned char *tiles = smem_raw + ((1024u - (raw & 1023u)) & 1023u);
  const int KB = P.kblocks;
  const unsigned u_lo = cid * P.sk_units / (unsigned)P.sk_ctas;              // fits in 32 bits (host)
  const unsigned u_hi = (cid + 1u) * P.sk_units / (unsigned)P.sk_ctas;
  const int n_units = (int)(u_hi - u_lo);
  const int n_epi = (int)(blockDim.x >> 5) - 2;
  constexpr int PARTS = CHAIN ? 1 : 2;                   // accumulators of 256 weight rows
  constexpr int ROWS = CHAIN ? CHAIN_ROWS : PAIR_ROWS;
  const int tt = P.tt;                                   // tokens per tile: a multiple of 32, at most 256
  const int x_part = (tt >> 1) * BK * 2;                  // this CTA's tokens, value or residual rows
  const int stage_bytes = PARTS * PAIR_PART_BYTES + 2 * x_part;
  const int n_stages = P.stages;

  auto tile_map = [&](int tile, int &row0) -> const CUtensorMap * {
    if (tile >= P.tiles1) { row0 = (tile - P.tiles1) * ROWS; return &tmW2; }
    if (tile >= P.tiles0) { row0 = (tile - P.tiles0) * ROWS; return &tmW1; }
    row0 = tile * ROWS;
    return &tmW0;
  };
  // The deal of tiles.  Up to 512 rows the token tiles of a weight tile lie next to one another; in chains, with
  // several tiles per cluster, a cluster would take them one after the other and the weights come from DRAM
  // once for each (1024 rows of the 7B gate and up: 755 MB for 180): there the weight tiles of a token tile do, and
  // groups of clusters, one per token tile, go through the weights side by side.
  auto weight_of = [&](int tile) { return CHAIN ? tile % P.wtiles : tile / P.ztiles; };
  auto tok_of = [&](int tile) { return CHAIN ? tile / P.wtiles : tile % P.ztiles; };
  const int pre = n_units < n_stages ? n_units : n_stages;

  pdl_launch_dependents();
  if (threadIdx.x == 0) {
#pragma unroll 1
    for (int s = 0; s < n_stages; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&acc_full[i], 1);
      mbar_init(&acc_empty[i], (uint32_t)(2 * n_epi));
    }
    mbar_init(&drain_bar, 1);
    s_error = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmW0) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmX) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmXlo) : "memory");
  }
  if (warp == 1) {
    // the same warp of both CTAs allocates all 512 columns in both tensor memories
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(&tmem_base_slot)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  cluster_barrier();            // both CTAs' barriers exist before anything signals them
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_acc = tmem_base_slot;

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer (both CTAs)
    if (lane == 0) {
      const uint64_t policy = stream_policy(P.ztiles == 1);
      uint32_t full_even[PAIR_MAX_STAGES];
      for (int s = 0; s < PAIR_MAX_STAGES; ++s) full_even[s] = cluster_addr_of(smem_u32(&full_bar[s]), 0);
      int tile = (int)(u_lo / KB), kb = (int)(u_lo % KB), row0;
      int tok0 = tok_of(tile) * tt;
      const CUtensorMap *tmW = tile_map(weight_of(tile), row0);
      auto next_unit = [&]() {
        if (++kb == KB) {
          kb = 0;
          ++tile;
          tok0 = tok_of(tile) * tt;
          tmW = tile_map(weight_of(tile), row0);
        }
      };
      auto load_w = [&](int s) {
        unsigned char *dst = tiles + (size_t)s * stage_bytes;
        if (rank == 0) mbar_expect_tx(&full_bar[s], 2u * (uint32_t)stage_bytes);
        tma_load_2d_pair_hint(tmW, full_even[s], dst, kb * BK, row0 + (int)rank * BM, policy);
        if (!CHAIN) tma_load_2d_pair_hint(tmW, full_even[s], dst + PAIR_PART_BYTES, kb * BK, row0 + 2 * BM + (int)rank * BM, policy);
      };
      auto load_x = [&](int s, int kbx, int tokx) {
        unsigned char *dst = tiles + (size_t)s * stage_bytes + PARTS * PAIR_PART_BYTES;
        tma_load_2d_pair(&tmX, full_even[s], dst, kbx * BK, tokx + (int)rank * (tt >> 1));
        tma_load_2d_pair(&tmXlo, full_even[s], dst + x_part, kbx * BK, tokx + (int)rank * (tt >> 1));
      };
      // the first stages' weights do not depend on the kernel before this one
      int kb_first[PAIR_MAX_STAGES], tok_first[PAIR_MAX_STAGES];
#pragma unroll 1
      for (int it = 0; it < pre; ++it) {
        kb_first[it] = kb;
        tok_first[it] = tok0;
        load_w(it);
        next_unit();
      }
      pdl_wait();
#pragma unroll 1
      for (int it = 0; it < pre; ++it) load_x(it, kb_first[it], tok_first[it]);
      bool ok = true;
      int s = pre % n_stages;
      uint32_t ph = (uint32_t)(pre / n_stages) & 1u;
#pragma unroll 1
      for (int it = pre; it < n_units; ++it) {
        ok = mbar_wait(&empty_bar[s], ph ^ 1u);
        if (!ok) break;
        load_w(s);
        load_x(s, kb, tok0);
        next_unit();
        if (++s == n_stages) { s = 0; ph ^= 1u; }
      }
      if (!ok) atomicExch(&s_error, 1);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (even CTA)
    if (lane == 0 && rank == 0) {
      // D fp32, A and B bf16, both K-major, N = tt, M = 256 over the two CTAs
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(tt >> 3) << 17) |
                             ((uint32_t)(256 >> 4) << 24);
      bool ok = true;
      int seg = 0, links = 0;              // CHAIN: a "segment" here is what goes into one accumulator set
      bool seg_start = true;
      int kb = (int)(u_lo % KB), s = 0, buf = 0;
      uint32_t ph = 0;
      for (int it = 0; it < n_units; ++it) {
        if (seg_start && seg >= P.nbuf) {
          ok = mbar_wait(&acc_empty[buf], (uint32_t)((seg / P.nbuf) - 1) & 1u);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        }
        ok = mbar_wait(&full_bar[s], ph);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t wa = smem_u32(tiles + (size_t)s * stage_bytes);
        const uint64_t da0 = smem_desc_sw128(wa);
        const uint64_t da1 = smem_desc_sw128(wa + PAIR_PART_BYTES);
        const uint64_t dbh = smem_desc_sw128(wa + PARTS * PAIR_PART_BYTES);
        const uint64_t dbl = smem_desc_sw128(wa + PARTS * PAIR_PART_BYTES + (uint32_t)x_part);
        const uint32_t d0 = tmem_acc + (uint32_t)(buf * PARTS * tt), d1 = d0 + (uint32_t)tt;
#pragma unroll
        for (int k = 0; k < BK / UMMA_K; ++k) {
          const uint32_t acc = (!seg_start || k > 0) ? 1u : 0u;
          umma2_bf16(d0, da0 + (uint64_t)(2 * k), dbh + (uint64_t)(2 * k), idesc, acc);
          umma2_bf16(d0, da0 + (uint64_t)(2 * k), dbl + (uint64_t)(2 * k), idesc, 1u);
          if (!CHAIN) {
            umma2_bf16(d1, da1 + (uint64_t)(2 * k), dbh + (uint64_t)(2 * k), idesc, acc);
            umma2_bf16(d1, da1 + (uint64_t)(2 * k), dbl + (uint64_t)(2 * k), idesc, 1u);
          }
        }
        umma2_commit_to(&empty_bar[s], 3);
        bool seg_end = (kb == KB - 1) || it == n_units - 1;
        if (CHAIN) {
          seg_end = ++links == CHAIN_KB || seg_end;
          if (seg_end) links = 0;
        }
        if (seg_end) {
          umma2_commit_to(&acc_full[buf], 3);
          ++seg;
          buf = (P.nbuf == 2) ? (buf ^ 1) : 0;
        }
        seg_start = seg_end;
        if (++kb == KB) kb = 0;
        if (++s == n_stages) { s = 0; ph ^= 1u; }
      }
      if (!ok) atomicExch(&s_error, 1);
    }
  } else {
    // ------------------------------------------------------------------ epilogue (both CTAs)
    const int quarter = warp & 3;
    const int n_ch = n_epi >> 2;
    const int c_per = (((tt >> 4) + n_ch - 1) / n_ch) << 4;   // token columns in steps of 16
    const int c_lo = min(((warp - 2) >> 2) * c_per, tt);
    const int c_hi = min(c_lo + c_per, tt);
    const uint32_t acc_empty_even[2] = {cluster_addr_of(smem_u32(&acc_empty[0]), 0),
                                        cluster_addr_of(smem_u32(&acc_empty[1]), 0)};
    bool dry = !CHAIN && P.epi_dry != 0; // a dry pass over the loop body first (nothing stored, nothing waited for)
    bool ok = true;
    int seg = 0;
    unsigned u = u_lo;
    while (u < u_hi && ok) {
      const int tile = (int)(u / KB);
      unsigned seg_hi = (unsigned)(tile + 1) * KB;
      if (seg_hi > u_hi) seg_hi = u_hi;
      int row0, col_off = 0, n_rows = P.n0;
      const int wt = weight_of(tile), tok0 = tok_of(tile) * tt;
      if (wt >= P.tiles1) { row0 = (wt - P.tiles1) * ROWS; col_off = P.n0 + P.n1; n_rows = P.n2; }
      else if (wt >= P.tiles0) { row0 = (wt - P.tiles0) * ROWS; col_off = P.n0; n_rows = P.n1; }
      else row0 = wt * ROWS;
      if (dry) n_rows = 0;
      // partial-sum slot = rank of this cluster among the tile's contributors
      const int slot = (int)cid - (int)sk_owner((unsigned)tile * KB, (unsigned)P.sk_ctas, P.sk_units);
      auto store16 = [&](int a, int c0, auto value) {
        const int feat = row0 + a * 2 * BM + (int)rank * BM + quarter * 32 + lane;
        const int left = feat < n_rows ? P.R - (tok0 + c0) : 0;
        float *yp = P.Y + (size_t)slot * P.split_stride + col_off + feat + (size_t)(tok0 + c0) * P.ldy;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          if (j < left) *yp = value(j);
          yp += P.ldy;
        }
      };
      if constexpr (CHAIN) {
        constexpr int GROUPS = 8;                          // steps of 16 columns per warp
        float sum[GROUPS][16];
#pragma unroll
        for (int i = 0; i < GROUPS; ++i)
#pragma unroll
          for (int j = 0; j < 16; ++j) sum[i][j] = 0.f;
#pragma unroll 1
        for (unsigned v = u; v < seg_hi; v += CHAIN_KB, ++seg) {
          const int buf = seg & 1;
          ok = mbar_wait(&acc_full[buf], (uint32_t)(seg >> 1) & 1u);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t from = tmem_acc + (uint32_t)(buf * tt + c_lo) + ((uint32_t)(quarter * 32) << 16);
#pragma unroll
          for (int i = 0; i < GROUPS; ++i) {
            if (c_lo + 16 * i >= c_hi) break;
            uint32_t va[16];
            tmem_ld16(from + 16u * i, va);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int j = 0; j < 16; ++j) sum[i][j] += __uint_as_float(va[j]);
          }
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(acc_empty_even[buf]);
        }
        if (!ok) break;
#pragma unroll
        for (int i = 0; i < GROUPS; ++i)
          if (c_lo + 16 * i < c_hi) store16(0, c_lo + 16 * i, [&](int j) { return sum[i][j]; });
      } else {
        const int buf = seg % P.nbuf;
        if (!dry) {
          ok = mbar_wait(&acc_full[buf], (uint32_t)(seg / P.nbuf) & 1u);
          if (!ok) break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
        for (int a = 0; a < 2; ++a) {
          const uint32_t lane_base = tmem_acc + (uint32_t)((buf * 2 + a) * tt) + ((uint32_t)(quarter * 32) << 16);
#pragma unroll 1
          for (int c0 = c_lo; c0 < c_hi; c0 += 16) {       // rolled, as in the one-CTA kernel
            uint32_t va[16];
            tmem_ld16(lane_base + (uint32_t)c0, va);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            store16(a, c0, [&](int j) { return __uint_as_float(va[j]); });
          }
        }
        if (dry) {                         // the same segment again, for real
          dry = false;
          continue;
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(acc_empty_even[buf]);
        ++seg;
      }
      u = seg_hi;
    }
    if (!ok) atomicExch(&s_error, 1);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1 && rank == 0 && s_error) {
    // a wait ran out: MMAs issued before that may still be running on both tensor memories
    if (lane == 0) {
      asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                   ::"r"(smem_u32(&drain_bar)) : "memory");
      (void)mbar_wait(&drain_bar, 0);
    }
    __syncwarp();
  }
  // neither CTA frees tensor memory or leaves while the other may still be signalled or read
  cluster_barrier();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_acc), "r"(512u) : "memory");
  }
  if (threadIdx.x == 0 && s_error && P.status) atomicMax(P.status, E_TIMEOUT);
}

// ------------------------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn g_encode = nullptr;
std::mutex g_mu;
std::map<std::tuple<const void *, int, int, int>, CUtensorMap> g_maps;   // (ptr, rows, K, box rows)
// Per-device facts and set-up: the kernel's shared-memory opt-in is an attribute of the function on
// one device, so every device the library is used on is prepared once (under g_mu).
constexpr int MAX_DEVICES = 64;
struct DevInfo {
  bool ready;
  int smem_optin, num_sms;
  int pair_clusters;    // CTA pairs of gemm_tc_pair_kernel that can be resident at once (0: not usable)
};
DevInfo g_dev[MAX_DEVICES] = {};
thread_local int t_dev = 0;          // the calling thread's current device as of its last use_current_device()
// Points the per-device facts at the calling thread's current device; false if that device was
// never prepared by tc_init_driver().
bool use_current_device() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES || !g_dev[dev].ready) return false;
  t_dev = dev;
  return true;
}
#define g_smem_optin (g_dev[t_dev].smem_optin)
#define g_num_sms (g_dev[t_dev].num_sms)
#define g_pair_clusters (g_dev[t_dev].pair_clusters)
int g_tune_stages = 0;      // 0 = as many as fit (at most 8)
int g_tune_max_split = 0;   // 0 = default rule
int g_tune_no_streamk = 0;  // 1 = always the per-tile decomposition
int g_tune_late_w = 0;      // 1 = weights wait for the dependency too
int g_tune_early_stages = -1; // < 0: EARLY_STAGES, or the whole ring without programmatic launch
int g_tune_no_wave_split = 0; // 1 = several token tiles keep the one-wave rule's split factor
int g_tune_no_accp = 0;      // 1 = pairs of more than 128 tokens as two 128-token tiles with extra columns
int g_tune_epi = 0;         // 1, 2: that many epilogue warps per lane quarter for 256-row weight tiles (default 4)
int g_tune_epi_narrow = 0;  // 1, 2, 4: epilogue warps per lane quarter for 128-row weight tiles (default by token tile)
int g_tune_no_pair2 = 0;    // 1 = no CTA-pair kernel; 2 = not for 65 to 128 tokens
int g_tune_pair_min = 0;    // > 0: fewest rows for the CTA-pair kernel
int g_tune_epi_dry = 1;
int g_tune_short_sums = 0;  // 1 = the CTA-pair kernel always sums in short chains, from 65 rows up
int g_tune_pace = PACE_CYCLES;      // 0 = the stages past the early ones come with their activations
int g_tune_no_wide = 0;      // 1 = 128 weight rows per CTA also for wide token tiles
int g_tune_traffic_div = 8; // split <= K_in / (div * tokens)

bool get_map(const void *ptr, int rows, int K_in, int box_rows, CUtensorMap *out) {
  std::lock_guard<std::mutex> lock(g_mu);
  auto key = std::make_tuple(ptr, rows, K_in, box_rows);
  auto it = g_maps.find(key);
  if (it != g_maps.end()) {
    *out = it->second;
    return true;
  }
  if (!g_encode) return false;
  CUtensorMap m;
  cuuint64_t dims[2] = {(cuuint64_t)K_in, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)K_in * 2};
  cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = g_encode(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(ptr), dims, strides,
                        box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return false;
  g_maps[key] = m;
  *out = m;
  return true;
}

}  // namespace

bool tc_get_map(const void *ptr, int rows, int K_in, int box_rows, CUtensorMap *out) {
  return get_map(ptr, rows, K_in, box_rows, out);
}
int tc_smem_optin() { return use_current_device() ? g_smem_optin : 0; }
int tc_num_sms() { return use_current_device() ? g_num_sms : 0; }
bool attn_tc_prepare(int smem_optin);

// Prepares the calling thread's current device (once per device) and remembers it for the
// launchers that follow on this thread.
int tc_init_driver(char *err, size_t errlen) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) {
    snprintf(err, errlen, "no usable current device: %s", cudaGetErrorString(e));
    return 1;
  }
  std::lock_guard<std::mutex> lock(g_mu);
  t_dev = dev;
  if (g_dev[dev].ready) return 0;
  if (!g_encode) {
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q);
    if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || fn == nullptr) {
      snprintf(err, errlen, "cuTensorMapEncodeTiled not available: %s", cudaGetErrorString(e));
      return 1;
    }
    g_encode = reinterpret_cast<EncodeTiledFn>(fn);
  }
  DevInfo d{};
  cudaDeviceGetAttribute(&d.smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaDeviceGetAttribute(&d.num_sms, cudaDevAttrMultiProcessorCount, dev);
  const void *forms[4] = {(const void *)gemm_tc_kernel<FORM_PLAIN, false>, (const void *)gemm_tc_kernel<FORM_COLS, false>,
                          (const void *)gemm_tc_kernel<FORM_ACC, false>, (const void *)gemm_tc_kernel<FORM_ACC, true>};
  for (const void *f : forms)
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, d.smem_optin - 1024);
  if (e != cudaSuccess) {
    snprintf(err, errlen, "cannot raise the GEMM kernel's shared memory: %s", cudaGetErrorString(e));
    return 1;
  }
  // the CTA-pair kernel: shared-memory opt-in, and how many pairs fit on this device at once
  {
    const size_t smem = (size_t)d.smem_optin - 1024;       // as many stages as fit, see gemm_tc()
    d.pair_clusters = 0;
    if ((size_t)d.smem_optin >= (size_t)3 * (2 * PAIR_PART_BYTES + 256 * BK * 2) + 2048 &&
        cudaFuncSetAttribute(gemm_tc_pair_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess &&
        cudaFuncSetAttribute(gemm_tc_pair_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(2 * (d.num_sms / 2));
      cfg.blockDim = dim3(PAIR_THREADS);
      cfg.dynamicSmemBytes = smem;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = 2;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, gemm_tc_pair_kernel<false>, &cfg) == cudaSuccess && n > 0)
        d.pair_clusters = n < d.num_sms / 2 ? n : d.num_sms / 2;
      (void)cudaGetLastError();
    }
  }
  if (!attn_tc_prepare(d.smem_optin)) {
    snprintf(err, errlen, "the attention kernels' shared memory is not laid out as they count on");
    return 1;
  }
  d.ready = true;
  g_dev[dev] = d;
  return 0;
}

void attn_tc_set_min_rows(int rows);
void attn_tc_set_chunks(int chunks);
void attn_tc_set_dry_pass(int on);
void attn_mma_set_chunks(int chunks);
void tc_set_tuning(int key, int value) {
  if (key == 9) attn_tc_set_min_rows(value);
  if (key == 12) attn_tc_set_chunks(value);
  if (key == 20) attn_tc_set_dry_pass(value);
  if (key == 1) g_tune_stages = value;
  if (key == 10) g_tune_no_wave_split = value;
  if (key == 11) g_tune_no_wide = value;
  if (key == 13) g_tune_no_accp = value;
  if (key == 15) g_tune_epi = value;
  if (key == 16) g_tune_epi_narrow = value;
  if (key == 17) g_tune_no_pair2 = value;
  if (key == 18) g_tune_pair_min = value;
  if (key == 21) g_tune_epi_dry = value;
  if (key == 22) attn_mma_set_chunks(value);
  if (key == 23) g_tune_short_sums = value;
  if (key == 24) g_tune_pace = value > 0 ? value : 0;      // exactly one thread requests those stages: pace > 0 or == 0
  if (key == 2) g_tune_max_split = value;
  if (key == 3) g_tune_no_streamk = value;
  if (key == 6) g_tune_late_w = value;
  if (key == 8) g_tune_early_stages = value;
  if (key == 7 && value > 0) g_tune_traffic_div = value;
}

void tc_forget_maps() {
  std::lock_guard<std::mutex> lock(g_mu);
  g_maps.clear();
}

bool tc_supported(const GemmMats &m, int K_in) {
  if (K_in % BK != 0 || K_in < BK) return false;
  for (int i = 0; i < m.n; ++i)
    if (m.n_out[i] < 1 || ((uintptr_t)m.W[i] & 15u)) return false;
  return g_encode != nullptr;
}

// Split-K factor: as many CTAs as fit in one wave of the co-resident slots (two per SM), while
// every split keeps at least 8 K-blocks and the fp32 partial sums written and re-read
// (split x tokens x 4 bytes per output) stay below about half of the weight bytes.
static int split_cap(int kblocks, int tokens) {
  int s = 12;
  const int by_k = kblocks / 8;
  const int by_traffic = (kblocks * 64) / (g_tune_traffic_div * (tokens > 0 ? tokens : 1));
  if (s > by_k) s = by_k;
  if (s > by_traffic) s = by_traffic;
  if (g_tune_max_split > 0 && s > g_tune_max_split) s = g_tune_max_split;
  return s < 1 ? 1 : s;
}

int tc_default_split(int n_tiles, int kblocks, int tokens) {
  if (!use_current_device()) return 1;
  const int slots = 2 * g_num_sms;
  int s = slots / (n_tiles > 0 ? n_tiles : 1);
  const int cap = split_cap(kblocks, tokens);
  if (s > cap) s = cap;
  return s < 1 ? 1 : s;
}

// Several token tiles (more than 128 rows as pairs): `ctas` = weight tiles x token tiles may exceed
// the co-resident slots, and then the launch runs in rounds whose last one can be nearly empty.
// The time goes as rounds(split) / split (each CTA covers K / split), so among the allowed factors
// take the one with the fewest round-lengths, but leave `split0` (the one-wave rule's choice)
// unless another is at least 10 % better.
static int wave_split(int ctas, int kblocks, int tokens, int split0, int slots) {
  const int cap = split_cap(kblocks, tokens);
  auto cost = [&](int sp) { return (double)((ctas * sp + slots - 1) / slots) / sp; };
  int best = split0 <= cap ? split0 : cap;
  if (best < 1) best = 1;
  double best_cost = cost(best);
  const double keep = 0.9 * best_cost;
  for (int sp = 1; sp <= cap; ++sp)
    if (cost(sp) < keep && cost(sp) < best_cost - 1e-9) { best = sp; best_cost = cost(sp); }
  return best;
}

// Stream-K plan: how many CTAs share the (tile, K-block) units.  At most two per SM, at least 8
// units per CTA, at most `max_slots` contributors to any tile, and the fp32 partial sums written
// and re-read stay below about half of the weight bytes.  Returns 0 when the classic per-tile
// decomposition is at least as good (one contributor per tile already fills the machine).
int tc_streamk_ctas(int n_tiles, int kblocks, int tokens, int max_slots, int *slots_out) {
  const long long units = (long long)n_tiles * kblocks;
  long long g = 2LL * g_num_sms;
  if (g > units / 8) g = units / 8;
  if (g < 1) g = 1;
  // average contributors per tile = kblocks * g / units; bound it by the traffic rule
  const long long by_traffic = (long long)(kblocks * 64) / ((long long)g_tune_traffic_div * (tokens > 0 ? tokens : 1));
  const long long avg_cap = by_traffic < 1 ? 1 : by_traffic;
  if ((long long)kblocks * g > avg_cap * units) g = avg_cap * units / kblocks;
  if (g_tune_max_split > 0 && (long long)kblocks * g > (long long)g_tune_max_split * units)
    g = (long long)g_tune_max_split * units / kblocks;
  if (g < 1) g = 1;
  auto slots_of = [&](long long gg) {
    const long long per = units / gg;                 // smallest run length
    return (int)((kblocks + per - 1) / per) + ((units % gg) || (kblocks % per) ? 1 : 0);
  };
  while (g > 1 && slots_of(g) > max_slots) --g;
  *slots_out = slots_of(g);
  return (int)g;
}

// The ring of the one-CTA form.  As many stages as fit, two CTAs per SM (each with half of the shared memory) where they get
// two each, so that one CTA's prologue and epilogue overlap the other's streaming.  Behind programmatic launch two weight
// tiles are requested at once, the rest of the ring one per PACE_CYCLES: the kernel before reads its partial sums while they are
// on their way, and behind a whole ring of every CTA at once (up to 28 MB) those reads took most of its time - the residual
// update at one row 4.9 us, 2.9 with two stages only; paced, the ring is as full when the activations come.  Six layers, us
// per pass, whole ring at once / two and one per 800 / 1200 / 1600 / 2000 / 2600 cycles: 7B one-token step 573 / 561 / 554 /
// 552 / 554 / 559, four sequences 644 / 628 / 623 / 622 / 626 / 630, chain of five 1266 / 1238 / 1223 / 1222 / 1225 / 1230, 64
// nodes 818 / 811 / 811 / 810 / 809 / 811, EAGLE iteration of 60 2016 / 1991 / 1978 / 1971 / 1970 / 1977.
// Without it nothing runs beforehand that could be spared: the whole ring at once, and not six stages, of which all CTAs
// begin together (us per call, six paced / six at once / five at once: pair of 8 rows, 12288 x 4096 26.0 / 26.0 / 24.7,
// 4096 x 11008 25.0 / 24.6 / 23.7, 5120 x 13824 32.2 / 32.2 / 31.0; 64 plain rows of 4096 x 4096, three stages, 17.6 paced,
// 16.9 at once).  Behind programmatic launch five are as fast as six (one-token step 560 / 557, chain 1230 / 1233).
TcRing tc_ring(int stage_bytes, int smem_optin, bool wide, bool pdl) {
  TcRing r;
  r.stages = (smem_optin - 2048) / stage_bytes;
  if (r.stages > MAX_STAGES) r.stages = MAX_STAGES;
  const int two_per_sm = (smem_optin / 2 - 2048) / stage_bytes;
  if (g_tune_stages == 0 && two_per_sm >= 2 && two_per_sm < r.stages && !wide)
    r.stages = !pdl && two_per_sm > ALONE_STAGES ? ALONE_STAGES : two_per_sm;
  if (g_tune_stages > 0 && g_tune_stages < r.stages) r.stages = g_tune_stages;
  const int early = g_tune_early_stages >= 0 ? g_tune_early_stages : (pdl ? EARLY_STAGES : r.stages);
  r.early = g_tune_late_w ? 0 : (early < r.stages ? early : r.stages);
  r.pace = r.early > 0 && r.early < r.stages ? g_tune_pace : 0;
  return r;
}

cudaError_t gemm_tc(Launch L, Operand X, int x_rows_alloc, GemmMats m, int K_in, int R,
                    float *Y, int ldy, int split, size_t split_stride, int *status, int max_slots,
                    SplitIn *out, bool short_sums, bool late_dependents) {
  if (!use_current_device()) return cudaErrorInitializationError;
  if (!tc_supported(m, K_in) || R < 1 || ((uintptr_t)X.hi & 15u) || ((uintptr_t)X.lo & 15u))
    return cudaErrorInvalidValue;
  TcParams P;
  memset(&P, 0, sizeof(P));
  const int pair = X.lo != nullptr ? 1 : 0;
  // A pair of more than 128 tokens keeps all of a tile's tokens in one accumulator (two accumulating
  // MMAs per K step, value rows then residual rows) so that a tile holds up to 256 tokens and the
  // weights are passed over once; up to 128 tokens the residual rows are extra accumulator columns.
  const int accp = (pair && R > 128 && !g_tune_no_accp) ? 1 : 0;
  const int tt_max = (pair && !accp) ? 128 : 256;
  // (A pair's tile is twice as many MMA columns, so up to 128 rows tokens come in eights: the bytes saved are weight
  // stages.  Sixteens / eights, six layers, us per pass: 7B one-token step 565 / 557, four sequences 636 / 627, chain of
  // five 1243 / 1233, 13B one token 794 / 781; before the stages were paced eight sequences 602 / 594, 40 rows 785 / 778, 72
  // rows 858 / 854, 100 rows 2184 / 2171.  Not 17 to 24 rows, where five stages come in the place of four: 7B 17, 20, 24
  // rows 713, 715, 718 / 710, 714, 717, but 13B 958, 959, 963 / 959, 962, 967, and without programmatic launch 893, 899, 901 /
  // 922, 930, 932.)
  const int unit = pair && R <= 128 && (R <= 16 || R > 24) ? 8 : 16;
  int tt = (R + unit - 1) / unit * unit;
  if (tt > tt_max) tt = tt_max;
  if (tt > x_rows_alloc) return cudaErrorInvalidValue;
  const int bn = (pair && !accp) ? 2 * tt : tt;
  const int x_bytes = (accp ? 2 : 1) * bn * BK * 2;      // activation bytes of a stage
  const int ztiles = (R + tt - 1) / tt;
  // the last token tile may reach past R: those rows must exist (they are read, results dropped)
  if (ztiles * tt > x_rows_alloc) return cudaErrorInvalidValue;
  P.tt = tt;
  P.ztiles = ztiles;
  int cols = 32;
  while (cols < bn) cols <<= 1;
  P.Y = Y;
  P.ldy = ldy;
  P.R = R;
  P.bn = bn;
  P.tmem_cols = cols;
  // wide mode: N = 256, every matrix a whole number of 256-row tiles, room for three 64 KB stages
  // (At exactly 128 tokens, where the extra-column form also reaches N = 256, 128 weight rows per CTA with
  // two CTAs per SM measured 6-7 % faster than 256 rows with one: 7B verify 5.7 against 6.1 ms.)
  bool wide = !g_tune_no_wide && accp && bn == 256 && g_smem_optin - 2048 >= 2 * (2 * W_STAGE_BYTES + x_bytes);
  for (int i = 0; i < m.n && wide; ++i) wide = (m.n_out[i] % (2 * BM)) == 0;
  // CTA pairs (512 weight rows per cluster, each CTA loading half of the tokens): 113 tokens and more
  // as a pair, stream-K over the clusters that fit on the device at once.  The last tile of a
  // matrix may be ragged (rows beyond the matrix are zero-filled by the loads and not stored).
  // Measured per verification, 7B shapes: 128 rows 5.67-5.85 against 5.78-5.90 ms, 2 x 64 rows
  // 5.50-5.85 against 5.76-5.90; the 128-token tile costs more than it saves below that (100 rows
  // 5.53 against 5.43, 80 rows 5.25 against 4.48, where the one-CTA form uses an 80-token tile;
  // with 32- and 64-token tiles the pair form measured 13-15 % slower at 16 to 64 rows, where two
  // independent CTAs per SM overlap each other's start and end).
  short_sums = short_sums || g_tune_short_sums != 0;
  const int pair_min_rows = short_sums ? 65 : (g_tune_pair_min > 0 ? g_tune_pair_min : 113);
  if (pair && R >= pair_min_rows && !(g_tune_no_pair2 & 1) && g_pair_clusters > 0 && split == 0 &&
      out != nullptr && max_slots >= 2 && m.n <= 3 && (R > 128 || short_sums || !(g_tune_no_pair2 & 2))) {
    const int zt = (R + 255) / 256, KB = K_in / BK;
    // Short chains: prompt forwards, which take the place of forwards of 64 rows; and where several token tiles
    // would sum over more of K than with one CTA per tile, whose split factor makes more parts (300 rows,
    // 27648 x 5120: 9.4e-6 against 5.7e-6, 0.6e-6 in chains).
    auto tiles_of = [&](int rows) {
      int n = 0;
      for (int i = 0; i < m.n; ++i) n += (m.n_out[i] + rows - 1) / rows;
      return n;
    };
    bool chain = short_sums;
    if (R > 256 && !chain) {
      const int one = wide ? wave_split(tiles_of(2 * BM) * ztiles, KB, R, 1, g_num_sms)
                           : wave_split(tiles_of(BM) * ztiles, KB, R, tc_default_split(tiles_of(BM), KB, R), 2 * g_num_sms);
      const int run = (tiles_of(PAIR_ROWS) * zt * KB + g_pair_clusters - 1) / g_pair_clusters;
      chain = (run < KB ? run : KB) > (KB + one - 1) / one;
    }
    const int rows = chain ? CHAIN_ROWS : PAIR_ROWS;
    const int q0 = (m.n_out[0] + rows - 1) / rows, q1 = m.n > 1 ? (m.n_out[1] + rows - 1) / rows : 0,
              q2 = m.n > 2 ? (m.n_out[2] + rows - 1) / rows : 0;
    // Token tiles: equal up to 32 rows (the MMA's N follows the tile, so 300 rows cost 320 and not 512), all in one
    // launch.
    int ptt = ((R + zt - 1) / zt + 31) / 32 * 32;
    if (ptt < 128 && !chain) ptt = 128;
    const int n_tiles = (q0 + q1 + q2) * zt;
    const long long units = (long long)n_tiles * KB;
    long long g = g_pair_clusters;
    if (g > units / 8) g = units / 8;
    if (g < 1) g = 1;
    auto slots_of = [&](long long gg) {
      const long long per = units / gg;
      return (int)((KB + per - 1) / per) + ((units % gg) || (KB % per) ? 1 : 0);
    };
    while (g > 1 && slots_of(g) > max_slots) --g;
    if (slots_of(g) <= max_slots && (g + 1) * units < (1LL << 32)) {
      P.tiles0 = q0;
      P.tiles1 = q0 + q1;
      P.n0 = m.n_out[0];
      P.n1 = m.n > 1 ? m.n_out[1] : 0;
      P.n2 = m.n > 2 ? m.n_out[2] : 0;
      P.kblocks = KB;
      P.tt = ptt;
      P.bn = ptt;
      P.nbuf = chain || ptt <= 128 ? 2 : 1;
      P.ztiles = zt;
      P.wtiles = q0 + q1 + q2;
      P.sk_ctas = (int)g;
      P.sk_units = (unsigned)units;
      P.split = 1;
      P.split_stride = split_stride;
      P.status = status;
      P.epi_dry = g_tune_epi_dry;
      CUtensorMap mw[3];
      for (int i = 0; i < 3; ++i) {
        const int j = i < m.n ? i : 0;
        if (!get_map(m.W[j], m.n_out[j], K_in, BM, &mw[i])) return cudaErrorInvalidValue;
      }
      SplitIn si{Y, slots_of(g), split_stride, ldy, (unsigned)g, (unsigned)units, (unsigned)KB, chain ? 1u : 2u};
      if (zt > 1) {
        si.sk_tt = (unsigned)ptt;
        si.sk_zt = chain ? 1u : (unsigned)zt;
        si.sk_wt = chain ? (unsigned)P.wtiles : 1u;
      }
      bool ragged = false;
      for (int i = 0; i + 1 < m.n; ++i) ragged = ragged || (m.n_out[i] % rows) != 0;
      if (ragged) {
        si.sk_m0 = (unsigned)P.n0;
        si.sk_m1 = m.n > 2 ? (unsigned)(P.n0 + P.n1) : 0xFFFFFFFFu;
        si.sk_t0 = (unsigned)q0;
        si.sk_t1 = (unsigned)(q0 + q1);
      }
      si.set_inverses();
      *out = si;
      const int stage = (chain ? 1 : 2) * PAIR_PART_BYTES + ptt * BK * 2;
      P.stages = (g_smem_optin - 2048) / stage < PAIR_MAX_STAGES ? (g_smem_optin - 2048) / stage : PAIR_MAX_STAGES;
      CUtensorMap mx, mxlo;
      if (!get_map(X.hi, x_rows_alloc, K_in, ptt / 2, &mx)) return cudaErrorInvalidValue;
      if (!get_map(X.lo, x_rows_alloc, K_in, ptt / 2, &mxlo)) return cudaErrorInvalidValue;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)(2 * g));
      cfg.blockDim = dim3(chain ? CHAIN_THREADS : PAIR_THREADS);
      cfg.dynamicSmemBytes = (size_t)P.stages * stage + 1024;
      cfg.stream = L.st;
      cudaLaunchAttribute attr[2];
      attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[0].val.programmaticStreamSerializationAllowed = L.pdl ? 1 : 0;
      attr[1].id = cudaLaunchAttributeClusterDimension;
      attr[1].val.clusterDim.x = 2;
      attr[1].val.clusterDim.y = 1;
      attr[1].val.clusterDim.z = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 2;
      ++g_launches;
      return chain ? cudaLaunchKernelEx(&cfg, gemm_tc_pair_kernel<true>, mw[0], mw[1], mw[2], mx, mxlo, P)
                   : cudaLaunchKernelEx(&cfg, gemm_tc_pair_kernel<false>, mw[0], mw[1], mw[2], mx, mxlo, P);
    }
    memset(&P, 0, sizeof(P));
    P.tt = tt; P.ztiles = ztiles; P.Y = Y; P.ldy = ldy; P.R = R; P.bn = bn; P.tmem_cols = cols;
  }
  const int bmw = wide ? 2 * BM : BM;
  const int t0 = (m.n_out[0] + bmw - 1) / bmw;
  const int t1 = m.n > 1 ? (m.n_out[1] + bmw - 1) / bmw : 0;
  const int t2 = m.n > 2 ? (m.n_out[2] + bmw - 1) / bmw : 0;
  const int n_tiles = t0 + t1 + t2;
  P.tiles0 = t0;
  P.tiles1 = t0 + t1;
  P.n0 = m.n_out[0];
  P.n1 = m.n > 1 ? m.n_out[1] : 0;
  P.n2 = m.n > 2 ? m.n_out[2] : 0;
  P.kblocks = K_in / BK;
  // stream-K (split == 0): needs a single token tile and 128-row-aligned matrices, so that a
  // column's tile (and with it the number of partial sums to add) follows from the column index
  bool sk = split == 0 && ztiles == 1 && 2LL * (g_num_sms + 1) * n_tiles * P.kblocks < (1LL << 32) && max_slots >= 2 && out != nullptr && !g_tune_no_streamk;
  for (int i = 0; i < m.n && sk; ++i) sk = (m.n_out[i] % bmw) == 0;
  // stream-K pays off where the per-tile decomposition cannot be split further and leaves the SMs
  // unevenly loaded (more tiles than SMs, not a whole number of two-per-SM waves); elsewhere
  // classic split-K gives the same balance with fewer partial sums per tile.  With 256-row tiles
  // (one CTA per SM, tensor-bound) it is taken whenever the best split factor would leave more
  // than a tenth of the SM-rounds empty.
  int sk_ctas = 0, sk_slots = 1;
  if (sk && wide) {
    const int sp = wave_split(n_tiles, P.kblocks, R, 1, g_num_sms);
    const int ctas = n_tiles * sp, rounds = (ctas + g_num_sms - 1) / g_num_sms;
    sk = (double)ctas < 0.9 * (double)rounds * g_num_sms;
    if (sk) {
      // every CTA at least 8 K-blocks, at most max_slots contributors per tile
      const long long units = (long long)n_tiles * P.kblocks;
      long long g = g_num_sms;
      if (g > units / 8) g = units / 8;
      if (g < 1) g = 1;
      auto slots_of = [&](long long gg) {
        const long long per = units / gg;
        return (int)((P.kblocks + per - 1) / per) + ((units % gg) || (P.kblocks % per) ? 1 : 0);
      };
      while (g > 1 && slots_of(g) > max_slots) --g;
      sk_ctas = (int)g;
      sk_slots = slots_of(g);
      if (sk_ctas <= ctas) sk = false;          // the classic decomposition uses as many CTAs
    }
  } else if (sk) {
    const int classic = tc_default_split(n_tiles, P.kblocks, R);
    sk = classic == 1 && n_tiles > g_num_sms && (n_tiles % (2 * g_num_sms)) != 0;
    if (sk) {
      sk_ctas = tc_streamk_ctas(n_tiles, P.kblocks, R, max_slots, &sk_slots);
      if (sk_ctas <= n_tiles) sk = false;         // nothing to share: one CTA per tile is the same thing
    }
  }
  if (!sk) {
    sk_ctas = 0;
    if (split < 1 && wide) {
      // one CTA per SM: the factor with the fewest round-lengths over the SMs
      split = wave_split(n_tiles * ztiles, P.kblocks, R, 1, g_num_sms);
    } else if (split < 1) {
      split = tc_default_split(n_tiles, P.kblocks, R);
      if (ztiles > 1 && !g_tune_no_wave_split) split = wave_split(n_tiles * ztiles, P.kblocks, R, split, 2 * g_num_sms);
    }
    if (split > P.kblocks) split = P.kblocks;
    if (max_slots > 0 && split > max_slots) split = max_slots;
  }
  P.split = sk ? 1 : split;
  P.sk_ctas = sk_ctas;
  P.sk_units = (unsigned)((long long)n_tiles * P.kblocks);
  P.split_stride = split_stride;
  P.status = status;
  P.nbuf = (sk && 2 * cols <= 256) ? 2 : 1;
  P.epi_dry = g_tune_epi_dry;
  P.late_dep = late_dependents ? 1 : 0;
  const int stage_bytes = (wide ? 2 : 1) * W_STAGE_BYTES + x_bytes;
  const TcRing ring = tc_ring(stage_bytes, g_smem_optin, wide, L.pdl);
  const int stages = ring.stages;
  if (stages < 2) return cudaErrorInvalidValue;
  P.stages = stages;
  P.early_w = ring.early;
  P.pace = ring.pace;
  CUtensorMap mw[3], mx, mxlo;
  for (int i = 0; i < 3; ++i) {
    const int j = i < m.n ? i : 0;
    if (!get_map(m.W[j], m.n_out[j], K_in, BM, &mw[i])) return cudaErrorInvalidValue;
  }
  if (!get_map(X.hi, x_rows_alloc, K_in, tt, &mx)) return cudaErrorInvalidValue;
  if (!get_map(pair ? X.lo : X.hi, x_rows_alloc, K_in, tt, &mxlo)) return cudaErrorInvalidValue;
  dim3 grid = sk ? dim3(sk_ctas, 1, 1) : dim3(n_tiles * ztiles, split, 1);
  const size_t smem = (size_t)stages * stage_bytes + 1024;
  if (out) {
    *out = SplitIn{Y, sk ? sk_slots : split, split_stride, ldy, sk ? (unsigned)sk_ctas : 0u, P.sk_units,
                   (unsigned)P.kblocks, (sk && wide) ? 1u : 0u};
    out->set_inverses();
  }
  // Epilogue warps per 32 accumulator lanes.  256-row tiles keep one accumulator set, so the MMAs
  // of a CTA's next tile wait for the epilogue: sixteen warps (13B-shaped verification of 256 rows:
  // 18.3 ms with four, 16.8 with eight, 16.3 with sixteen).  128-row tiles: four warps (eight: 7B
  // Medusa iteration of 64 rows + 1.5 %, EAGLE iteration + 0.8 %, sampled chain + 1.5 %, one-token
  // step + 0.1 %; sixteen + 20 %).
  int groups = wide ? 4 : 1;
  const int forced = wide ? g_tune_epi : g_tune_epi_narrow;
  if (forced == 1 || forced == 2 || forced == 4) groups = forced;
  auto go = [&](auto *kern) {
    return launch_k(kern, grid, dim3(64 + 128 * groups), smem, L.st, L.pdl, mw[0], mw[1], mw[2], mx, mxlo, P);
  };
  if (!pair) return go(gemm_tc_kernel<FORM_PLAIN, false>);
  if (!accp) return go(gemm_tc_kernel<FORM_COLS, false>);
  return wide ? go(gemm_tc_kernel<FORM_ACC, true>) : go(gemm_tc_kernel<FORM_ACC, false>);
}

}  // namespace koala
