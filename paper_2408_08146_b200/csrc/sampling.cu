// Speculative sampling on chain drafts (Section 2.2 of the paper, the paragraph after Eq. 3):
// drafted tokens are DRAWN from the head's distributions d_i, token i is accepted with probability
// min(1, q_i(x_i) / d_i(x_i)), the first rejected position is redrawn from norm(max(0, q_f - d_f)),
// and if every token is accepted one more is drawn from q_{t+1}.  All random numbers are inputs
// (uniforms in [0, 1)); every draw is an inverse-CDF walk in token-id order.
//   sample_rows_kernel     one row of draft logits -> softmax d (kept), token ~ d, log d(token)
//   accept_sampled_kernel  one sequence: judges the chain, draws the extra token, commits the path
//                          (the same bookkeeping as the greedy acceptance kernel)
#include "common.cuh"

namespace koala {
namespace {

constexpr int NT = 1024;

struct Scratch {          // shared-memory scratch of a block-wide draw
  double wsum[NT / 32];   // per-warp sums of the segment sums
  int owner, last_pos, result;
  float red[32];
};

__device__ __forceinline__ float block_max_f(float v, float *red) {
  v = warp_max(v);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  float r = red[lane];
  r = warp_max(r);
  return r;
}
__device__ __forceinline__ float block_sum_f(float v, float *red) {
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  float r = red[lane];
  r = warp_sum(r);
  return r;
}

// Inverse-CDF draw in index order from the non-negative weights w[0..V-1] in shared memory: the
// smallest j with w[0] + .. + w[j] > u * total.  Thread t owns the contiguous ids [t*seg, (t+1)*seg);
// the 1024 segment sums are scanned in double (shuffles inside a warp, the 32 warp sums by every warp),
// the first segment whose inclusive sum exceeds the target is walked by its thread.  If rounding leaves
// no such j, the last id with a positive weight.  Every thread of the block calls this with the weights
// written and a barrier behind them; every thread gets the result.
// The row is in shared memory with consecutive segments a multiple of the bank count apart at the usual
// vocabulary (32 words): a thread starts its sum at a place of its own in the segment, so that the lanes
// of a warp read 32 different banks.  (A first version let one thread add the 1024 sums one after the
// other and all lanes read one bank: 85 us per drawn row of 32000 against 13 now.)
__device__ int block_draw(const float *w, int V, float u, Scratch *sc) {
  const int seg = (V + NT - 1) / NT;
  const int lo = min((int)threadIdx.x * seg, V), hi = min(lo + seg, V), n = hi - lo;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  double local = 0.0;
  if (n > 0) {
    int j = lo + (int)(threadIdx.x % (unsigned)n);
    for (int i = 0; i < n; ++i) {
      local += (double)w[j];
      if (++j == hi) j = lo;
    }
  }
  double incl = local;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (threadIdx.x == 0) { sc->owner = NT; sc->last_pos = 0; sc->result = 0; }
  if (lane == 31) sc->wsum[wp] = incl;
  __syncthreads();
  double wincl = sc->wsum[lane];               // NT / 32 = 32 warps: lane l holds warp l's sum
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double y = __shfl_up_sync(0xffffffffu, wincl, o);
    if (lane >= o) wincl += y;
  }
  const double total = __shfl_sync(0xffffffffu, wincl, 31);
  const double before_warp = wp > 0 ? __shfl_sync(0xffffffffu, wincl, wp > 0 ? wp - 1 : 0) : 0.0;
  double up = __shfl_up_sync(0xffffffffu, incl, 1);
  if (lane == 0) up = 0.0;
  const double base = before_warp + up;        // weight before this thread's segment
  const double target = (double)u * total;
  if (local > 0.0) {
    atomicMax(&sc->last_pos, (int)threadIdx.x);
    if (before_warp + incl > target) atomicMin(&sc->owner, (int)threadIdx.x);
  }
  __syncthreads();
  const int owner = sc->owner < NT ? sc->owner : sc->last_pos;   // none: rounding; the last positive id
  if ((int)threadIdx.x == owner) {
    int res = -1, last = lo;
    double acc = base;
    for (int j = lo; j < hi; ++j) {
      const float x = w[j];
      if (x > 0.f) last = j;
      acc += (double)x;
      if (res < 0 && sc->owner < NT && acc > target) res = j;
    }
    sc->result = res >= 0 ? res : last;
  }
  __syncthreads();
  return sc->result;
}

// grid R, block 1024, dynamic shared memory V floats.  Row r of the logits belongs to sequence r
// (chain drafts: one row per sequence); its uniform is u[r * u_stride + u_off], its distribution
// goes to probs[(r * u_stride + u_off) * V ..].
__global__ void __launch_bounds__(NT)
sample_rows_kernel(const float *logits, const float *u, int u_stride, int u_off, int32_t *tok, float *logp,
                   float *probs, int V) {
  extern __shared__ float srow[];
  __shared__ Scratch sc;
  pdl_launch_dependents();
  pdl_wait();
  const int r = blockIdx.x;
  const float *row = logits + (size_t)r * V;
  float mx = -INFINITY;
  for (int j = threadIdx.x; j < V; j += NT) {
    srow[j] = row[j];
    mx = fmaxf(mx, srow[j]);
  }
  mx = block_max_f(mx, sc.red);
  float se = 0.f;
  for (int j = threadIdx.x; j < V; j += NT) {
    const float e = expf(srow[j] - mx);
    srow[j] = e;
    se += e;
  }
  se = block_sum_f(se, sc.red);
  float *pr = probs + ((size_t)r * u_stride + u_off) * V;
  const float inv = 1.f / se;
  for (int j = threadIdx.x; j < V; j += NT) {
    const float p = srow[j] * inv;
    srow[j] = p;
    pr[j] = p;
  }
  __syncthreads();
  const int idx = block_draw(srow, V, u[(size_t)r * u_stride + u_off], &sc);
  if (threadIdx.x == 0) {
    tok[r] = idx;
    logp[r] = (row[idx] - mx) - logf(se);
  }
}

// grid B, block 1024, dynamic shared memory V floats.
__global__ void __launch_bounds__(NT)
accept_sampled_kernel(TreeBufs t, const float *verify_logits, const float *chain_d,
                      const float *u_accept, const float *u_bonus, int32_t *seq_len, int32_t *out_tokens,
                      int out_stride, int32_t *out_len, int N, int V, int D, int *status) {
  extern __shared__ float srow[];
  __shared__ Scratch sc;
  __shared__ int s_tok[128];
  __shared__ int s_accept;
  pdl_launch_dependents();
  pdl_wait();
  const int b = blockIdx.x;
  int n = t.tree_n[b] < 128 ? t.tree_n[b] : 128;
  if (n > D + 1) n = D + 1;                       // a chain of at most D drafted tokens
  for (int v = threadIdx.x; v < n; v += NT) {
    s_tok[v] = t.tree_tok[b * N + v];
    if (t.tree_parent[b * N + v] != v - 1 && status) atomicMax(status, 1);     // not a chain: invalid input
  }
  __syncthreads();
  int a = 0;                                      // accepted drafted tokens
  int bonus = 0;
  bool done = false;
  for (int i = 1; i <= n && !done; ++i) {
    // q = softmax of the target's logits at node i - 1 (judges drafted token i, or gives the extra token)
    const float *row = verify_logits + ((size_t)b * N + i - 1) * V;
    float mx = -INFINITY;
    for (int j = threadIdx.x; j < V; j += NT) {
      srow[j] = row[j];
      mx = fmaxf(mx, srow[j]);
    }
    mx = block_max_f(mx, sc.red);
    float se = 0.f;
    for (int j = threadIdx.x; j < V; j += NT) {
      const float e = expf(srow[j] - mx);
      srow[j] = e;
      se += e;
    }
    se = block_sum_f(se, sc.red);
    const float inv = 1.f / se;
    const float *d = chain_d + ((size_t)b * D + i - 1) * V;     // read only while i < n
    const bool last = i == n;                     // every drafted token was accepted: draw from q_{t+1}
    __syncthreads();
    if (threadIdx.x == 0) {
      bool acc = false;
      if (!last) {
        const int x = s_tok[i];
        acc = u_accept[(size_t)b * D + i - 1] * d[x] < srow[x] * inv;
      }
      s_accept = acc ? 1 : 0;
    }
    __syncthreads();
    if (s_accept) {
      ++a;
    } else {                                      // first rejection: redraw from norm(max(0, q - d))
      for (int j = threadIdx.x; j < V; j += NT) {
        const float q = srow[j] * inv;
        srow[j] = last ? q : fmaxf(0.f, q - d[j]);
      }
      __syncthreads();
      bonus = block_draw(srow, V, u_bonus[b], &sc);
      done = true;
    }
    __syncthreads();
  }
  const int len = a + 1;
  if (threadIdx.x == 0) {
    const int S = seq_len[b];
    for (int i = 0; i < len; ++i) {
      t.acc_path[b * N + i] = i;
      if (i >= 1) {
        t.pend_tok[b * N + i - 1] = s_tok[i];
        if (i - 1 < out_stride) out_tokens[(size_t)b * out_stride + i - 1] = s_tok[i];
      }
    }
    if (len - 1 < out_stride) out_tokens[(size_t)b * out_stride + len - 1] = bonus;
    out_len[b] = len;
    t.acc_len[b] = len;
    t.acc_S[b] = S;
    t.n_pend[b] = len;
    t.root_tok[b] = bonus;
    seq_len[b] = S + len;
    if (t.alpha_hits != nullptr) {
      for (int i = 1; i < len; ++i) {
        atomicAdd(&t.alpha_hits[i - 1], 1ull);
        atomicAdd(&t.alpha_trials[i - 1], 1ull);
      }
      if (len < n) atomicAdd(&t.alpha_trials[len - 1], 1ull);
    }
  }
}

}  // namespace

cudaError_t sample_rows(Launch L, const float *logits, const float *u, int u_stride, int u_off, int32_t *tok,
                        float *logp, float *probs, int R, int V) {
  static SmemOptIn optin;
  const size_t smem = (size_t)V * sizeof(float);
  cudaError_t e = optin.ensure((const void *)sample_rows_kernel, smem);
  if (e != cudaSuccess) return e;
  return launch_k(sample_rows_kernel, dim3(R), dim3(NT), smem, L.st, L.pdl, logits, u, u_stride, u_off, tok, logp,
                  probs, V);
}

cudaError_t accept_sampled(Launch L, TreeBufs t, const float *verify_logits, const float *chain_d,
                           const float *u_accept, const float *u_bonus, int32_t *seq_len,
                           int32_t *out_tokens, int out_stride, int32_t *out_len, int B, int N, int V, int D, int *status) {
  static SmemOptIn optin;
  const size_t smem = (size_t)V * sizeof(float);
  cudaError_t e = optin.ensure((const void *)accept_sampled_kernel, smem);
  if (e != cudaSuccess) return e;
  return launch_k(accept_sampled_kernel, dim3(B), dim3(NT), smem, L.st, L.pdl, t, verify_logits, chain_d,
                  u_accept, u_bonus, seq_len, out_tokens, out_stride, out_len, N, V, D, status);
}

}  // namespace koala
