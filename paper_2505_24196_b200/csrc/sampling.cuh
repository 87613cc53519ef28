// Non-greedy decoding (Sec. 4, Table 1 "Temperature = 1"): draws of softmax(logits / T) by the
// Gumbel-max rule and the accept / resample rule of speculative sampling (Leviathan et al. 2023,
// which the paper cites for losslessness), on full rows of logits the forwards leave in global memory.
//
// Random numbers: Philox4x32-10 (Salmon et al., SC'11), key = the caller's 64-bit seed, counter =
// (index, position, purpose, round).  A uniform is ((x >> 8) + 0.5) / 2^24 of the first output word:
// exact in float, never 0 or 1.  Every draw is a pure function of where it is used, so no generator
// state lives anywhere and a round can be replayed.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace clasp {
namespace smp {

enum { DRAW_DRAFT = 0, DRAW_ACCEPT = 1, DRAW_RESIDUAL = 2, DRAW_TARGET = 3 };
constexpr int THREADS = 256;
constexpr int MAX_DRAFTS = 63;
constexpr int PER = 8;                    // values a thread holds at a time
constexpr int MAX_CHUNKS = 64;            // parts of a row of logits, one CTA each

__device__ __forceinline__ uint32_t philox_first_word(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0,
                                                      uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
    const uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
    c0 = n0; c1 = lo1; c2 = n2; c3 = lo0;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return c0;
}
__device__ __forceinline__ float uniform24(unsigned long long seed, uint32_t index, uint32_t pos, uint32_t purpose,
                                           uint32_t rnd) {
  const uint32_t x = philox_first_word(index, pos, purpose, rnd, (uint32_t)seed, (uint32_t)(seed >> 32));
  return ((float)(x >> 8) + 0.5f) * (1.0f / 16777216.0f);
}
__device__ __forceinline__ float gumbel(unsigned long long seed, uint32_t index, uint32_t pos, uint32_t purpose,
                                        uint32_t rnd) {
  return -logf(-logf(uniform24(seed, index, pos, purpose, rnd)));
}

// A row is cut into at most MAX_CHUNKS parts of equal length (a multiple of a CTA's stride), so that one row keeps as many
// SMs busy: a draw is bound by the arithmetic of its Philox rounds and logarithms (about 130 instructions per value), and
// the arg-max of the parts' maxima is that of the row whatever the cut.  At 128256 values, 63 parts: a round of four drafts
// and their verification on the 8B shape 12575 -> 12016 us (one CTA of 1024 threads per row: 121 us per draw, 297 us for the
// five rows of the verification).
inline int chunks_of(int vocab) {
  const int n = (vocab + THREADS * PER - 1) / (THREADS * PER);
  return n < MAX_CHUNKS ? n : MAX_CHUNKS;
}
struct Span {
  int lo, hi;
  __device__ __forceinline__ Span(int vocab, int chunk, int n_chunks) {
    const int len = ((vocab + n_chunks - 1) / n_chunks + THREADS - 1) / THREADS * THREADS;
    lo = min(vocab, chunk * len);
    hi = min(vocab, lo + len);
  }
};

// (value, index) maximum over the block, lowest index on ties; result valid in thread 0
struct Best { float v; int i; };
__device__ __forceinline__ Best better(Best a, Best b) { return (b.v > a.v || (b.v == a.v && b.i < a.i)) ? b : a; }
__device__ __forceinline__ Best warp_best(Best mine) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    Best other{__shfl_xor_sync(0xffffffffu, mine.v, o), __shfl_xor_sync(0xffffffffu, mine.i, o)};
    mine = better(mine, other);
  }
  return mine;
}
__device__ Best block_argmax(Best mine) {
  __shared__ Best part[THREADS / 32];
  mine = warp_best(mine);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = mine;
  __syncthreads();
  if (threadIdx.x == 0)
    for (int w = 1; w < THREADS / 32; ++w) mine = better(mine, part[w]);
  return mine;
}
// maximum of a span of a row scaled by inv_t and the sum of exp(x - maximum); valid in thread 0
__device__ float2 block_max_sum(const float* __restrict__ row, Span s, float inv_t) {
  __shared__ float part[2][THREADS / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float mx = -INFINITY;
  for (int c = s.lo + threadIdx.x; c < s.hi; c += THREADS) mx = fmaxf(mx, row[c] * inv_t);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  __syncthreads();
  if (lane == 0) part[0][warp] = mx;
  __syncthreads();
  mx = part[0][0];
  for (int w = 1; w < THREADS / 32; ++w) mx = fmaxf(mx, part[0][w]);
  float sum = 0.f;
  for (int c = s.lo + threadIdx.x; c < s.hi; c += THREADS) {
    const float x = row[c] * inv_t;
    sum += x == -INFINITY ? 0.f : expf(x - mx);   // (a span may hold nothing but -inf)
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) part[1][warp] = sum;
  __syncthreads();
  float tot = 0.f;
  for (int w = 0; w < THREADS / 32; ++w) tot += part[1][w];   // fixed order
  return make_float2(mx, tot);
}

// scratch of the rows of one call (in the workspace); every entry is written before it is read
struct AcceptScratch {
  Best best[MAX_DRAFTS + 1][MAX_CHUNKS];        // per row and part: the draw's candidate
  float2 norm_p[MAX_DRAFTS + 1][MAX_CHUNKS];    // (maximum, sum of exp) of the full model's row
  float2 norm_q[MAX_DRAFTS + 1][MAX_CHUNKS];    // ... of the draft model's row
};

// the span's part of a draw of softmax(logits / T): arg-max of logits / T + Gumbel noise, lowest index on ties
__device__ Best span_draw(const float* __restrict__ row, Span s, float inv_t, unsigned long long seed, int pos, int purpose,
                          int rnd) {
  Best mine{-INFINITY, 0x7fffffff};
  for (int c0 = s.lo + threadIdx.x; c0 < s.hi; c0 += THREADS * PER) {
    float l[PER];
#pragma unroll
    for (int e = 0; e < PER; ++e) l[e] = c0 + e * THREADS < s.hi ? row[c0 + e * THREADS] : -INFINITY;
#pragma unroll
    for (int e = 0; e < PER; ++e)
      if (l[e] != -INFINITY) {
        const int c = c0 + e * THREADS;
        mine = better(mine, Best{l[e] * inv_t + gumbel(seed, (uint32_t)c, (uint32_t)pos, (uint32_t)purpose, (uint32_t)rnd), c});
      }
  }
  return block_argmax(mine);
}

// grid: parts of the row
__global__ void __launch_bounds__(THREADS)
gumbel_argmax_kernel(const float* __restrict__ logits, int vocab, float inv_t, unsigned long long seed, int pos,
                     int purpose, int rnd, AcceptScratch* __restrict__ out) {
  const Best b = span_draw(logits, Span(vocab, blockIdx.x, gridDim.x), inv_t, seed, pos, purpose, rnd);
  if (threadIdx.x == 0) out->best[0][blockIdx.x] = b;
}
// the candidate of the parts' candidates of one row, by one warp
__device__ __forceinline__ Best merge_parts(const Best* __restrict__ part, int n_chunks) {
  Best mine{-INFINITY, 0x7fffffff};
  for (int c = threadIdx.x & 31; c < n_chunks; c += 32) mine = better(mine, part[c]);
  return warp_best(mine);
}
__global__ void gumbel_merge_kernel(const AcceptScratch* __restrict__ in, int n_chunks, int32_t* __restrict__ token_out) {
  const Best b = merge_parts(in->best[0], n_chunks);
  if (threadIdx.x == 0) token_out[0] = b.i;
}

// Grid (parts, n_drafts + 1).  Rows k < n_drafts: the part's share of both log normalisers; row n_drafts: its candidate for
// the token of the position after the last draft.  p: full model's logits [n_drafts + 1, vocab], q: the draft model's
// [n_drafts, vocab]; draft k sits at position pos0 + k.
__global__ void __launch_bounds__(THREADS)
spec_norm_kernel(const float* __restrict__ p, const float* __restrict__ q, int n_drafts, int vocab, float inv_t,
                 unsigned long long seed, int pos0, int rnd, AcceptScratch* __restrict__ out) {
  const int k = blockIdx.y;
  const Span s(vocab, blockIdx.x, gridDim.x);
  const float* pr = p + (long long)k * vocab;
  if (k == n_drafts) {
    const Best b = span_draw(pr, s, inv_t, seed, pos0 + k, DRAW_TARGET, rnd);
    if (threadIdx.x == 0) out->best[k][blockIdx.x] = b;
    return;
  }
  const float2 zp = block_max_sum(pr, s, inv_t), zq = block_max_sum(q + (long long)k * vocab, s, inv_t);
  if (threadIdx.x == 0) {
    out->norm_p[k][blockIdx.x] = zp;
    out->norm_q[k][blockIdx.x] = zq;
  }
}
// log normaliser of a row from its parts, by one warp: every lane the same value
__device__ __forceinline__ float log_norm(const float2* __restrict__ part, int n_chunks) {
  const int lane = threadIdx.x & 31;
  float mx = -INFINITY, sum = 0.f;
  for (int c = lane; c < n_chunks; c += 32) mx = fmaxf(mx, part[c].x);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  for (int c = lane; c < n_chunks; c += 32) {
    const float2 v = part[c];
    sum += v.x == -INFINITY ? v.y : v.y * expf(v.x - mx);   // (nothing but -inf: v.y = 0)
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  return mx + logf(sum);
}

// Grid (parts, n_drafts): the part's candidate for the replacement of draft k, a draw of norm(max(0, p_k - q_k))
__global__ void __launch_bounds__(THREADS)
spec_rows_kernel(const float* __restrict__ p, const float* __restrict__ q, int vocab, float inv_t, unsigned long long seed,
                 int pos0, int rnd, AcceptScratch* __restrict__ out) {
  const int k = blockIdx.y;
  const Span s(vocab, blockIdx.x, gridDim.x);
  const float* pr = p + (long long)k * vocab;
  const float* qr = q + (long long)k * vocab;
  const float zp = log_norm(out->norm_p[k], gridDim.x), zq = log_norm(out->norm_q[k], gridDim.x);
  Best mine{-INFINITY, 0x7fffffff};
  for (int c = s.lo + threadIdx.x; c < s.hi; c += THREADS) {
    const float resid = expf(pr[c] * inv_t - zp) - expf(qr[c] * inv_t - zq);
    if (resid > 0.f)
      mine = better(mine, Best{logf(resid) + gumbel(seed, (uint32_t)c, (uint32_t)(pos0 + k), DRAW_RESIDUAL, (uint32_t)rnd), c});
  }
  mine = block_argmax(mine);
  if (threadIdx.x == 0) out->best[k][blockIdx.x] = mine;
}

// One CTA, a warp per row in turn: acceptance probability min(1, p_k(x_k) / q_k(x_k)) of draft k and its replacement; then
// one thread walks the drafts, accepts while u_k < the probability, and commits the replacement.
__global__ void __launch_bounds__(THREADS)
spec_commit_kernel(const AcceptScratch* __restrict__ in, const float* __restrict__ p, const float* __restrict__ q,
                   const int32_t* __restrict__ drafts, int n_drafts, int n_chunks, int vocab, float inv_t,
                   unsigned long long seed, int pos0, int rnd, int32_t* __restrict__ n_accepted,
                   int32_t* __restrict__ committed) {
  __shared__ float acc_prob[MAX_DRAFTS + 1];
  __shared__ int repl[MAX_DRAFTS + 1];
  for (int k = threadIdx.x >> 5; k <= n_drafts; k += THREADS / 32) {
    const Best b = merge_parts(in->best[k], n_chunks);
    if (k == n_drafts) {
      if ((threadIdx.x & 31) == 0) repl[k] = b.i;
      continue;
    }
    const float zp = log_norm(in->norm_p[k], n_chunks), zq = log_norm(in->norm_q[k], n_chunks);
    if ((threadIdx.x & 31) == 0) {
      const int x = drafts[k];
      const float lr = (p[(long long)k * vocab + x] * inv_t - zp) - (q[(long long)k * vocab + x] * inv_t - zq);
      acc_prob[k] = expf(fminf(lr, 0.f));
      repl[k] = b.i < vocab ? b.i : x;   // (no positive residual: p == q, the draft cannot be rejected)
    }
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  int a = 0;
  while (a < n_drafts && uniform24(seed, 0u, (uint32_t)(pos0 + a), DRAW_ACCEPT, (uint32_t)rnd) < acc_prob[a]) {
    committed[a] = drafts[a];
    ++a;
  }
  committed[a] = repl[a];
  n_accepted[0] = a;
}

}  // namespace smp
}  // namespace clasp
