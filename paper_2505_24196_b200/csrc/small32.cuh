// fp32 models whose layers fit the shared memory of one thread-block cluster: a whole call (layer search, verification,
// draft token) is ONE launch of one cluster of 16 CTAs.
//
// The work of a call is a chain of small dependent steps (at 256 columns a product over two rows is 0.3 MFLOP), so what
// bounds it is the hand-off between steps, not any unit of the chip: as one kernel per step a step took 4 us (launch,
// ramp, tail), here a step ends in a hardware cluster barrier.  Every CTA owns a slice of each matrix's output features;
// its slices of the next layer are on their way to shared memory (bulk copies) while the current one is multiplied.
// Activations cross between the CTAs through global memory (L2).
// Measured on 256 columns, 8 layers: search over 64 positions 396 -> 146 us, draft token 310 -> 108, verification of five
// rows 474 -> 176.  A layer takes about 15 us: five hand-offs of about 2000 cycles (stores to L2 before the barrier, the
// barrier, loads from L2 behind it) and as much again for what the 16 SMs read from shared memory and shuffle.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "gemm_tc.cuh"
#include "kernels.cuh"

namespace clasp {
namespace s32 {

constexpr int CTAS = 16;
constexpr int WARPS = 16;
constexpr int THREADS = WARPS * 32;
constexpr int NR = 8;              // rows per pass of a product
constexpr int MAX_F = 6;           // features per warp and product
constexpr int MAX_L = 32;
constexpr int MAX_STATES = 64;
constexpr uint32_t GAVE_UP = 1u << 4;
constexpr int MAX_ROWS = 128;      // rows of a call: an Eq. 2 step keeps two doubles of each in the attention's area

struct LayerPtrs {
  const float *attn_norm, *wq, *wk, *wv, *wo, *mlp_norm, *wg, *wu, *wd;
  float *ck, *cv;
};

struct Params {
  LayerPtrs layer[MAX_L];   // search: all layers; forward: the kept ones in order
  int n_layers;
  int d, qd, kvd, nq, nkv, dffn, vocab;
  float eps;
  double theta;
  int T, C, pos0;
  float *qkv, *attn, *x1, *act, *logits;
  float2* rope;
  // forward (search == 0): T rows, one state, K/V written to the cache at C
  int search;
  const int32_t* tokens;
  const float* embed;
  float* x_base[2];         // layer input k at x_base[0] + k * x_step when x_step > 0, else ping-pong
  long long x_step, ldx;
  const float *final_norm, *lm_head;
  int head_rows;            // last rows that go through the head (0: none)
  int32_t* argmax_out;
  float *top1_out, *logits_out;
  // search
  const float* hidden;
  long long layer_stride, token_stride;
  int M, prune;             // prune: only states that can reach (L, M)
  float* G;                 // layer output of state j, row t at row (j - 1) * T + t
  float* g[2];
  float *scores, *margins, *g_final;
  const uint8_t* forced;
  uint8_t* skip_mask;
  int* status;
  uint32_t spin_fast, spin_slow;
};
static_assert(sizeof(Params) < 4000, "kernel parameters");
static_assert(MAX_ROWS * 2 * (int)sizeof(double) <= WARPS * (2 * 64 + 4) * (int)sizeof(float), "cosines of a step's rows");

__host__ __device__ __forceinline__ int slice_cap(int n) { return (n + CTAS - 1) / CTAS; }
// floats of dynamic shared memory: weight slices (the gate/up area also takes the head's slice), rows, attention, tables
__host__ __device__ inline int smem_floats(int d, int qd, int kvd, int dffn, int hd, int L, int M) {
  const int kmax = d > qd ? (d > dffn ? d : dffn) : (qd > dffn ? qd : dffn);
  return slice_cap(qd + 2 * kvd) * d + slice_cap(d) * qd + 2 * slice_cap(dffn) * d + slice_cap(d) * dffn + NR * kmax +
         WARPS * (2 * hd + 4) + MAX_STATES + ((L + 1) * (M + 1) + 15) / 16 * 4;
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_barrier() {
  cluster_arrive();
  cluster_wait();
}
// consecutive floats from global to shared memory (a multiple of 16 bytes, both ends 16-byte aligned)
__device__ __forceinline__ void bulk_copy(float* dst, const float* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(tc::smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

// one rotated pair; spelled out so that a key rotated for the cache and one rotated on the fly are the same bits
__device__ __forceinline__ float rot_lo(float a, float b, float2 cs) { return __fmaf_rn(a, cs.x, -__fmul_rn(b, cs.y)); }
__device__ __forceinline__ float rot_hi(float a, float b, float2 cs) { return __fmaf_rn(b, cs.x, __fmul_rn(a, cs.y)); }

// Sums over the warp of the N <= 8 values of v: lane l returns the total of v[l & (N - 1)].  Partners are 4, 2, 1, 8, 16
// lanes away for every N, so a row's sum is the same however many rows share the pass.
template <int N>
__device__ __forceinline__ float reduce_rows(float (&v)[N], int lane) {
#pragma unroll
  for (int w = 4; w >= 1; w >>= 1) {
    if (w >= N) {
#pragma unroll
      for (int i = 0; i < N; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], w);
      continue;
    }
    const bool up = (lane & w) != 0;
#pragma unroll
    for (int i = 0; i < w; ++i) {
      const float send = up ? v[i] : v[i + w];
      const float keep = up ? v[i + w] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, w);
    }
  }
  float t = v[0];
  t += __shfl_xor_sync(0xffffffffu, t, 8);
  t += __shfl_xor_sync(0xffffffffu, t, 16);
  return t;
}

template <int HD>
struct Call {
  const Params& p;
  int rank, tid, warp, lane;
  float *w_qkv, *w_o, *w_gu, *w_d, *xs, *att_q, *att_p;
  int* s_take;
  uint8_t* s_choice;
  uint64_t* bars;           // per product: its slices of the layer at hand have arrived
  mutable uint32_t parity;  // bit ph: parity of the next wait on bars[ph]; GAVE_UP: a wait of this thread ran out
  int kmax;
  int lo_qkv, n_qkv, lo_d, n_d, lo_f, n_f, lo_v, n_v;

  __device__ __forceinline__ Call(const Params& p_, float* sm, uint64_t* bars_, int rank_)
      : p(p_), rank(rank_), bars(bars_), parity(0) {
    tid = threadIdx.x;
    warp = tid >> 5;
    lane = tid & 31;
    auto part = [&](int n, int& lo, int& cnt) {
      lo = n * rank / CTAS;
      cnt = n * (rank + 1) / CTAS - lo;
    };
    part(p.qd + 2 * p.kvd, lo_qkv, n_qkv);
    part(p.d, lo_d, n_d);
    part(p.dffn, lo_f, n_f);
    part(p.vocab, lo_v, n_v);
    kmax = max(p.d, max(p.qd, p.dffn));
    w_qkv = sm;
    w_o = w_qkv + slice_cap(p.qd + 2 * p.kvd) * p.d;
    w_gu = w_o + slice_cap(p.d) * p.qd;
    w_d = w_gu + 2 * slice_cap(p.dffn) * p.d;
    xs = w_d + slice_cap(p.d) * p.dffn;
    att_q = xs + NR * kmax;
    att_p = att_q + WARPS * HD;
    s_take = reinterpret_cast<int*>(att_p + WARPS * (HD + 4));
    s_choice = reinterpret_cast<uint8_t*>(s_take + MAX_STATES);
  }

  // ---- weight slices of a layer from global to shared memory (one thread; a slice is consecutive rows of a matrix)
  __device__ void fetch(int ph, int l) const {
    if (tid != 0 || (parity & GAVE_UP)) return;   // (a barrier whose phase may still be open is not armed again)
    const uint32_t bar = tc::smem_u32(bars + ph);
    auto rows = [&](float* dst, const float* w, int first, int n, int K) {
      if (n > 0) bulk_copy(dst, w + (long long)first * K, (uint32_t)n * K * 4u, bar);
    };
    if (l < p.n_layers) {
      const LayerPtrs& w = p.layer[l];
      const int n = ph == 0 ? n_qkv : (ph == 2 ? 2 * n_f : n_d), K = ph == 1 ? p.qd : (ph == 3 ? p.dffn : p.d);
      tc::mbar_expect_tx(bar, (uint32_t)n * K * 4u);
      if (ph == 0) {
        const int hi = lo_qkv + n_qkv, k0 = p.qd, v0 = p.qd + p.kvd;   // features of q, k, v
        const int nq_ = min(hi, k0) - lo_qkv, nk0 = max(lo_qkv, k0), nv0 = max(lo_qkv, v0);
        rows(w_qkv, w.wq, lo_qkv, nq_, K);
        rows(w_qkv + (nk0 - lo_qkv) * K, w.wk, nk0 - k0, min(hi, v0) - nk0, K);
        rows(w_qkv + (nv0 - lo_qkv) * K, w.wv, nv0 - v0, hi - nv0, K);
      } else if (ph == 1) {
        rows(w_o, w.wo, lo_d, n_d, K);
      } else if (ph == 2) {
        rows(w_gu, w.wg, lo_f, n_f, K);
        rows(w_gu + n_f * K, w.wu, lo_f, n_f, K);
      } else {
        rows(w_d, w.wd, lo_d, n_d, K);
      }
    } else if (ph == 2 && p.head_rows > 0 && l == p.n_layers) {
      tc::mbar_expect_tx(bar, (uint32_t)n_v * p.d * 4u);
      rows(w_gu, p.lm_head, lo_v, n_v, p.d);
    }
  }
  // The slices of product ph have arrived.  A wait that runs out is reported and the call carries on to its end through the
  // hardware barriers of its other hand-offs: the thread polls once per product from then on, and when it is the one that
  // fetches slices it fetches none (whoever still waits for those runs out in turn, once).
  __device__ __forceinline__ void arrived(int ph) const {
    const uint32_t bar = tc::smem_u32(bars + ph), par = (parity >> ph) & 1u;
    if (!tc::mbar_test(bar, par) && ((parity & GAVE_UP) || !tc::mbar_wait(bar, par, p.status, p.spin_fast, p.spin_slow))) {
      parity |= GAVE_UP;
      return;
    }
    parity ^= 1u << ph;
  }

  // ---- rows [r0, r0 + nr) into shared memory, as they are or (w != null) RMS-normed; one warp per row
  template <typename Src>
  __device__ __forceinline__ void stage(int r0, int nr, int K, const float* w, Src src) const {
    for (int k = warp; k < nr; k += WARPS) {
      const float* x = src(r0 + k);
      float* dst = xs + k * K;
      if (w) {
        // (rows of up to 256 columns stay in registers, their norm weights come in the same trip)
        float4 v[2], g[2];
        float ss = 0.f;
        double tail = 0.0;   // (past 256 columns: a lane's sum of many groups of four loses what a small group adds)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int c = lane * 4 + q * 128;
          v[q] = g[q] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (c < K) {
            v[q] = __ldcg(reinterpret_cast<const float4*>(x + c));
            g[q] = __ldg(reinterpret_cast<const float4*>(w + c));
          }
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) ss += v[q].x * v[q].x + v[q].y * v[q].y + v[q].z * v[q].z + v[q].w * v[q].w;
        for (int c = lane * 4 + 256; c < K; c += 128) {
          const float4 u = __ldcg(reinterpret_cast<const float4*>(x + c));
          tail += (double)(u.x * u.x + u.y * u.y + u.z * u.z + u.w * u.w);
          *reinterpret_cast<float4*>(dst + c) = u;
        }
        if (K > 256) ss = (float)((double)ss + tail);
        const float sc = rsqrtf(warp_sum(ss) / (float)K + p.eps);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int c = lane * 4 + q * 128;
          if (c < K)
            *reinterpret_cast<float4*>(dst + c) =
                make_float4(v[q].x * sc * g[q].x, v[q].y * sc * g[q].y, v[q].z * sc * g[q].z, v[q].w * sc * g[q].w);
        }
        for (int c = lane * 4 + 256; c < K; c += 128) {
          const float4 u = *reinterpret_cast<const float4*>(dst + c), h = __ldg(reinterpret_cast<const float4*>(w + c));
          *reinterpret_cast<float4*>(dst + c) = make_float4(u.x * sc * h.x, u.y * sc * h.y, u.z * sc * h.z, u.w * sc * h.w);
        }
      } else {
        for (int c = lane * 4; c < K; c += 128)
          *reinterpret_cast<float4*>(dst + c) = __ldcg(reinterpret_cast<const float4*>(x + c));
      }
    }
    __syncthreads();
  }

  // ---- sums over K of N rows in shared memory with the warp's features warp, warp + 16, ... (F at most) of a slice:
  // out(feature in the slice, row of the block, sum, addend) is called by the lane that holds it, with the addend
  // pre(feature, row) that was fetched before the products.  The order of a sum depends on
  // K only, never on the number of rows.
  template <int F, int N, typename Pre, typename Out>
  __device__ __forceinline__ void product_fn(const float* w, int n, int K, int nr, Pre pre, Out out) const {
    float acc[F][N], add[F];
#pragma unroll
    for (int i = 0; i < F; ++i) {
      const int f = warp + i * WARPS;
      add[i] = f < n && lane < nr ? pre(f, lane) : 0.f;
    }
#pragma unroll
    for (int i = 0; i < F; ++i)
#pragma unroll
      for (int r = 0; r < N; ++r) acc[i][r] = 0.f;
    for (int c = lane * 4; c < K; c += 128) {
      float4 x[N];
#pragma unroll
      for (int r = 0; r < N; ++r) x[r] = *reinterpret_cast<const float4*>(xs + r * K + c);
#pragma unroll
      for (int i = 0; i < F; ++i) {
        const int f = min(warp + i * WARPS, n - 1);
        const float4 v = *reinterpret_cast<const float4*>(w + f * K + c);
#pragma unroll
        for (int r = 0; r < N; ++r) {
          acc[i][r] = fmaf(x[r].x, v.x, acc[i][r]);
          acc[i][r] = fmaf(x[r].y, v.y, acc[i][r]);
          acc[i][r] = fmaf(x[r].z, v.z, acc[i][r]);
          acc[i][r] = fmaf(x[r].w, v.w, acc[i][r]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < F; ++i) {
      const float tot = reduce_rows<N>(acc[i], lane);
      const int f = warp + i * WARPS;
      if (f < n && lane < nr) out(f, lane, tot, add[i]);
    }
  }
  template <int F, typename Pre, typename Out>
  __device__ __forceinline__ void product_n(const float* w, int n, int K, int nr, Pre pre, Out out) const {
    if (nr <= 2) product_fn<F, 2>(w, n, K, nr, pre, out);
    else product_fn<F, NR>(w, n, K, nr, pre, out);
  }
  template <typename Pre, typename Out>
  __device__ __forceinline__ void product(const float* w, int n, int K, int nr, Pre pre, Out out) const {
    if (n <= 0) return;
    const int f = (n + WARPS - 1) / WARPS;
    if (f <= 1) product_n<1>(w, n, K, nr, pre, out);
    else if (f <= 2) product_n<2>(w, n, K, nr, pre, out);
    else if (f <= 4) product_n<4>(w, n, K, nr, pre, out);
    else product_n<MAX_F>(w, n, K, nr, pre, out);
  }
  struct NoAdd {
    __device__ __forceinline__ float operator()(int, int) const { return 0.f; }
  };

  // ---- attention of (row, query head) items over cache keys and the row's own state.  Bound by trips to L2, so an item's
  // keys go to up to 16 warps in blocks of eight (four lanes per key: all loads of a block are in flight at once) and the
  // warps' partial results are added in warp order.  Blocks are counted over cache and own keys alike: a position's sums
  // are the same whether its keys come from the cache or from this call.
  __device__ void attention(const LayerPtrs& w, int R) const {
    constexpr int KB = 8, DL = HD / 4;   // keys per block, dims of a key per lane
    const int Gq = p.nq / p.nkv, qkvd = p.qd + 2 * p.kvd;
    const int nb_max = (p.C + p.T + KB - 1) / KB;
    const int S = min(nb_max, WARPS), IG = WARPS / S;
    const int n_items = R * p.nq;
    const float scale = rsqrtf((float)HD) * 1.4426950408889634f;
    for (int base = rank; base < n_items; base += CTAS * IG) {
      const int it = base + (warp / S) * CTAS, sp = warp % S;
      const bool on = warp / S < IG && it < n_items;
      float m = -INFINITY, l = 0.f;
      float acc[HD / 32];
#pragma unroll
      for (int e = 0; e < HD / 32; ++e) acc[e] = 0.f;
      if (on) {
        const int r = it / p.nq, hq = it % p.nq, kvh = hq / Gq, t = r % p.T, s0 = r - t;
        float* q = att_q + warp * HD;
        const float* qr = p.qkv + (long long)r * qkvd + hq * HD;
        for (int i = lane; i < HD / 2; i += 32) {
          const float a = __ldcg(qr + i), b = __ldcg(qr + i + HD / 2);
          const float2 cs = __ldcg(p.rope + t * (HD / 2) + i);
          q[i] = rot_lo(a, b, cs) * scale;
          q[i + HD / 2] = rot_hi(a, b, cs) * scale;
        }
        __syncwarp();
        const int nk = p.C + t + 1, Sr = min((nk + KB - 1) / KB, WARPS);   // (warps past the row's own blocks stay idle)
        for (int k0 = sp < Sr ? sp * KB : nk; k0 < nk; k0 += Sr * KB) {
          // values of the block: HD / 32 dims per lane, all keys in flight (weight 0 past the last key)
          float v[KB][HD / 32];
#pragma unroll
          for (int k = 0; k < KB; ++k) {
            const int kk = min(k0 + k, nk - 1);
            const float* vr = (kk < p.C ? w.cv + (long long)kk * p.kvd : p.qkv + (long long)(s0 + kk - p.C) * qkvd + p.qd + p.kvd) +
                              kvh * HD + lane * (HD / 32);
            if constexpr (HD == 64) {
              const float2 u = __ldcg(reinterpret_cast<const float2*>(vr));
              v[k][0] = u.x; v[k][1] = u.y;
            } else {
              const float4 u = __ldcg(reinterpret_cast<const float4*>(vr));
              v[k][0] = u.x; v[k][1] = u.y; v[k][2] = u.z; v[k][3] = u.w;
            }
          }
          // scores: lane = (key lane / 4, dims of quarter lane % 4)
          const int key = k0 + (lane >> 2), d0 = (lane & 3) * DL;
          float s = 0.f;
          if (key < p.C) {
            const float* kr = w.ck + (long long)key * p.kvd + kvh * HD + d0;
#pragma unroll
            for (int i = 0; i < DL; i += 4) {
              const float4 k4 = __ldcg(reinterpret_cast<const float4*>(kr + i)), q4 = *reinterpret_cast<const float4*>(q + d0 + i);
              s = __fmaf_rn(k4.x, q4.x, s); s = __fmaf_rn(k4.y, q4.y, s);
              s = __fmaf_rn(k4.z, q4.z, s); s = __fmaf_rn(k4.w, q4.w, s);
            }
          } else if (key < nk) {
            const int tk = key - p.C, h = d0 & (HD / 2 - 1);
            const float* kr = p.qkv + (long long)(s0 + tk) * qkvd + p.qd + kvh * HD + h;
            const float2* cr = p.rope + tk * (HD / 2) + h;
            const bool low = d0 < HD / 2;
#pragma unroll
            for (int i = 0; i < DL; i += 4) {
              const float4 a = __ldcg(reinterpret_cast<const float4*>(kr + i)), b = __ldcg(reinterpret_cast<const float4*>(kr + i + HD / 2));
              const float4 c0 = __ldcg(reinterpret_cast<const float4*>(cr + i)), c1 = __ldcg(reinterpret_cast<const float4*>(cr + i + 2));
              const float4 q4 = *reinterpret_cast<const float4*>(q + d0 + i);
              const float2 e0 = make_float2(c0.x, c0.y), e1 = make_float2(c0.z, c0.w), e2 = make_float2(c1.x, c1.y), e3 = make_float2(c1.z, c1.w);
              s = __fmaf_rn(low ? rot_lo(a.x, b.x, e0) : rot_hi(a.x, b.x, e0), q4.x, s);
              s = __fmaf_rn(low ? rot_lo(a.y, b.y, e1) : rot_hi(a.y, b.y, e1), q4.y, s);
              s = __fmaf_rn(low ? rot_lo(a.z, b.z, e2) : rot_hi(a.z, b.z, e2), q4.z, s);
              s = __fmaf_rn(low ? rot_lo(a.w, b.w, e3) : rot_hi(a.w, b.w, e3), q4.w, s);
            }
          }
          s += __shfl_xor_sync(0xffffffffu, s, 1);
          s += __shfl_xor_sync(0xffffffffu, s, 2);
          if (key >= nk) s = -INFINITY;
          float mx = s;
#pragma unroll
          for (int o = 4; o < 32; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
          const float m_new = fmaxf(m, mx);
          const float corr = exp2f(m - m_new);
          const float pe = s == -INFINITY ? 0.f : exp2f(s - m_new);
          float sum = pe;
#pragma unroll
          for (int o = 4; o < 32; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
          l = l * corr + sum;
          m = m_new;
#pragma unroll
          for (int e = 0; e < HD / 32; ++e) acc[e] *= corr;
#pragma unroll
          for (int k = 0; k < KB; ++k) {
            const float pk = __shfl_sync(0xffffffffu, pe, k * 4);
#pragma unroll
            for (int e = 0; e < HD / 32; ++e) acc[e] = __fmaf_rn(pk, v[k][e], acc[e]);
          }
        }
      }
      float* mine = att_p + warp * (HD + 4);
#pragma unroll
      for (int e = 0; e < HD / 32; ++e) mine[lane * (HD / 32) + e] = acc[e];
      if (lane == 0) {
        mine[HD] = m;
        mine[HD + 1] = l;
      }
      __syncthreads();
      for (int idx = tid; idx < IG * HD; idx += THREADS) {
        const int gi = idx / HD, c = idx % HD, item = base + gi * CTAS;
        if (item < n_items) {
          const float* pp = att_p + gi * S * (HD + 4);
          float mx = -INFINITY;
          for (int s = 0; s < S; ++s) mx = fmaxf(mx, pp[s * (HD + 4) + HD]);
          float num = 0.f, den = 0.f;
          for (int s = 0; s < S; ++s) {
            const float ms = pp[s * (HD + 4) + HD];
            if (ms == -INFINITY) continue;   // no key of this row in the warp's blocks
            const float wg = exp2f(ms - mx);
            num = fmaf(wg, pp[s * (HD + 4) + c], num);
            den = fmaf(wg, pp[s * (HD + 4) + HD + 1], den);
          }
          __stcg(p.attn + (long long)item * HD + c, num / den);
        }
      }
      __syncthreads();
    }
  }
  // the rows' keys and values into the cache (nothing in this call reads them back; rows of a search stay out of it)
  __device__ void write_cache(const LayerPtrs& w, int R) const {
    const int qkvd = p.qd + 2 * p.kvd;
    for (int idx = rank * THREADS + tid; idx < R * p.nkv * (HD / 2); idx += CTAS * THREADS) {
      const int i = idx % (HD / 2), rh = idx / (HD / 2), r = rh / p.nkv, h = rh - r * p.nkv;
      const float* kr = p.qkv + (long long)r * qkvd + p.qd + h * HD + i;
      const float a = __ldcg(kr), b = __ldcg(kr + HD / 2), va = __ldcg(kr + p.kvd), vb = __ldcg(kr + p.kvd + HD / 2);
      const float2 cs = __ldcg(p.rope + r * (HD / 2) + i);
      const long long o = (long long)(p.C + r) * p.kvd + h * HD + i;
      w.ck[o] = rot_lo(a, b, cs);
      w.ck[o + HD / 2] = rot_hi(a, b, cs);
      w.cv[o] = va;
      w.cv[o + HD / 2] = vb;
    }
  }

  // ---- one decoder layer over R rows; src(r): the rows that go in (also the residual, as resid(r) after two barriers)
  template <typename Src, typename Res, typename Dst>
  __device__ void layer(int l, int R, bool uniform, Src src, Res resid, Dst dst) const {
    const LayerPtrs& w = p.layer[l];
    const int qkvd = p.qd + 2 * p.kvd;
    arrived(0);
    for (int r0 = 0; r0 < R; r0 += NR) {
      const int nr = min(NR, R - r0);
      stage(r0, nr, p.d, w.attn_norm, src);
      product(w_qkv, n_qkv, p.d, nr, NoAdd(),
              [&](int f, int r, float v, float) { __stcg(p.qkv + (long long)(r0 + r) * qkvd + lo_qkv + f, v); });
      __syncthreads();
    }
    cluster_arrive();
    fetch(0, l + 1);
    cluster_wait();
    attention(w, R);
    cluster_arrive();
    if (uniform) write_cache(w, R);
    cluster_wait();
    arrived(1);
    for (int r0 = 0; r0 < R; r0 += NR) {
      const int nr = min(NR, R - r0);
      stage(r0, nr, p.qd, nullptr, [&](int r) { return p.attn + (long long)r * p.qd; });
      product(w_o, n_d, p.qd, nr, [&](int f, int r) { return __ldcg(resid(r0 + r) + lo_d + f); },
              [&](int f, int r, float v, float x) { __stcg(p.x1 + (long long)(r0 + r) * p.d + lo_d + f, x + v); });
      __syncthreads();
    }
    cluster_arrive();
    fetch(1, l + 1);
    cluster_wait();
    arrived(2);
    for (int r0 = 0; r0 < R; r0 += NR) {
      const int nr = min(NR, R - r0);
      stage(r0, nr, p.d, w.mlp_norm, [&](int r) { return p.x1 + (long long)r * p.d; });
      // the slice holds the gate rows, then the up rows: the two sums of a feature meet in shared memory
      product(w_gu, 2 * n_f, p.d, nr, NoAdd(), [&](int f, int r, float v, float) { pair_s(r)[f] = v; });
      __syncthreads();
      for (int r = warp; r < nr; r += WARPS)
        for (int f = lane; f < n_f; f += 32)
          __stcg(p.act + (long long)(r0 + r) * p.dffn + lo_f + f, silu_f(pair_s(r)[f]) * pair_s(r)[n_f + f]);
      __syncthreads();
    }
    cluster_arrive();
    fetch(2, l + 1);
    cluster_wait();
    arrived(3);
    for (int r0 = 0; r0 < R; r0 += NR) {
      const int nr = min(NR, R - r0);
      stage(r0, nr, p.dffn, nullptr, [&](int r) { return p.act + (long long)r * p.dffn; });
      product(w_d, n_d, p.dffn, nr, [&](int f, int r) { return __ldcg(p.x1 + (long long)(r0 + r) * p.d + lo_d + f); },
              [&](int f, int r, float v, float x) { __stcg(dst(r0 + r) + lo_d + f, x + v); });
      __syncthreads();
    }
    cluster_arrive();
    fetch(3, l + 1);
    cluster_wait();
  }
  // gate / up sums of a row of the pass: the attention's area is free then (WARPS * (2 HD + 4) floats >= NR * 2 * MAX_F * 16 / 2)
  __device__ __forceinline__ float* pair_s(int r) const { return att_q + r * (MAX_F * WARPS); }

  __device__ void rope_table() const {
    const int half = HD / 2, n = p.T * half;
    // (the upper half of the warps: the lower one goes on to the first rows)
    constexpr int H = THREADS / 2;
    for (int idx = rank * H + tid - H; tid >= H && idx < n; idx += CTAS * H) {
      const int t = idx / half, i = idx % half;
      const double inv = exp2(-(2.0 * i / (2.0 * half)) * log2(p.theta));
      double s, c;
      sincos((double)(p.pos0 + t) * inv, &s, &c);
      __stcg(p.rope + idx, make_float2((float)c, (float)s));
    }
  }

  __device__ void forward() const {
    const int R = p.T;
    auto x_at = [&](int k, int r) { return (p.x_step > 0 ? p.x_base[0] + k * p.x_step : p.x_base[k & 1]) + r * p.ldx; };
    auto token_row = [&](int r) {
      const int tok = min(max(__ldg(p.tokens + r), 0), p.vocab - 1);
      return p.embed + (long long)tok * p.d;
    };
    for (int r = rank * WARPS + warp; r < R; r += CTAS * WARPS) {   // the first layer's residual
      const float* e = token_row(r);
      for (int c = lane * 4; c < p.d; c += 128) __stcg(reinterpret_cast<float4*>(x_at(0, r) + c), __ldg(reinterpret_cast<const float4*>(e + c)));
    }
    rope_table();
    for (int l = 0; l < p.n_layers; ++l) {
      auto in = [&](int r) -> const float* { return l == 0 ? token_row(r) : x_at(l, r); };
      auto res = [&](int r) -> const float* { return x_at(l, r); };
      layer(l, R, true, in, res, [&](int r) { return x_at(l + 1, r); });
    }
    if (p.head_rows == 0) return;
    if (p.n_layers == 0) cluster_barrier();   // the embedding rows are the head's input
    // LM head (its slice came into the gate/up area), then the greedy token of each row
    arrived(2);
    for (int r0 = 0; r0 < p.head_rows; r0 += NR) {
      const int nr = min(NR, p.head_rows - r0);
      stage(r0, nr, p.d, p.final_norm, [&](int r) -> const float* { return x_at(p.n_layers, R - p.head_rows + r); });
      product(w_gu, n_v, p.d, nr, NoAdd(), [&](int f, int r, float v, float) {
        __stcg(p.logits + (long long)(r0 + r) * p.vocab + lo_v + f, v);
        if (p.logits_out) p.logits_out[(long long)(r0 + r) * p.vocab + lo_v + f] = v;
      });
      __syncthreads();
    }
    cluster_barrier();
    for (int r = rank + warp * CTAS; r < p.head_rows; r += CTAS * WARPS) {
      const float* row = p.logits + (long long)r * p.vocab;
      float best = -INFINITY;
      int bi = 0x7fffffff;
#pragma unroll 8
      for (int c = lane; c < p.vocab; c += 32) {
        const float v = __ldcg(row + c);
        if (v > best || (v == best && c < bi)) { best = v; bi = c; }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
      }
      if (lane == 0) p.argmax_out[r] = bi;
      if (p.top1_out) {
        float sum = 0.f;
#pragma unroll 8
        for (int c = lane; c < p.vocab; c += 32) sum += __expf(__ldcg(row + c) - best);
        sum = warp_sum(sum);
        if (lane == 0) p.top1_out[r] = 1.0f / sum;
      }
    }
  }

  // ---- Eq. 2 step i over the candidate states j_lo..n (plus the diagonal one): every CTA computes all sums and decides alike.
  // Layer outputs in G, skip candidates in g_prev (state 1's: the objective rows of step i - 1).  Rows are counted from state
  // 1's on, whatever j_lo.
  __device__ __forceinline__ const float* skip_row(const float* g_prev, int i, int r) const {
    return r < p.T ? p.hidden + (long long)(i - 1) * p.layer_stride + r * p.token_stride : g_prev + (long long)r * p.d;
  }
  __device__ void select(int i, int j_lo, int n, bool diag, const float* g_prev, float* g_next) const {
    const int states = n + (diag ? 1 : 0), r0 = (j_lo - 1) * p.T, r1 = states * p.T;
    double2* row_cos = reinterpret_cast<double2*>(att_q);   // per row (cosine of the layer output, of the skip candidate)
    for (int r = r0 + warp; r < r1; r += WARPS) {
      const int j = r / p.T + 1, t = r % p.T;
      const float* x = p.hidden + (long long)i * p.layer_stride + t * p.token_stride;
      const float* s = skip_row(g_prev, i, r);
      const float* y = j <= n ? p.G + (long long)r * p.d : s;
      double q[5] = {0.0, 0.0, 0.0, 0.0, 0.0};   // x.x, y.y, x.y, s.s, x.s: four products in fp32, the rest in double
#pragma unroll 2
      for (int c = lane * 4; c < p.d; c += 128) {
        const float4 a = __ldg(reinterpret_cast<const float4*>(x + c));
        const float4 b = __ldcg(reinterpret_cast<const float4*>(y + c)), e = __ldcg(reinterpret_cast<const float4*>(s + c));
        q[0] += (double)(a.x * a.x + a.y * a.y + a.z * a.z + a.w * a.w);
        q[1] += (double)(b.x * b.x + b.y * b.y + b.z * b.z + b.w * b.w);
        q[2] += (double)(a.x * b.x + a.y * b.y + a.z * b.z + a.w * b.w);
        q[3] += (double)(e.x * e.x + e.y * e.y + e.z * e.z + e.w * e.w);
        q[4] += (double)(a.x * e.x + a.y * e.y + a.z * e.z + a.w * e.w);
      }
#pragma unroll
      for (int k = 0; k < 5; ++k) q[k] = warp_sum_d(q[k]);
      if (lane == 0) {
        const double nx = fmax(sqrt(q[0]), 1e-12);
        row_cos[r - r0] = make_double2(q[2] / (nx * fmax(sqrt(q[1]), 1e-12)), q[4] / (nx * fmax(sqrt(q[3]), 1e-12)));
      }
    }
    __syncthreads();
    for (int j = j_lo + tid; j <= states; j += THREADS) {
      double s_app = 0.0, s_skip = 0.0;
      for (int t = 0; t < p.T; ++t) {
        const double2 q = row_cos[(j - 1) * p.T - r0 + t];
        s_app += q.x;
        s_skip += q.y;
      }
      const float a = (float)(s_app / p.T), s = (float)(s_skip / p.T);
      int take = 0;
      const long long cell = (long long)i * (p.M + 1) + j;
      if (j <= n) {
        take = a > s;
        if (p.forced && p.forced[cell] != 255) take = p.forced[cell] == 0;
      }
      s_take[j - 1] = take;
      s_choice[cell] = take ? 0 : 1;
      if (rank == 0) {
        p.scores[cell] = take ? a : s;
        if (p.margins && j <= n) p.margins[cell] = a - s;
      }
    }
    __syncthreads();
    if (tid == 0) {
      s_choice[(long long)i * (p.M + 1)] = 0;
      if (rank == 0) p.scores[(long long)i * (p.M + 1)] = 1.0f;
    }
    __syncthreads();
    for (int r = r0 + rank + warp * CTAS; r < r1; r += CTAS * WARPS) {
      const int j = r / p.T + 1, t = r % p.T;
      const float* src = s_take[j - 1] ? p.G + (long long)r * p.d : skip_row(g_prev, i, r);
      for (int c = lane * 4; c < p.d; c += 128) {
        const float4 v = __ldcg(reinterpret_cast<const float4*>(src + c));
        __stcg(reinterpret_cast<float4*>(g_next + (long long)(r + p.T) * p.d + c), v);
        if (i == p.n_layers && j == p.M && p.g_final) *reinterpret_cast<float4*>(p.g_final + (long long)t * p.d + c) = v;
      }
    }
  }

  __device__ void search() const {
    const int L = p.n_layers, M = p.M;
    rope_table();
    if (rank == 0) {
      const float nan = __int_as_float(0x7fc00000);
      for (int c = tid; c < (L + 1) * (M + 1); c += THREADS) {
        p.scores[c] = c == 0 ? 1.0f : nan;
        if (p.margins) p.margins[c] = nan;
      }
    }
    for (int c = tid; c < (L + 1) * (M + 1); c += THREADS) s_choice[c] = c == 0 ? 0 : 255;
    __syncthreads();
    // Layer 0 is never applied (its only input would be x_0, whose image is x_1): its slices were not fetched.  Nor are any
    // when pruning leaves the diagonal only (M = L).  Pruned steps carry states j_lo..n: from j < M - (L - i) there is no way
    // to (L, M).  Rows and their sums are the same as without.
    const float* g_prev = p.g[0];
    float* g_next = p.g[1];
    for (int i = 1; i <= L; ++i) {
      const int n = min(i - 1, M), j_lo = p.prune ? max(1, M - (L - i)) : 1;
      const int sh = (j_lo - 1) * p.T;   // rows before state j_lo
      if (n >= j_lo) {
        // the rows the last step chose, straight from where they are (g[i-1] itself is on its way to memory)
        const float* gp = g_next;      // g[i - 2] (ping-pong: the buffer this step overwrites)
        auto in = [&](int k) -> const float* {
          const int r = sh + k;
          return s_take[r / p.T] ? p.G + (long long)r * p.d : skip_row(gp, i - 1, r);
        };
        auto res = [&](int k) -> const float* { return g_prev + (long long)(sh + k + p.T) * p.d; };
        layer(i - 1, n * p.T - sh, false, in, res, [&](int k) { return p.G + (long long)(sh + k) * p.d; });
      } else if (i > 1) {
        cluster_barrier();   // the rows the last step wrote
      }
      select(i, j_lo, n, i <= M, g_prev, g_next);
      const float* t = g_prev;
      g_prev = g_next;
      g_next = const_cast<float*>(t);
    }
    if (rank == 0) {
      __syncthreads();
      if (tid == 0) {   // backtrack of Algorithm 1
        for (int l = 0; l < L; ++l) p.skip_mask[l] = 0;
        int i = L, j = M;
        while (i > 0 && j > 0) {
          if (s_choice[i * (M + 1) + j] == 1) {
            p.skip_mask[i - 1] = 1;
            --j;
          }
          --i;
        }
      }
    }
  }
};

template <int HD>
__global__ void __launch_bounds__(THREADS, 1) call_kernel(const __grid_constant__ Params p) {
  extern __shared__ __align__(16) float s32_smem[];
  __shared__ uint64_t bars[4];
  uint32_t rank;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  Call<HD> c(p, s32_smem, bars, (int)rank);
  if (threadIdx.x == 0) {
    for (int ph = 0; ph < 4; ++ph) tc::mbar_init(tc::smem_u32(bars + ph), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    for (int ph = 0; ph < 4; ++ph) c.fetch(ph, !p.search ? 0 : (p.prune && p.M == p.n_layers ? p.n_layers : 1));
  }
  __syncthreads();
  if (p.search) c.search();
  else c.forward();
  if (c.parity & GAVE_UP)   // a wait ran out: copies still in flight land before the shared memory is given back
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);
}

}  // namespace s32
}  // namespace clasp
